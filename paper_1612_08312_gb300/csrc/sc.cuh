// sc.cuh -- Swendsen-Wang sweep of the Ising model on the simple-cubic lattice
// with implicit bonds (Sec. 3.4, the comparison lattice of Eq. 5-6), optionally
// diluted, tile by tile like the pyrochlore sweep.
//
// Spins are bit-packed: a row of L sites is cut into segments of 16, one
// 16-bit word each (bit 1 = -1; the last segment of a row may be short).  A
// thread takes a segment: its 48 bonds 3 s + d are consecutive, three BOND calls
// (four where the row does not start at a multiple of 16), compared four bytes
// at a time and sorted by direction; bonds along x join the sites of a
// segment into runs without any union; the others, and a segment's last one
// along x, are united in shared memory within a tile of segments, and through
// the tiles' slots where they cross its faces (sweep_core.cuh).
//
// Against one global union-find over all sites (the generic path, which this
// replaced on the simple-cubic Ising lattice) the unions' chains run in shared
// memory and a site costs two bytes of HBM instead of fourteen.
#pragma once

#include "sweep_core.cuh"

namespace pyro {

struct ScDev {
    int64_t N, nsegs;
    int L, SX;                       // sites per edge, segments per row
    int TX, TY, TZ, lTX, lTY, lTZ;   // tile: segments along x, rows, planes
    int ntx, nty, ntz, nslot;        // tiles per axis, slots reserved per tile
    uint16_t *spins;                 // per segment
    uint16_t *code;                  // 16 per segment
    uint32_t *P;                     // slots, nslot per tile (as Rep::P)
    int32_t *nslots;
    uint16_t *sflip;                 // nslot / 16 per tile
    unsigned long long *cross;       // per segment: active bonds that leave the tile, bit 0 x (its last
                                     // site's), bits 16-31 y, 32-47 z
    uint32_t *fb;                    // FLIP stream, 4 words per 128 sites, and one word more
    const uint16_t *px, *py, *pz;    // present bonds of each direction per segment, or null
    const uint16_t *occ;             // occupied sites per segment, or null
    int8_t *bytes;                   // N spins of +-1, for the copies to and from the host
    int32_t *labels;                 // canonical labels, written when asked for
    double *partials;
    DevStats *st;
    uint64_t seed, thr;
};

// Segment of the calling thread in its tile and lattice.
struct ScCtx {
    int lx, ly, lz, gx, y, z, nt, t, tile;
    int nv;        // its valid sites
    uint32_t vm;   // mask of them; 0 past the lattice
    int64_t seg;   // clamped into the lattice
};

__device__ __forceinline__ int64_t sc_seg(const ScDev &S, int gx, int y, int z)
{
    return gx + (int64_t)S.SX * (y + (int64_t)S.L * z);
}
// First site of a segment.
__device__ __forceinline__ int64_t sc_site(const ScDev &S, int gx, int y, int z)
{
    return 16 * gx + (int64_t)S.L * (y + (int64_t)S.L * z);
}

__device__ __forceinline__ ScCtx sc_ctx(const ScDev &S, int tile, int t)
{
    ScCtx c;
    c.nt = S.TX * S.TY * S.TZ;
    c.t = t;
    c.tile = tile;
    const uint32_t tl = (uint32_t)tile, txy = tl / (uint32_t)S.ntx;
    c.lx = t & (S.TX - 1);
    c.ly = (t >> S.lTX) & (S.TY - 1);
    c.lz = t >> (S.lTX + S.lTY);
    const int gx = (int)(tl - txy * (uint32_t)S.ntx) * S.TX + c.lx, y = (int)(txy % (uint32_t)S.nty) * S.TY + c.ly,
              z = (int)(txy / (uint32_t)S.nty) * S.TZ + c.lz;
    const bool valid = gx < S.SX && y < S.L && z < S.L;
    c.gx = min(gx, S.SX - 1);
    c.y = min(y, S.L - 1);
    c.z = min(z, S.L - 1);
    c.nv = min(16, S.L - 16 * c.gx);
    c.vm = valid ? 0xFFFFu >> (16 - c.nv) : 0u;
    c.seg = sc_seg(S, c.gx, c.y, c.z);
    return c;
}

// A segment's spin word, and those of its sites' neighbours along +x, +y, +z.
struct ScSpins {
    uint32_t w, wx, wy, wz;
};
__device__ __forceinline__ ScSpins sc_spins(const ScDev &S, const ScCtx &c)
{
    const int yp = c.y + 1 == S.L ? 0 : c.y + 1, zp = c.z + 1 == S.L ? 0 : c.z + 1;
    const int xp = c.gx + 1 == S.SX ? 0 : c.gx + 1;
    ScSpins s;
    s.w = S.spins[c.seg];
    const uint32_t nx = S.spins[sc_seg(S, xp, c.y, c.z)] & 1u;
    s.wx = (s.w >> 1) | (nx << (c.nv - 1));
    s.wy = S.spins[sc_seg(S, c.gx, yp, c.z)];
    s.wz = S.spins[sc_seg(S, c.gx, c.y, zp)];
    return s;
}

// Bits 0, 3, 6 .. 45 of x as 16 bits.
__host__ __device__ __forceinline__ uint32_t every_third(unsigned long long x)
{
    x &= 0x249249249249ull;
    x = (x ^ (x >> 2)) & 0x0C30C30C30C3ull;
    x = (x ^ (x >> 4)) & 0xF00F00F00Full;
    x = (x ^ (x >> 8)) & 0xFF0000FFull;
    return (uint32_t)((x ^ (x >> 16)) & 0xFFFFull);
}

// 16 bits of a bit stream from bit i on.
__device__ __forceinline__ uint32_t stream_bits(const uint32_t *words, int64_t i)
{
    return __funnelshift_r(words[i >> 5], words[(i >> 5) + 1], (uint32_t)(i & 31)) & 0xFFFFu;
}

__global__ void __launch_bounds__(256, 4) sc_local_kernel(const __grid_constant__ ScDev S)
{
    extern __shared__ __align__(16) int smem[];
    const int nt = S.TX * S.TY * S.TZ;
    const CoreSmem s = core_smem(smem, nt);
    if (threadIdx.x == 0) {
        s.pcount[0] = 0;
        s.pcount[1] = 0;
    }
    overlap_begin();
    const ScCtx c = sc_ctx(S, blockIdx.x, threadIdx.x);
    const uint32_t sweep = (uint32_t)S.st->sweep;
    const int64_t call = (int64_t)blockIdx.x * nt + threadIdx.x;
    if (128 * call < S.N) reinterpret_cast<uint4 *>(S.fb)[call] = philox_call(S.seed, sweep, TAG_FLIP, (uint64_t)call);

    // ---- bonds
    const ScSpins sp = sc_spins(S, c);
    uint32_t sat[3] = {~(sp.w ^ sp.wx) & c.vm, ~(sp.w ^ sp.wy) & c.vm, ~(sp.w ^ sp.wz) & c.vm};
    if (S.px) {
        sat[0] &= S.px[c.seg];
        sat[1] &= S.py[c.seg];
        sat[2] &= S.pz[c.seg];
    }
    uint32_t act[3] = {0, 0, 0};
    const ByteCompare bc(S.thr);
    const uint64_t b0 = 3 * (uint64_t)sc_site(S, c.gx, c.y, c.z);  // id of the first site's bond along x
    if (bc.all) {
        act[0] = sat[0];
        act[1] = sat[1];
        act[2] = sat[2];
    } else if (!bc.none && c.vm) {
        const uint32_t t4 = bc.t8 * 0x01010101u;
        unsigned long long lt = 0, eq = 0;
        const int off = (int)(b0 & 15u);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (k == 3 && off == 0) break;
            const uint4 w = philox_call(S.seed, sweep, TAG_BOND, (b0 >> 4) + k);
            const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
            uint32_t l = 0, e = 0;
#pragma unroll
            for (int f = 0; f < 4; ++f) {
                l |= byte_flags_to_nibble(bytes_lt(ww[f], t4)) << (4 * f);
                e |= byte_flags_to_nibble(bytes_eq(ww[f], t4)) << (4 * f);
            }
            lt |= (unsigned long long)l << (16 * k);
            eq |= (unsigned long long)e << (16 * k);
        }
        lt >>= off;
        eq = (eq >> off) & 0xFFFFFFFFFFFFull;
#pragma unroll
        for (int d = 0; d < 3; ++d) act[d] = every_third(lt >> d) & sat[d];
        // top bytes equal: compare the low 24 bits
#pragma unroll 1
        while (eq) {
            const int k = __ffsll((long long)eq) - 1;
            eq &= eq - 1;
            const int j = k / 3, d = k - 3 * j;
            const uint32_t sd = d == 0 ? sat[0] : d == 1 ? sat[1] : sat[2];
            if (!((sd >> j) & 1u)) continue;
            const uint64_t id = b0 + (uint32_t)k;
            const uint4 w = philox_call(S.seed, sweep, TAG_TIE, id >> 2);
            if ((word_of(w, (int)(id & 3u)) & 0xFFFFFFu) < bc.t24) {
                act[0] |= d == 0 ? 1u << j : 0u;
                act[1] |= d == 1 ? 1u << j : 0u;
                act[2] |= d == 2 ? 1u << j : 0u;
            }
        }
    }

    // ---- runs along x: every site starts under its run's first one
    const int me = s.lab + CELL_BYTES * c.t;
    const uint32_t last = c.vm ? (act[0] >> (c.nv - 1)) & 1u : 0u;  // the bond to the next segment
    const uint32_t reps = ~((act[0] & (c.vm >> 1)) << 1) & 0xFFFFu;
    {
        int r = me;
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            if ((reps >> q) & 1u) r = me + 4 * q;
            label_set(me + 4 * q, r);
        }
    }
    // the next segments along the axes: in the tile unless a step leaves it
    // (a tile that covers an axis wraps onto itself)
    const bool wrapx = c.gx + 1 == S.SX, wrapy = c.y + 1 == S.L, wrapz = c.z + 1 == S.L;
    const bool inx = wrapx ? S.ntx == 1 : c.lx + 1 < S.TX;
    const bool iny = wrapy ? S.nty == 1 : c.ly + 1 < S.TY;
    const bool inz = wrapz ? S.ntz == 1 : c.lz + 1 < S.TZ;
    const int nextx = me + CELL_BYTES * (wrapx ? -c.lx : 1);
    const int nexty = me + CELL_BYTES * (wrapy ? -c.ly * S.TX : S.TX);
    const int nextz = me + CELL_BYTES * (wrapz ? -c.lz * S.TX * S.TY : S.TX * S.TY);
    const unsigned long long cross = (!inx && last ? 1ull : 0ull) | (iny ? 0ull : (unsigned long long)act[1] << 16) |
                                     (inz ? 0ull : (unsigned long long)act[2] << 32);
    __syncthreads();  // labels initialised
    // ---- first pass over the bonds in the tile, as in local_core: the larger
    // of the ends' parents is linked under the other if it is a root still,
    // else the pair is listed; four bonds at a time.  At low temperatures there
    // are more pairs than the list holds: the bonds left then have a pass of
    // their own after the list is united.  (United at once, lane by lane: at
    // beta = 1 L = 16 150 us a sweep, now 64, and L = 256 1,446, now 546.)
    const bool unite = c_unite_bound > 0;
    bool ok = true;
    const auto link_or_list = [&](int a, int b) {  // false: the list is full
        const int lo = min(a, b), hi = max(a, b);
        int old = label_link_if(unite && lo != hi, hi, lo);
        if (!unite) old = lo;
        if (old == hi || (old == lo && unite)) return true;
        const int pos = atomicAdd(s.pcount, 1);
        if (pos >= list_room(nt)) return false;
        s.plist[pos] = (uint32_t)lo | ((uint32_t)old << 16);
        return true;
    };
    const auto pass = [&](uint32_t bits, int next) {  // the bonds left
        uint32_t left = 0;
#pragma unroll 1
        while (bits) {
            int a[4], b[4], q[4];
            const int q0 = __ffs(bits) - 1;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                q[k] = bits ? __ffs(bits) - 1 : q0;
                bits &= bits - 1;
                a[k] = label_get(me + 4 * q[k]);
                b[k] = label_get(next + 4 * q[k]);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (!link_or_list(a[k], b[k])) left |= 1u << q[k];
        }
        return left;
    };
    uint32_t ybits = iny ? act[1] : 0u, zbits = inz ? act[2] : 0u;
    bool xbit = inx && last;
#pragma unroll 1
    for (;;) {
        ybits = pass(ybits, nexty);
        zbits = pass(zbits, nextz);
        if (xbit) xbit = !link_or_list(label_get(me + 4 * (c.nv - 1)), label_get(nextx));
        __syncthreads();  // pairs listed
        // (every pass but the last lists a whole list of pairs, so they end)
        if (s.pcount[0] <= list_room(nt)) break;
        ok &= unite_listed(s, nt);
        __syncthreads();
        if (threadIdx.x == 0) s.pcount[0] = 0;
        __syncthreads();
    }
    if (!ok) atomicOr(&S.st->status, ST_NOCONVERGE);
    // sites a crossing bond may end on: those of segments on a face that is not
    // the tile's own continuation; along x a segment's last or first
    const auto ends = [&] {
        uint32_t m = 0;
        if (S.ntx > 1) m |= (inx ? 0u : 1u << (c.nv - 1)) | (c.lx == 0 ? 1u : 0u);
        if (S.nty > 1 && (!iny || c.ly == 0)) m = 0xFFFFu;
        if (S.ntz > 1 && (!inz || c.lz == 0)) m = 0xFFFFu;
        return m & c.vm;
    };
    int ent[16];
    finish_labels(s, nt, me, reps, ends, (int32_t)sc_site(S, c.gx, c.y, c.z),
                  reinterpret_cast<int32_t *>(S.P) + (int64_t)c.tile * S.nslot, S.nslots + c.tile, &S.st->status, ent);
    if (!c.vm) return;
    uint32_t packed[8];
    uint32_t code = 0;
#pragma unroll
    for (int q = 0; q < 16; ++q) {
        if ((reps >> q) & 1u)
            code = ent[q] < IS_CODE ? (uint32_t)(ent[q] - s.lab) >> 2 : (uint32_t)(ent[q] - IS_CODE);
        if (q & 1) packed[q >> 1] |= code << 16;
        else packed[q >> 1] = code;
    }
    uint4 *dst = reinterpret_cast<uint4 *>(S.code + 16 * c.seg);
    dst[0] = make_uint4(packed[0], packed[1], packed[2], packed[3]);
    dst[1] = make_uint4(packed[4], packed[5], packed[6], packed[7]);
    S.cross[c.seg] = cross;
}

// Slot of site q of segment (gx, y, z), an end of a crossing bond.
__device__ __forceinline__ uint32_t sc_slot(const ScDev &S, int gx, int y, int z, int q, int nt)
{
    const uint32_t tile = (uint32_t)(gx >> S.lTX) +
                          (uint32_t)S.ntx * ((uint32_t)(y >> S.lTY) + (uint32_t)S.nty * (uint32_t)(z >> S.lTZ));
    return tile * (uint32_t)S.nslot + (uint32_t)(S.code[16 * sc_seg(S, gx, y, z) + q] - slot_code(nt));
}

// Unites the clusters joined by the active bonds that leave a tile, a block per
// tile, its bonds listed first so that every thread takes an equal share.
__global__ void __launch_bounds__(256, 8) sc_unite_kernel(const __grid_constant__ ScDev S)
{
    extern __shared__ uint16_t list[];  // (thread << 6) | (direction << 4) | site; up to 33 per segment
    __shared__ int count;
    const int nt = S.TX * S.TY * S.TZ;
    if (threadIdx.x == 0) count = 0;
    __syncthreads();
    overlap_begin();
    const ScCtx c = sc_ctx(S, blockIdx.x, threadIdx.x);
    unsigned long long todo = c.vm ? S.cross[c.seg] : 0ull;
    const int n = __popcll(todo);
    int pos = n ? atomicAdd(&count, n) : 0;
    while (todo) {
        const int k = __ffsll((long long)todo) - 1;
        todo &= todo - 1;
        const int d = k >> 4, q = d == 0 ? c.nv - 1 : k & 15;
        list[pos++] = (uint16_t)((c.t << 6) | (d << 4) | q);
    }
    __syncthreads();
    const int np = count;
    bool ok = true;
    for (int i = threadIdx.x; i < np; i += nt) {
        const int e = list[i], q = e & 15, d = (e >> 4) & 3;
        const ScCtx a = sc_ctx(S, blockIdx.x, e >> 6);
        int gx = a.gx, y = a.y, z = a.z, qb = q;
        if (d == 0) {
            gx = gx + 1 == S.SX ? 0 : gx + 1;
            qb = 0;
        } else if (d == 1) {
            y = y + 1 == S.L ? 0 : y + 1;
        } else {
            z = z + 1 == S.L ? 0 : z + 1;
        }
        const uint32_t g0 = sc_slot(S, a.gx, a.y, a.z, q, nt), g1 = sc_slot(S, gx, y, z, qb, nt);
        if (g0 != g1) ok &= slot_unite(S.P, g0, g1);
    }
    if (!ok) atomicOr(&S.st->status, ST_NOCONVERGE);
}

// The flip bit of every slot's cluster, 16 slots to a word (read-only loads of
// the flip bits as in boundary_flip_kernel).
__global__ void __launch_bounds__(SLOT_BLOCK) sc_slot_flip_kernel(const __grid_constant__ ScDev S)
{
    overlap_begin();
    const int n = S.nslots[blockIdx.x];
    const uint32_t *own = S.P + (int64_t)blockIdx.x * S.nslot;
    uint16_t *out = S.sflip + (int64_t)blockIdx.x * (S.nslot / 16);
    slot_flips(own, S.P, n, out, [&](uint32_t site) { return (__ldg(S.fb + (site >> 5)) >> (site & 31)) & 1u; });
}

// Flips every occupied site whose cluster's flip bit is set.
__global__ void __launch_bounds__(256) sc_flip_kernel(const __grid_constant__ ScDev S)
{
    extern __shared__ uint32_t bits[];
    const int nt = S.TX * S.TY * S.TZ, words = slot_code(nt) >> 5;
    overlap_begin();
    const ScCtx c = sc_ctx(S, blockIdx.x, threadIdx.x);
    const uint32_t was = S.spins[c.seg];
    const uint4 *src = reinterpret_cast<const uint4 *>(S.code + 16 * c.seg);
    const uint4 a0 = src[0], a1 = src[1];
    const uint32_t w[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
    const uint32_t f = stream_bits(S.fb, sc_site(S, c.gx, c.y, c.z));
    const int n = (S.nslots[blockIdx.x] + 15) >> 4;
    const uint16_t *sf = S.sflip + (int64_t)blockIdx.x * (S.nslot / 16);
    for (int i = threadIdx.x; i < n; i += nt) reinterpret_cast<uint16_t *>(bits + words)[i] = sf[i];
    place_flip_bits(bits, f, c.t, nt);
    __syncthreads();
    if (!c.vm) return;
    uint32_t flip = 0;
#pragma unroll
    for (int q = 0; q < 16; ++q) {
        const int code = (int)((w[q >> 1] >> (16 * (q & 1))) & 0xFFFFu);
        if (q < c.nv) flip |= ((bits[code >> 5] >> (code & 31)) & 1u) << q;
    }
    if (S.occ) flip &= S.occ[c.seg];
    S.spins[c.seg] = (uint16_t)(was ^ (flip & c.vm));
}

// Sum over present bonds of s_i s_j and magnetisation of the occupied sites,
// per block (exact integers, held in FP64).
__global__ void __launch_bounds__(256) sc_measure_kernel(const __grid_constant__ ScDev S, int ntiles)
{
    overlap_begin();
    int e = 0, m = 0;
    const int nt = S.TX * S.TY * S.TZ;
    const int lnt = S.lTX + S.lTY + S.lTZ;
    const int64_t total = (int64_t)ntiles * nt, stride = (int64_t)gridDim.x * blockDim.x;
#pragma unroll 2
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += stride) {
        const ScCtx c = sc_ctx(S, (int)(i >> lnt), (int)(i & (nt - 1)));
        if (!c.vm) continue;
        const ScSpins s = sc_spins(S, c);
        const uint32_t px = S.px ? S.px[c.seg] : c.vm, py = S.px ? S.py[c.seg] : c.vm, pz = S.px ? S.pz[c.seg] : c.vm;
        const uint32_t occ = S.occ ? S.occ[c.seg] : c.vm;
        e += __popc(px) + __popc(py) + __popc(pz) -
             2 * (__popc((s.w ^ s.wx) & px) + __popc((s.w ^ s.wy) & py) + __popc((s.w ^ s.wz) & pz));
        m += __popc(occ) - 2 * __popc(s.w & occ);
    }
    __shared__ double red[2][256];
    double v[2] = {(double)__reduce_add_sync(0xffffffffu, e), (double)__reduce_add_sync(0xffffffffu, m)};
    if (threadIdx.x & 31) v[0] = v[1] = 0.0;
    block_sums<double, 2, 256>(v, red);
    if (threadIdx.x == 0) {
        double *o = S.partials + 4 * (int64_t)blockIdx.x;
        o[0] = v[0];
        o[1] = v[1];
        o[2] = 0.0;
        o[3] = 0.0;
    }
}

// Ordered or random start (bit i of the INIT stream, as in graph_init_kernel).
__global__ void __launch_bounds__(256) sc_init_kernel(const __grid_constant__ ScDev S, int random)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= S.nsegs) return;
    const int gx = (int)(i % S.SX), nv = min(16, S.L - 16 * gx);
    uint32_t w = 0;
    if (random) {
        const int64_t yz = i / S.SX, s0 = 16 * gx + (int64_t)S.L * yz;
        for (int q = 0; q < nv; ++q) {
            const uint4 p = philox_call(S.seed, INIT_SWEEP_FIELD, TAG_INIT, (uint64_t)(s0 + q) >> 7);
            w |= ((word_of(p, (int)(((s0 + q) & 127) >> 5)) >> ((s0 + q) & 31)) & 1u) << q;
        }
    }
    S.spins[i] = (uint16_t)w;
}

// Segment words from the N spins of +-1 in S.bytes, and back.
__global__ void __launch_bounds__(256) sc_pack_kernel(const __grid_constant__ ScDev S)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= S.nsegs) return;
    const int gx = (int)(i % S.SX), nv = min(16, S.L - 16 * gx);
    const int8_t *b = S.bytes + 16 * gx + (int64_t)S.L * (i / S.SX);
    uint32_t w = 0;
    for (int q = 0; q < nv; ++q) w |= (b[q] < 0 ? 1u : 0u) << q;
    S.spins[i] = (uint16_t)w;
}

__global__ void __launch_bounds__(256) sc_unpack_kernel(const __grid_constant__ ScDev S)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= S.nsegs) return;
    const int gx = (int)(i % S.SX), nv = min(16, S.L - 16 * gx);
    int8_t *b = S.bytes + 16 * gx + (int64_t)S.L * (i / S.SX);
    const uint32_t w = S.spins[i];
    if (S.L % 16 == 0) {  // whole, 16-byte aligned segments
        uint32_t o[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            // bit j -> byte j: 1 or, for -1, 0xFF
            const uint32_t f = (((w >> (4 * k)) & 0xFu) * 0x00204081u) & 0x01010101u;
            o[k] = 0x01010101u | (f * 0xFFu);
        }
        *reinterpret_cast<uint4 *>(b) = make_uint4(o[0], o[1], o[2], o[3]);
    } else {
        for (int q = 0; q < nv; ++q) b[q] = ((w >> q) & 1u) ? -1 : 1;
    }
}

// Canonical label of every site from the last sweep's codes and slots; before
// the first sweep every site is its own cluster.
__global__ void __launch_bounds__(256) sc_labels_kernel(const __grid_constant__ ScDev S, int swept)
{
    const int nt = S.TX * S.TY * S.TZ;
    const ScCtx c = sc_ctx(S, blockIdx.x, threadIdx.x);
    if (!c.vm) return;
    const int64_t s0 = sc_site(S, c.gx, c.y, c.z);
    for (int q = 0; q < c.nv; ++q) {
        int label = (int)(s0 + q);
        if (swept) {
            const int code = S.code[16 * c.seg + q];
            if (code >= slot_code(nt)) {
                label = (int)slot_root(S.P, S.P[(int64_t)c.tile * S.nslot + (code - slot_code(nt))]);
            } else {
                const int t = word_cell(code);
                const ScCtx r = sc_ctx(S, blockIdx.x, t);
                label = (int)sc_site(S, r.gx, r.y, r.z) + (code - 17 * t);
            }
        }
        S.labels[s0 + q] = label;
    }
}

}  // namespace pyro
