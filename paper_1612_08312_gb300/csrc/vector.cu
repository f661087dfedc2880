// vector.cu -- Swendsen-Wang sweep of the pyrochlore XY (n = 2) and
// Heisenberg (n = 3) models with Wolff's embedded-cluster construction
// (Sec. 2): per sweep one random unit axis r; the projections p_i = s_i.r
// define an Ising model with couplings J p_i p_j; bonds with p_i p_j > 0 are
// activated with probability 1 - exp(-2 beta J p_i p_j); flipped clusters
// reflect their spins, s -> s - 2 (s.r) r.
//
// Spins are stored as n component planes of N values of T (float or
// double).  A bond with p_i p_j > 0 is active iff its 32-bit uniform
// w < floor(p 2^32), w drawn like the Ising bonds' (sweep_core.cuh).  The FP64
// path rounds every operation as IEEE does, in the order of the definition, so
// projections, reflections and the axis are bit-identical to a straightforward
// FP64 evaluation without fused multiply-add.  The FP32 path stores and updates spins in float; its
// measurements are accumulated in FP64.
//
// Kernels (each over a Batch of lattices): vec_local (projections of the
// tile + halo staged in shared memory, bond activation, tile-local
// labelling), the global union of tile-crossing clusters (boundary_unite and
// boundary_flip, shared with the Ising sweep), vec_flip (root, flip,
// reflection) and vec_measure (E and M per block in FP64).
#include <algorithm>

#include "nvec.cuh"
#include "sweep_core.cuh"

namespace pyro {

// 4 consecutive values of T (16-byte aligned) in 16-byte accesses.
template <typename T>
__device__ __forceinline__ void load4(const T *p, T out[4])
{
    const uint4 *q = reinterpret_cast<const uint4 *>(p);
#pragma unroll
    for (int k = 0; k < (int)(sizeof(T)) / 4; ++k) {
        const uint4 w = q[k];
        memcpy(&out[k * 16 / (int)sizeof(T)], &w, 16);
    }
}

// The local kernel's staging area (the projections of the tile and its halo,
// in FP32) is dead once the bonds are decided, before the labelling writes its
// labels and pair list: when it fits in their room (32 words a cell, the
// start of the core area) it shares it, which halves the shared memory of the
// common tiles.
__host__ __device__ constexpr size_t vec_stage_bytes(int TX, int TY, int TZ)
{
    return (size_t)16 * halo_cells(TX, TY, TZ) * 4;
}

__host__ __device__ constexpr bool vec_stage_shared(int TX, int TY, int TZ)
{
    return vec_stage_bytes(TX, TY, TZ) <= (size_t)core_shared_words(TX * TY * TZ) * 4;
}

// Margin of the bond shortcut below, in units of 1/256 of probability.  With
// 256 exp(-y) = 2^(8 - y log2 e) the evaluation errs by at most 2e-4 there:
// 256 * 2^-22 of ex2, 2^-22 in its argument (256 ln 2 * 2^-22), four roundings
// of y log2 e (256 y exp(-y) * 2^-22 <= 94 * 2^-22) and that of q.
// FP64 projections are staged in FP32 as sums of rounded terms, for spins of
// length 1 3e-7 off at most (six roundings of 2^-24), so y = K2 p p' errs by
// 6e-7 K2 more and q by 1.6e-4 K2.  A caller may set spins of any length: a
// block that stages one whose squared length exceeds LENGTH2_MAX (or is no
// number) decides all its bonds by the FP64 rule.  (FP32 projections are the
// rule's own, whatever the length.)
constexpr float LENGTH2_MAX = 1.0001f;
template <typename T>
__device__ __forceinline__ float shortcut_margin(double K2, bool any_long)
{
    return sizeof(T) == 4 ? SHORTCUT_MARGIN : any_long ? INFINITY : SHORTCUT_MARGIN + 4e-4f * (float)K2;
}

// Registers: two 512-thread blocks' worth of warps per SM.
template <int NC, typename T>
__global__ void __launch_bounds__(512, 2) vec_local_kernel(const __grid_constant__ Batch B)
{
    using A = Ar<T>;
    extern __shared__ __align__(16) int smem[];
    const CoreSmem sm = core_smem(smem, B.TX * B.TY * B.TZ);
    core_prologue(sm);
    overlap_wait();
    if (sizeof(T) == 8) overlap_next();  // (FP32: 0.4 % slower; FP64 L = 50: 211 us a sweep with, 220 without)
    const int rep = find_rep(B.tile_begin, B.R, blockIdx.x);
    const Rep &R = B.reps[rep];
    const int tile = (int)(blockIdx.x - B.tile_begin[rep]);
    const TileCtx c = tile_ctx(B, R, tile);
    const bool shared_stage = vec_stage_shared(c.TX, c.TY, c.TZ);
    float *proj = reinterpret_cast<float *>(shared_stage ? reinterpret_cast<unsigned char *>(smem) : sm.stage);
    const T *spins = static_cast<const T *>(R.spins);
    const int64_t N = R.N;
    const uint32_t sweep = (uint32_t)R.st->sweep;
    const uint64_t seed = R.seed;

    // Projections s_i . r of the tile's sites and the backward halo, in FP32
    // (for FP64 spins an approximation that the shortcut's margin covers: FP64
    // arithmetic here cost more than the whole FP32 kernel).  Site-major layout
    // (site s of halo cell h at s nh + h): a warp's consecutive cells read
    // consecutive words.  A thread takes four consecutive sites at a time, each
    // component read in 16 bytes, two loads of each in flight; of a halo cell only the sites a
    // down tetrahedron of the tile can reach are read: two groups of four across
    // a face, one across an edge, none at the corner.  One group after the
    // other, every halo site and the axis drawn here, the staging took a third
    // of the kernel (337 us at L = 128, n = 3, FP32, now 287).
    const int nh = halo_cells(c.TX, c.TY, c.TZ), HX = c.TX + 1, HY = c.TY + 1;
    const int nt = c.nt, L = c.L;
    constexpr int BATCH = 2;
    T v[BATCH][NC][4];
    auto own_load = [&](int b, int k) {
        const int t = (threadIdx.x + k * nt) >> 2;
        const int x = min(c.ox + (t & (c.TX - 1)), L - 1), y = min(c.oy + ((t >> c.lTX) & (c.TY - 1)), L - 1),
                  z = min(c.oz + (t >> (c.lTX + c.lTY)), L - 1);
        const int i0 = 16 * (x + L * (y + L * z)) + 4 * (threadIdx.x + k * nt & 3);
#pragma unroll
        for (int m = 0; m < NC; ++m) load4(spins + m * N + i0, v[b][m]);
    };
#pragma unroll
    for (int b = 0; b < BATCH; ++b) own_load(b, b);
    const double *axis = R.st->axis;
    const float rf[3] = {(float)axis[0], (float)axis[1], (float)axis[2]};
    bool is_long = false;  // (FP64) a spin staged by this thread
    auto put = [&](const T w[NC][4], int h, int s0) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float pr = (float)w[0][q] * rf[0];  // in the order of project()
#pragma unroll
            for (int k = 1; k < NC; ++k) pr = Ar<float>::add(pr, Ar<float>::mul((float)w[k][q], rf[k]));
            proj[(s0 + q) * nh + h] = pr;
            if (sizeof(T) == 8) {
                float len2 = 0.0f;
#pragma unroll
                for (int k = 0; k < NC; ++k) len2 = fmaf((float)w[k][q], (float)w[k][q], len2);
                is_long |= !(len2 <= LENGTH2_MAX);
            }
        }
    };
#pragma unroll
    for (int b0 = 0; b0 < 4; b0 += BATCH) {
        if (b0 > 0)
#pragma unroll
            for (int b = 0; b < BATCH; ++b) own_load(b, b0 + b);
#pragma unroll
        for (int b = 0; b < BATCH; ++b) {
            const int idx = threadIdx.x + (b0 + b) * nt, t = idx >> 2;
            const int lx = t & (c.TX - 1), ly = (t >> c.lTX) & (c.TY - 1), lz = t >> (c.lTX + c.lTY);
            put(v[b], lx + 1 + HX * (ly + 1 + HY * (lz + 1)), 4 * (idx & 3));
        }
    }
    // halo: faces x, y, z (two groups a cell), then edges xy, xz, yz
    const int fx = 2 * c.TY * c.TZ, fy = 2 * c.TX * c.TZ, fz = 2 * c.TX * c.TY;
    const int nhalo = fx + fy + fz + c.TX + c.TY + c.TZ;
    auto halo_load = [&](int e, T w[NC][4], int &h, int &s0) {
        int lx = -1, ly = -1, lz = -1, g;
        if (e < fx) {
            ly = (e >> 1) & (c.TY - 1);
            lz = e >> (1 + c.lTY);
            g = 2 + (e & 1);
        } else if ((e -= fx) < fy) {
            lx = (e >> 1) & (c.TX - 1);
            lz = e >> (1 + c.lTX);
            g = 1 + 2 * (e & 1);
        } else if ((e -= fy) < fz) {
            lx = (e >> 1) & (c.TX - 1);
            ly = e >> (1 + c.lTX);
            g = 1 + (e & 1);
        } else if ((e -= fz) < c.TZ) {
            lz = e;
            g = 3;
        } else if ((e -= c.TZ) < c.TY) {
            ly = e;
            g = 2;
        } else {
            lx = e - c.TY;
            g = 1;
        }
        h = lx + 1 + HX * (ly + 1 + HY * (lz + 1));
        s0 = 4 * g;
        // a step back from the lattice's first cell wraps, and a tile may
        // reach past the last
        int x = c.ox + lx, y = c.oy + ly, z = c.oz + lz;
        x = x < 0 ? L - 1 : min(x, L - 1);
        y = y < 0 ? L - 1 : min(y, L - 1);
        z = z < 0 ? L - 1 : min(z, L - 1);
        const int i0 = 16 * (x + L * (y + L * z)) + s0;
#pragma unroll
        for (int m = 0; m < NC; ++m) load4(spins + m * N + i0, w[m]);
    };
    for (int e = threadIdx.x; e < nhalo; e += 2 * nt) {
        int h[2], s0[2];
        halo_load(e, v[0], h[0], s0[0]);
        const bool two = e + nt < nhalo;
        if (two) halo_load(e + nt, v[1], h[1], s0[1]);
        put(v[0], h[0], s0[0]);
        if (two) put(v[1], h[1], s0[1]);
    }
    bool any_long = false;
    if (sizeof(T) == 8) any_long = __syncthreads_or(is_long);
    else __syncthreads();

    uint32_t act[3] = {0, 0, 0};
    if (R.K2 > 0.0 && c.valid) {
        // A bond with p = 1 - exp(-K2 p_i p_j) and top byte b of its uniform is
        // on whatever the low bits if 256 p > b + 1, off if 256 p < b (or p
        // <= 0): q = 256 p - b from one fast exponential decides all bonds but
        // those within the margin of [0, 1], about 1 in 250 of the positive
        // ones.  They take the exact path below, all of them in one loop: with
        // the exact path expanded at each of the 48 bonds the kernel had
        // 145 KB of code (now 54) and waited for instructions: L = 128, n = 3, FP32
        // 534 -> 327 us; FP64, whose projections and exponentials all ran in
        // FP64, L = 64 862 -> 97 us.
        const float K2l = (float)R.K2 * 1.44269504f;
        const float margin = shortcut_margin<T>(R.K2, any_long);
        // (three calls together; then tetrahedron by tetrahedron, so that each
        // projection is loaded once)
        uint32_t ww[3][4];
#pragma unroll
        for (int g = 0; g < 3; ++g) {
            const uint4 wd = philox_call(seed, sweep, TAG_BOND, 3 * (uint64_t)c.cell + g);
            ww[g][0] = wd.x;
            ww[g][1] = wd.y;
            ww[g][2] = wd.z;
            ww[g][3] = wd.w;
        }
        uint32_t und[3] = {0, 0, 0};
        const int h0 = halo_index(c, 0);
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            float up[4], dn[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                up[v] = proj[(4 * f + v) * nh + h0];
                dn[v] = v == 0 ? up[0] : proj[down_bit(f, v) * nh + halo_index(c, down_mask(f, v))];
            }
            float ups[3], dns[3];  // the first vertex's, times -K2 log2 e
#pragma unroll
            for (int v = 0; v < 3; ++v) {
                ups[v] = -(up[v] * K2l);
                dns[v] = -(dn[v] * K2l);
            }
#pragma unroll
            for (int g = 0; g < 3; ++g)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int va = slot_a(g, q), vb = slot_b(g, q);
                    const float e = exp2_approx(slot_up(g, q) ? fmaf(ups[va], up[vb], 8.0f) : fmaf(dns[va], dn[vb], 8.0f));
                    // -q: 256 exp(-y) less 256 - b, the latter from the float
                    // whose low mantissa bits are b
                    const float nq =
                        e - (8388864.0f - __uint_as_float(__byte_perm(ww[g][f], 0x4B000000u, 0x7440u | (uint32_t)q)));
                    const uint32_t bit = 1u << (4 * f + q);
                    // (a NaN, from an infinite K2l, is neither on nor off)
                    if (nq < -1.0f - margin) act[g] |= bit;
                    if (!(nq > margin)) und[g] |= bit;
                }
        }
#pragma unroll
        for (int g = 0; g < 3; ++g) und[g] &= ~act[g];
        const T K2 = (T)R.K2;
        unsigned long long todo =
            (unsigned long long)(und[0] | (und[1] << 16)) | ((unsigned long long)und[2] << 32);
#pragma unroll 1
        while (todo) {
            const int k = __ffsll((long long)todo) - 1;
            todo &= todo - 1;
            const int g = k >> 4, f = (k >> 2) & 3, q = k & 3;
            T pr[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int v = e == 0 ? slot_a(g, q) : slot_b(g, q);
                const int m = slot_up(g, q) ? 0 : down_mask(f, v);
                const int s = slot_up(g, q) ? 4 * f + v : down_bit(f, v);
                if (sizeof(T) == 4) {
                    pr[e] = (T)proj[s * nh + halo_index(c, m)];
                } else {
                    const T r[3] = {(T)axis[0], (T)axis[1], (T)axis[2]};
                    const int cx = (m & 1) ? wrap_back(c.x, L) : c.x, cy = (m & 2) ? wrap_back(c.y, L) : c.y,
                              cz = (m & 4) ? wrap_back(c.z, L) : c.z;
                    pr[e] = project<NC, T>(spins, N, 16 * (int64_t)(cx + L * (cy + L * cz)) + s, r);
                }
            }
            const T x = A::mul(pr[0], pr[1]);
            if (!(x > (T)0)) continue;
            const ByteCompare bc(prob_threshold(A::bond_p(K2, x)));
            const uint64_t id = 48 * (uint64_t)c.cell + (uint32_t)k;
            const uint4 wd = philox_call(seed, sweep, TAG_BOND, id >> 4);
            const uint32_t byte = (word_of(wd, f) >> (8 * q)) & 0xFFu;
            bool on = bc.all || byte < bc.t8;
            if (!on && byte == bc.t8) {
                const uint4 w4 = philox_call(seed, sweep, TAG_TIE, id >> 2);
                on = (word_of(w4, q) & 0xFFFFFFu) < bc.t24;
            }
            if (on && !bc.none) {
                const uint32_t bit = 1u << (k & 15);
                act[0] |= g == 0 ? bit : 0u;
                act[1] |= g == 1 ? bit : 0u;
                act[2] |= g == 2 ? bit : 0u;
            }
        }
    }
    if (shared_stage) __syncthreads();  // the staging area is read no more: the labels may take it
    local_core(c, R, sm, act[0], act[1], act[2], sweep, tile);
}

// s <- the reflection s - 2 (s . r) r, normalised.
template <int NC, typename T>
__device__ __forceinline__ void reflect(T t[NC], const T r[3])
{
    using A = Ar<T>;
    T pr = A::mul(t[0], r[0]);  // the projection, in the order of project()
#pragma unroll
    for (int k = 1; k < NC; ++k) pr = A::add(pr, A::mul(t[k], r[k]));
    const T d2 = A::mul((T)2, pr);
#pragma unroll
    for (int k = 0; k < NC; ++k) t[k] = A::sub(t[k], A::mul(d2, r[k]));
    normalise<NC>(t);
}

// Reflection of the flipped sites.  Every thread first finds its cell's flip
// mask.  FP32: the block then walks its cells' sites in the order of memory,
// 16 bytes of every component per thread, so that a warp reads and writes
// whole lines (a thread per cell stored half sectors, 2.7 times the sectors
// the spins have) and groups without a flipped site are not touched: bound by
// HBM, 805 MB in 134 us at L = 128, n = 3 (210 us before).  FP64: bound by the
// FP64 units, so the flipped sites are listed and every lane takes one.
template <int NC, typename T>
__global__ void __launch_bounds__(512) vec_flip_kernel(const __grid_constant__ Batch B)
{
    extern __shared__ __align__(16) int smem[];
    overlap_begin();
    const int rep = find_rep(B.tile_begin, B.R, blockIdx.x);
    const Rep &R = B.reps[rep];
    const int tile = (int)(blockIdx.x - B.tile_begin[rep]);
    const TileCtx c = tile_ctx(B, R, tile);
    const double *axis = R.st->axis;
    T *spins = static_cast<T *>(R.spins);
    const int64_t N = R.N;
    if (sizeof(T) == 8) {
        // the tile's flipped sites in the order of memory along its rows
        int *list = smem;
        __shared__ int wtotal[17];
        uint32_t mask = cell_flip_mask(c, R, tile, smem + 16 * c.nt);
        if (!c.valid) mask = 0;
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (c.nt + 31) >> 5;
        const unsigned lanes = lanes_mask(c.nt);
        const int n = __popc(mask);
        int incl = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(lanes, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31 || (int)threadIdx.x == c.nt - 1) wtotal[wid] = incl;
        __syncthreads();
        int total = 0, base = 0;
        for (int w = 0; w < nw; ++w) {
            if (w == wid) base = total;
            total += wtotal[w];
        }
        int pos = base + incl - n;
        while (mask) {
            list[pos++] = (int)(16 * c.cell) + __ffs(mask) - 1;
            mask &= mask - 1;
        }
        __syncthreads();
        const T r[3] = {(T)axis[0], (T)axis[1], (T)axis[2]};
        for (int e = threadIdx.x; e < total; e += c.nt) {
            T *p = spins + list[e];
            T t[NC];
#pragma unroll
            for (int k = 0; k < NC; ++k) t[k] = p[k * N];
            reflect<NC, T>(t, r);
#pragma unroll
            for (int k = 0; k < NC; ++k) p[k * N] = t[k];
        }
        return;
    }
    // per cell: its first site and its flip mask (0 past the lattice)
    int2 *todo = reinterpret_cast<int2 *>(smem);
    const uint32_t mask = cell_flip_mask(c, R, tile, smem + 2 * c.nt);
    todo[c.t] = make_int2((int)(16 * c.cell), c.valid ? (int)mask : 0);
    __syncthreads();
    const T r[3] = {(T)axis[0], (T)axis[1], (T)axis[2]};
    for (int idx = threadIdx.x; idx < 4 * c.nt; idx += blockDim.x) {
        const int2 cell = todo[idx >> 2];
        const int s0 = 4 * (idx & 3);
        const uint32_t flip = ((uint32_t)cell.y >> s0) & 0xFu;
        if (!flip) continue;
        T *p = spins + cell.x + s0;
        T sv[NC][4];
#pragma unroll
        for (int k = 0; k < NC; ++k) load4(p + k * N, sv[k]);
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            if (!((flip >> s) & 1u)) continue;
            T t[NC];
#pragma unroll
            for (int k = 0; k < NC; ++k) t[k] = sv[k][s];
            reflect<NC, T>(t, r);
#pragma unroll
            for (int k = 0; k < NC; ++k) sv[k][s] = t[k];
        }
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            uint4 w;
            memcpy(&w, sv[k], 16);
            *reinterpret_cast<uint4 *>(p + k * N) = w;
        }
    }
}

constexpr int VEC_MEASURE_BLOCK = 128;

// Energy (Eq. 1) and magnetisation of the current configuration: every
// cell sums the 48 bonds it owns and its 16 spins (FP64 spins in FP64; FP32
// spins in FP32 within the cell, since FP64 adds and conversions run at a
// small fraction of the FP32 rate on this GPU), then in FP64; one partial
// (E, M_x, M_y, M_z) per tile, summed in a fixed order.
//
// Four threads per cell, one per FCC point f: a warp's sites are consecutive
// in memory (one thread per cell read half sectors at a stride of a cell and
// moved 4.6 times the spins' sectors).  FP32: the cell's sums run over f =
// 0..3 in turn, handed from thread to thread, and are added in FP64, every
// lane its own quantity; FP64, bound by the FP64 units: every thread its own
// sums.  A block of 128 threads takes 32 cells at a time.
template <int NC, typename T>
__global__ void __launch_bounds__(VEC_MEASURE_BLOCK) vec_measure_kernel(const __grid_constant__ Batch B)
{
    extern __shared__ __align__(16) int smem[];
    overlap_begin();
    double *scratch = reinterpret_cast<double *>(smem);  // blockDim values (FP64: 4 blockDim)
    const int rep = find_rep(B.tile_begin, B.R, blockIdx.x);
    const Rep &R = B.reps[rep];
    const int L = R.L, TX = B.TX, TY = B.TY, nt = B.TX * B.TY * B.TZ;
    const uint32_t tile = (uint32_t)(blockIdx.x - B.tile_begin[rep]);
    const uint32_t txy = tile / (uint32_t)R.ntx;
    const int ox = (int)(tile - txy * (uint32_t)R.ntx) * TX;
    const int oy = (int)(txy % (uint32_t)R.nty) * TY;
    const int oz = (int)(txy / (uint32_t)R.nty) * B.TZ;
    const int64_t N = R.N;
    const T *sp = static_cast<const T *>(R.spins);
    const int f = threadIdx.x & 3;
    const unsigned lanes = lanes_mask((int)blockDim.x);
    // FP32: thread f < 3 sums M_f and thread 3 E; FP64: every thread all four
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    // blockDim is a multiple of 4 and at most 4 nt; every thread makes the same rounds
    for (int c0 = 0; c0 < nt; c0 += blockDim.x >> 2) {
        const int t = c0 + (threadIdx.x >> 2);
        const int x = ox + (t & (TX - 1)), y = oy + ((t >> B.lTX) & (TY - 1)), z = oz + (t >> (B.lTX + B.lTY));
        const bool valid = t < nt && max(x, max(y, z)) < L;
        T u[NC][4] = {}, w[NC][4] = {};
        if (valid) {
            const int own = 16 * (x + L * (y + L * z));
#pragma unroll
            for (int k = 0; k < NC; ++k) load4(sp + k * N + own + 4 * f, u[k]);
            // the down tetrahedron's vertices nu = 1..3: basis nu of FCC point
            // f ^ nu, a cell back along the axes where a(f) is 0 and a(nu) 1
#pragma unroll
            for (int nu = 1; nu < 4; ++nu) {
                const int bx = (nu >> 1) & 1 & ~(f >> 1), by = nu & 1 & ~f, bz = ((nu ^ (nu >> 1)) & 1) & ~(f ^ (f >> 1));
                const int cx = bx ? wrap_back(x, L) : x, cy = by ? wrap_back(y, L) : y, cz = bz ? wrap_back(z, L) : z;
                const int site = 16 * (cx + L * (cy + L * cz)) + 4 * (f ^ nu) + nu;
#pragma unroll
                for (int k = 0; k < NC; ++k) w[k][nu] = sp[k * N + site];
            }
#pragma unroll
            for (int k = 0; k < NC; ++k) w[k][0] = u[k][0];
        }
        if (sizeof(T) == 8) {
#pragma unroll
            for (int k = 0; k < 6; ++k)
#pragma unroll
                for (int q = 0; q < NC; ++q) {
                    acc[0] = fma((double)u[q][pair_a(k)], (double)u[q][pair_b(k)], acc[0]);
                    acc[0] = fma((double)w[q][pair_a(k)], (double)w[q][pair_b(k)], acc[0]);
                }
#pragma unroll
            for (int k = 0; k < NC; ++k)
                acc[1 + k] += ((double)u[k][0] + (double)u[k][1]) + ((double)u[k][2] + (double)u[k][3]);
            continue;
        }
        T v[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const int va = pair_a(k), vb = pair_b(k);
            T du = u[0][va] * u[0][vb];
#pragma unroll
            for (int q = 1; q < NC; ++q) du += u[q][va] * u[q][vb];
            T dd = w[0][va] * w[0][vb];
#pragma unroll
            for (int q = 1; q < NC; ++q) dd += w[q][va] * w[q][vb];
            v[k] = du + dd;
        }
        T ec = (T)0, Mc[3] = {(T)0, (T)0, (T)0};
#pragma unroll
        for (int st = 0; st < 4; ++st) {
            if (f == st) {
#pragma unroll
                for (int k = 0; k < 6; ++k) ec += v[k];
#pragma unroll
                for (int k = 0; k < NC; ++k)
#pragma unroll
                    for (int q = 0; q < 4; ++q) Mc[k] += u[k][q];
            }
            ec = __shfl_sync(lanes, ec, st, 4);
#pragma unroll
            for (int k = 0; k < NC; ++k) Mc[k] = __shfl_sync(lanes, Mc[k], st, 4);
        }
        // (a cell past the lattice has zeros)
        acc[0] += (double)(f == 0 ? Mc[0] : f == 1 ? Mc[1] : f == 2 ? Mc[2] : ec);
    }
    const int per = sizeof(T) == 8 ? (int)blockDim.x : (int)blockDim.x >> 2;
    if (sizeof(T) == 8) {
#pragma unroll
        for (int q = 0; q < 4; ++q) scratch[q * per + threadIdx.x] = acc[q];
    } else {
        scratch[((f + 1) & 3) * per + (threadIdx.x >> 2)] = acc[0];
    }
    __syncthreads();
    double tot[4];
    tile_sum4_f64(tot, per, scratch);
    if (threadIdx.x == 0) {
        double *o = B.partials + 4 * (int64_t)blockIdx.x;
#pragma unroll
        for (int q = 0; q < 4; ++q) o[q] = tot[q];
    }
}

// Ordered start (e_x) or Philox-random start: site i takes attempt a of
// call index (i << 8) | a of the INIT stream.
template <int NC, typename T>
__global__ void __launch_bounds__(CELL_BLOCK) vec_init_kernel(const __grid_constant__ Batch B, int random)
{
    const int rep = find_rep(B.block_begin, B.R, blockIdx.x);
    const Rep &R = B.reps[rep];
    const int64_t cell = (blockIdx.x - B.block_begin[rep]) * CELL_BLOCK + threadIdx.x;
    if (cell >= R.ncells) return;
    T *spins = static_cast<T *>(R.spins);
    for (int s = 0; s < 16; ++s) {
        const int64_t i = 16 * cell + s;
        double r[3] = {1.0, 0.0, 0.0};
        if (random) unit_vector_dev<NC>(R.seed, INIT_SWEEP_FIELD, TAG_INIT, (uint64_t)i << 8, r);
#pragma unroll
        for (int k = 0; k < NC; ++k) spins[k * R.N + i] = (T)r[k];
    }
}

// ------------------------------------------------------------ launchers --
cudaError_t vec_set_unite_bound(int bound) { return cudaMemcpyToSymbol(c_unite_bound, &bound, sizeof(int)); }

size_t resolve_smem(const TileShape &t);
void launch_boundary(const Batch &B, int64_t ntiles, cudaStream_t s);

size_t vec_local_smem(const TileShape &t)
{
    const size_t core = core_smem_bytes(t.TX * t.TY * t.TZ);
    return vec_stage_shared(t.TX, t.TY, t.TZ) ? core : core + vec_stage_bytes(t.TX, t.TY, t.TZ);
}

// FP32: per cell its first site and flip mask; FP64: the flipped sites' list;
// then the flip stage's own words.
static size_t vec_flip_smem(const TileShape &t, size_t es)
{
    return (es == 8 ? (size_t)64 : (size_t)8) * t.TX * t.TY * t.TZ + resolve_smem(t);
}

template <int NC, typename T>
struct VecOps {
    static cudaError_t prepare(const TileShape &t)
    {
        cudaError_t e = allow_dynamic_smem(vec_local_kernel<NC, T>, vec_local_smem(t));
        if (e == cudaSuccess) e = allow_dynamic_smem(vec_flip_kernel<NC, T>, vec_flip_smem(t, sizeof(T)));
        return e;
    }
    static void init(const Batch &B, int64_t nblocks, int random, cudaStream_t s)
    {
        vec_init_kernel<NC, T><<<(unsigned)nblocks, CELL_BLOCK, 0, s>>>(B, random);
    }
    static void phase(int p, const Batch &B, int64_t ntiles, cudaStream_t s)
    {
        const TileShape t{B.TX, B.TY, B.TZ};
        const int nt = B.TX * B.TY * B.TZ;
        if (p == 0) launch_overlapped(vec_local_kernel<NC, T>, (unsigned)ntiles, nt, vec_local_smem(t), s, B);
        else if (p == 1) launch_boundary(B, ntiles, s);
        else launch_overlapped(vec_flip_kernel<NC, T>, (unsigned)ntiles, nt, vec_flip_smem(t, sizeof(T)), s, B);
    }
    static void measure(const Batch &B, int64_t ntiles, cudaStream_t s)
    {
        const int threads = std::min(VEC_MEASURE_BLOCK, 4 * B.TX * B.TY * B.TZ);
        launch_overlapped(vec_measure_kernel<NC, T>, (unsigned)ntiles, threads,
                          threads * sizeof(double) * (sizeof(T) == 8 ? 4 : 1), s, B);
    }
};

#define PYRO_VEC_DISPATCH(model, prec, call)                                       \
    do {                                                                            \
        if ((model) == PYRO_XY) {                                                   \
            if ((prec) == PYRO_FP64) VecOps<2, double>::call; else VecOps<2, float>::call; \
        } else {                                                                    \
            if ((prec) == PYRO_FP64) VecOps<3, double>::call; else VecOps<3, float>::call; \
        }                                                                           \
    } while (0)

cudaError_t ising_prepare(const TileShape &t);

cudaError_t vec_prepare(int model, int prec, const TileShape &t)
{
    // the labels kernel (compiled with the Ising sweep) serves every model
    const cudaError_t e = ising_prepare(t);
    if (e != cudaSuccess) return e;
    if (model == PYRO_XY) return prec == PYRO_FP64 ? VecOps<2, double>::prepare(t) : VecOps<2, float>::prepare(t);
    return prec == PYRO_FP64 ? VecOps<3, double>::prepare(t) : VecOps<3, float>::prepare(t);
}

void vec_launch_init(int model, int prec, const Batch &B, int64_t nblocks, int random, cudaStream_t s)
{
    PYRO_VEC_DISPATCH(model, prec, init(B, nblocks, random, s));
}

// Phase p of a sweep: 0 local labelling, 1 crossing unions, 2 flip.
void vec_launch_phase(int p, int model, int prec, const Batch &B, int64_t ntiles, cudaStream_t s)
{
    PYRO_VEC_DISPATCH(model, prec, phase(p, B, ntiles, s));
}

void vec_launch_measure(int model, int prec, const Batch &B, int64_t ntiles, cudaStream_t s)
{
    PYRO_VEC_DISPATCH(model, prec, measure(B, ntiles, s));
}

}  // namespace pyro
