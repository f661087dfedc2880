// ising.cu -- Swendsen-Wang sweep of the pyrochlore Ising model (Sec. 2).
//
// Spins are bit-packed, one uint16 per cubic cell (bit s of cell c is site
// 16 c + s; 1 means s = -1).  Every kernel runs over a Batch of one or more
// lattices, one CTA per tile of TX x TY x TZ cells, one thread per cell.
//
//   ising_local     reads its cell's spin word and those of the backward
//                   neighbour cells, forms the 48 bonds' antiparallel bits by
//                   shift-XOR, draws one Philox call per 16 bonds and
//                   compares its bytes with the threshold four at a time
//                   (a satisfied bond is active with p = 1 - exp(-2 beta J),
//                   the SW bond rule), then runs the tile-local labelling.
//   ising_flip      flips every site whose cluster's flip bit is set: the
//                   bit of its tile-local root, or of its slot's cluster
//                   where the cluster may cross a tile face.
//   ising_measure   counts antiparallel bonds and -1 spins per tile, a warp
//                   per tile, four cells of a row at a time (exact integers;
//                   energy of Eq. 1, magnetisation of Eq. 2).
//   boundary_unite, boundary_flip  unite the clusters that cross tile faces and
//                   find their flip bits (all models).
//   labels_kernel   writes the canonical label of every site on demand.
#include <algorithm>

#include "sweep_core.cuh"

namespace pyro {

// Threads of a measurement block: four tiles of up to 256 cells, a warp each,
// or a tile of up to 512, four cells per thread.
constexpr int MEASURE_BLOCK = 128;

__global__ void __launch_bounds__(512) ising_local_kernel(const __grid_constant__ Batch B)
{
    extern __shared__ __align__(16) int smem[];
    const CoreSmem s = core_smem(smem, B.TX * B.TY * B.TZ);
    core_prologue(s);
    overlap_wait();
    const int r = find_rep(B.tile_begin, B.R, blockIdx.x);
    const Rep &R = B.reps[r];
    const int tile = (int)(blockIdx.x - B.tile_begin[r]);
    const TileCtx c = tile_ctx(B, R, tile);
    const uint32_t sweep = (uint32_t)R.st->sweep;
    const uint64_t seed = R.seed;
    const ByteCompare bc(R.thr);
    if (bc.none) {
        local_identity(c, R, sweep, tile);
        return;
    }
    // the cell's spin word and those of the cells one step back along the
    // axes of each mask m (read straight from global memory, L1-cached)
    const uint16_t *spins = static_cast<const uint16_t *>(R.spins);
    uint32_t w[7];
    {
        const int L = c.L;
        const int x = c.x, y = c.y, z = c.z;
        const int xm = wrap_back(x, L), ym = wrap_back(y, L), zm = wrap_back(z, L);
#pragma unroll
        for (int m = 0; m < 7; ++m) {
            const int cx = (m & 1) ? xm : x, cy = (m & 2) ? ym : y, cz = (m & 4) ? zm : z;
            w[m] = spins[(uint32_t)cx + (uint32_t)L * ((uint32_t)cy + (uint32_t)L * (uint32_t)cz)];
        }
    }
    __syncthreads();  // table and pair counters ready
    uint32_t anti[3];
    antiparallel_groups(w[0], down_word(w), anti[0], anti[1], anti[2]);
    const uint32_t vmask = c.valid ? 0xFFFFu : 0u;  // no bond past the lattice
    uint32_t act[3];
    if (bc.all) {
#pragma unroll
        for (int g = 0; g < 3; ++g) act[g] = ~anti[g] & vmask;
    } else {
        // bond 48 c + 16 g + 4 f + q: byte 4 f + q of BOND call 3 c + g; the
        // three calls are drawn together (independent chains interleave)
        uint4 wd[3];
#pragma unroll
        for (int g = 0; g < 3; ++g) wd[g] = philox_call(seed, sweep, TAG_BOND, 3 * (uint64_t)c.cell + g);
        const uint32_t t4 = bc.t8 * 0x01010101u;
        uint32_t tie[3];
#pragma unroll
        for (int g = 0; g < 3; ++g) {
            const uint32_t sat = ~anti[g] & vmask;
            const uint32_t ww[4] = {wd[g].x, wd[g].y, wd[g].z, wd[g].w};
            uint32_t a = 0, e = 0;
#pragma unroll
            for (int f = 0; f < 4; ++f) {
                a |= byte_flags_to_nibble(bytes_lt(ww[f], t4)) << (4 * f);
                e |= byte_flags_to_nibble(bytes_eq(ww[f], t4)) << (4 * f);
            }
            act[g] = a & sat;
            tie[g] = e & sat;
        }
        // top bytes equal (1 bond in 256): compare the low 24 bits.  All of a
        // cell's ties share one loop: a loop per word, twelve copies of the
        // draw, ran 3.6 draws a warp instead of about 2 and made up a quarter
        // of the kernel's code (47 KB, now 34): local 1,871 -> 1,656 us at L = 256
        unsigned long long ties =
            (unsigned long long)(tie[0] | (tie[1] << 16)) | ((unsigned long long)tie[2] << 32);
#pragma unroll 1
        while (ties) {
            const int k = __ffsll((long long)ties) - 1;
            ties &= ties - 1;
            // bond 48 c + k: word k & 3 of TIE call 12 c + (k >> 2)
            const uint4 w4 = philox_call(seed, sweep, TAG_TIE, 12 * (uint64_t)c.cell + (uint32_t)(k >> 2));
            if ((word_of(w4, k & 3) & 0xFFFFFFu) < bc.t24) {
                const uint32_t bit = 1u << (k & 15);
                act[0] |= (k >> 4) == 0 ? bit : 0u;
                act[1] |= (k >> 4) == 1 ? bit : 0u;
                act[2] |= (k >> 4) == 2 ? bit : 0u;
            }
        }
    }
    local_core(c, R, s, act[0], act[1], act[2], sweep, tile);
}

__global__ void __launch_bounds__(512) ising_flip_kernel(const __grid_constant__ Batch B)
{
    extern __shared__ __align__(16) int smem[];
    overlap_begin();
    const int r = find_rep(B.tile_begin, B.R, blockIdx.x);
    const Rep &R = B.reps[r];
    const int tile = (int)(blockIdx.x - B.tile_begin[r]);
    const TileCtx c = tile_ctx(B, R, tile);
    uint16_t *spins = static_cast<uint16_t *>(R.spins);
    const uint32_t was = spins[c.cell];
    const uint32_t flip = cell_flip_mask(c, R, tile, smem);
    if (c.valid) spins[c.cell] = (uint16_t)(was ^ flip);
}

// Canonical label (global index of the cluster root) of every site.
__global__ void __launch_bounds__(512) labels_kernel(const __grid_constant__ Batch B)
{
    const int r = find_rep(B.tile_begin, B.R, blockIdx.x);
    const Rep &R = B.reps[r];
    const int tile = (int)(blockIdx.x - B.tile_begin[r]);
    const TileCtx c = tile_ctx(B, R, tile);
    int root[16];
    if (!c.valid) return;
    resolve_cell(c, R, tile, root);
    int4 *dst = reinterpret_cast<int4 *>(R.labels + 16 * c.cell);
#pragma unroll
    for (int q = 0; q < 4; ++q) dst[q] = make_int4(root[4 * q], root[4 * q + 1], root[4 * q + 2], root[4 * q + 3]);
}

// Antiparallel bonds (48 per cell) and -1 spins: exact integer counts per
// tile, written to the tile's partial slot.  WARPS: a warp per tile, four tiles
// per block, since with a block per tile the blocks' latency bounded large
// lattices (32 resident on an SM): L = 256 71 -> 57 us, L = 192 37 -> 29, 48
// replicas of L = 16 .. 96 twice swept 3,307 -> 3,281.  Tiles of more than 256
// cells, by default the one tile of a small lattice, take a block each: L = 8
// 8.53 us a sweep, 8.86 with one warp.
template <bool WARPS>
__global__ void __launch_bounds__(MEASURE_BLOCK) ising_measure_kernel(const __grid_constant__ Batch B)
{
    overlap_begin();
    const int64_t b = WARPS ? (int64_t)blockIdx.x * (MEASURE_BLOCK / 32) + (threadIdx.x >> 5) : (int64_t)blockIdx.x;
    if (WARPS && b >= B.tile_begin[B.R]) return;
    const int me = WARPS ? threadIdx.x & 31 : threadIdx.x, all = WARPS ? 32 : blockDim.x;
    const int r = find_rep(B.tile_begin, B.R, b);
    const Rep &R = B.reps[r];
    const TileCtx c = tile_ctx(B, R, b - B.tile_begin[r]);  // the tile's origin
    const uint16_t *spins = static_cast<const uint16_t *>(R.spins);
    const int L = c.L;
    unsigned anti = 0, ndown = 0;
    if (((c.TX | L) & 3) == 0 && (reinterpret_cast<uintptr_t>(spins) & 7) == 0) {
        // a run of four cells of a row: 8 bytes of each of the four rows and
        // the words before three of them, 7 loads for 28, worked on as two
        // pairs (L = 256 78 -> 71 us, with a block per tile).  A caller's own
        // array may start on any cell.
        for (int t = me << 2; t < c.nt; t += all << 2) {
            const int x = c.ox + (t & (c.TX - 1)), y = c.oy + ((t >> c.lTX) & (c.TY - 1)), z = c.oz + (t >> (c.lTX + c.lTY));
            if (max(x, max(y, z)) >= L) continue;
            const int xm = wrap_back(x, L), ym = wrap_back(y, L), zm = wrap_back(z, L);
            uint2 row[4];
            uint32_t before[3];
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const uint16_t *p = spins + (uint32_t)L * ((uint32_t)(m & 1 ? ym : y) + (uint32_t)L * (uint32_t)(m & 2 ? zm : z));
                row[m] = *reinterpret_cast<const uint2 *>(p + x);
                if (m < 3) before[m] = p[xm];
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint32_t w[7];
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    w[2 * m] = h ? row[m].y : row[m].x;
                    if (m < 3) w[2 * m + 1] = h ? __funnelshift_l(row[m].x, row[m].y, 16) : before[m] | row[m].x << 16;
                }
                uint32_t A, Bg, C;
                antiparallel_groups<0x10001u>(w[0], down_word<0x10001u>(w), A, Bg, C);
                anti += (unsigned)(__popc(A) + __popc(Bg) + __popc(C));
                ndown += (unsigned)__popc(w[0]);
            }
        }
    } else {
        // up to four cells per thread: their 28 spin-word loads are independent
#pragma unroll 4
        for (int t = me; t < c.nt; t += all) {
            const int x = c.ox + (t & (c.TX - 1)), y = c.oy + ((t >> c.lTX) & (c.TY - 1)), z = c.oz + (t >> (c.lTX + c.lTY));
            if (max(x, max(y, z)) >= L) continue;
            const int xm = wrap_back(x, L), ym = wrap_back(y, L), zm = wrap_back(z, L);
            uint32_t w[7];
#pragma unroll
            for (int m = 0; m < 7; ++m) {
                const int cx = (m & 1) ? xm : x, cy = (m & 2) ? ym : y, cz = (m & 4) ? zm : z;
                w[m] = spins[(uint32_t)cx + (uint32_t)L * ((uint32_t)cy + (uint32_t)L * (uint32_t)cz)];
            }
            uint32_t A, Bg, C;
            antiparallel_groups(w[0], down_word(w), A, Bg, C);
            anti += (unsigned)(__popc(A) + __popc(Bg) + __popc(C));
            ndown += (unsigned)__popc(w[0]);
        }
    }
    anti = __reduce_add_sync(0xffffffffu, anti);  // blockDim is a multiple of 32
    ndown = __reduce_add_sync(0xffffffffu, ndown);
    unsigned long long *o = reinterpret_cast<unsigned long long *>(B.partials + 4 * b);
    if (WARPS) {
        if (me == 0) *reinterpret_cast<ulonglong2 *>(o) = make_ulonglong2(anti, ndown);
        return;
    }
    __shared__ unsigned red[2][MEASURE_BLOCK / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) {
        red[0][wid] = anti;
        red[1][wid] = ndown;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long sa = 0, sd = 0;
        for (int q = 0; q < (int)(blockDim.x >> 5); ++q) {
            sa += red[0][q];
            sd += red[1][q];
        }
        o[0] = sa;
        o[1] = sd;
    }
}

// Ordered or Philox-random start: site i is -1 iff bit i of the INIT stream
// (bit i & 127 of call i >> 7) is 1.
__global__ void __launch_bounds__(CELL_BLOCK) ising_init_kernel(const __grid_constant__ Batch B, int random)
{
    const int r = find_rep(B.block_begin, B.R, blockIdx.x);
    const Rep &R = B.reps[r];
    const int64_t cell = (blockIdx.x - B.block_begin[r]) * CELL_BLOCK + threadIdx.x;
    if (cell >= R.ncells) return;
    uint32_t word = 0;
    if (random) {
        const uint4 wd = philox_call(R.seed, INIT_SWEEP_FIELD, TAG_INIT, (uint64_t)cell >> 3);
        word = (word_of(wd, (int)((cell & 7) >> 1)) >> (16 * (int)(cell & 1))) & 0xFFFFu;
    }
    static_cast<uint16_t *>(R.spins)[cell] = (uint16_t)word;
}

// A listed crossing pair: its cell in the tile, nine bits a coordinate (a tile
// has at most 512 cells, so an edge may have as many), and the pair 6 f + k.
__host__ __device__ constexpr uint32_t cell_entry(int lx, int ly, int lz)
{
    return (uint32_t)lx | ((uint32_t)ly << 9) | ((uint32_t)lz << 18);
}
__host__ __device__ constexpr uint32_t pair_entry(uint32_t cell, int pair) { return cell | ((uint32_t)pair << 27); }
__host__ __device__ constexpr int entry_x(uint32_t e) { return (int)(e & 511u); }
__host__ __device__ constexpr int entry_y(uint32_t e) { return (int)((e >> 9) & 511u); }
__host__ __device__ constexpr int entry_z(uint32_t e) { return (int)((e >> 18) & 511u); }
__host__ __device__ constexpr int entry_pair(uint32_t e) { return (int)(e >> 27); }
constexpr bool entry_holds(int lx, int ly, int lz, int pair)
{
    const uint32_t e = pair_entry(cell_entry(lx, ly, lz), pair);
    return entry_x(e) == lx && entry_y(e) == ly && entry_z(e) == lz && entry_pair(e) == pair;
}
static_assert(entry_holds(511, 0, 0, 23) && entry_holds(0, 511, 0, 23) && entry_holds(0, 0, 511, 23) &&
                  entry_holds(511, 511, 511, 0),
              "a pair entry holds every cell of the longest tile");

// Phase 1, first launch, over the face cells of every tile (one thread each):
// unites the clusters joined by the union pairs that leave the tile.  Model-
// independent: used by the n-vector sweeps too.  Latency-bound chains of
// scattered loads: at most 32 registers, for occupancy.
__global__ void __launch_bounds__(512, 4) boundary_unite_kernel(const __grid_constant__ Batch B)
{
    // the block's crossing pairs, compacted so that every thread takes an
    // equal share (at most three pairs per tetrahedron span it)
    extern __shared__ uint32_t blist[];
    __shared__ int bcount;
    __shared__ uint32_t ends[24];
    if (threadIdx.x < 24) ends[threadIdx.x] = pair_table.e[threadIdx.x];
    overlap_begin();
    const int r = find_rep(B.tile_begin, B.R, blockIdx.x);
    const Rep &R = B.reps[r];
    const int nface = face_cells(B.TX, B.TY, B.TZ);
    const uint32_t tile = (uint32_t)(blockIdx.x - B.tile_begin[r]);
    const uint32_t txy = tile / (uint32_t)R.ntx;
    const int L = R.L;
    const int ox = (int)(tile - txy * (uint32_t)R.ntx) * B.TX;
    const int oy = (int)(txy % (uint32_t)R.nty) * B.TY;
    const int oz = (int)(txy / (uint32_t)R.nty) * B.TZ;
    if (threadIdx.x == 0) bcount = 0;
    __syncthreads();
    uint32_t todo = 0, here = 0;
    if ((int)threadIdx.x < nface) {
        int lx, ly, lz;
        face_cell_coords(B, threadIdx.x, lx, ly, lz);
        if (max(ox + lx, max(oy + ly, oz + lz)) < L)
            todo = R.dmask[(int64_t)(ox + lx) + (int64_t)L * ((int64_t)(oy + ly) + (int64_t)L * (oz + lz))];
        here = cell_entry(lx, ly, lz);
    }
    const int lane = threadIdx.x & 31;
    const int n = __popc(todo);
    int incl = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    const int wtotal = __shfl_sync(0xffffffffu, incl, 31);
    int base = 0;
    if (lane == 31 && wtotal) base = atomicAdd(&bcount, wtotal);
    int pos = __shfl_sync(0xffffffffu, base, 31) + incl - n;
    while (todo) {
        const int bit = __ffs(todo) - 1;
        todo &= todo - 1;
        blist[pos++] = pair_entry(here, bit);
    }
    __syncthreads();
    const int np = bcount;
    uint32_t *P = reinterpret_cast<uint32_t *>(R.P);
    bool ok = true;
    for (int i = threadIdx.x; i < np; i += blockDim.x) {
        const uint32_t en = blist[i];
        const int x = ox + entry_x(en), y = oy + entry_y(en), z = oz + entry_z(en);
        uint32_t pr = ends[entry_pair(en)];
        uint32_t g[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int cx = (pr & 1u) ? wrap_back(x, L) : x;
            const int cy = (pr & 2u) ? wrap_back(y, L) : y;
            const int cz = (pr & 4u) ? wrap_back(z, L) : z;
            g[e] = crossing_slot(R, B, cx, cy, cz, (int)((pr >> 4) & 15u));
            pr >>= 16;
        }
        if (g[0] != g[1]) ok &= slot_unite(P, g[0], g[1]);
    }
    if (!ok) atomicOr(&R.st->status, ST_NOCONVERGE);
}

// Phase 1, second launch: the flip bit of every slot's cluster (that of its
// root site), 16 slots to a word.  The flip bits may be read through the read-
// only path: the local kernel, which wrote them, had ended before this one
// could start (its predecessor lets it start only after waiting for that end).
__global__ void __launch_bounds__(SLOT_BLOCK) boundary_flip_kernel(const __grid_constant__ Batch B)
{
    overlap_begin();
    const int r = find_rep(B.tile_begin, B.R, blockIdx.x);
    const Rep &R = B.reps[r];
    const int64_t tile = blockIdx.x - B.tile_begin[r];
    const int nt = B.TX * B.TY * B.TZ;
    const int n = R.nslots[tile];
    const uint32_t *P = reinterpret_cast<const uint32_t *>(R.P);
    const uint32_t *own = P + tile * (16 * nt);
    // (a tile of one cell has half a word of slots)
    uint16_t *out = reinterpret_cast<uint16_t *>(R.sflip) + tile * nt;
    slot_flips(own, P, n, out, [&](uint32_t site) { return ((uint32_t)__ldg(R.F + (site >> 4)) >> (site & 15)) & 1u; });
}

// ------------------------------------------------------------ launchers --
cudaError_t ising_set_unite_bound(int bound) { return cudaMemcpyToSymbol(c_unite_bound, &bound, sizeof(int)); }

size_t ising_local_smem(const TileShape &t) { return core_smem_bytes(t.TX * t.TY * t.TZ); }

size_t resolve_smem(const TileShape &t) { return resolve_smem_bytes(t.TX * t.TY * t.TZ); }

cudaError_t ising_prepare(const TileShape &t)
{
    cudaError_t e = allow_dynamic_smem(ising_local_kernel, ising_local_smem(t));
    if (e == cudaSuccess) e = allow_dynamic_smem(ising_flip_kernel, resolve_smem(t));
    return e;
}

void ising_launch_init(const Batch &B, int64_t nblocks, int random, cudaStream_t s)
{
    ising_init_kernel<<<(unsigned)nblocks, CELL_BLOCK, 0, s>>>(B, random);
}

void launch_boundary(const Batch &B, int64_t ntiles, cudaStream_t s)
{
    const int nf = face_cells(B.TX, B.TY, B.TZ);
    // a thread per face cell where the grid fills the GPU; up to four per cell
    // (a pair each) where it does not and the longest thread's chain of finds
    // is the kernel's time (L = 16: 41 -> 36 us a sweep, L = 45: 62 -> 53; four
    // at L = 256: crossing 685 -> 955 us)
    int threads = (nf + 31) & ~31;
    while (2 * threads <= 512 && 2 * threads <= 4 * ((nf + 31) & ~31) && ntiles * (2 * threads) <= GPU_THREADS) threads *= 2;
    const size_t smem = (size_t)nf * 12 * sizeof(uint32_t);
    launch_overlapped(boundary_unite_kernel, (unsigned)ntiles, threads, smem, s, B);
    launch_overlapped(boundary_flip_kernel, (unsigned)ntiles, SLOT_BLOCK, 0, s, B);
}

void launch_labels(const Batch &B, int64_t ntiles, cudaStream_t s)
{
    labels_kernel<<<(unsigned)ntiles, B.TX * B.TY * B.TZ, 0, s>>>(B);
}

// Phase p of a sweep: 0 local labelling, 1 crossing unions, 2 flip.
void ising_launch_phase(int p, const Batch &B, int64_t ntiles, cudaStream_t s)
{
    const TileShape t{B.TX, B.TY, B.TZ};
    const int nt = B.TX * B.TY * B.TZ;
    if (p == 0) launch_overlapped(ising_local_kernel, (unsigned)ntiles, nt, ising_local_smem(t), s, B);
    else if (p == 1) launch_boundary(B, ntiles, s);
    else launch_overlapped(ising_flip_kernel, (unsigned)ntiles, nt, resolve_smem(t), s, B);
}

void ising_launch_measure(const Batch &B, int64_t ntiles, cudaStream_t s)
{
    const int nt = B.TX * B.TY * B.TZ;
    constexpr int per = MEASURE_BLOCK / 32;
    if (nt <= 256) launch_overlapped(ising_measure_kernel<true>, (unsigned)((ntiles + per - 1) / per), MEASURE_BLOCK, 0, s, B);
    else launch_overlapped(ising_measure_kernel<false>, (unsigned)ntiles, MEASURE_BLOCK, 0, s, B);
}

}  // namespace pyro
