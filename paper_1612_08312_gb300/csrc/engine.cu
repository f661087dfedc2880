// engine.cu -- host side of a set of lattices updated together: device
// memory, the replica table, the launch sequence of a sweep, CUDA graphs of
// multi-sweep chunks, and the per-replica measurement / accumulation kernel.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>

#include "engine.h"
#include "launch.cuh"
#include "nvec.cuh"

namespace pyro {

// ising.cu
size_t ising_local_smem(const TileShape &t);
void launch_labels(const Batch &B, int64_t ntiles, cudaStream_t s);
cudaError_t ising_prepare(const TileShape &t);
void ising_launch_init(const Batch &B, int64_t nblocks, int random, cudaStream_t s);
void ising_launch_phase(int p, const Batch &B, int64_t ntiles, cudaStream_t s);
void ising_launch_measure(const Batch &B, int64_t ntiles, cudaStream_t s);
// vector.cu
size_t vec_local_smem(const TileShape &t);
cudaError_t vec_prepare(int model, int prec, const TileShape &t);
void vec_launch_init(int model, int prec, const Batch &B, int64_t nblocks, int random, cudaStream_t s);
void vec_launch_phase(int p, int model, int prec, const Batch &B, int64_t ntiles, cudaStream_t s);
void vec_launch_measure(int model, int prec, const Batch &B, int64_t ntiles, cudaStream_t s);

// With B.fold groups per replica, a first kernel sums each group of a
// replica's tile partials (a contiguous range, fixed order) on its own
// block, so that the accumulation reads B.fold values per replica instead of
// one per tile; one block reading tens of thousands of partials, in FP64 for
// the n-vector models, was the accumulation's whole cost.
template <bool ISING>
__global__ void __launch_bounds__(ACC_THREADS) fold_kernel(const __grid_constant__ Batch B)
{
    overlap_begin();
    const int r = blockIdx.x / B.fold, k = blockIdx.x - r * B.fold;
    const int64_t b0 = B.tile_begin[r], n = B.tile_begin[r + 1] - b0;
    const int64_t lo = b0 + n * k / B.fold, hi = b0 + n * (k + 1) / B.fold;
    if (ISING) {
        __shared__ unsigned long long red[2][ACC_THREADS];
        unsigned long long v[2] = {0, 0};
#pragma unroll 4
        for (int64_t b = lo + threadIdx.x; b < hi; b += ACC_THREADS) {
            const ulonglong2 p = *reinterpret_cast<const ulonglong2 *>(B.partials + 4 * b);
            v[0] += p.x;
            v[1] += p.y;
        }
        block_sums<unsigned long long, 2, ACC_THREADS>(v, red);
        if (threadIdx.x == 0) *reinterpret_cast<ulonglong2 *>(B.folded + 4 * (int64_t)blockIdx.x) = make_ulonglong2(v[0], v[1]);
    } else {
        __shared__ double red[4][ACC_THREADS];
        double v[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
        for (int64_t b = lo + threadIdx.x; b < hi; b += ACC_THREADS) {
            const double2 p = *reinterpret_cast<const double2 *>(B.partials + 4 * b);
            const double2 q = *reinterpret_cast<const double2 *>(B.partials + 4 * b + 2);
            v[0] += p.x;
            v[1] += p.y;
            v[2] += q.x;
            v[3] += q.y;
        }
        block_sums<double, 4, ACC_THREADS>(v, red);
        if (threadIdx.x == 0)
#pragma unroll
            for (int q = 0; q < 4; ++q) B.folded[4 * (int64_t)blockIdx.x + q] = v[q];
    }
}

// The n-vector axis of a replica's next sweep, part of its chain's state like
// the sweep counter: drawn by one thread when the counter moves.  (Every block
// of the local and the flip kernels drew it before: the FP64 roots and
// quotients, with a barrier behind them, were 2 to 4 thousand cycles of each.)
__device__ void draw_axis(const Rep &R, unsigned long long sweep, int nc)
{
    double r[3];
    if (nc == 2) unit_vector_dev<2>(R.seed, (uint32_t)sweep, TAG_AXIS, 0, r);
    else unit_vector_dev<3>(R.seed, (uint32_t)sweep, TAG_AXIS, 0, r);
    for (int k = 0; k < 3; ++k) R.st->axis[k] = r[k];
}

// Per replica (one block each): sum the tiles' partials of the measurement
// kernel in a fixed order, form E, m = |M|/N, m^2, m^4 (Eq. 1, Eq. 2) and, in
// mode 1, add them to the Neumaier sums, append the trace record and advance
// the sweep counter; mode 2 only records them as the last measurement.
// A block per replica, bound by its own latency: few threads (a replica has
// at most FOLD_MIN_TILES partials, or its FOLD_GROUPS folded ones) and one
// tree for all four sums.  With 1,024 threads and a shuffle tree per sum it
// took 10 us (Ising) and 16 us (n-vector) whatever the lattice.
template <bool ISING>
__global__ void __launch_bounds__(ACC_THREADS) accumulate_kernel(const __grid_constant__ Batch B, int mode, int nc)
{
    overlap_begin();
    const int r = blockIdx.x;
    const Rep &R = B.reps[r];
    DevStats *st = R.st;
    // the replica's tile partials, or its folded groups
    const double *src = B.fold ? B.folded : B.partials;
    const int64_t b0 = B.fold ? (int64_t)r * B.fold : B.tile_begin[r];
    const int64_t b1 = B.fold ? (int64_t)(r + 1) * B.fold : B.tile_begin[r + 1];
    // the record's fields, read ahead of the sums they are needed after
    const int t = threadIdx.x;
    const unsigned long long sweep = st->sweep, count = st->count;
    double acc_s = t < 5 ? st->acc_s[t] : 0.0, acc_c = t < 5 ? st->acc_c[t] : 0.0;
    double tot[4] = {0.0, 0.0, 0.0, 0.0};
    if (ISING) {
        __shared__ unsigned long long red[2][ACC_THREADS];
        unsigned long long v[2] = {0, 0};
#pragma unroll 4
        for (int64_t b = b0 + threadIdx.x; b < b1; b += ACC_THREADS) {
            const ulonglong2 p = *reinterpret_cast<const ulonglong2 *>(src + 4 * b);
            v[0] += p.x;
            v[1] += p.y;
        }
        block_sums<unsigned long long, 2, ACC_THREADS>(v, red);
        if (t >= 32) return;
        const long long anti = (long long)v[0];
        const long long M = R.N - 2 * (long long)v[1];
        tot[0] = (double)(3 * R.N - 2 * anti);  // sum over bonds of s_i s_j
        tot[1] = (double)M;
    } else {
        __shared__ double red[4][ACC_THREADS];
        // (thread 0 moves the counter after the sums' barriers)
        if (mode == 1 && threadIdx.x == ACC_THREADS - 1) draw_axis(R, sweep + 1, nc);
#pragma unroll 4
        for (int64_t b = b0 + threadIdx.x; b < b1; b += ACC_THREADS) {
            const double2 p = *reinterpret_cast<const double2 *>(src + 4 * b);
            const double2 q = *reinterpret_cast<const double2 *>(src + 4 * b + 2);
            tot[0] += p.x;
            tot[1] += p.y;
            tot[2] += q.x;
            tot[3] += q.y;
        }
        block_sums<double, 4, ACC_THREADS>(tot, red);
        if (t >= 32) return;
    }
    // every lane of the first warp forms the observables; lane k < 5 keeps sum k
    const double E = __dmul_rn(-R.J, tot[0]);
    double m;
    if (ISING) {
        m = __ddiv_rn(fabs(tot[1]), (double)R.N);
    } else {
        double msq = __dmul_rn(tot[1], tot[1]);
        for (int k = 1; k < nc; ++k) msq = __dadd_rn(msq, __dmul_rn(tot[1 + k], tot[1 + k]));
        m = __ddiv_rn(__dsqrt_rn(msq), (double)R.N);
    }
    const double m2 = __dmul_rn(m, m);
    const double m4 = __dmul_rn(m2, m2);
    if (t == 0) {
        st->last[0] = E;
        st->last[1] = m2;
        st->last[2] = m4;
        st->last[3] = tot[1];
    }
    if (mode != 1) return;
    if (t < 5) {
        const double x = t == 0 ? E : t == 1 ? __dmul_rn(E, E) : t == 2 ? m2 : t == 3 ? m4 : __dsqrt_rn(m2);
        nsum_add(acc_s, acc_c, x);
        st->acc_s[t] = acc_s;
        st->acc_c[t] = acc_c;
    }
    if (t != 0) return;
    if (R.trace && R.trace_cap > 0) {
        double *rec = R.trace + 4 * (int64_t)(count % (unsigned long long)R.trace_cap);
        rec[0] = E;
        rec[1] = m2;
        rec[2] = m4;
        rec[3] = tot[1];
    }
    st->count = count + 1;
    st->sweep = sweep + 1;
}

__global__ void set_params_kernel(Rep *reps, int r, uint64_t thr, double K2)
{
    reps[r].thr = thr;
    reps[r].K2 = K2;
}

__global__ void set_trace_kernel(Rep *reps, int r, double *trace, int64_t cap)
{
    reps[r].trace = trace;
    reps[r].trace_cap = cap;
}

__global__ void set_sweep_kernel(const __grid_constant__ Batch B, unsigned long long sweep, int nc)
{
    if ((int)threadIdx.x >= B.R) return;
    B.reps[threadIdx.x].st->sweep = sweep;
    if (nc > 1) draw_axis(B.reps[threadIdx.x], sweep, nc);
}

// Host launcher of the accumulation kernel for callers outside this file.
void launch_accumulate(const Batch &B, bool ising, int mode, int nc, cudaStream_t s)
{
    if (ising) launch_overlapped(accumulate_kernel<true>, B.R, ACC_THREADS, 0, s, B, mode, nc);
    else launch_overlapped(accumulate_kernel<false>, B.R, ACC_THREADS, 0, s, B, mode, nc);
}

// ------------------------------------------------------------------ host --
int g_fail_allocs = 0;

cudaError_t engine_malloc(void **p, size_t bytes)
{
    if (g_fail_allocs > 0) {
        --g_fail_allocs;
        *p = nullptr;
        return cudaErrorMemoryAllocation;
    }
    return cudaMalloc(p, bytes);
}

uint64_t ising_threshold(double beta, double J)
{
    if (!(beta > 0.0)) return 0;
    const double p = -expm1(-2.0 * beta * J);
    if (!(p > 0.0)) return 0;
    const double tq = floor(p * 4294967296.0);
    return tq >= 4294967296.0 ? (1ull << 32) : (uint64_t)tq;
}

static int log2i(int v)
{
    int l = 0;
    while ((1 << l) < v) ++l;
    return l;
}

static bool is_pow2(int v) { return v > 0 && (v & (v - 1)) == 0; }

// Tiles along an axis of L cells with tile edge T (the last may reach past
// the lattice).
static int tiles_along(int L, int T) { return (L + T - 1) / T; }

static int64_t tiles_of(int L, const TileShape &t)
{
    return (int64_t)tiles_along(L, t.TX) * tiles_along(L, t.TY) * tiles_along(L, t.TZ);
}

// The tile whose modelled sweep is cheapest over the set of lattices, among
// the power-of-two tiles of at most `cap` cells.  The edges need not divide L.
// Model: every tile costs its cells, padded to the lattice's edge and to a
// warp, times 1 + w (1/TX + 1/TY + 1/TZ) over the axes it does not cover, for the
// crossing unions of its faces; w is the measured cost of the crossing phase
// per face cell over the local phase's per cell (Ising L = 256: 640 us over 0.5
// face cells per cell against 1,449; n = 3, L = 128: 91 over 0.5 against 268).
// Edges that divide L would be one cell for odd L, tiles of one thread (Ising
// L = 45 938 us a sweep, 87 with this rule).
//
// cap.  Sets that do not fill the GPU are bound by a block's latency, which
// grows with its threads; sets that do, by the crossing work, which falls with
// the tile.  A sweep in us at 64 / 128 / 256 cells: Ising L = 16 30.2 / 30.1 / 32.4,
// L = 32 35.6 / 33.1 / 36.0, L = 64 73.2 / 68.1 / 70.1, L = 72 94.8 / 80.0 / 85.5, L = 96
// 181 / 151 / 149, L = 128 401 / 324 / 311 and 322 at 512: 128 and 256 meet between
// L = 80 and 96, past the line at L = 66.  n = 3, FP32 L = 16 39.8 / 42.3 / 47.5, L = 32
// 47.0 / 48.9 / 52.0, L = 48 65.5 / 64.3 / 66.3, L = 64 109 / 106 / 106, L = 80
// 192 / 182 / 176; FP64 L = 32 90 / 95 / 104, L = 48 182 / 192 / 211, L = 64
// 318 / 313 / 323: 64 and 256 meet near the line at L = 40 for FP32, near L = 64 for FP64.
// One lattice that a block of 512 cells covers has no crossing work at all: L = 8
// 21.4, and 24.3 with two tiles of 256.
TileShape default_tile(const int *Ls, int R, int model)
{
    int64_t cells = 0;
    int size[MAX_REPS], times[MAX_REPS], n = 0;  // the distinct sizes
    for (int r = 0; r < R; ++r) {
        cells += (int64_t)Ls[r] * Ls[r] * Ls[r];
        int k = 0;
        while (k < n && size[k] != Ls[r]) ++k;
        if (k == n) {
            size[n] = Ls[r];
            times[n++] = 0;
        }
        ++times[k];
    }
    const int cap = model == PYRO_ISING ? (cells <= 512 ? 512 : cells <= 300000 ? 128 : 256)
                                        : (cells <= 512 ? 256 : cells <= 65536 ? 64 : 256);
    const double w = model == PYRO_ISING ? 0.9 : 0.66;
    TileShape best{1, 1, 1};
    double best_cost = -1.0;
    for (int tx = 32; tx >= 1; tx /= 2)
        for (int ty = 32; ty >= 1; ty /= 2)
            for (int tz = 32; tz >= 1; tz /= 2) {
                const int nt = tx * ty * tz;
                if (nt > cap) continue;
                double cost = 0.0;
                for (int k = 0; k < n; ++k) {
                    double f = 1.0;
                    if (tx < size[k]) f += w / tx;
                    if (ty < size[k]) f += w / ty;
                    if (tz < size[k]) f += w / tz;
                    cost += f * times[k] * (double)tiles_of(size[k], TileShape{tx, ty, tz}) * std::max(nt, 32);
                }
                // equal costs: fewer threads, then the longer x edge
                if (best_cost < 0.0 || cost < best_cost * (1.0 - 1e-9) ||
                    (cost < best_cost * (1.0 + 1e-9) && nt < best.TX * best.TY * best.TZ)) {
                    best_cost = cost;
                    best = TileShape{tx, ty, tz};
                }
            }
    return best;
}

size_t local_smem(int model, int prec, const TileShape &t)
{
    return model == PYRO_ISING ? ising_local_smem(t) : vec_local_smem(t);
}

// The edges of a caller's tile divide every L; the default tile's need not.
std::string check_tile(const int *Ls, int R, int model, int prec, const TileShape &t, bool callers)
{
    if (!is_pow2(t.TX) || !is_pow2(t.TY) || !is_pow2(t.TZ)) return "tile edges must be powers of two";
    for (int r = 0; r < R && callers; ++r)
        if (Ls[r] % t.TX || Ls[r] % t.TY || Ls[r] % t.TZ) return "tile edges must divide every L";
    const int nt = t.TX * t.TY * t.TZ;
    if (nt > 512) return "tile has too many cells (at most 512)";
    if (local_smem(model, prec, t) > 200 * 1024) return "tile needs too much shared memory";
    return "";
}

static size_t spin_bytes_of(int model, int prec, int64_t N)
{
    if (model == PYRO_ISING) return (size_t)(N / 16) * sizeof(uint16_t);
    return (size_t)N * model * (prec == PYRO_FP64 ? 8 : 4);
}

size_t Engine::spin_bytes(int r) const { return spin_bytes_of(model, prec, reps[r].N); }

static size_t ws_align(size_t x) { return (x + 255) & ~(size_t)255; }

// The replicas' statistics records (contiguous); per replica: spins, slots,
// slot counts and flip bits, codes, flip words, face masks, canonical labels;
// then the tiles' partial sums and the replica table.
size_t workspace_bytes(int R, const int *Ls, int model, int prec, const TileShape &t)
{
    size_t total = ws_align((size_t)R * sizeof(DevStats));
    int64_t ntiles = 0;
    for (int r = 0; r < R; ++r) {
        const int64_t ncells = (int64_t)Ls[r] * Ls[r] * Ls[r], N = 16 * ncells;
        const size_t nt = (size_t)t.TX * t.TY * t.TZ, nrt = (size_t)tiles_of(Ls[r], t);
        total += ws_align(spin_bytes_of(model, prec, N)) + ws_align(nrt * nt * 16 * sizeof(int32_t)) +
                 ws_align(nrt * sizeof(int32_t)) + ws_align(nrt * nt * 2 + 4) + ws_align((size_t)N * sizeof(uint16_t)) + ws_align((size_t)ncells * sizeof(uint16_t)) +
                 ws_align((size_t)ncells * sizeof(uint32_t)) + ws_align((size_t)N * sizeof(int32_t));
        ntiles += tiles_of(Ls[r], t);
    }
    return total + ws_align((size_t)(ntiles + (int64_t)R * FOLD_GROUPS) * 4 * sizeof(double)) +
           ws_align((size_t)R * sizeof(Rep));
}

// One device array: carved from the caller's workspace when there is one,
// else allocated (and freed by release()).
cudaError_t Engine::alloc(void **p, size_t bytes)
{
    if (ws) {
        const size_t need = ws_align(bytes);
        if (ws_used + need > ws_bytes) {
            *p = nullptr;
            return cudaErrorMemoryAllocation;
        }
        *p = ws + ws_used;
        ws_used += need;
        return cudaSuccess;
    }
    const cudaError_t e = engine_malloc(p, bytes);
    if (e == cudaSuccess) owned.push_back(*p);
    return e;
}

cudaError_t Engine::setup(int R_, const int *Ls, const double *betas, int model_, int prec_, int start_, double J,
                          const uint64_t *seeds, cudaStream_t user_stream, const TileShape &t, std::string &err,
                          void *workspace, size_t workspace_bytes_)
{
    ws = static_cast<unsigned char *>(workspace);
    ws_bytes = workspace ? workspace_bytes_ : 0;
    ws_used = 0;
    R = R_;
    model = model_;
    prec = model_ == PYRO_ISING ? PYRO_FP64 : prec_;
    start = start_;
    tile = t;
    cudaError_t e = cudaSuccess;
    if (user_stream) {
        stream = user_stream;
        own_stream = false;
    } else {
        e = cudaStreamCreateWithFlags(&stream, cudaStreamNonBlocking);
        if (e != cudaSuccess) {
            err = "stream create";
            return e;
        }
        own_stream = true;
    }
    std::memset(&B, 0, sizeof(B));
    B.R = R;
    B.TX = t.TX;
    B.TY = t.TY;
    B.TZ = t.TZ;
    B.lTX = log2i(t.TX);
    B.lTY = log2i(t.TY);
    B.lTZ = log2i(t.TZ);
    reps.assign(R, Rep{});
    ntiles = 0;
    nblocks = 0;
    // every replica's statistics in one block, so that they can be read in
    // one copy
    DevStats *stats = nullptr;
    e = alloc((void **)&stats, (size_t)R * sizeof(DevStats));
    if (e != cudaSuccess) {
        err = ws ? "workspace too small" : "device allocation failed";
        return e;
    }
    for (int r = 0; r < R; ++r) {
        Rep &p = reps[r];
        p.L = Ls[r];
        p.ncells = (int64_t)Ls[r] * Ls[r] * Ls[r];
        p.N = 16 * p.ncells;
        p.ntx = tiles_along(Ls[r], t.TX);
        p.nty = tiles_along(Ls[r], t.TY);
        p.seed = seeds[r];
        p.J = J;
        p.thr = ising_threshold(betas ? betas[r] : 0.0, J);
        p.K2 = 2.0 * (betas ? betas[r] : 0.0) * J;
        beta.push_back(betas ? betas[r] : 0.0);
        B.tile_begin[r] = ntiles;
        B.block_begin[r] = nblocks;
        const size_t nt = (size_t)t.TX * t.TY * t.TZ, nrt = (size_t)tiles_of(Ls[r], t);
        ntiles += (int64_t)nrt;
        nblocks += (p.ncells + CELL_BLOCK - 1) / CELL_BLOCK;
        struct {
            void **ptr;
            size_t bytes;
        } al[] = {{&p.spins, spin_bytes_of(model, prec, p.N)},
                  {(void **)&p.P, nrt * nt * 16 * sizeof(int32_t)},
                  {(void **)&p.nslots, nrt * sizeof(int32_t)},
                  {(void **)&p.sflip, nrt * nt * 2 + 4},
                  {(void **)&p.L16, (size_t)p.N * sizeof(uint16_t)},
                  {(void **)&p.F, (size_t)p.ncells * sizeof(uint16_t)},
                  {(void **)&p.dmask, (size_t)p.ncells * sizeof(uint32_t)},
                  {(void **)&p.labels, ws ? (size_t)p.N * sizeof(int32_t) : 0}};
        p.st = stats + r;
        for (auto &a : al) {
            if (!a.bytes) continue;  // canonical labels: allocated on first use, unless in a workspace
            e = alloc(a.ptr, a.bytes);
            if (e != cudaSuccess) {
                err = ws ? "workspace too small" : "device allocation failed";
                return e;
            }
        }
        e = cudaMemsetAsync(p.st, 0, sizeof(DevStats), stream);
        if (e != cudaSuccess) return e;
    }
    B.tile_begin[R] = ntiles;
    B.block_begin[R] = nblocks;
    // lattices of many tiles first fold their partials (see fold_kernel)
    int64_t max_tiles = 0;
    for (int r = 0; r < R; ++r) max_tiles = std::max(max_tiles, B.tile_begin[r + 1] - B.tile_begin[r]);
    B.fold = max_tiles >= FOLD_MIN_TILES ? FOLD_GROUPS : 0;
    e = alloc((void **)&B.partials, (size_t)(ntiles + (int64_t)R * FOLD_GROUPS) * 4 * sizeof(double));
    B.folded = B.partials ? B.partials + 4 * ntiles : nullptr;
    if (e == cudaSuccess) e = alloc((void **)&d_reps, (size_t)R * sizeof(Rep));
    if (e != cudaSuccess) {
        err = ws ? "workspace too small" : "device allocation failed";
        return e;
    }
    B.reps = d_reps;
    e = cudaMemcpyAsync(d_reps, reps.data(), (size_t)R * sizeof(Rep), cudaMemcpyHostToDevice, stream);
    if (e != cudaSuccess) return e;
    e = model == PYRO_ISING ? ising_prepare(tile) : vec_prepare(model, prec, tile);
    if (e != cudaSuccess) {
        err = "kernel attributes";
        return e;
    }
    if (model == PYRO_ISING) ising_launch_init(B, nblocks, start == PYRO_START_RANDOM, stream);
    else vec_launch_init(model, prec, B, nblocks, start == PYRO_START_RANDOM, stream);
    launches += 1;
    if (model != PYRO_ISING) {  // the first sweep's axis
        set_sweep_kernel<<<1, MAX_REPS, 0, stream>>>(B, 0, model);
        launches += 1;
    }
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) err = "initial state";
    return e;
}

void Engine::release()
{
    if (stream) cudaStreamSynchronize(stream);
    for (auto &g : graphs)
        if (g.exec) cudaGraphExecDestroy(g.exec);
    graphs.clear();
    for (void *p : owned) cudaFree(p);
    owned.clear();
    for (auto &r : reps)
        if (r.trace) cudaFree(r.trace);
    if (own_stream && stream) cudaStreamDestroy(stream);
    stream = nullptr;
}

cudaError_t Engine::set_beta(int r, double b)
{
    if (beta[r] == b) return cudaSuccess;
    beta[r] = b;
    reps[r].thr = ising_threshold(b, reps[r].J);
    reps[r].K2 = 2.0 * b * reps[r].J;
    set_params_kernel<<<1, 1, 0, stream>>>(d_reps, r, reps[r].thr, reps[r].K2);
    launches += 1;
    return cudaGetLastError();
}

// Phase p of a sweep: 0 tile-local labelling (with bond activation),
// 1 crossing unions, 2 flip, 3 measurement, 4 accumulation (mode as in
// accumulate_kernel).
void Engine::enqueue_phase(int p, int mode)
{
    if (p < 3) {
        if (model == PYRO_ISING) ising_launch_phase(p, B, ntiles, stream);
        else vec_launch_phase(p, model, prec, B, ntiles, stream);
    } else if (p == 3) {
        if (model == PYRO_ISING) ising_launch_measure(B, ntiles, stream);
        else vec_launch_measure(model, prec, B, ntiles, stream);
    } else {
        if (B.fold) {
            if (model == PYRO_ISING) launch_overlapped(fold_kernel<true>, R * B.fold, ACC_THREADS, 0, stream, B);
            else launch_overlapped(fold_kernel<false>, R * B.fold, ACC_THREADS, 0, stream, B);
        }
        if (model == PYRO_ISING) launch_overlapped(accumulate_kernel<true>, R, ACC_THREADS, 0, stream, B, mode, 1);
        else launch_overlapped(accumulate_kernel<false>, R, ACC_THREADS, 0, stream, B, mode, model);
    }
}

void Engine::enqueue_sweeps(int n)
{
    for (int s = 0; s < n; ++s)
        for (int p = 0; p < NPHASE; ++p) enqueue_phase(p, 1);
}

void Engine::enqueue_measure(int mode)
{
    enqueue_phase(3, mode);
    enqueue_phase(4, mode);
}

cudaError_t Engine::compute_labels()
{
    bool changed = false;
    for (auto &r : reps)
        if (!r.labels) {
            const cudaError_t e = cudaMalloc(&r.labels, (size_t)r.N * sizeof(int32_t));
            if (e != cudaSuccess) return e;
            owned.push_back(r.labels);
            changed = true;
        }
    if (changed) {
        const cudaError_t e = cudaMemcpyAsync(d_reps, reps.data(), (size_t)R * sizeof(Rep), cudaMemcpyHostToDevice, stream);
        if (e != cudaSuccess) return e;
    }
    launch_labels(B, ntiles, stream);
    launches += 1;
    return cudaGetLastError();
}

cudaError_t Engine::profile(int n, double *phase_ms)
{
    cudaEvent_t ev[NPHASE + 1];
    for (auto &x : ev)
        if (cudaEventCreate(&x) != cudaSuccess) return cudaGetLastError();
    double acc[NPHASE] = {};
    cudaError_t e = cudaSuccess;
    for (int s = 0; s < n && e == cudaSuccess; ++s) {
        cudaEventRecord(ev[0], stream);
        for (int p = 0; p < NPHASE; ++p) {
            enqueue_phase(p, 1);
            cudaEventRecord(ev[p + 1], stream);
        }
        launches += launches_per_sweep();
        e = cudaEventSynchronize(ev[NPHASE]);
        for (int p = 0; p < NPHASE && e == cudaSuccess; ++p) {
            float ms = 0.f;
            e = cudaEventElapsedTime(&ms, ev[p], ev[p + 1]);
            acc[p] += ms;
        }
    }
    for (auto &x : ev) cudaEventDestroy(x);
    sweep += n;
    labels_valid = true;
    for (int p = 0; p < NPHASE; ++p) phase_ms[p] = n > 0 ? acc[p] / n : 0.0;
    return e;
}

// Kernel launches of one sweep: one per phase, the crossing phase is two
// (unions, then the slots' flip bits), and the accumulation two when
// the partials are folded first.
int Engine::launches_per_sweep() const { return NPHASE + 1 + (B.fold ? 1 : 0); }

cudaGraphExec_t Engine::graph_for(int n)
{
    for (auto &g : graphs)
        if (g.n == n) return g.exec;
    cudaGraph_t graph = nullptr;
    if (cudaStreamBeginCapture(stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    enqueue_sweeps(n);
    if (cudaStreamEndCapture(stream, &graph) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    cudaGraphExec_t exec = nullptr;
    const cudaError_t e = cudaGraphInstantiate(&exec, graph, 0);
    cudaGraphDestroy(graph);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    graphs.push_back(GraphEntry{n, exec});
    return exec;
}

cudaError_t Engine::sweeps(int n)
{
    if (n <= 0) return cudaSuccess;
    // A call replays graphs: of whole chunks, and of one sweep for what is left.
    // Six or seven launches a sweep cost the host 10 us, more than a small
    // lattice's sweep costs a GPU that several handles share, and a graph 1:
    // eight Ising lattices of L = 8 driven by one thread in calls of 2 to 31
    // sweeps take 3.6 us a sweep, launched plainly 11; FP32 XY of L = 16 6.5 and
    // 11.  One handle alone pays for it, since plain launches overlap from sweep to
    // sweep and graphs do not: L = 8 23.7 us for 21.5, L = 24 34.3 for 32.2.
    int left = n;
    if (use_graphs && own_stream) {
        for (const int chunk : {GRAPH_CHUNK, 1}) {
            if (left < chunk) continue;
            cudaGraphExec_t g = graph_for(chunk);
            for (; g && left >= chunk; left -= chunk) {
                const cudaError_t e = cudaGraphLaunch(g, stream);
                if (e != cudaSuccess) return e;
            }
        }
    }
    enqueue_sweeps(left);
    launches += (uint64_t)n * launches_per_sweep();
    sweep += n;
    labels_valid = true;
    return cudaGetLastError();
}

cudaError_t Engine::time_sweeps(int n, double &ms)
{
    cudaEvent_t a, b;
    cudaError_t e = cudaEventCreate(&a);
    if (e != cudaSuccess) return e;
    e = cudaEventCreate(&b);
    if (e != cudaSuccess) {
        cudaEventDestroy(a);
        return e;
    }
    cudaEventRecord(a, stream);
    e = sweeps(n);
    cudaEventRecord(b, stream);
    if (e == cudaSuccess) e = cudaEventSynchronize(b);
    float f = 0.f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&f, a, b);
    ms = n > 0 ? (double)f / n : 0.0;
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    return e;
}

cudaError_t Engine::measure()
{
    enqueue_measure(2);
    launches += 2;
    return cudaGetLastError();
}

cudaError_t Engine::set_sweep(uint64_t s)
{
    set_sweep_kernel<<<1, MAX_REPS, 0, stream>>>(B, s, model);
    launches += 1;
    sweep = s;
    return cudaGetLastError();
}

cudaError_t Engine::set_trace(int r, int64_t cap)
{
    cudaError_t e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) return e;
    if (reps[r].trace) cudaFree(reps[r].trace);
    reps[r].trace = nullptr;
    reps[r].trace_cap = 0;
    if (cap > 0) {
        e = cudaMalloc(&reps[r].trace, (size_t)cap * 4 * sizeof(double));
        if (e != cudaSuccess) return e;
        reps[r].trace_cap = cap;
    }
    set_trace_kernel<<<1, 1, 0, stream>>>(d_reps, r, reps[r].trace, reps[r].trace_cap);
    launches += 1;
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    return e;
}

int Engine::read_status(std::string &err)
{
    // the replicas' records are contiguous: one copy reads every status
    std::vector<DevStats> d((size_t)R);
    cudaError_t e = cudaMemcpyAsync(d.data(), reps[0].st, d.size() * sizeof(DevStats), cudaMemcpyDeviceToHost, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) {
        err = cudaGetErrorString(e);
        return -1;
    }
    int st = 0;
    for (const auto &x : d) st |= x.status;
    return st;
}

}  // namespace pyro
