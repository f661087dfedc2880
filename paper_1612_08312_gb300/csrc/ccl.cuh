// ccl.cuh -- connected-component labelling helpers shared by the Ising and
// n-vector sweeps.
//
// Labels are union-find parent pointers.  Linking always hangs the larger
// root under the smaller one (atomicMin on the larger root's parent), so the
// root of a finished cluster is its minimum index -- the canonical label.
// This file holds the tile-local level, in shared memory, over tile-local
// site indices (inside a tile the local index order agrees with the global
// one); the global level for clusters that cross tile faces is in
// sweep_core.cuh.  Every loop is bounded; exceeding a bound sets a status
// bit instead of spinning forever.
#pragma once

#include "pyro_internal.cuh"

namespace pyro {

// A tile-local site (cell t, offset s) is named by the address of its label in
// the shared window, base + 4 (17 t + s): the names grow with the site index
// 16 t + s, following a label is one load without any address arithmetic, and
// since a cell takes 17 words the 32 threads of a warp (consecutive cells)
// touch 32 different banks for any fixed s.
constexpr int CELL_BYTES = 68;
__device__ __forceinline__ int label_get(int name)
{
    int v;
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(name) : "memory");
    return v;
}
__device__ __forceinline__ void label_set(int name, int v)
{
    asm volatile("st.shared.b32 [%0], %1;" ::"r"(name), "r"(v) : "memory");
}
// The same under a predicate: one instruction, no branch.
__device__ __forceinline__ void label_set_if(bool on, int name, int v)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %2, 0;\n\t@p st.shared.b32 [%0], %1;\n\t}" ::"r"(name), "r"(v),
                 "r"((int)on)
                 : "memory");
}
// If on, links root hi under lo; hi if it was a root still (or not on), else
// its entry.
__device__ __forceinline__ int label_link_if(bool on, int hi, int lo)
{
    int old = hi;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %3, 0;\n\t@p atom.shared.cas.b32 %0, [%1], %1, %2;\n\t}"
                 : "+r"(old)
                 : "r"(hi), "r"(lo), "r"((int)on)
                 : "memory");
    return old;
}
// Cell t of a label's word 17 t + s (exact for up to 512 cells).
__device__ __forceinline__ int word_cell(int word) { return (word * 61681) >> 20; }

// Iteration bound of one union (4096).  A test can lower it (to 0) through
// pyro_debug_set to exercise the bound-exceeded status path.
static __constant__ int c_unite_bound = 4096;

// Unions of the clusters of a0 and b0 and of a1 and b1 in shared memory.  All
// four finds walk in lockstep, one step of each per iteration (the label of a
// root is its own name, so a find that has arrived stays); they write nothing
// on the way.  Returns false if the iteration bound was hit.
__device__ __forceinline__ bool sunite2(int a0, int b0, int a1, int b1)
{
    int a[2] = {a0, a1}, b[2] = {b0, b1};
    const int bound = c_unite_bound * 16;
#pragma unroll 1
    for (int it = 0; it < bound; ++it) {
        int ga[2], gb[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            ga[k] = label_get(a[k]);
            gb[k] = label_get(b[k]);
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const bool arrived = ga[k] == a[k] && gb[k] == b[k];
            const int lo = min(ga[k], gb[k]), hi = max(ga[k], gb[k]);
            // (not a root any more: its new parent)
            const int old = label_link_if(arrived && lo != hi, hi, lo);
            a[k] = lo;
            b[k] = old == hi && arrived ? lo : old;  // united: the same twice
        }
        if (a[0] == b[0] && a[1] == b[1]) return true;
    }
    return false;
}

// Pair index k of vertices (a, b), a < b.
__host__ __device__ constexpr int pair_index(int a, int b) { return a == 0 ? b - 1 : (a == 1 ? b + 1 : 5); }

// Threads of an accumulation block.
constexpr int ACC_THREADS = 128;

// Sums of NV values over a block of THREADS (a power of two from 64) threads,
// a fixed tree in shared memory, one barrier per level for all; results valid
// in the first warp.  (A shuffle tree adds in FP64 on every lane at every
// level; FP64 adds are scarce on this GPU.)
template <typename V, int NV, int THREADS>
__device__ __forceinline__ void block_sums(V v[NV], V (*red)[THREADS])
{
    const int t = threadIdx.x;
#pragma unroll
    for (int q = 0; q < NV; ++q) red[q][t] = v[q];
    __syncthreads();
#pragma unroll
    for (int o = THREADS / 2; o > 0; o >>= 1) {
        if (t < o)
#pragma unroll
            for (int q = 0; q < NV; ++q) red[q][t] += red[q][t + o];
        if (o > 16) __syncthreads();
        else __syncwarp();
    }
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] = red[q][0];
}

// Neumaier step with explicitly rounded operations (no contraction).
__device__ __forceinline__ void nsum_add(double &s, double &c, double x)
{
    const double t = __dadd_rn(s, x);
    if (fabs(s) >= fabs(x)) c = __dadd_rn(c, __dadd_rn(__dadd_rn(s, -t), x));
    else c = __dadd_rn(c, __dadd_rn(__dadd_rn(x, -t), s));
    s = t;
}

}  // namespace pyro
