// graph.cu -- Swendsen-Wang sweep on a generic lattice: an explicit list of
// nearest-neighbour bonds (Sec. 2: the program needs only each site's
// neighbour table), the simple-cubic lattice with implicit bonds (Sec. 3.4,
// the comparison lattice of Eq. 5-6), either one optionally diluted by a
// site mask and a bond mask (Sec. 4).  Ising (n = 1) and the embedded-
// cluster n-vector models (n = 2, 3), conventions as in include/pyro.h.  The
// Ising model on the simple-cubic lattice has a sweep of its own (sc.cuh).
//
// A sweep is four launches (five for n > 1):
//   graph_proj   (n > 1) the sweep's axis r and every projection s_i . r;
//   graph_bond   one thread per 16 consecutive bond ids: one Philox call
//                gives their top bytes, the tie call is drawn only when a
//                top byte equals the threshold's; active bonds are united
//                in a global union-find array (atomicMin, larger root under
//                the smaller, so a finished cluster's root is its minimum
//                site, the canonical label).  The same threads draw the
//                sweep's flip bits, 128 sites per call;
//   graph_flip   one thread per site: root, canonical label, flip
//                (Ising: negate; n > 1: reflect and renormalise), and the
//                identity labels of the next sweep's array (two arrays
//                alternate, so no separate reset launch is needed);
//   graph_measure / graph_accumulate   E over present bonds and M over
//                occupied sites, per block in a fixed order, then one block
//                forms E, m^2, m^4 and adds them to the Neumaier sums.
#include <cmath>
#include <cstdint>
#include <cstring>
#include <algorithm>
#include <new>
#include <string>
#include <vector>

#include "bonds.cuh"
#include "engine.h"
#include "launch.cuh"
#include "nvec.cuh"
#include "sc.cuh"

namespace pyro {

struct GraphDev {
    int64_t N, NB, nocc;
    int L;     // simple-cubic edge (n > 1; Ising: sc.cuh); 0 = explicit bond list
    int nc;    // spin components
    const int32_t *bi, *bj;
    const uint32_t *present;  // bond bit set (bond mask and both ends occupied), or null
    const uint32_t *occ;      // site bit set, or null
    void *spins;              // Ising int8 +-1; n > 1 nc planes of N values of T
    int32_t *lab, *lab_next;
    uint32_t *fb;             // flip bits, 4 words per 128 sites
    void *proj;               // n > 1: projections s_i . r (T)
    double *axis;             // n > 1: the sweep's axis
    double *partials;         // 4 per measurement block
    DevStats *st;
    uint64_t seed, thr;
    double K2, J;
};

constexpr int GB_THREADS = 256;

// Simple cubic: coordinates of site s and its neighbour one step along
// +axis d (32-bit arithmetic: N < 2^31).
__device__ __forceinline__ void sc_coords(int L, int s, int &x, int &y, int &z)
{
    const unsigned us = (unsigned)s, uL = (unsigned)L, t = us / uL;
    x = (int)(us - t * uL);
    z = (int)(t / uL);
    y = (int)(t - (unsigned)z * uL);
}

__device__ __forceinline__ int sc_next(int L, int s, int x, int y, int z, int d)
{
    if (d == 0) return x + 1 == L ? s - x : s + 1;
    if (d == 1) return y + 1 == L ? s - y * L : s + L;
    return z + 1 == L ? s - z * L * L : s + L * L;
}

// Sites joined by bond e.
__device__ __forceinline__ void bond_ends(const GraphDev &G, int64_t e, int &i, int &j)
{
    if (G.L) {
        const int64_t s = e / 3;
        int x, y, z;
        sc_coords(G.L, (int)s, x, y, z);
        i = (int)s;
        j = sc_next(G.L, i, x, y, z, (int)(e - 3 * s));
    } else {
        i = G.bi[e];
        j = G.bj[e];
    }
}

__device__ __forceinline__ bool bit_of(const uint32_t *set, int64_t k) { return (set[k >> 5] >> (k & 31)) & 1u; }

// Union of the clusters of a and b in the global array (path halving in
// both finds).  The finds read through L1: a stale entry still names an
// ancestor, links are decided by the atomic, and from L2 all finds met at the
// entry of the largest cluster's root.  False if the union's iteration bound
// was hit.
__device__ __forceinline__ bool gunite(int32_t *lab, int a, int b)
{
    const int bound = c_unite_bound;
    int pa = __ldca(lab + a), pb = __ldca(lab + b);
#pragma unroll 1
    for (int it = 0; it < bound; ++it) {
#pragma unroll 1
        for (int st = 0; (pa != a || pb != b) && st < (1 << 20); ++st) {
            const int ga = __ldca(lab + pa), gb = __ldca(lab + pb);
            if (ga != pa) lab[a] = ga;
            if (gb != pb) lab[b] = gb;
            a = pa;
            pa = ga;
            b = pb;
            pb = gb;
        }
        if (a == b) return true;
        const int lo = min(a, b), hi = max(a, b);
        const int old = atomicMin(&lab[hi], lo);
        if (old == hi) return true;
        // hi had been linked meanwhile: unite lo with its new parent
        a = lo;
        b = old;
        pa = __ldca(lab + a);
        pb = __ldca(lab + b);
    }
    return false;
}

template <int NC, typename T>
__global__ void __launch_bounds__(GB_THREADS) graph_init_kernel(const __grid_constant__ GraphDev G, int random)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= G.N) return;
    G.lab[i] = (int32_t)i;
    G.lab_next[i] = (int32_t)i;
    if (NC == 1) {
        int neg = 0;
        if (random) {
            const uint4 w = philox_call(G.seed, INIT_SWEEP_FIELD, TAG_INIT, (uint64_t)i >> 7);
            neg = (word_of(w, (int)((i & 127) >> 5)) >> (i & 31)) & 1;
        }
        static_cast<int8_t *>(G.spins)[i] = neg ? -1 : 1;
    } else {
        double r[3] = {1.0, 0.0, 0.0};
        if (random) unit_vector_dev<NC>(G.seed, INIT_SWEEP_FIELD, TAG_INIT, (uint64_t)i << 8, r);
#pragma unroll
        for (int k = 0; k < NC; ++k) static_cast<T *>(G.spins)[k * G.N + i] = (T)r[k];
    }
}

template <int NC, typename T>
__global__ void __launch_bounds__(GB_THREADS) graph_proj_kernel(const __grid_constant__ GraphDev G)
{
    overlap_begin();
    __shared__ double rs[3];
    if (threadIdx.x == 0) {
        unit_vector_dev<NC>(G.seed, (uint32_t)G.st->sweep, TAG_AXIS, 0, rs);
        if (blockIdx.x == 0)
            for (int k = 0; k < 3; ++k) G.axis[k] = rs[k];
    }
    __syncthreads();
    const T r[3] = {(T)rs[0], (T)rs[1], (T)rs[2]};
    const T *sp = static_cast<const T *>(G.spins);
    T *proj = static_cast<T *>(G.proj);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < G.N; i += (int64_t)gridDim.x * blockDim.x)
        proj[i] = project<NC, T>(sp, G.N, i, r);
}

// Thread c takes the 16 bonds 16 c .. 16 c + 15 (one BOND call) and draws
// the FLIP call c.  (One bond per lane with the words passed by shuffles was
// measured slower: a warp's lanes then unite the bonds of the same few sites
// at once.)  The bonds are decided first, all sites and spins loaded together
// (bond after bond, each waited for its own sites, spins and unions), then the
// active ones are united in a loop of their own: chains of dependent reads,
// for which every warp the SM holds counts (Ising, a simple-cubic bond list, a
// sweep with 48, 40 and 32 registers: L = 256 727, 674 and 615 us, L = 128 124,
// 117 and 117; below L = 100, where the SMs are not full, 32 are 1 to 4 % slower).
template <int NC, typename T>
__global__ void __launch_bounds__(GB_THREADS, NC == 1 ? 8 : 4) graph_bond_kernel(const __grid_constant__ GraphDev G)
{
    overlap_begin();
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t sweep = (uint32_t)G.st->sweep;
    if (128 * c < G.N) reinterpret_cast<uint4 *>(G.fb)[c] = philox_call(G.seed, sweep, TAG_FLIP, (uint64_t)c);
    const int64_t e0 = 16 * c;
    if (e0 >= G.NB) return;
    const uint4 w = philox_call(G.seed, sweep, TAG_BOND, (uint64_t)c);
    const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
    const int nq = (int)(G.NB - e0 < 16 ? G.NB - e0 : 16);
    uint32_t pres = 0xFFFFu >> (16 - nq);
    if (G.present) pres &= G.present[e0 >> 5] >> (e0 & 31);
    // simple cubic: bond 3 s + d, from the chunk's first
    int s0 = 0, d0 = 0, x0 = 0, y0 = 0, z0 = 0;
    if (NC > 1 && G.L) {
        const uint64_t s = (uint64_t)e0 / 3u;
        s0 = (int)s;
        d0 = (int)((uint64_t)e0 - 3u * s);
        sc_coords(G.L, s0, x0, y0, z0);
    }
    const auto ends = [&](int q, int &i, int &j) {  // of bond e0 + q, q < nq
        if (NC > 1 && G.L) {
            int x = x0, y = y0, z = z0, ds = (d0 + q) / 3;
            const int d = d0 + q - 3 * ds;
            i = s0 + ds;
            for (x += ds; x >= G.L; x -= G.L)
                if (++y == G.L) {
                    y = 0;
                    ++z;
                }
            j = sc_next(G.L, i, x, y, z, d);
        } else {
            i = G.bi[e0 + q];
            j = G.bj[e0 + q];
        }
    };
    uint32_t act = 0, tie = 0;
    if (NC == 1) {
        // bonds whose top byte is below (equals) the threshold's, then those
        // between equal spins
        const ByteCompare bc(G.thr);
        if (bc.all) {
            act = 0xFFFFu;
        } else if (!bc.none) {
            const uint32_t t4 = bc.t8 * 0x01010101u;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                act |= byte_flags_to_nibble(bytes_lt(ww[k], t4)) << (4 * k);
                tie |= byte_flags_to_nibble(bytes_eq(ww[k], t4)) << (4 * k);
            }
        }
        const uint32_t cand = (act | tie) & pres;
        const int8_t *sp = static_cast<const int8_t *>(G.spins);
        uint32_t same = 0;
#pragma unroll
        for (int h = 0; h < 16; h += 8) {
            int si[8], sj[8];
            if (nq == 16) {  // the list in 16-byte loads
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const int4 i = __ldg(reinterpret_cast<const int4 *>(G.bi + e0 + h) + k);
                    const int4 j = __ldg(reinterpret_cast<const int4 *>(G.bj + e0 + h) + k);
                    si[4 * k] = i.x;
                    si[4 * k + 1] = i.y;
                    si[4 * k + 2] = i.z;
                    si[4 * k + 3] = i.w;
                    sj[4 * k] = j.x;
                    sj[4 * k + 1] = j.y;
                    sj[4 * k + 2] = j.z;
                    sj[4 * k + 3] = j.w;
                }
            } else {
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    si[q] = sj[q] = 0;
                    if ((cand >> (h + q)) & 1u) ends(h + q, si[q], sj[q]);
                }
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                if (!((cand >> (h + q)) & 1u)) continue;
                si[q] = sp[si[q]];
                sj[q] = sp[sj[q]];
            }  // (a bond that is no candidate is masked out below)
#pragma unroll
            for (int q = 0; q < 8; ++q) same |= (si[q] == sj[q] ? 1u : 0u) << (h + q);
        }
        act &= same & pres;
        tie &= same & pres;
        for (uint32_t k = tie; k; k &= k - 1) {
            const int q = __ffs(k) - 1;
            const uint4 t = philox_call(G.seed, sweep, TAG_TIE, (uint64_t)(e0 + q) >> 2);
            if ((word_of(t, q & 3) & 0xFFFFFFu) < bc.t24) act |= 1u << q;
        }
    } else {
        const T *p = static_cast<const T *>(G.proj);
        T xp[16];
#pragma unroll
        for (int h = 0; h < 16; h += 8) {
            int si[8], sj[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                si[q] = sj[q] = -1;
                if ((pres >> (h + q)) & 1u) ends(h + q, si[q], sj[q]);
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) xp[h + q] = si[q] >= 0 ? Ar<T>::mul(p[si[q]], p[sj[q]]) : (T)0;
        }
        // the pyrochlore kernel's shortcut: 256 p - b from one fast exponential
        // decides all bonds but those within the margin of [0, 1]
        const float K2l = (float)G.K2 * 1.44269504f;
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            if (!(xp[q] > (T)0)) continue;
            const float nq2 = exp2_approx(fmaf(-K2l, (float)xp[q], 8.0f)) -
                              (8388864.0f - __uint_as_float(__byte_perm(ww[q >> 2], 0x4B000000u, 0x7440u | (q & 3))));
            if (nq2 < -1.0f - SHORTCUT_MARGIN) act |= 1u << q;
            else if (!(nq2 > SHORTCUT_MARGIN)) tie |= 1u << q;
        }
        if (!(G.K2 > 0.0)) act = tie = 0;
        for (uint32_t k = tie; k; k &= k - 1) {
            const int q = __ffs(k) - 1;
            int i, j;
            ends(q, i, j);
            const ByteCompare bc(prob_threshold(Ar<T>::bond_p((T)G.K2, Ar<T>::mul(p[i], p[j]))));
            const uint32_t byte = (word_of(w, q >> 2) >> (8 * (q & 3))) & 0xFFu;
            bool on = bc.all || byte < bc.t8;
            if (!on && byte == bc.t8) {
                const uint4 t = philox_call(G.seed, sweep, TAG_TIE, (uint64_t)(e0 + q) >> 2);
                on = (word_of(t, q & 3) & 0xFFFFFFu) < bc.t24;
            }
            if (on && !bc.none) act |= 1u << q;
        }
    }
    bool ok = true;
#pragma unroll 1
    for (; act; act &= act - 1) {
        int i, j;
        ends(__ffs(act) - 1, i, j);
        ok &= gunite(G.lab, i, j);
    }
    if (!ok) atomicOr(&G.st->status, ST_NOCONVERGE);
}

template <int NC, typename T>
__global__ void __launch_bounds__(GB_THREADS) graph_flip_kernel(const __grid_constant__ GraphDev G)
{
    overlap_begin();
    using A = Ar<T>;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= G.N) return;
    int r = __ldca(G.lab + i);  // (stale entries are ancestors)
    int steps = 0;
#pragma unroll 1
    for (;;) {
        const int p = __ldca(G.lab + r);
        if (p == r) break;
        r = p;
        if (++steps > UF_MAX_ITERS) {
            atomicOr(&G.st->status, ST_NOCONVERGE);
            break;
        }
    }
    G.lab_next[i] = (int32_t)i;
    G.lab[i] = r;
    if (G.occ && !bit_of(G.occ, i)) return;
    if (!bit_of(G.fb, r)) return;
    if (NC == 1) {
        int8_t *s = static_cast<int8_t *>(G.spins);
        s[i] = (int8_t)(-s[i]);
    } else {
        T *sp = static_cast<T *>(G.spins);
        const T rr[3] = {(T)G.axis[0], (T)G.axis[1], (T)G.axis[2]};
        const T d2 = A::mul((T)2, static_cast<const T *>(G.proj)[i]);
        T sv[3];
#pragma unroll
        for (int k = 0; k < NC; ++k) sv[k] = A::sub(sp[k * G.N + i], A::mul(d2, rr[k]));
        T q = A::mul(sv[0], sv[0]);
#pragma unroll
        for (int k = 1; k < NC; ++k) q = A::add(q, A::mul(sv[k], sv[k]));
        q = A::sqrt_(q);
#pragma unroll
        for (int k = 0; k < NC; ++k) sp[k * G.N + i] = A::div(sv[k], q);
    }
}

// Per block: sum over present bonds of s_i . s_j and the occupied sites'
// magnetisation components, in a fixed order (grid-stride, then a fixed
// shuffle tree).  Ising sums are integers, exact in FP64.
template <int NC, typename T>
__global__ void __launch_bounds__(GB_THREADS) graph_measure_kernel(const __grid_constant__ GraphDev G)
{
    overlap_begin();
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    if (NC == 1) {
        const int8_t *s = static_cast<const int8_t *>(G.spins);
        long long e = 0, m = 0;
#pragma unroll 4
        for (int64_t i = t0; i < G.N; i += stride)
            if (!G.occ || bit_of(G.occ, i)) m += s[i];
        // four bonds per thread in 16-byte loads, two fours in flight
        const int4 *bi = reinterpret_cast<const int4 *>(G.bi), *bj = reinterpret_cast<const int4 *>(G.bj);
#pragma unroll 2
        for (int64_t b = t0; b < G.NB >> 2; b += stride) {
            const int4 i = __ldg(bi + b), j = __ldg(bj + b);
            const uint32_t pres = G.present ? (G.present[b >> 3] >> (4 * (b & 7))) & 0xFu : 0xFu;
            const uint32_t diff = (s[i.x] != s[j.x] ? 1u : 0u) | (s[i.y] != s[j.y] ? 2u : 0u) |
                                  (s[i.z] != s[j.z] ? 4u : 0u) | (s[i.w] != s[j.w] ? 8u : 0u);
            e += __popc(pres) - 2 * __popc(pres & diff);
        }
        const int64_t b = (G.NB & ~(int64_t)3) + t0;
        if (b < G.NB && (!G.present || bit_of(G.present, b))) e += s[G.bi[b]] == s[G.bj[b]] ? 1 : -1;
        v[0] = (double)e;
        v[1] = (double)m;
    } else {
        const T *sp = static_cast<const T *>(G.spins);
        for (int64_t i = t0; i < G.N; i += stride)
            if (!G.occ || bit_of(G.occ, i))
#pragma unroll
                for (int k = 0; k < NC; ++k) v[1 + k] = __dadd_rn(v[1 + k], (double)sp[k * G.N + i]);
        for (int64_t b = t0; b < G.NB; b += stride) {
            if (G.present && !bit_of(G.present, b)) continue;
            int i, j;
            bond_ends(G, b, i, j);
            double d = __dmul_rn((double)sp[i], (double)sp[j]);
#pragma unroll
            for (int k = 1; k < NC; ++k) d = __dadd_rn(d, __dmul_rn((double)sp[k * G.N + i], (double)sp[k * G.N + j]));
            v[0] = __dadd_rn(v[0], d);
        }
    }
    __shared__ double red[4][GB_THREADS];
    block_sums<double, 4, GB_THREADS>(v, red);
    if (threadIdx.x == 0)
#pragma unroll
        for (int q = 0; q < 4; ++q) G.partials[4 * blockIdx.x + q] = v[q];
}

// One block: the partials in a fixed order, E = -J sum s_i . s_j,
// m = |M| / N_occ, m^2, m^4; mode 1 adds them to the Neumaier sums and
// advances the sweep counter, mode 2 only records them.
__global__ void __launch_bounds__(ACC_THREADS) graph_accumulate_kernel(const __grid_constant__ GraphDev G, int nblocks,
                                                                       int mode)
{
    overlap_begin();
    const int t = threadIdx.x;
    DevStats *st = G.st;
    // the record's fields, read ahead of the sums they are needed after
    const unsigned long long sweep = st->sweep, count = st->count;
    double acc_s = t < 5 ? st->acc_s[t] : 0.0, acc_c = t < 5 ? st->acc_c[t] : 0.0;
    __shared__ double red[4][ACC_THREADS];
    double tot[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
    for (int b = t; b < nblocks; b += ACC_THREADS)
#pragma unroll
        for (int q = 0; q < 4; ++q) tot[q] += G.partials[4 * b + q];
    block_sums<double, 4, ACC_THREADS>(tot, red);
    if (t >= 32) return;
    // every lane of the first warp forms the observables; lane k < 5 keeps sum k
    const double E = __dmul_rn(-G.J, tot[0]);
    double m = 0.0;
    if (G.nocc > 0) {
        if (G.nc == 1) {
            m = __ddiv_rn(fabs(tot[1]), (double)G.nocc);
        } else {
            double msq = __dmul_rn(tot[1], tot[1]);
            for (int k = 1; k < G.nc; ++k) msq = __dadd_rn(msq, __dmul_rn(tot[1 + k], tot[1 + k]));
            m = __ddiv_rn(__dsqrt_rn(msq), (double)G.nocc);
        }
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
    if (t == 0) {
        st->count = count + 1;
        st->sweep = sweep + 1;
    }
}

__global__ void graph_set_sweep_kernel(DevStats *st, unsigned long long s) { st->sweep = s; }

cudaError_t graph_set_unite_bound(int bound) { return cudaMemcpyToSymbol(c_unite_bound, &bound, sizeof(int)); }

// ------------------------------------------------------------ host side --
static int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }

// Kernels of one (model, precision).
struct GraphKernels {
    void (*init)(GraphDev, int, cudaStream_t, unsigned);
    void (*sweep)(const GraphDev &, cudaStream_t, unsigned, unsigned, unsigned, unsigned);
    void (*measure)(const GraphDev &, cudaStream_t, unsigned);
};

template <int NC, typename T>
struct GraphOps {
    static void init(GraphDev G, int random, cudaStream_t s, unsigned nsite_blocks)
    {
        graph_init_kernel<NC, T><<<nsite_blocks, GB_THREADS, 0, s>>>(G, random);
    }
    static void sweep(const GraphDev &G, cudaStream_t s, unsigned nproj, unsigned nbond, unsigned nsite,
                      unsigned nmeas)
    {
        if (NC > 1) launch_overlapped(graph_proj_kernel<NC, T>, nproj, GB_THREADS, 0, s, G);
        launch_overlapped(graph_bond_kernel<NC, T>, nbond, GB_THREADS, 0, s, G);
        launch_overlapped(graph_flip_kernel<NC, T>, nsite, GB_THREADS, 0, s, G);
        launch_overlapped(graph_measure_kernel<NC, T>, nmeas, GB_THREADS, 0, s, G);
    }
    static void measure(const GraphDev &G, cudaStream_t s, unsigned nmeas)
    {
        launch_overlapped(graph_measure_kernel<NC, T>, nmeas, GB_THREADS, 0, s, G);
    }
};

static GraphKernels kernels_for(int model, int prec)
{
    if (model == PYRO_ISING) return {GraphOps<1, double>::init, GraphOps<1, double>::sweep, GraphOps<1, double>::measure};
    if (model == PYRO_XY) {
        if (prec == PYRO_FP64) return {GraphOps<2, double>::init, GraphOps<2, double>::sweep, GraphOps<2, double>::measure};
        return {GraphOps<2, float>::init, GraphOps<2, float>::sweep, GraphOps<2, float>::measure};
    }
    if (prec == PYRO_FP64) return {GraphOps<3, double>::init, GraphOps<3, double>::sweep, GraphOps<3, double>::measure};
    return {GraphOps<3, float>::init, GraphOps<3, float>::sweep, GraphOps<3, float>::measure};
}

struct GraphEngine {
    GraphDev G{};
    int model = 0, prec = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    std::vector<void *> owned;
    int32_t *lab_a = nullptr, *lab_b = nullptr, *lab_last = nullptr;
    uint64_t launches = 0;
    double beta = -1.0;
    unsigned nproj = 1, nbond = 1, nsite = 1, nmeas = 1;
    GraphKernels k{};
    ScDev sc{};               // Ising on the simple-cubic lattice
    unsigned sc_tiles = 0;    // its tiles; 0 = the generic kernels
    bool swept = false;

    cudaError_t alloc(void **p, size_t bytes)
    {
        const cudaError_t e = engine_malloc(p, bytes ? bytes : 16);
        if (e == cudaSuccess) owned.push_back(*p);
        return e;
    }

    void release()
    {
        if (stream) cudaStreamSynchronize(stream);
        for (void *p : owned) cudaFree(p);
        owned.clear();
        if (own_stream && stream) cudaStreamDestroy(stream);
        stream = nullptr;
    }

    size_t spin_elem() const { return model == PYRO_ISING ? 1 : (prec == PYRO_FP64 ? 8 : 4); }

    cudaError_t setup(const pyro_graph_config &c, int64_t N, int64_t NB, const std::vector<uint32_t> &present,
                      const std::vector<uint32_t> &occ, int64_t nocc, std::string &err)
    {
        model = c.model;
        prec = model == PYRO_ISING ? PYRO_FP64 : c.precision;
        k = kernels_for(model, prec);
        cudaError_t e;
        if (c.stream) {
            stream = static_cast<cudaStream_t>(c.stream);
        } else {
            e = cudaStreamCreateWithFlags(&stream, cudaStreamNonBlocking);
            if (e != cudaSuccess) return err = "stream creation", e;
            own_stream = true;
        }
        if (c.sc_L && model == PYRO_ISING) return sc_setup(c, N, present, occ, nocc, err);
        G.N = N;
        G.NB = NB;
        G.nocc = nocc;
        G.L = c.sc_L;
        G.nc = model;
        G.seed = c.seed;
        G.J = c.J;
        const int64_t nchunk = std::max(cdiv(NB, 16), cdiv(N, 128));
        nbond = (unsigned)std::max<int64_t>(1, cdiv(nchunk, GB_THREADS));
        nsite = (unsigned)cdiv(N, GB_THREADS);
        nproj = (unsigned)std::min<int64_t>(cdiv(N, GB_THREADS), GPU_SMS * 8);
        nmeas = (unsigned)std::min<int64_t>(cdiv(std::max(N, NB), GB_THREADS), model == PYRO_ISING ? GPU_SMS * 4 : GPU_SMS * 8);
        struct {
            void **p;
            size_t bytes;
        } al[] = {{&G.spins, (size_t)N * model * spin_elem()},
                  {(void **)&lab_a, (size_t)N * 4},
                  {(void **)&lab_b, (size_t)N * 4},
                  {(void **)&G.fb, (size_t)cdiv(N, 128) * 16},
                  {&G.proj, model == PYRO_ISING ? 0 : (size_t)N * spin_elem()},
                  {(void **)&G.axis, 3 * sizeof(double)},
                  {(void **)&G.partials, (size_t)nmeas * 4 * sizeof(double)},
                  {(void **)&G.st, sizeof(DevStats)},
                  {(void **)&G.bi, c.sc_L ? 0 : (size_t)NB * 4},
                  {(void **)&G.bj, c.sc_L ? 0 : (size_t)NB * 4},
                  {(void **)&G.present, present.size() * 4},
                  {(void **)&G.occ, occ.size() * 4}};
        for (auto &a : al) {
            if (!a.bytes) {
                *a.p = nullptr;
                continue;
            }
            e = alloc(a.p, a.bytes);
            if (e != cudaSuccess) return err = "device allocation failed", e;
        }
        if (!c.sc_L && NB) {
            e = cudaMemcpyAsync(const_cast<int32_t *>(G.bi), c.bond_i, (size_t)NB * 4, cudaMemcpyHostToDevice, stream);
            if (e == cudaSuccess)
                e = cudaMemcpyAsync(const_cast<int32_t *>(G.bj), c.bond_j, (size_t)NB * 4, cudaMemcpyHostToDevice, stream);
            if (e != cudaSuccess) return err = "bond list copy", e;
        }
        if (!present.empty()) {
            e = cudaMemcpyAsync(const_cast<uint32_t *>(G.present), present.data(), present.size() * 4,
                                cudaMemcpyHostToDevice, stream);
            if (e != cudaSuccess) return err = "bond mask copy", e;
        }
        if (!occ.empty()) {
            e = cudaMemcpyAsync(const_cast<uint32_t *>(G.occ), occ.data(), occ.size() * 4, cudaMemcpyHostToDevice, stream);
            if (e != cudaSuccess) return err = "site mask copy", e;
        }
        e = cudaMemsetAsync(G.st, 0, sizeof(DevStats), stream);
        if (e != cudaSuccess) return err = "stats reset", e;
        G.lab = lab_a;
        G.lab_next = lab_b;
        lab_last = lab_b;
        k.init(G, c.start == PYRO_START_RANDOM, stream, nsite);
        ++launches;
        e = cudaGetLastError();
        if (e != cudaSuccess) return err = "init launch", e;
        // the host-side copies above read pageable host memory that the
        // caller may free on return
        e = cudaStreamSynchronize(stream);
        if (e != cudaSuccess) return err = "set-up", e;
        return cudaSuccess;
    }

    cudaError_t set_beta(double b)
    {
        if (b == beta) return cudaSuccess;
        beta = b;
        G.thr = sc.thr = ising_threshold(b, G.J);
        G.K2 = 2.0 * b * G.J;
        return cudaSuccess;
    }

    // Tile of the simple-cubic sweep: the power-of-two tile of at most `cap`
    // segments whose padded cost is least, each axis it does not cover adding its
    // crossing faces (as default_tile in engine.cu).
    //
    // cap.  A sweep in us at 64 / 128 / 256 segments, at the critical temperature:
    // L = 16 (a lone tile at 256) 29.0 / 26.6 / 21.7, L = 32 36.4 / 36.0 / 34.8, L = 64
    // 47.0 / 40.3 / 39.4, L = 128 66.2 / 61.2 / 60.0, L = 256 226 / 213 / 213; at
    // beta = 1, where the trees are deep: L = 16 49 / 53 / 62, L = 32 51 / 57 / 78,
    // L = 64 63 / 63 / 71, L = 128 91 / 99 / 112.  Lattices of several tiles that do
    // not fill the GPU, bound by a block's latency, take 64: up to a sixth slower at
    // the transition, up to a third faster below it.
    void sc_tile()
    {
        const int64_t segs = (int64_t)sc.SX * sc.L * sc.L;
        const int cap = segs > 256 && segs <= 16384 ? 64 : 256;
        const auto along = [](int n, int t) { return (n + t - 1) / t; };
        double best = -1.0;
        for (int tx = 1; tx <= 8; tx *= 2)
            for (int ty = 32; ty >= 1; ty /= 2)
                for (int tz = 32; tz >= 1; tz /= 2) {
                    const int nt = tx * ty * tz;
                    if (nt > cap) continue;
                    const int ax = along(sc.SX, tx), ay = along(sc.L, ty), az = along(sc.L, tz);
                    double f = 1.0;
                    if (ax > 1) f += 1.0 / (16.0 * tx);
                    if (ay > 1) f += 1.0 / ty;
                    if (az > 1) f += 1.0 / tz;
                    const double cost = f * (double)ax * ay * az * std::max(nt, 32);
                    if (best >= 0.0 && cost >= best * (1.0 - 1e-9)) continue;
                    best = cost;
                    sc.TX = tx;
                    sc.TY = ty;
                    sc.TZ = tz;
                    sc.ntx = ax;
                    sc.nty = ay;
                    sc.ntz = az;
                }
        for (sc.lTX = 0; (1 << sc.lTX) < sc.TX;) ++sc.lTX;
        for (sc.lTY = 0; (1 << sc.lTY) < sc.TY;) ++sc.lTY;
        for (sc.lTZ = 0; (1 << sc.lTZ) < sc.TZ;) ++sc.lTZ;
        // slots: every site of the segments on y and z faces, two of the others
        const int face = sc.TX * (sc.TY * sc.TZ - std::max(0, sc.TY - 2) * std::max(0, sc.TZ - 2));
        sc.nslot = (16 * face + 2 * (sc.TX * sc.TY * sc.TZ - face) + 31) & ~31;
    }

    size_t sc_flip_smem() const { return (size_t)slot_code(sc.TX * sc.TY * sc.TZ) / 8 + (size_t)sc.nslot / 8; }
    unsigned sc_seg_blocks() const { return (unsigned)cdiv(sc.nsegs, 256); }

    cudaError_t sc_setup(const pyro_graph_config &c, int64_t N, const std::vector<uint32_t> &present,
                         const std::vector<uint32_t> &occ, int64_t nocc, std::string &err)
    {
        G.N = sc.N = N;
        G.NB = 3 * N;
        G.nocc = nocc;
        G.nc = 1;
        G.J = c.J;
        sc.L = c.sc_L;
        sc.SX = (sc.L + 15) / 16;
        sc.nsegs = (int64_t)sc.SX * sc.L * sc.L;
        sc.seed = c.seed;
        sc_tile();
        const int nt = sc.TX * sc.TY * sc.TZ;
        sc_tiles = (unsigned)sc.ntx * (unsigned)sc.nty * (unsigned)sc.ntz;
        nmeas = (unsigned)std::min<int64_t>(cdiv((int64_t)sc_tiles * nt, 256), GPU_SMS * 4);
        const size_t segs = (size_t)sc.nsegs, mask = present.empty() ? 0 : segs * 2;
        struct {
            void **p;
            size_t bytes;
        } al[] = {{(void **)&sc.spins, segs * 2},
                  {(void **)&sc.code, segs * 32},
                  {(void **)&sc.P, (size_t)sc_tiles * sc.nslot * 4},
                  {(void **)&sc.nslots, (size_t)sc_tiles * 4},
                  {(void **)&sc.sflip, (size_t)sc_tiles * (sc.nslot / 8)},
                  {(void **)&sc.cross, segs * 8},
                  {(void **)&sc.fb, (size_t)cdiv(N, 128) * 16 + 16},
                  {(void **)&sc.px, mask},
                  {(void **)&sc.py, mask},
                  {(void **)&sc.pz, mask},
                  {(void **)&sc.occ, occ.empty() ? 0 : segs * 2},
                  {(void **)&sc.bytes, (size_t)N},
                  {(void **)&sc.labels, (size_t)N * 4},  // (asking for them later can't fail)
                  {(void **)&G.partials, (size_t)nmeas * 4 * sizeof(double)},
                  {(void **)&G.st, sizeof(DevStats)}};
        cudaError_t e;
        for (auto &a : al) {
            if (!a.bytes) continue;
            e = alloc(a.p, a.bytes);
            if (e != cudaSuccess) return err = "device allocation failed", e;
        }
        sc.partials = G.partials;
        sc.st = G.st;
        // the masks per segment, from 16 bits of the site set and 48 of the
        // bond set each (site by site this took 92 ms more at L = 256, of 469)
        if (mask || !occ.empty()) {
            std::vector<uint16_t> w[4];
            for (auto &v : w) v.assign(segs, 0);
            const auto bits64 = [](const std::vector<uint32_t> &set, int64_t i) {
                const size_t k = (size_t)(i >> 5);
                const unsigned sh = (unsigned)(i & 31);
                const auto word = [&](size_t j) { return j < set.size() ? (uint64_t)set[j] : 0; };
                const uint64_t lo = word(k) | word(k + 1) << 32;
                return sh ? lo >> sh | word(k + 2) << (64 - sh) : lo;
            };
            size_t seg = 0;
            for (int64_t row = 0; row < (int64_t)sc.L * sc.L; ++row)
                for (int gx = 0; gx < sc.SX; ++gx, ++seg) {
                    const int64_t i = row * sc.L + 16 * gx;
                    const uint32_t valid = 0xFFFFu >> (16 - std::min(16, sc.L - 16 * gx));
                    if (mask) {
                        const uint64_t b = bits64(present, 3 * i);
                        for (int d = 0; d < 3; ++d) w[d][seg] = (uint16_t)(every_third(b >> d) & valid);
                    }
                    if (!occ.empty()) w[3][seg] = (uint16_t)(bits64(occ, i) & valid);
                }
            const uint16_t *dst[4] = {sc.px, sc.py, sc.pz, sc.occ};
            for (int d = 0; d < 4; ++d) {
                if (!dst[d]) continue;
                e = cudaMemcpyAsync(const_cast<uint16_t *>(dst[d]), w[d].data(), segs * 2, cudaMemcpyHostToDevice, stream);
                if (e == cudaSuccess) e = cudaStreamSynchronize(stream);  // (pageable source)
                if (e != cudaSuccess) return err = "mask copy", e;
            }
        }
        e = cudaMemsetAsync(G.st, 0, sizeof(DevStats), stream);
        if (e != cudaSuccess) return err = "stats reset", e;
        sc_init_kernel<<<sc_seg_blocks(), 256, 0, stream>>>(sc, c.start == PYRO_START_RANDOM);
        ++launches;
        e = cudaGetLastError();
        if (e != cudaSuccess) return err = "init launch", e;
        e = cudaStreamSynchronize(stream);
        if (e != cudaSuccess) return err = "set-up", e;
        return cudaSuccess;
    }

    cudaError_t sc_sweeps(int64_t n)
    {
        const unsigned nt = (unsigned)(sc.TX * sc.TY * sc.TZ);
        for (int64_t s = 0; s < n; ++s) {
            launch_overlapped(sc_local_kernel, sc_tiles, nt, core_smem_bytes((int)nt), stream, sc);
            launch_overlapped(sc_unite_kernel, sc_tiles, nt, (size_t)nt * 33 * 2, stream, sc);
            launch_overlapped(sc_slot_flip_kernel, sc_tiles, SLOT_BLOCK, 0, stream, sc);
            launch_overlapped(sc_flip_kernel, sc_tiles, nt, sc_flip_smem(), stream, sc);
            launch_overlapped(sc_measure_kernel, nmeas, 256, 0, stream, sc, (int)sc_tiles);
            launch_overlapped(graph_accumulate_kernel, 1, ACC_THREADS, 0, stream, G, (int)nmeas, 1);
            launches += 6;
            swept = true;
        }
        return cudaGetLastError();
    }

    // The spins as N bytes of +-1 in sc.bytes.
    cudaError_t sc_unpack()
    {
        sc_unpack_kernel<<<sc_seg_blocks(), 256, 0, stream>>>(sc);
        ++launches;
        return cudaGetLastError();
    }
    cudaError_t sc_pack()
    {
        sc_pack_kernel<<<sc_seg_blocks(), 256, 0, stream>>>(sc);
        ++launches;
        return cudaGetLastError();
    }

    cudaError_t sc_labels()
    {
        sc_labels_kernel<<<sc_tiles, sc.TX * sc.TY * sc.TZ, 0, stream>>>(sc, swept);
        ++launches;
        lab_last = sc.labels;
        return cudaGetLastError();
    }

    cudaError_t sweeps(int64_t n)
    {
        if (sc_tiles) return sc_sweeps(n);
        for (int64_t s = 0; s < n; ++s) {
            k.sweep(G, stream, nproj, nbond, nsite, nmeas);
            launch_overlapped(graph_accumulate_kernel, 1, ACC_THREADS, 0, stream, G, (int)nmeas, 1);
            launches += model == PYRO_ISING ? 4 : 5;
            lab_last = G.lab;
            std::swap(G.lab, G.lab_next);
        }
        return cudaGetLastError();
    }

    cudaError_t measure()
    {
        if (sc_tiles) launch_overlapped(sc_measure_kernel, nmeas, 256, 0, stream, sc, (int)sc_tiles);
        else k.measure(G, stream, nmeas);
        launch_overlapped(graph_accumulate_kernel, 1, ACC_THREADS, 0, stream, G, (int)nmeas, 2);
        launches += 2;
        return cudaGetLastError();
    }

    int read_status(std::string &err)
    {
        int st = 0;
        cudaError_t e = cudaMemcpyAsync(&st, &G.st->status, sizeof(int), cudaMemcpyDeviceToHost, stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
        if (e != cudaSuccess) {
            err = std::string("device status read: ") + cudaGetErrorString(e);
            return -1;
        }
        if (st) cudaMemsetAsync(&G.st->status, 0, sizeof(int), stream);
        return st;
    }
};

}  // namespace pyro

// ------------------------------------------------------------------ C ABI --
struct pyro_graph_ctx {
    pyro::GraphEngine g;
};

namespace pyro {

void set_error(const std::string &msg);

static int gfail(int code, const std::string &msg)
{
    set_error(msg);
    return code;
}

#define GRAPH_CUDA(call, what)                                                                     \
    do {                                                                                           \
        const cudaError_t e_ = (call);                                                             \
        if (e_ != cudaSuccess) return gfail(PYRO_E_CUDA, std::string(what) + ": " + cudaGetErrorString(e_)); \
    } while (0)

static int gfinish(GraphEngine &g)
{
    std::string err;
    const int st = g.read_status(err);
    if (st < 0) return gfail(PYRO_E_CUDA, err);
    if (st & ST_NOCONVERGE) return gfail(PYRO_E_NOCONVERGE, "union-find exceeded its iteration bound");
    return PYRO_OK;
}

// Bond list of a neighbour table; -1 on a bad table (see pyro.h).
static int64_t bonds_from_table(int64_t N, int z, const int32_t *nbr, int32_t *bi, int32_t *bj, std::string &why)
{
    int64_t E = 0;
    for (int64_t i = 0; i < N; ++i)
        for (int k = 0; k < z; ++k) {
            const int32_t j = nbr[i * z + k];
            if (j < 0) continue;
            if (j >= N || j == i) {
                why = "neighbour table entry out of range or naming its own row (site " + std::to_string(i) + ")";
                return -1;
            }
            if (i < j) {
                // j must appear in i's row as often as i appears in j's row
                int a = 0, b = 0;
                for (int q = 0; q < z; ++q) {
                    a += nbr[i * z + q] == j;
                    b += nbr[(int64_t)j * z + q] == i;
                }
                if (a != b) {
                    why = "neighbour table is not symmetric (sites " + std::to_string(i) + ", " + std::to_string(j) + ")";
                    return -1;
                }
                if (bi) {
                    bi[E] = (int32_t)i;
                    bj[E] = j;
                }
                ++E;
            } else {
                int a = 0, b = 0;
                for (int q = 0; q < z; ++q) {
                    a += nbr[i * z + q] == j;
                    b += nbr[(int64_t)j * z + q] == i;
                }
                if (a != b) {
                    why = "neighbour table is not symmetric (sites " + std::to_string(j) + ", " + std::to_string(i) + ")";
                    return -1;
                }
            }
        }
    return E;
}

}  // namespace pyro

using namespace pyro;

extern "C" {

int64_t pyro_graph_bonds_from_table(int64_t N, int z, const int32_t *nbr, int32_t *bond_i, int32_t *bond_j)
{
    if (N < 1 || N > INT32_MAX || z < 0 || (z > 0 && !nbr) || ((bond_i == nullptr) != (bond_j == nullptr)))
        return gfail(PYRO_E_INVAL, "bad argument");
    std::string why;
    const int64_t E = bonds_from_table(N, z, nbr, bond_i, bond_j, why);
    if (E < 0) return gfail(PYRO_E_INVAL, why);
    return E;
}

int pyro_graph_init(pyro_graph *out, const pyro_graph_config *c)
{
    if (!out || !c) return gfail(PYRO_E_INVAL, "NULL argument");
    *out = nullptr;
    if (c->model < PYRO_ISING || c->model > PYRO_HEIS) return gfail(PYRO_E_INVAL, "model must be 1, 2 or 3");
    if (c->model != PYRO_ISING && c->precision != PYRO_FP32 && c->precision != PYRO_FP64)
        return gfail(PYRO_E_INVAL, "precision must be PYRO_FP32 or PYRO_FP64");
    if (c->start != PYRO_START_UP && c->start != PYRO_START_RANDOM)
        return gfail(PYRO_E_INVAL, "start must be PYRO_START_UP or PYRO_START_RANDOM");
    if (!(c->J > 0.0) || !std::isfinite(c->J)) return gfail(PYRO_E_INVAL, "J must be positive and finite");
    int64_t N, NB;
    if (c->sc_L) {
        if (c->sc_L < 2 || c->sc_L > 1290) return gfail(PYRO_E_INVAL, "sc_L must be in [2, 1290]");
        if (c->bond_i || c->bond_j) return gfail(PYRO_E_INVAL, "a simple-cubic lattice takes no bond list");
        N = (int64_t)c->sc_L * c->sc_L * c->sc_L;
        NB = 3 * N;
    } else {
        N = c->nsites;
        NB = c->nbonds;
        if (N < 1 || N > INT32_MAX) return gfail(PYRO_E_INVAL, "nsites must be in [1, 2^31)");
        if (NB < 0 || NB >= ((int64_t)1 << 35)) return gfail(PYRO_E_INVAL, "nbonds must be in [0, 2^35)");
        if (NB && (!c->bond_i || !c->bond_j)) return gfail(PYRO_E_INVAL, "NULL bond list");
        for (int64_t e = 0; e < NB; ++e) {
            const int64_t i = c->bond_i[e], j = c->bond_j[e];
            if (i < 0 || i >= N || j < 0 || j >= N) return gfail(PYRO_E_INVAL, "bond " + std::to_string(e) + ": site out of range");
            if (i == j) return gfail(PYRO_E_INVAL, "bond " + std::to_string(e) + ": self-loop");
        }
    }
    // occupied-site and present-bond bit sets (only with a mask)
    std::vector<uint32_t> occ, present;
    int64_t nocc = N;
    if (c->site_mask) {
        occ.assign((size_t)((N + 31) / 32), 0u);
        nocc = 0;
        for (int64_t i = 0; i < N; ++i)
            if (c->site_mask[i]) {
                occ[(size_t)(i >> 5)] |= 1u << (i & 31);
                ++nocc;
            }
    }
    if (c->site_mask || c->bond_mask) {
        present.assign((size_t)((NB + 31) / 32), 0u);
        const int64_t L = c->sc_L;
        for (int64_t e = 0; e < NB; ++e) {
            if (c->bond_mask && !c->bond_mask[e]) continue;
            int64_t i, j;
            if (L) {
                const int64_t s = e / 3, d = e % 3, x = s % L, y = (s / L) % L, z = s / (L * L);
                i = s;
                j = d == 0 ? (x + 1) % L + L * (y + L * z) : d == 1 ? x + L * ((y + 1) % L + L * z)
                                                                    : x + L * (y + L * ((z + 1) % L));
            } else {
                i = c->bond_i[e];
                j = c->bond_j[e];
            }
            if (c->site_mask && (!c->site_mask[i] || !c->site_mask[j])) continue;
            present[(size_t)(e >> 5)] |= 1u << (e & 31);
        }
    }
    pyro_graph_ctx *h = new (std::nothrow) pyro_graph_ctx;
    if (!h) return gfail(PYRO_E_NOMEM, "host allocation failed");
    std::string err;
    const cudaError_t ce = h->g.setup(*c, N, NB, present, occ, nocc, err);
    if (ce != cudaSuccess) {
        cudaGetLastError();
        h->g.release();
        delete h;
        return gfail(ce == cudaErrorMemoryAllocation ? PYRO_E_NOMEM : PYRO_E_CUDA,
                     err + ": " + cudaGetErrorString(ce));
    }
    *out = h;
    return PYRO_OK;
}

int pyro_graph_sweep(pyro_graph g, double beta, int64_t n)
{
    if (!g) return gfail(PYRO_E_INVAL, "NULL handle");
    if (!(beta >= 0.0) || !std::isfinite(beta)) return gfail(PYRO_E_INVAL, "beta must be finite and >= 0");
    if (n < 0) return gfail(PYRO_E_INVAL, "n must be >= 0");
    g->g.set_beta(beta);
    GRAPH_CUDA(g->g.sweeps(n), "sweep launch");
    return PYRO_OK;
}

int pyro_graph_measure(pyro_graph g, double *E, double *m2, double *m4)
{
    if (!g) return gfail(PYRO_E_INVAL, "NULL handle");
    GRAPH_CUDA(g->g.measure(), "measure launch");
    double last[4];
    GRAPH_CUDA(cudaMemcpyAsync(last, g->g.G.st->last, sizeof(last), cudaMemcpyDeviceToHost, g->g.stream), "measure copy");
    const int rc = gfinish(g->g);
    if (rc) return rc;
    if (E) *E = last[0];
    if (m2) *m2 = last[1];
    if (m4) *m4 = last[2];
    return PYRO_OK;
}

int pyro_graph_stats(pyro_graph g, pyro_stats_t *s)
{
    if (!g || !s) return gfail(PYRO_E_INVAL, "NULL argument");
    DevStats d;
    GRAPH_CUDA(cudaMemcpyAsync(&d, g->g.G.st, sizeof(d), cudaMemcpyDeviceToHost, g->g.stream), "stats copy");
    const int rc = gfinish(g->g);
    if (rc) return rc;
    s->count = d.count;
    double *dst[5] = {&s->sum_E, &s->sum_E2, &s->sum_m2, &s->sum_m4, &s->sum_absm};
    for (int k = 0; k < 5; ++k) *dst[k] = d.acc_s[k] + d.acc_c[k];
    return PYRO_OK;
}

int pyro_graph_reset_stats(pyro_graph g)
{
    if (!g) return gfail(PYRO_E_INVAL, "NULL handle");
    DevStats *d = g->g.G.st;
    GRAPH_CUDA(cudaMemsetAsync(d->acc_s, 0, sizeof(d->acc_s), g->g.stream), "reset");
    GRAPH_CUDA(cudaMemsetAsync(d->acc_c, 0, sizeof(d->acc_c), g->g.stream), "reset");
    GRAPH_CUDA(cudaMemsetAsync(&d->count, 0, sizeof(d->count), g->g.stream), "reset");
    return PYRO_OK;
}

int pyro_graph_get_spins(pyro_graph g, void *host, size_t bytes)
{
    if (!g || !host) return gfail(PYRO_E_INVAL, "NULL argument");
    GraphEngine &e = g->g;
    const int64_t N = e.G.N;
    if (e.model == PYRO_ISING) {
        if (bytes != (size_t)N) return gfail(PYRO_E_INVAL, "Ising spins need N bytes");
        if (e.sc_tiles) GRAPH_CUDA(e.sc_unpack(), "spins unpacking");
        GRAPH_CUDA(cudaMemcpyAsync(host, e.sc_tiles ? e.sc.bytes : e.G.spins, (size_t)N, cudaMemcpyDeviceToHost, e.stream),
                   "spins copy");
        return gfinish(e);
    }
    const int n = e.model;
    if (bytes != (size_t)N * n * sizeof(double)) return gfail(PYRO_E_INVAL, "n-vector spins need 8 n N bytes");
    std::vector<unsigned char> raw((size_t)N * n * e.spin_elem());
    GRAPH_CUDA(cudaMemcpyAsync(raw.data(), e.G.spins, raw.size(), cudaMemcpyDeviceToHost, e.stream), "spins copy");
    const int rc = gfinish(e);
    if (rc) return rc;
    double *o = static_cast<double *>(host);
    for (int64_t i = 0; i < N; ++i)
        for (int k = 0; k < n; ++k)
            o[i * n + k] = e.prec == PYRO_FP64 ? reinterpret_cast<const double *>(raw.data())[(size_t)k * N + i]
                                               : (double)reinterpret_cast<const float *>(raw.data())[(size_t)k * N + i];
    return PYRO_OK;
}

int pyro_graph_set_spins(pyro_graph g, const void *host, size_t bytes)
{
    if (!g || !host) return gfail(PYRO_E_INVAL, "NULL argument");
    GraphEngine &e = g->g;
    const int64_t N = e.G.N;
    if (e.model == PYRO_ISING) {
        if (bytes != (size_t)N) return gfail(PYRO_E_INVAL, "Ising spins need N bytes");
        const int8_t *s = static_cast<const int8_t *>(host);
        unsigned bad = 0;  // branch-free, so that the check vectorises
        for (int64_t i = 0; i < N; ++i) bad |= (unsigned)((uint8_t)(s[i] + 1) & 0xFDu);  // 0 for -1 and +1 only
        if (bad) return gfail(PYRO_E_INVAL, "Ising spins must be +1 or -1");
        GRAPH_CUDA(cudaMemcpyAsync(e.sc_tiles ? e.sc.bytes : e.G.spins, host, (size_t)N, cudaMemcpyHostToDevice, e.stream),
                   "spins copy");
        if (e.sc_tiles) GRAPH_CUDA(e.sc_pack(), "spins packing");
        GRAPH_CUDA(cudaStreamSynchronize(e.stream), "stream synchronize");
        return PYRO_OK;
    }
    const int n = e.model;
    if (bytes != (size_t)N * n * sizeof(double)) return gfail(PYRO_E_INVAL, "n-vector spins need 8 n N bytes");
    const double *s = static_cast<const double *>(host);
    std::vector<unsigned char> raw((size_t)N * n * e.spin_elem());
    for (int64_t i = 0; i < N; ++i)
        for (int k = 0; k < n; ++k) {
            if (e.prec == PYRO_FP64) reinterpret_cast<double *>(raw.data())[(size_t)k * N + i] = s[i * n + k];
            else reinterpret_cast<float *>(raw.data())[(size_t)k * N + i] = (float)s[i * n + k];
        }
    GRAPH_CUDA(cudaMemcpyAsync(e.G.spins, raw.data(), raw.size(), cudaMemcpyHostToDevice, e.stream), "spins copy");
    GRAPH_CUDA(cudaStreamSynchronize(e.stream), "stream synchronize");
    return PYRO_OK;
}

int pyro_graph_get_labels(pyro_graph g, int32_t *host, int64_t n)
{
    if (!g || !host) return gfail(PYRO_E_INVAL, "NULL argument");
    if (n != g->g.G.N) return gfail(PYRO_E_INVAL, "labels need N entries");
    if (g->g.sc_tiles) GRAPH_CUDA(g->g.sc_labels(), "labels");
    GRAPH_CUDA(cudaMemcpyAsync(host, g->g.lab_last, (size_t)n * 4, cudaMemcpyDeviceToHost, g->g.stream), "labels copy");
    return gfinish(g->g);
}

int pyro_graph_set_sweep(pyro_graph g, uint64_t sweep)
{
    if (!g) return gfail(PYRO_E_INVAL, "NULL handle");
    graph_set_sweep_kernel<<<1, 1, 0, g->g.stream>>>(g->g.G.st, sweep);
    GRAPH_CUDA(cudaGetLastError(), "set sweep");
    return PYRO_OK;
}

uint64_t pyro_graph_get_sweep(pyro_graph g)
{
    if (!g) return 0;
    unsigned long long s = 0;
    if (cudaMemcpyAsync(&s, &g->g.G.st->sweep, sizeof(s), cudaMemcpyDeviceToHost, g->g.stream) != cudaSuccess) return 0;
    cudaStreamSynchronize(g->g.stream);
    return s;
}

int64_t pyro_graph_num_sites(pyro_graph g) { return g ? g->g.G.N : 0; }
int64_t pyro_graph_num_bonds(pyro_graph g) { return g ? g->g.G.NB : 0; }

int pyro_graph_sync(pyro_graph g)
{
    if (!g) return gfail(PYRO_E_INVAL, "NULL handle");
    return gfinish(g->g);
}

void *pyro_graph_get_stream(pyro_graph g) { return g ? static_cast<void *>(g->g.stream) : nullptr; }
uint64_t pyro_graph_launch_count(pyro_graph g) { return g ? g->g.launches : 0; }

void pyro_graph_destroy(pyro_graph g)
{
    if (!g) return;
    g->g.release();
    delete g;
}

}  // extern "C"
