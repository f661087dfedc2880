// sweep_core.cuh -- the model-independent parts of a Swendsen-Wang sweep:
// tile geometry, tile-local labelling in shared memory, the global union of
// tile-crossing clusters, and the resolution of every site to its cluster's
// canonical root.
//
// Bonds of a cell.  Each of the cell's four FCC points f owns an "up"
// tetrahedron (its sites 4 f .. 4 f + 3) and a "down" tetrahedron (its
// site 4 f and three sites of backward neighbour cells).  The 48 bonds are
// kept as three 16-bit groups, bit 4 f + q of group g:
//   g = 0 (A): up pairs    q = 0 (0,1)  1 (1,2)  2 (2,3)  3 (0,3)
//   g = 1 (B): up (0,2), up (1,3), down (0,2), down (1,3)
//   g = 2 (C): down pairs  q = 0 (0,1)  1 (1,2)  2 (2,3)  3 (0,3)
// so that shift-XOR of a 16-bit spin word yields four bonds at once, and
// the bond with random-number id b = 48 c + 16 g + 4 f + q draws the top
// byte of its uniform from byte (b & 15) of BOND call b >> 4 = 3 c + g.
#pragma once

#include "bonds.cuh"
#include "ccl.cuh"
#include "launch.cuh"

namespace pyro {

// Position of the calling thread's cell in its tile and in the lattice.
// Tile edges are powers of two (shifts, no divisions) and need not divide L:
// the last tile of an axis may reach past the lattice.  A thread whose cell
// lies there has valid = false; its coordinates are clamped into the lattice
// (so that its loads stay in bounds), it activates no bond and stores
// nothing.  A tile that covers a whole axis wraps onto itself along it.
struct TileCtx {
    int TX, TY, TZ, lTX, lTY, nt, L;
    int ox, oy, oz;
    int lx, ly, lz, t;
    int x, y, z;  // the cell's coordinates (clamped)
    bool valid;
    int64_t cell;
    // local cell offset of a backward step along each axis (valid only if
    // the step stays in the tile), and whether it leaves the tile
    int dxm, dym, dzm;
    bool bx, by, bz;
};

__device__ __forceinline__ TileCtx tile_ctx(const Batch &B, const Rep &R, int64_t tile)
{
    TileCtx c;
    c.TX = B.TX;
    c.TY = B.TY;
    c.TZ = B.TZ;
    c.lTX = B.lTX;
    c.lTY = B.lTY;
    c.nt = B.TX * B.TY * B.TZ;
    c.L = R.L;
    // a lattice has fewer than 2^31 tiles (L <= 511): 32-bit divisions
    const uint32_t tl = (uint32_t)tile, ntx = (uint32_t)R.ntx, nty = (uint32_t)R.nty;
    const uint32_t txy = tl / ntx;
    c.ox = (int)(tl - txy * ntx) * c.TX;
    c.oy = (int)(txy % nty) * c.TY;
    c.oz = (int)(txy / nty) * c.TZ;
    c.t = threadIdx.x;
    c.lx = c.t & (c.TX - 1);
    c.ly = (c.t >> c.lTX) & (c.TY - 1);
    c.lz = c.t >> (c.lTX + c.lTY);
    c.x = c.ox + c.lx;
    c.y = c.oy + c.ly;
    c.z = c.oz + c.lz;
    c.valid = max(c.x, max(c.y, c.z)) < c.L;
    c.x = min(c.x, c.L - 1);
    c.y = min(c.y, c.L - 1);
    c.z = min(c.z, c.L - 1);
    c.cell = (int64_t)c.x + (int64_t)c.L * ((int64_t)c.y + (int64_t)c.L * c.z);
    c.bx = c.lx == 0 && c.TX < c.L;
    c.by = c.ly == 0 && c.TY < c.L;
    c.bz = c.lz == 0 && c.TZ < c.L;
    c.dxm = c.lx > 0 ? -1 : c.L - 1;
    c.dym = c.ly > 0 ? -c.TX : (c.L - 1) * c.TX;
    c.dzm = c.lz > 0 ? -c.TX * c.TY : (c.L - 1) * c.TX * c.TY;
    return c;
}

// Lanes of the calling thread's warp that exist in a block of nt threads.
__device__ __forceinline__ unsigned lanes_mask(int nt)
{
    const int cnt = min(32, nt - (int)(threadIdx.x & ~31u));
    return cnt >= 32 ? 0xffffffffu : ((1u << cnt) - 1u);
}

// Deterministic sums of the four groups of nt doubles in scratch (written by
// the block and published by a barrier; group q at q nt): a fixed tree in
// shared memory (any nt), one barrier per level for all four; results valid
// in thread 0.  (A warp-shuffle tree would add in FP64 on every lane at every
// level; FP64 adds are scarce on this GPU.)
__device__ __forceinline__ void tile_sum4_f64(double v[4], int nt, double *scratch)
{
    for (int lo = 30 - __clz(max(2 * nt - 1, 2)); lo >= 0; --lo) {
        const int o = 1 << lo;  // half the span of nt values still to add
        // the threads share the 4 o additions of a level
        for (int e = threadIdx.x; e < 4 * o; e += blockDim.x) {
            const int q = e >> lo, t = e & (o - 1);
            if (t + o < nt) scratch[q * nt + t] = __dadd_rn(scratch[q * nt + t], scratch[q * nt + t + o]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = scratch[q * nt];
}

// Tile-local cell of a vertex whose cell is this cell stepped back along
// the axes of mask m (only meaningful if the vertex is inside the tile).
__device__ __forceinline__ int vertex_local_cell(const TileCtx &c, int m)
{
    return c.t + ((m & 1) ? c.dxm : 0) + ((m & 2) ? c.dym : 0) + ((m & 4) ? c.dzm : 0);
}

__device__ __forceinline__ int wrap_back(int v, int L) { return v == 0 ? L - 1 : v - 1; }

// Cells of the backward halo staged by the tile kernels.
__host__ __device__ constexpr int halo_cells(int TX, int TY, int TZ) { return (TX + 1) * (TY + 1) * (TZ + 1); }

__device__ __forceinline__ int halo_index(const TileCtx &c, int m)
{
    const int HX = c.TX + 1, HY = c.TY + 1;
    return (c.lx + 1 - (m & 1)) + HX * ((c.ly + 1 - ((m >> 1) & 1)) + HY * (c.lz + 1 - ((m >> 2) & 1)));
}

// ------------------------------------------------------ bond bit layout --
// Vertex pair of slot q of group g (see the header comment); up = whether
// the pair belongs to the up tetrahedron.
__host__ __device__ constexpr int slot_a(int g, int q) { return g == 1 ? (q & 1) : (q == 3 ? 0 : q); }
__host__ __device__ constexpr int slot_b(int g, int q) { return g == 1 ? (q & 1) + 2 : (q == 3 ? 3 : q + 1); }
__host__ __device__ constexpr bool slot_up(int g, int q) { return g == 0 || (g == 1 && q < 2); }

// Index into the tetrahedron table from a tetrahedron's bond bits: bits
// 0..3 pairs (0,1) (1,2) (2,3) (0,3), bits 4..5 pairs (0,2) (1,3).
__device__ __forceinline__ uint32_t up_tet_index(uint32_t A, uint32_t Bg, int f)
{
    return ((A >> (4 * f)) & 0xFu) | (((Bg >> (4 * f)) & 0x3u) << 4);
}
__device__ __forceinline__ uint32_t down_tet_index(uint32_t C, uint32_t Bg, int f)
{
    return ((C >> (4 * f)) & 0xFu) | (((Bg >> (4 * f + 2)) & 0x3u) << 4);
}

// Tetrahedron table, by bond pattern idx (order as above): bits 0-7 the
// smallest vertex connected to each vertex (2 bits each), bits 8-11 the
// component representatives, bits 16-21 the spanning pairs (pair index k of
// (smallest vertex, v) for every non-representative v).
struct TetTable {
    uint32_t e[64];
};
constexpr TetTable make_tet_table()
{
    TetTable t{};
    const int pa[6] = {0, 1, 2, 0, 0, 1}, pb[6] = {1, 2, 3, 3, 2, 3};
    for (uint32_t idx = 0; idx < 64; ++idx) {
        int rr[4] = {0, 1, 2, 3};
        for (int pass = 0; pass < 3; ++pass)
            for (int k = 0; k < 6; ++k)
                if ((idx >> k) & 1u) {
                    const int m = rr[pa[k]] < rr[pb[k]] ? rr[pa[k]] : rr[pb[k]];
                    rr[pa[k]] = m;
                    rr[pb[k]] = m;
                }
        uint32_t w = 1u << 8;
        for (int v = 0; v < 4; ++v) {
            w |= (uint32_t)rr[v] << (2 * v);
            if (v > 0 && rr[v] == v) w |= 1u << (8 + v);
            if (rr[v] != v) w |= 1u << (16 + pair_index(rr[v], v));
        }
        t.e[idx] = w;
    }
    return t;
}
static __device__ const TetTable tet_table = make_tet_table();

// The four spins of the down tetrahedron of each FCC point f of a cell,
// gathered into one 16-bit word (bit 4 f + v = vertex v).  w[m] = spin word
// of the cell stepped back along the axes of mask m.  ONE = 0x10001: two
// cells at once, one in each half of the words.
template <uint32_t ONE = 1u>
__device__ __forceinline__ uint32_t down_word(const uint32_t w[7])
{
    uint32_t D = 0;
#pragma unroll
    for (int f = 0; f < 4; ++f)
#pragma unroll
        for (int v = 0; v < 4; ++v) D |= ((w[down_mask(f, v)] >> down_bit(f, v)) & ONE) << (4 * f + v);
    return D;
}

// Antiparallel bits of the three bond groups from the up and down spin
// words (shift-XOR within each nibble, so halves of a word stay apart).
template <uint32_t ONE = 1u>
__device__ __forceinline__ void antiparallel_groups(uint32_t U, uint32_t D, uint32_t &A, uint32_t &Bg, uint32_t &C)
{
    const uint32_t u1 = U ^ (U >> 1), u2 = U ^ (U >> 2), u3 = U ^ (U >> 3);
    const uint32_t d1 = D ^ (D >> 1), d2 = D ^ (D >> 2), d3 = D ^ (D >> 3);
    A = (u1 & (0x7777u * ONE)) | ((u3 & (0x1111u * ONE)) << 3);
    Bg = (u2 & (0x3333u * ONE)) | ((d2 & (0x3333u * ONE)) << 2);
    C = (d1 & (0x7777u * ONE)) | ((d3 & (0x1111u * ONE)) << 3);
}

// Flip bits of the tile's sites: bits 16 c .. 16 c + 15 of the FLIP stream
// (bit i = bit i & 127 of call i >> 7) for cell c.  One Philox call serves 8
// cells: where those are a run of the tile's rows (TX and L multiples of 8)
// one thread draws and stores them, one warp of the tile's; else every thread
// draws its own cell's.
__device__ __forceinline__ void store_flip_bits(const TileCtx &c, const Rep &R, uint32_t sweep)
{
    if (((c.TX | c.L) & 7) == 0) {
        if (c.t >= c.nt >> 3) return;
        const int t = c.t << 3;  // first cell of the run
        const int x = c.ox + (t & (c.TX - 1)), y = c.oy + ((t >> c.lTX) & (c.TY - 1)), z = c.oz + (t >> (c.lTX + c.lTY));
        if (max(x, max(y, z)) >= c.L) return;
        const int64_t cell = (int64_t)x + (int64_t)c.L * ((int64_t)y + (int64_t)c.L * z);
        *reinterpret_cast<uint4 *>(R.F + cell) = philox_call(R.seed, sweep, TAG_FLIP, (uint64_t)cell >> 3);
    } else if (c.valid) {
        const uint4 w = philox_call(R.seed, sweep, TAG_FLIP, (uint64_t)c.cell >> 3);
        R.F[c.cell] = (uint16_t)(word_of(w, (int)((c.cell & 7) >> 1)) >> (16 * (int)(c.cell & 1)));
    }
}

// --------------------------------------------------- tile-local labelling --
// Shared memory of the local kernels: labels (17 nt ints), union pairs
// (15 nt words), the pair and the slot counter, tetrahedron table
// (64 words); the model's staging area follows at the next 16-byte boundary
// (it holds 16-byte vectors).
__host__ __device__ constexpr int core_words(int nt) { return (32 * nt + 4 + 64 + 3) & ~3; }
__host__ __device__ constexpr size_t core_smem_bytes(int nt) { return (size_t)core_words(nt) * 4; }
static_assert(core_smem_bytes(1) % 16 == 0 && core_smem_bytes(2) % 16 == 0 && core_smem_bytes(8) % 16 == 0 &&
                  core_smem_bytes(512) % 16 == 0 && core_words(1) >= 32 + 68 && core_words(2) >= 64 + 68,
              "staging area must start on a 16-byte boundary after the core area");
// Words that hold labels and pairs, dead until the labelling starts.
__host__ __device__ constexpr int core_shared_words(int nt) { return 32 * nt; }

// Pairs k of the down tetrahedron of f with a vertex whose cell is a
// backward step along axis d (bit k).
__host__ __device__ constexpr uint32_t pair_axis_mask(int f, int d)
{
    uint32_t m = 0;
    for (int k = 0; k < 6; ++k)
        if (((down_mask(f, pair_a(k)) | down_mask(f, pair_b(k))) >> d) & 1) m |= 1u << k;
    return m;
}

// Ends of pair 6 f + k of a cell's down tetrahedra: the cells' shift masks
// (bits 0-2 and 16-18) and sites (bits 4-7 and 20-23).
struct PairTable {
    uint32_t e[24];
};
constexpr PairTable make_pair_table()
{
    PairTable t{};
    for (int f = 0; f < 4; ++f)
        for (int k = 0; k < 6; ++k) {
            const int a = pair_a(k), b = pair_b(k);
            t.e[6 * f + k] = (uint32_t)(down_mask(f, a) | (down_bit(f, a) << 4) | (down_mask(f, b) << 16) | (down_bit(f, b) << 20));
        }
    return t;
}
static __device__ const PairTable pair_table = make_pair_table();

// The same of all four tetrahedra (bit 6 f + k).
__host__ __device__ constexpr uint32_t leaving_pairs(int d)
{
    return pair_axis_mask(0, d) | (pair_axis_mask(1, d) << 6) | (pair_axis_mask(2, d) << 12) | (pair_axis_mask(3, d) << 18);
}

// Sites (bit 4 g + v) of a cell that belong to down tetrahedra reaching across
// the low (high) face of axis d from a cell on that face: the tetrahedron of
// f = g ^ v extends along d iff a_d(f) = 0, i.e. a_d(g) = a_d(v); its vertices
// with a_d(v) = 1 are a cell back along d.
__host__ __device__ constexpr uint32_t face_sites(int d, int high)
{
    uint32_t m = 0;
    for (int g = 0; g < 4; ++g)
        for (int v = 0; v < 4; ++v)
            if (afcc(g, d) == high && afcc(v, d) == high) m |= 1u << (4 * g + v);
    return m;
}

// Sites of the calling thread's cell whose down tetrahedron reaches into
// another tile: the possible ends of the bonds that cross tile faces.
__device__ __forceinline__ uint32_t crossing_sites(const TileCtx &c)
{
    uint32_t m = 0;
    if (c.TX < c.L) m |= (c.lx == 0 ? face_sites(0, 0) : 0u) | (c.lx == c.TX - 1 || c.x == c.L - 1 ? face_sites(0, 1) : 0u);
    if (c.TY < c.L) m |= (c.ly == 0 ? face_sites(1, 0) : 0u) | (c.ly == c.TY - 1 || c.y == c.L - 1 ? face_sites(1, 1) : 0u);
    if (c.TZ < c.L) m |= (c.lz == 0 ? face_sites(2, 0) : 0u) | (c.lz == c.TZ - 1 || c.z == c.L - 1 ? face_sites(2, 1) : 0u);
    return c.valid ? m : 0u;
}

// A slot's entry with this bit set is a link: the low 31 bits are the slot
// (16 nt tile + slot in the tile, below 2^31) it points at.  Without it the
// entry is the root site of the slot's cluster so far.
constexpr uint32_t SLOT_LINK = 0x80000000u;

struct CoreSmem {
    int lab;  // base of the labels: their address in the shared window
    uint32_t *plist;
    int *pcount;
    uint32_t *lut;  // the block's copy of tet_table
    unsigned char *stage;  // model staging area (16-byte aligned)
};

__device__ __forceinline__ CoreSmem core_smem(int *smem, int nt)
{
    CoreSmem s;
    s.lab = (int)__cvta_generic_to_shared(smem);
    s.plist = reinterpret_cast<uint32_t *>(smem + 17 * nt);
    s.pcount = smem + 32 * nt;  // counters of the listed pairs and of the slots
    s.lut = reinterpret_cast<uint32_t *>(smem + 32 * nt + 4);
    s.stage = reinterpret_cast<unsigned char *>(smem + core_words(nt));
    return s;
}

// Called by every thread before the model's staging (covered by the same
// __syncthreads): clears the counters and fills the table.
__device__ __forceinline__ void core_prologue(const CoreSmem &s)
{
    if (threadIdx.x == 0) {  // the block may be a single thread
        s.pcount[0] = 0;
        s.pcount[1] = 0;
    }
    for (int i = threadIdx.x; i < 64; i += blockDim.x) s.lut[i] = tet_table.e[i];
}

// The code of a tile-local root without a slot is its label's word, 17 t + s; the
// codes of the slots follow from the next multiple of 32.
__host__ __device__ constexpr int slot_code(int nt) { return (17 * nt + 31) & ~31; }
static_assert(slot_code(512) + 16 * 512 < 65536, "codes are 16-bit");

// Entries at or above this are codes, not names.
constexpr int IS_CODE = 1 << 20;
// Synchronous rounds of the resolution before the walks.
constexpr int RESOLVE_ROUNDS = 1;

// Pairs the list has room for.
__device__ __forceinline__ int list_room(int nt) { return 15 * nt; }

// Unites the listed pairs, two at a time per thread (after a barrier behind the
// listing, before one ahead of the labels' next use).  False if a bound was hit.
__device__ __forceinline__ bool unite_listed(const CoreSmem &s, int nt)
{
    bool ok = true;
    const int np = min(s.pcount[0], list_room(nt));
    for (int e = threadIdx.x; e < np; e += 2 * nt) {
        const uint32_t p0 = s.plist[e], p1 = e + nt < np ? s.plist[e + nt] : p0;
        ok &= sunite2((int)(p0 & 0xFFFFu), (int)(p0 >> 16), (int)(p1 & 0xFFFFu), (int)(p1 >> 16));
    }
    return ok;
}

// The second half of a tile's labelling, for a thread's 16 sites named me, me +
// 4, ..: unites the listed pairs, resolves every representative (reps) to its
// root, gives the roots of the sites in `ends` (which a crossing bond may end
// on) a slot each in P (the root's site: site0 + q for the thread's q-th), and
// returns in ent the codes of the representatives (entries below IS_CODE are
// names of roots without a slot).  Called by every thread of the block, after a
// barrier behind the listing.
template <typename Ends>
__device__ __forceinline__ void finish_labels(const CoreSmem &s, int nt, int me, uint32_t reps, const Ends &ends_of,
                                              int32_t site0, int32_t *P, int32_t *nslots, int *status, int ent[16])
{
    const bool ok = unite_listed(s, nt);
    __syncthreads();  // all unions done
    if (!ok) atomicOr(status, ST_NOCONVERGE);
    // Resolution: every representative's entry becomes its root's name.  No
    // union changes the trees any more, and entries only move up them.
    // RESOLVE_ROUNDS times all entries move to their grandparents together, a
    // barrier after each; a representative whose parent is a root is done for
    // good.  The few left on deeper chains are walked to their roots by their
    // threads, three at a time, read-only (whatever the others write meanwhile,
    // an entry is an ancestor).  The loads of a step are issued together: one
    // representative after the other took 31 % of the kernel.  Ising local kernel
    // at L = 256 with 0, 1, 2 rounds: 1,698, 1,595, 1,684 us (a round between the
    // first pass and the listed pairs besides: 60 us slower than without).
    uint32_t todo = reps;
#pragma unroll 1
    for (int it = 0; it < RESOLVE_ROUNDS; ++it) {
        int p[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) p[q] = label_get(me + 4 * q);
        todo = 0;
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            const int gp = label_get(p[q]);
            const bool move = ((reps >> q) & 1u) && gp != p[q];
            label_set_if(move, me + 4 * q, gp);
            todo |= (move ? 1u : 0u) << q;
        }
        __syncthreads();
    }
    bool walked = true;
#pragma unroll 1
    while (todo) {
        int x[3], r[3];
        const int q0 = __ffs(todo) - 1;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            x[k] = me + 4 * (todo ? __ffs(todo) - 1 : q0);
            todo &= todo - 1;
            r[k] = label_get(x[k]);
        }
#pragma unroll 1
        for (int st = 0;; ++st) {
            int p[3];
            bool there = true;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                p[k] = label_get(r[k]);
                there &= p[k] == r[k];
            }
            if (there) break;
#pragma unroll
            for (int k = 0; k < 3; ++k) r[k] = p[k];
            if (st == 16 * nt) {
                walked = false;
                break;
            }
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) label_set(x[k], r[k]);
    }
    if (!walked) atomicOr(status, ST_NOCONVERGE);
    __syncthreads();
    // Mark the roots of the sites a crossing bond may end on: the root's own
    // entry, its name, gets bit 0 set (every marker stores the same value).
    // A site's entry is its root's name or its representative's, so two loads
    // lead to the root whatever is marked meanwhile.
    const uint32_t ends = ends_of();
#pragma unroll
    for (int q = 0; q < 16; ++q) ent[q] = label_get(me + 4 * q) & ~1;
    if (ends) {
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            const bool end = (ends >> q) & 1u;
            const int r = label_get(end ? ent[q] : me) & ~1;
            label_set_if(end, r, r | 1);
        }
    }
    __syncthreads();
    // number the marked roots; a marked root's own entry becomes its code
    {
        uint32_t marked = 0;
#pragma unroll
        for (int q = 0; q < 16; ++q) marked |= (uint32_t)(label_get(me + 4 * q) & 1) << q;
        const unsigned lanes = lanes_mask(nt);
        const int lane = threadIdx.x & 31, last = 31 - __clz(lanes);
        const int n = __popc(marked);
        int incl = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(lanes, incl, o);
            if (lane >= o) incl += v;
        }
        int base = 0;
        if (lane == last && incl) base = atomicAdd(s.pcount + 1, incl);
        int slot = __shfl_sync(lanes, base, last) + incl - n;
#pragma unroll 1
        while (marked) {
            const int q = __ffs(marked) - 1;
            marked &= marked - 1;
            P[slot] = site0 + q;
            label_set(me + 4 * q, IS_CODE + slot_code(nt) + slot);
            ++slot;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) *nslots = s.pcount[1];
    // every site takes the code of its component's representative: the entry
    // of its root (a code, or the name of a root without a slot)
#pragma unroll
    for (int q = 0; q < 16; ++q)
        ent[q] = label_get(ent[q]);
}

// The labelling where no bond can be active (beta = 0): every site is a cluster
// of its own, none needs a slot and no pair leaves the tile.  (The general form
// gives every site on a face a slot: L = 256 at beta = 0 1,205 us a sweep, with
// this 482.)
__device__ __forceinline__ void local_identity(const TileCtx &c, const Rep &R, uint32_t sweep, int tile)
{
    if (c.t == 0) R.nslots[tile] = 0;
    store_flip_bits(c, R, sweep);
    if (!c.valid) return;
    uint32_t packed[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) packed[k] = (uint32_t)(17 * c.t + 2 * k) * 0x10001u + 0x10000u;
    uint4 *dst = reinterpret_cast<uint4 *>(R.L16 + 16 * c.cell);
    dst[0] = make_uint4(packed[0], packed[1], packed[2], packed[3]);
    dst[1] = make_uint4(packed[4], packed[5], packed[6], packed[7]);
    if (c.lx == 0 || c.ly == 0 || c.lz == 0) R.dmask[c.cell] = 0;
}

// Tile-local labelling of one cell's sites from its active-bond groups.
// Writes L16 (the code of each site), F (flip bits), the tile's slots and, for
// face cells, dmask (the union pairs that leave the tile: bit 6 f + k, k the
// pair index of (a, b) in the order (0,1) (0,2) (0,3) (1,2) (1,3) (2,3)).
//
// Slots: the tile-local clusters with a site that a crossing bond may end on
// are numbered 0, 1, .. in each tile, and the crossing unions run on a table
// of four bytes per slot, dense in every tile (about 350 slots of a 8 x 8 x 4
// tile's 4,096 sites).  That table stays in L2; links kept at the roots' sites
// took a DRAM sector for every entry.
// Called by every thread of the block after the staging barrier.
__device__ __forceinline__ void local_core(const TileCtx &c, const Rep &R, const CoreSmem &s, uint32_t A, uint32_t Bg,
                                           uint32_t C, uint32_t sweep, int tile)
{
    const int nt = c.nt;
    const uint32_t out = (c.bx ? 1u : 0u) | (c.by ? 2u : 0u) | (c.bz ? 4u : 0u);  // axes whose backward step leaves
    const int me = s.lab + CELL_BYTES * c.t;  // name of the cell's site 0
    // every site starts under its representative in its up tetrahedron
    uint32_t uptab[4];
    uint32_t reps = 0;  // bit 4 f + v: site is its component's representative
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        uptab[f] = s.lut[up_tet_index(A, Bg, f)];
        reps |= ((uptab[f] >> 8) & 0xFu) << (4 * f);
#pragma unroll
        for (int v = 0; v < 4; ++v)
            label_set(me + 4 * (4 * f + v), me + 16 * f + 4 * (int)((uptab[f] >> (2 * v)) & 3u));
    }
    // the down tetrahedra join every vertex v to the smallest vertex connected
    // to it: pairs with a vertex across a backward tile face are left to the
    // crossing unions, the others are united here
    uint32_t span = 0, leave = 0;  // bit 6 f + k: pair k of tetrahedron f
#pragma unroll
    for (int f = 0; f < 4; ++f) span |= ((s.lut[down_tet_index(C, Bg, f)] >> 16) & 0x3Fu) << (6 * f);
    if (out & 1u) leave |= leaving_pairs(0);
    if (out & 2u) leave |= leaving_pairs(1);
    if (out & 4u) leave |= leaving_pairs(2);
    const uint32_t in = span & ~leave, cross = span & leave;
    __syncthreads();  // labels initialised
    // First pass over all pairs, without finds: each links the larger of its
    // ends' parents under the other if that is a root still (seven pairs of
    // ten), else it is listed, as the pair of that root's new parent and the
    // smaller one.  (All pairs listed and united with full finds took three
    // rounds, whose barriers waited for the longest chains.)
    uint32_t rest[12];
    uint32_t nrest = 0;
    const bool unite = c_unite_bound > 0;
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        int name[4];
#pragma unroll
        for (int v = 0; v < 4; ++v)
            name[v] = s.lab + CELL_BYTES * vertex_local_cell(c, down_mask(f, v)) + 4 * down_bit(f, v);
        int a[3], b[3];
#pragma unroll
        for (int v = 1; v < 4; ++v) {
            // at most one pair (u, v), u < v, spans; none: the same label twice
            int ea = me, eb = me;
#pragma unroll
            for (int u = 0; u < v; ++u)
                if ((in >> (6 * f + pair_index(u, v))) & 1u) {
                    ea = name[u];
                    eb = name[v];
                }
            a[v - 1] = label_get(ea);
            b[v - 1] = label_get(eb);
        }
#pragma unroll
        for (int v = 0; v < 3; ++v) {
            const int lo = min(a[v], b[v]), hi = max(a[v], b[v]);
            int old = label_link_if(unite && lo != hi, hi, lo);
            if (!unite) old = lo;
            const uint32_t r = old != hi ? (uint32_t)lo | ((uint32_t)old << 16) : 0u;
            rest[3 * f + v] = r;
            nrest += r ? 1u : 0u;
        }
    }
    if (nrest) {
        int pos = atomicAdd(s.pcount, (int)nrest);
#pragma unroll
        for (int k = 0; k < 12; ++k)
            if (rest[k]) s.plist[pos++] = rest[k];
    }
    __syncthreads();  // pairs listed
    int ent[16];
    finish_labels(s, nt, me, reps, [&] { return crossing_sites(c); }, (int32_t)(16 * c.cell), R.P + (int64_t)tile * (16 * nt),
                  R.nslots + tile, &R.st->status, ent);
    uint32_t packed[8];
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        uint32_t code[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const uint32_t rv = (uptab[f] >> (2 * v)) & 3u;
            const int e = ent[4 * f + v];
            uint32_t r = e < IS_CODE ? (uint32_t)(e - s.lab) >> 2 : (uint32_t)(e - IS_CODE);
#pragma unroll
            for (int u = 0; u < v; ++u)
                if (rv == (uint32_t)u) r = code[u];
            code[v] = r;
        }
        packed[2 * f] = code[0] | (code[1] << 16);
        packed[2 * f + 1] = code[2] | (code[3] << 16);
    }
    store_flip_bits(c, R, sweep);
    if (!c.valid) return;
    uint4 *dst = reinterpret_cast<uint4 *>(R.L16 + 16 * c.cell);
    dst[0] = make_uint4(packed[0], packed[1], packed[2], packed[3]);
    dst[1] = make_uint4(packed[4], packed[5], packed[6], packed[7]);
    if (c.lx == 0 || c.ly == 0 || c.lz == 0) R.dmask[c.cell] = cross;
}

// ------------------------------------------------------ crossing clusters --
// A root's entry is its cluster's smallest site so far, a link's the slot it
// points at (SLOT_LINK).  The root with the larger site is always hung under
// the other one, so a cluster's root keeps its minimum site index.  The local
// kernel writes every slot in use, so nothing is left over from earlier
// sweeps.
//
// No load of the table takes the read-only path (__ldg), the walks after the
// last union included: that path asks for data nobody writes while the kernel
// exists, and an overlapped kernel exists while the one before it still links
// slots; what overlap_wait makes visible, ordinary loads see.
__device__ __forceinline__ bool slot_linked(uint32_t v) { return (v & SLOT_LINK) != 0; }

// One find step with path splitting: x (entry v, a link) moves to its parent,
// whose entry is returned in v; x's entry is pointed at its grandparent if the
// parent is itself linked.  One dependent load per level.
__device__ __forceinline__ void slot_step(uint32_t *P, uint32_t &x, uint32_t &v)
{
    const uint32_t p = v & ~SLOT_LINK;
    const uint32_t gv = __ldca(P + p);
    if (slot_linked(gv)) __stcg(P + x, gv);
    x = p;
    v = gv;
}

// Union of the crossing clusters of slots a and b.  Both finds walk in
// lockstep (their loads overlap); a root is linked by a compare-and-swap from
// the entry its walk ended on.  Returns false if the bound was hit.
__device__ __forceinline__ bool slot_unite(uint32_t *P, uint32_t a, uint32_t b)
{
    uint32_t va = __ldca(P + a), vb = __ldca(P + b);
#pragma unroll 1
    for (int it = 0; it < (1 << 20); ++it) {
        const bool la = slot_linked(va), lb = slot_linked(vb);
        if (la || lb) {
            if (la) slot_step(P, a, va);
            if (lb) slot_step(P, b, vb);
            continue;
        }
        if (a == b) return true;
        if (va > vb) {  // roots: sites
            uint32_t t = a;
            a = b;
            b = t;
            t = va;
            va = vb;
            vb = t;
        }
        const uint32_t old = atomicCAS(P + b, vb, SLOT_LINK | a);
        if (old == vb) return true;
        vb = old;  // b was linked meanwhile: walk on from its new entry
    }
    return false;
}

// Root site of slot entry v after all unions of the sweep (cached loads).
__device__ __forceinline__ uint32_t slot_root(const uint32_t *P, uint32_t v)
{
#pragma unroll 1
    for (int it = 0; it < (1 << 20) && slot_linked(v); ++it) v = P[v & ~SLOT_LINK];
    return v;
}

// Threads of a slot block.
constexpr int SLOT_BLOCK = 128;

// The flip bits of the clusters of a tile's n slots, 16 to a word: three slots
// per thread at a time, their walks in lockstep.
template <typename FlipBit>
__device__ __forceinline__ void slot_flips(const uint32_t *own, const uint32_t *P, int n, uint16_t *out,
                                           const FlipBit &flip_bit)
{
    const int lane = threadIdx.x & 31;
    for (int k0 = threadIdx.x & ~31; k0 < n; k0 += 3 * SLOT_BLOCK) {
        uint32_t v[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const int k = k0 + j * SLOT_BLOCK + lane;
            v[j] = k < n ? own[k] : 0u;
        }
#pragma unroll 1
        for (int it = 0; it < (1 << 20) && ((v[0] | v[1] | v[2]) & SLOT_LINK); ++it)
#pragma unroll
            for (int j = 0; j < 3; ++j)
                if (slot_linked(v[j])) v[j] = P[v[j] & ~SLOT_LINK];
        uint32_t bit[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) bit[j] = flip_bit(v[j]);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const int k = k0 + j * SLOT_BLOCK + lane;
            const uint32_t word = __ballot_sync(0xffffffffu, bit[j]);
            if ((lane & 15) == 0 && k < n) out[k >> 4] = (uint16_t)(word >> (lane & 16));
        }
    }
}

// Index of the tile of cell (x, y, z) in its lattice.
__device__ __forceinline__ uint32_t tile_of(const Rep &R, const Batch &B, int x, int y, int z)
{
    return (uint32_t)(x >> B.lTX) + (uint32_t)R.ntx * ((uint32_t)(y >> B.lTY) + (uint32_t)R.nty * (uint32_t)(z >> B.lTZ));
}

// Slot of site s of cell (x, y, z), an end of a crossing bond.
__device__ __forceinline__ uint32_t crossing_slot(const Rep &R, const Batch &B, int x, int y, int z, int s)
{
    const uint32_t L = (uint32_t)R.L, nt = (uint32_t)(B.TX * B.TY * B.TZ);  // (N < 2^31)
    const uint32_t code = R.L16[16 * ((uint32_t)x + L * ((uint32_t)y + L * (uint32_t)z)) + (uint32_t)s];
    return tile_of(R, B, x, y, z) * (16 * nt) + (code - (uint32_t)slot_code((int)nt));
}

// Shared-memory bytes of the flip stage: a bit per code.
__host__ __device__ constexpr size_t resolve_smem_bytes(int nt) { return (size_t)slot_code(nt) / 8 + (size_t)nt * 2 + 16; }

// Global index of the cluster root of every site of the calling thread's
// (valid) cell.
__device__ __forceinline__ void resolve_cell(const TileCtx &c, const Rep &R, int tile, int root[16])
{
    const uint4 *src = reinterpret_cast<const uint4 *>(R.L16 + 16 * c.cell);
    const uint4 a0 = src[0], a1 = src[1];
    const uint32_t w[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
    const uint32_t *P = reinterpret_cast<const uint32_t *>(R.P);
    const int base = slot_code(c.nt);
#pragma unroll
    for (int s = 0; s < 16; ++s) {
        const int code = (int)((w[s >> 1] >> (16 * (s & 1))) & 0xFFFFu);
        if (code >= base) {
            root[s] = (int)slot_root(P, P[(int64_t)tile * (16 * c.nt) + (code - base)]);
        } else {
            const int lc = word_cell(code);
            const int rx = c.ox + (lc & (c.TX - 1));
            const int ry = c.oy + ((lc >> c.lTX) & (c.TY - 1));
            const int rz = c.oz + (lc >> (c.lTX + c.lTY));
            root[s] = 16 * (rx + c.L * (ry + c.L * rz)) + (code - 17 * lc);
        }
    }
}

// Writes the 16 flip bits f of every cell to 17 bits a cell of fx.  The 17 words of
// a warp's 32 cells are put together from its lanes' f: three cells reach
// into a word.  Called by every thread of the block.  The flip stage is bound by
// its blocks' latency between barriers: zeroing the words and OR-ing the bits
// in by shared atomics took a barrier more and two lanes contended for a word
// (with the spins' load before the barrier, flip at L = 256: 190 -> 156 us).
__device__ __forceinline__ void place_flip_bits(uint32_t *fx, uint32_t f, int t, int nt)
{
    const int lane = t & 31, n = min(32, nt - (t - lane));  // (tiles are powers of two: n = 32 or nt)
    const int c0 = 32 * lane / 17, o = 32 * lane - 17 * c0;
    const unsigned lanes = lanes_mask(nt);
    const uint32_t a = __shfl_sync(lanes, f, min(c0, n - 1)), b = __shfl_sync(lanes, f, min(c0 + 1, n - 1)),
                   d = __shfl_sync(lanes, f, min(c0 + 2, n - 1));
    if (32 * lane >= 17 * n) return;
    uint32_t word = a >> o;
    if (c0 + 1 < n) word |= b << (17 - o);
    if (c0 + 2 < n && o > 2) word |= d << (34 - o);
    fx[17 * (t >> 5) + lane] = word;
}

// Flip mask of the calling thread's cell (bit s = site 16 c + s flips): each
// site's code indexes a bit array the block shares, the flip bits of the
// tile's sites (17 bits a cell), then those of its slots' clusters.  Called by
// every thread of the block.
__device__ __forceinline__ uint32_t cell_flip_mask(const TileCtx &c, const Rep &R, int tile, int *smem)
{
    uint32_t *fx = reinterpret_cast<uint32_t *>(smem);
    const int words = slot_code(c.nt) >> 5;
    const uint4 *src = reinterpret_cast<const uint4 *>(R.L16 + 16 * c.cell);
    const uint4 a0 = src[0], a1 = src[1];
    const uint32_t w[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
    const uint32_t f = R.F[c.cell];
    const uint16_t *sf = reinterpret_cast<const uint16_t *>(R.sflip) + (int64_t)tile * c.nt;
    if (16 * c.t < R.nslots[tile]) reinterpret_cast<uint16_t *>(fx + words)[c.t] = sf[c.t];
    place_flip_bits(fx, f, c.t, c.nt);
    __syncthreads();
    uint32_t flip = 0;
#pragma unroll
    for (int s = 0; s < 16; ++s) {
        const int code = (int)((w[s >> 1] >> (16 * (s & 1))) & 0xFFFFu);
        flip |= ((fx[code >> 5] >> (code & 31)) & 1u) << s;
    }
    return flip;
}

// ------------------------------------------------------- face-cell grid --
// Cells of a tile with lx == 0, ly == 0 or lz == 0 (the cells that own the
// tetrahedra leaving the tile), enumerated compactly: the lz == 0 plane,
// then for each lz > 0 the row ly == 0 and the column lx == 0.
__host__ __device__ constexpr int face_cells(int TX, int TY, int TZ) { return TX * TY * TZ - (TX - 1) * (TY - 1) * (TZ - 1); }

__device__ __forceinline__ void face_cell_coords(const Batch &B, int i, int &lx, int &ly, int &lz)
{
    const int plane = B.TX * B.TY;
    if (i < plane) {
        lz = 0;
        ly = i >> B.lTX;
        lx = i & (B.TX - 1);
        return;
    }
    const int per = B.TX + B.TY - 1;
    const int j = i - plane;
    lz = 1 + j / per;
    const int k = j - (lz - 1) * per;
    if (k < B.TX) {
        ly = 0;
        lx = k;
    } else {
        ly = k - B.TX + 1;
        lx = 0;
    }
}

}  // namespace pyro
