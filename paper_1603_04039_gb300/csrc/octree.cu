// octree.cu -- Section 4: Morton keys, key sort, error-balance refinement,
// minimal 2:1 face balance, leaves, boundary nodes and face adjacency.
//
// GB300 design.  The paper builds the tree with a sequential queue and
// incremental neighbour lists (Section 4.3).  Here the node set is computed
// as a closure over the set of opened cells, a hash set for all levels:
//   * every cell at level l < max_depth that holds N' > 0 particles with
//     N' h_l^2 >= c^2 opens (the criterion is monotone down the tree, so the
//     criterion tree is exactly this set); with the particles sorted by key
//     that is a look T_l - 1 particles ahead at every cell's first particle,
//     T_l the least count that opens a cell of level l -- one pass over the
//     keys for all levels;
//   * an opened cell at level l+1 forces its parent and the parents of its
//     six same-level face neighbours to open (this is the 2:1 face balance
//     rule: the children of the opened cell need face neighbours no more than
//     one level coarser), one launch per level from the deepest up;
// so O_l = Crit_l U parent(O_{l+1}) U parent(faces(O_{l+1})).  The result is
// the unique minimal balanced refinement, the set the paper's
// deepest-level-first loop produces.  The leaves are the children of opened
// cells that are not opened themselves, ordered by one sort of their anchors.
// The order in which cells enter the set does not show in the result.
//
// Nothing here waits for the host but the number of opened cells (it gives the
// number of leaves) and the number of boundary nodes.  A sort, a scan and two
// host reads per level took 1.18 ms for 1e5 particles at depth 8 (15324
// leaves), 3.16 ms for 1e7 at depth 10 (1.05e6 leaves) and 4.0 ms for 2e7 at
// depth 9 (2.6e5 leaves); now 0.23, 1.37 and 1.49 ms (GB300, whole call).  What
// is left: launches and two host reads for the small tree; the sort (0.58 ms
// of the large one, bound by the ranking of equal digits: see prims.cu), the
// particle maps (0.31 ms) and the keys (0.20).
//
// Batches: several independent problems (beams) on the same cubic domain are
// one tree whose cell keys carry the beam index above the 3l Morton bits of
// level l, so one sort and one closure serve all beams and no neighbour
// relation crosses from one beam to another.
#include <algorithm>
#include <cmath>

#include "fpconv.cuh"
#include "internal.cuh"

namespace apc {

namespace {

constexpr int T = 256;

// beam of particle i from the batch offsets (nb + 1 entries, offs[0] = 0)
__device__ __forceinline__ uint64_t beam_of(const int64_t *offs, int nb, int64_t i) {
    int lo = 0, hi = nb;
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (offs[mid] <= i) lo = mid; else hi = mid;
    }
    return (uint64_t)lo;
}

// The cell coordinate floor((p - lo) 2^21 / (hi - lo)) of depth 21, no
// contraction, clamped into the cube, with bit 31 set for a p outside [lo, hi]
__device__ __noinline__ uint32_t cell_coord_f64(double p, double lo, double hi, double s) {
    const double t = __dmul_rn(__dsub_rn(p, lo), s);
    return f64_floor_clamp_u32(t, (1u << KEY_DEPTH) - 1u) | (f64_in_range(p, lo, hi) ? 0u : 0x80000000u);
}

// The same in integers.  With hi - lo a power of two the product with s is
// exact, so the cell is that of the rounded difference p - lo.  In units of
// 2^-f (lo and hi whole numbers of them) the difference is exact but for the
// bits of a small p below the unit, and it rounds across a cell boundary only
// when it lies within the guard (the widest rounding step) under one; there,
// and where lost bits could matter (a unit above one), cell_coord_f64 decides.
// FP64 runs at two lanes per clock and SM: the subtraction and the product of
// three coordinates held 2e7 keys at 352 us; 201 us now.
struct KeyFix {
    int on, f, sh;      // cell edge 2^sh units
    int64_t lo;
    uint64_t ext, guard;
};
__device__ __forceinline__ uint32_t cell_coord(double p, double lo, double hi, double s, const KeyFix &k) {
    const uint64_t b = (uint64_t)__double_as_longlong(p);
    const int E = (int)(b >> 52 & 0x7FFu);
    const uint64_t m = (b & 0xFFFFFFFFFFFFFull) | (E ? 1ull << 52 : 0ull);
    const int sft = E - 1075 + k.f;
    const uint64_t mag = sft >= 0 ? m << (sft & 63) : (sft > -64 ? m >> (-sft & 63) : 0ull);
    const uint64_t d = (b >> 63 ? 0ull - mag : mag) - (uint64_t)k.lo;
    const uint64_t edge = 1ull << k.sh, frac = d & (edge - 1);
    if (!k.on || sft > 10 || frac - 2 >= edge - 2 - k.guard) return cell_coord_f64(p, lo, hi, s);
    if (d >= k.ext)   // outside (below lo wraps around), or at hi but for bits lost below the unit
        return d > k.ext ? 0x80000000u : cell_coord_f64(p, lo, hi, s);
    const uint32_t q = (uint32_t)(d >> k.sh);   // hi - lo may exceed its rounded value
    return q < (1u << KEY_DEPTH) ? q : (1u << KEY_DEPTH) - 1u;
}

__device__ __forceinline__ uint32_t spread3_10(uint32_t x) {   // 10 bits, two apart
    x = (x | x << 16) & 0x030000FFu;
    x = (x | x << 8) & 0x0300F00Fu;
    x = (x | x << 4) & 0x030C30C3u;
    return (x | x << 2) & 0x09249249u;
}

// Keys at depth L (K: 32 bits while 3 L and the beam bits fit) and the counts
// of every digit the sort will take them by.
template <class K>
__global__ void __launch_bounds__(512) k_keys(const double *__restrict__ x, const double *__restrict__ y,
                                              const double *__restrict__ z, int64_t n, double lo0, double lo1,
                                              double lo2, double hi0, double hi1, double hi2, double s, int shift,
                                              KeyFix fix, const int64_t *__restrict__ offs, int nb, int L,
                                              K *__restrict__ key, RadixDigits dg, uint32_t *__restrict__ hist, unsigned *err) {
    extern __shared__ uint32_t h[];
    for (int i = threadIdx.x; i < dg.passes * RS_BINS; i += blockDim.x) h[i] = 0;
    __syncthreads();
    const double lo[3] = {lo0, lo1, lo2}, hi[3] = {hi0, hi1, hi2};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double p[3] = {__ldg(x + i), __ldg(y + i), __ldg(z + i)};
        uint32_t cc[3], bad = 0u;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const uint32_t q = cell_coord(p[d], lo[d], hi[d], s, fix);
            bad |= q;
            cc[d] = (q & 0x7FFFFFFFu) >> shift;
        }
        if (bad >> 31) atomicOr(err, ERR_DOMAIN);
        const uint64_t beam = nb > 1 ? beam_of(offs, nb, i) << (3 * L) : 0ull;
        K k;
        if (sizeof(K) == 4)   // L <= 10
            k = (K)((uint32_t)beam | spread3_10(cc[0]) << 2 | spread3_10(cc[1]) << 1 | spread3_10(cc[2]));
        else
            k = (K)(beam | morton(cc[0], cc[1], cc[2]));
        key[i] = k;
        rs_count(k, dg, h);
    }
    __syncthreads();
    rs_flush(h, dg, hist);
}

__global__ void k_iota(uint32_t *__restrict__ v, int64_t n) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) v[i] = (uint32_t)i;
}

// ---- the set of opened cells.  A cell of level l is the code
// 1 << (3 l + beam bits) | key: parents and children are shifts by 3, and no
// two levels share a code.  The list keeps the cells in the order they came;
// a slot not written yet reads 0.
struct CellSet {
    uint64_t *table, *list;
    uint32_t mask, cap;
    int shift;          // 64 - log2(table size)
    uint32_t *count;
    unsigned *err;
};

__device__ __forceinline__ uint32_t cell_slot(const CellSet &t, uint64_t code) {
    return (uint32_t)((code * 0x9E3779B97F4A7C15ull) >> t.shift);
}

__device__ __forceinline__ void cell_insert(const CellSet &t, uint64_t code) {
    uint32_t h = cell_slot(t, code);
    for (uint32_t probe = 0; probe <= t.mask && probe < 1024u; ++probe) {   // far past what half a table needs
        uint64_t cur = __ldcg(t.table + h);
        if (cur == 0ull) cur = atomicCAS(reinterpret_cast<unsigned long long *>(t.table + h), 0ull, code);
        if (cur == code) return;
        if (cur == 0ull) {   // new: append it (one counter update per warp)
            const unsigned m = __activemask(), lane = threadIdx.x & 31;
            const int leader = __ffs(m) - 1;
            uint32_t base = 0;
            if ((int)lane == leader) base = atomicAdd(t.count, (uint32_t)__popc(m));
            base = __shfl_sync(m, base, leader);
            const uint32_t pos = base + __popc(m & ((1u << lane) - 1u));
            if (pos < t.cap) t.list[pos] = code;
            else atomicOr(t.err, ERR_CELLS);
            return;
        }
        h = (h + 1) & t.mask;
    }
    atomicOr(t.err, ERR_CELLS);
}

__device__ __forceinline__ bool cell_in(const CellSet &t, uint64_t code) {
    uint32_t h = cell_slot(t, code);
    for (uint32_t probe = 0; probe <= t.mask; ++probe) {
        const uint64_t cur = __ldg(t.table + h);
        if (cur == code) return true;
        if (cur == 0ull) return false;
        h = (h + 1) & t.mask;
    }
    return false;
}

struct Thresholds {
    uint32_t t[KEY_DEPTH];   // particles that open a cell of level l
};

// Error-balance criterion (Section 4.3, k = 2: open iff N' > 0 and N' h^2 >=
// c^2).  Particle i is the first of its cell at every level from the one where
// its key leaves the key before it; such a cell of level l holds T_l particles
// iff particle i + T_l - 1 is still in it.  A cell that does not open has no
// child that does.
template <class K>
__global__ void k_crit(const K *__restrict__ key, int64_t n, int L, int bb, Thresholds th, CellSet set) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint64_t k = key[i];
    int l = 0;
    if (i > 0) {
        const uint64_t x = k ^ (uint64_t)key[i - 1];
        if (x == 0ull) return;
        const int top = (63 - __clzll((long long)x)) / 3;
        l = top >= L ? 0 : L - top;
    }
    // only the deepest cell that opens is entered: the closure opens its ancestors
    uint64_t deepest = 0ull;
    for (; l < L; ++l) {
        const int64_t j = i + th.t[l] - 1;
        const int sh = 3 * (L - l);
        if (j >= n || ((uint64_t)key[j] >> sh) != (k >> sh)) break;
        deepest = 1ull << (3 * l + bb) | k >> sh;
    }
    if (deepest) cell_insert(set, deepest);
}

// Eight threads per opened cell of level lev1: its parent and the parents of
// its six face neighbours inside the cube open too.
__global__ void k_close(CellSet set, int lev1, int bb) {
    const uint32_t cnt = *set.count < set.cap ? *set.count : set.cap;
    const int lead = 3 * lev1 + bb;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < (int64_t)cnt * 8;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int f = (int)(t & 7);
        const uint64_t code = __ldcg(set.list + (t >> 3));
        if (code >> lead != 1ull || f == 7) continue;   // another level's (or not written yet: a lower level's)
        uint64_t nb = code;
        if (f > 0) {
            const int d = (f - 1) >> 1, up = (f - 1) & 1;
            const uint64_t pre = code >> (3 * lev1) << (3 * lev1);   // leading one and beam bits
            uint32_t c[3];
            unmorton(code ^ pre, c[0], c[1], c[2]);
            const uint32_t lim = 1u << lev1;
            if (up ? c[d] + 1 >= lim : c[d] == 0) continue;
            c[d] = up ? c[d] + 1 : c[d] - 1;
            nb = pre | morton(c[0], c[1], c[2]);
        }
        cell_insert(set, nb >> 3);
    }
}

// Leaves in any order: the children of opened cells that are not opened, and
// the roots (one per beam) that are not; anchors (first key at depth L) and
// the digit counts for their sort.
template <class K>
__global__ void __launch_bounds__(512) k_leaf_emit(CellSet set, uint32_t nopen, int nb, int L, int bb,
                                                   K *__restrict__ anchor, uint32_t *__restrict__ count,
                                                   RadixDigits dg, uint32_t *__restrict__ hist) {
    extern __shared__ uint32_t h[];
    for (int i = threadIdx.x; i < dg.passes * RS_BINS; i += blockDim.x) h[i] = 0;
    __syncthreads();
    const int64_t all = (int64_t)nopen * 8 + nb;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < all; t += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t code = t < nb ? (1ull << bb | (uint64_t)t)
                                     : (set.list[(t - nb) >> 3] << 3 | (uint64_t)((t - nb) & 7));
        const int lev = (63 - __clzll((long long)code) - bb) / 3;
        if (lev < L && cell_in(set, code)) continue;
        const K a = (K)((code ^ 1ull << (3 * lev + bb)) << (3 * (L - lev)));
        const unsigned m = __activemask(), lane = threadIdx.x & 31;
        const int leader = __ffs(m) - 1;
        uint32_t base = 0;
        if ((int)lane == leader) base = atomicAdd(count, (uint32_t)__popc(m));
        base = __shfl_sync(m, base, leader);
        anchor[base + __popc(m & ((1u << lane) - 1u))] = a;
        rs_count(a, dg, h);
    }
    __syncthreads();
    rs_flush(h, dg, hist);
}

template <class K>
__device__ __forceinline__ int64_t lower_bound_key(const K *a, int64_t n, uint64_t v) {
    int64_t lo = 0, hi = n;
    while (lo < hi) {
        int64_t mid = (lo + hi) >> 1;
        if ((uint64_t)a[mid] < v) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// index of the leaf whose anchor is the largest one <= v, looked for from leaf
// j outwards in doubling steps (face neighbours are mostly a few leaves away in
// Morton order)
__device__ __forceinline__ int64_t leaf_of(const uint64_t *anchor, int64_t n, uint64_t v, int64_t j) {
    int64_t lo, hi, step = 2;
    if (anchor[j] <= v) {
        lo = j;
        hi = j + 1;
        while (hi < n && anchor[hi] <= v) {
            lo = hi;
            hi += step;
            step *= 2;
        }
        if (hi > n) hi = n;
    } else {
        hi = j;
        lo = j - 1;
        while (lo >= 0 && anchor[lo] > v) {
            hi = lo;
            lo -= step;
            step *= 2;
        }
        if (lo < -1) lo = -1;
    }
    while (hi - lo > 1) {   // anchor[lo] <= v < anchor[hi]
        const int64_t mid = (lo + hi) >> 1;
        if (anchor[mid] <= v) lo = mid; else hi = mid;
    }
    return lo;
}

// is face f (0..5 = -x, +x, ...) of a leaf on the domain boundary?
__device__ __forceinline__ bool on_face(const int4 &q, int f) {
    const int v = (f >> 1) == 0 ? q.x : ((f >> 1) == 1 ? q.y : q.z);
    const int c = v >> (KEY_DEPTH + 1 - q.w);   // cell coordinate at the leaf's level
    return c == ((f & 1) ? (1 << q.w) - 1 : 0);
}

// Leaves in order: level (the leaves tile the key space, so the gap to the
// next anchor is 8^(L - level)), particle range, integer centre, beam, and the
// block's boundary faces per direction.
template <class K>
__global__ void __launch_bounds__(T) k_leaf_geom(const K *__restrict__ sorted, int64_t n, int L, int nb,
                                                 const K *__restrict__ skeys, int64_t npart,
                                                 uint64_t *__restrict__ anchor, int8_t *__restrict__ level,
                                                 int32_t *__restrict__ first, int32_t *__restrict__ count,
                                                 int4 *__restrict__ ic, int32_t *__restrict__ beam,
                                                 uint32_t *__restrict__ bcnt, int nblk) {
    __shared__ int sf[T + 1];
    __shared__ uint32_t sc[6];
    const int64_t j = (int64_t)blockIdx.x * T + threadIdx.x;
    if (threadIdx.x < 6) sc[threadIdx.x] = 0u;
    uint64_t a = 0, nx = 0;
    if (j < n) {
        a = sorted[j];
        nx = j + 1 < n ? (uint64_t)sorted[j + 1] : (uint64_t)nb << (3 * L);
        sf[threadIdx.x] = (int)lower_bound_key(skeys, npart, a);
        if (threadIdx.x == T - 1 || j + 1 == n)
            sf[threadIdx.x + 1] = j + 1 < n ? (int)lower_bound_key(skeys, npart, nx) : (int)npart;
    }
    __syncthreads();
    int4 q = make_int4(0, 0, 0, 0);
    if (j < n) {
        const int lev = L - (63 - __clzll((long long)(nx - a))) / 3;
        anchor[j] = a;
        level[j] = (int8_t)lev;
        first[j] = sf[threadIdx.x];
        count[j] = sf[threadIdx.x + 1] - sf[threadIdx.x];
        beam[j] = (int32_t)(a >> (3 * L));
        uint32_t c[3];
        unmorton((a >> (3 * (L - lev))) & ((1ull << (3 * lev)) - 1ull), c[0], c[1], c[2]);
        const int sh = KEY_DEPTH - lev;
        q = make_int4((int)((2u * c[0] + 1u) << sh), (int)((2u * c[1] + 1u) << sh), (int)((2u * c[2] + 1u) << sh), lev);
        ic[j] = q;
    }
#pragma unroll
    for (int f = 0; f < 6; ++f) {
        const unsigned b = __ballot_sync(0xffffffffu, j < n && on_face(q, f));
        if ((threadIdx.x & 31) == 0 && b) atomicAdd(&sc[f], (uint32_t)__popc(b));
    }
    __syncthreads();
    if (threadIdx.x < 6) bcnt[(int64_t)threadIdx.x * nblk + blockIdx.x] = sc[threadIdx.x];
}

// leaf of key-sorted particle i: the last one whose first is <= i (an empty
// leaf shares its first with the next and is never the last)
__device__ __forceinline__ int leaf_at(const int32_t *first, int lo, int hi, int i) {   // in [lo, hi)
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (first[mid] <= i) lo = mid; else hi = mid;
    }
    return lo;
}

// Leaf and key-sorted position of every particle in the caller's order (read
// by the gather and the deposit, so that neither needs a search or a gather
// through the permutation), a tile of sorted particles per block.  While the
// two arrays fit L2 the 4-byte stores go straight to their random places (tiles
// of PL_SMALL, so that small sets reach all SMs: 15 us for 1e5 particles, 26 in
// tiles of 8192; 187 and 202 for 1e7, 200 with windows).  Larger sets (BUCKET)
// would fetch and write back a 32-byte sector per store: the tile is ordered by
// destination window first and appended to the windows' lists (a permutation
// fills every window exactly), and k_particle_place stores window by window,
// inside L2.  A list entry is one word; as three words in a row it took 402
// instead of 310 us for 2e7 particles, both kernels.  Sets whose three fields
// need more than 64 bits are stored directly.
constexpr int PL_SMALL = 1024, PL_TILE = 8192, PL_T = 1024, PL_WIN = 2048;   // most windows
constexpr int PL_WBITS = 14;                               // particles per window: 128 KB of the two arrays
// A particle of a window's list in one word: its place in the window, its leaf
// and its key-sorted position (w, l and s bits)
struct PackBits {
    int w, l, s;
    __device__ __forceinline__ uint64_t pack(uint32_t p, int leaf, int64_t pos) const {
        return (uint64_t)(p & ((1u << w) - 1u)) << (l + s) | (uint64_t)leaf << s | (uint64_t)pos;
    }
    __device__ __forceinline__ uint32_t low(uint64_t e) const { return (uint32_t)(e >> (l + s)) & ((1u << w) - 1u); }
    __device__ __forceinline__ int32_t leaf(uint64_t e) const { return (int32_t)(e >> s & ((1ull << l) - 1ull)); }
    __device__ __forceinline__ int32_t pos(uint64_t e) const { return (int32_t)(e & ((1ull << s) - 1ull)); }
};
static int bits_of(uint64_t v) {
    int b = 0;
    while (v >> b) ++b;
    return b;
}
template <bool BUCKET>
__global__ void __launch_bounds__(PL_T) k_particle_leaf(const int32_t *__restrict__ first, int n_leaf,
                                                        const uint32_t *__restrict__ perm, int64_t n,
                                                        int32_t *__restrict__ pleaf, int32_t *__restrict__ spos,
                                                        int tile, PackBits pb, uint32_t *__restrict__ cursor,
                                                        uint64_t *__restrict__ bp) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int range[2];
    __shared__ uint32_t wtot[PL_T / 32];
    const int64_t i0 = (int64_t)blockIdx.x * tile;   // BUCKET: tile = PL_TILE
    const int m = (int)(n - i0 < tile ? n - i0 : tile);
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    uint32_t *cnt = reinterpret_cast<uint32_t *>(smem), *gof = cnt + PL_WIN;
    if (tid < 2) range[tid] = leaf_at(first, 0, n_leaf, (int)(tid == 0 ? i0 : i0 + m - 1));
    if (BUCKET)
        for (int q = tid; q < PL_WIN; q += PL_T) cnt[q] = 0u;
    __syncthreads();
    const int ja = range[0], jb = range[1] + 1;
    if (!BUCKET) {
#pragma unroll 4
        for (int t = tid; t < m; t += blockDim.x) {
            const int i = (int)(i0 + t);
            const uint32_t p = __ldcs(perm + i);
            if (p >= n) continue;   // only after a sort that gave up
            pleaf[p] = leaf_at(first, ja, jb, i);
            spos[p] = i;
        }
        return;
    }
    uint64_t *sw = reinterpret_cast<uint64_t *>(gof + PL_WIN);
    uint16_t *win_of = reinterpret_cast<uint16_t *>(sw + PL_TILE);
    const int wbits = pb.w;
    constexpr int PER = PL_TILE / PL_T, WPT = PL_WIN / PL_T;
    uint32_t p[PER], r[PER];
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        const int t = tid + u * PL_T;
        p[u] = t < m ? __ldcs(perm + i0 + t) : 0u;
        if (p[u] >= n) p[u] = 0u;   // only after a sort that gave up
    }
#pragma unroll
    for (int u = 0; u < PER; ++u)
        if (tid + u * PL_T < m) r[u] = atomicAdd(&cnt[p[u] >> wbits], 1u);
    __syncthreads();
    // windows tid * WPT ..: their places in the staged tile and in their lists
    uint32_t v[WPT], sum = 0;
#pragma unroll
    for (int q = 0; q < WPT; ++q) {
        v[q] = cnt[tid * WPT + q];
        sum += v[q];
    }
    uint32_t inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) wtot[w] = inc;
    __syncthreads();
    uint32_t base = inc - sum;
    for (int q = 0; q < w; ++q) base += wtot[q];
#pragma unroll
    for (int q = 0; q < WPT; ++q) {
        const int win = tid * WPT + q;
        cnt[win] = base;
        gof[win] = v[q] ? ((uint32_t)win << wbits) + atomicAdd(cursor + win, v[q]) - base : 0u;
        base += v[q];
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        const int t = tid + u * PL_T;
        if (t < m) {
            const uint32_t at = cnt[p[u] >> wbits] + r[u];
            sw[at] = pb.pack(p[u], leaf_at(first, ja, jb, (int)(i0 + t)), i0 + t);
            win_of[at] = (uint16_t)(p[u] >> wbits);
        }
    }
    __syncthreads();
    for (int t = tid; t < m; t += PL_T) {
        const uint32_t dst = gof[win_of[t]] + (uint32_t)t;
        if (dst < n) bp[dst] = sw[t];   // else only after a sort that gave up
    }
}

// A window's list into the two arrays, ordered in shared memory (WBITS = 14)
__global__ void __launch_bounds__(1024) k_particle_place(const uint64_t *__restrict__ bp, int64_t n, PackBits pb,
                                                         int32_t *__restrict__ pleaf, int32_t *__restrict__ spos) {
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int W = 1 << PL_WBITS;
    int32_t *sl = reinterpret_cast<int32_t *>(smem), *ss = sl + W;
    const int64_t p0 = (int64_t)blockIdx.x << PL_WBITS;
    const int m = (int)(n - p0 < W ? n - p0 : W);
#pragma unroll 4
    for (int t = threadIdx.x; t < m; t += 1024) {
        const uint64_t e = __ldcs(bp + p0 + t);
        const uint32_t at = pb.low(e);   // pb.w = PL_WBITS
        sl[at] = pb.leaf(e);
        ss[at] = pb.pos(e);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < m; t += 1024) {
        pleaf[p0 + t] = sl[t];
        spos[p0 + t] = ss[t];
    }
}

// The same for more particles than PL_WIN such windows hold: larger windows,
// the stores to random places of a window that stays in L2
__global__ void __launch_bounds__(T) k_particle_place_l2(const uint64_t *__restrict__ bp, int64_t n, PackBits pb,
                                                         int32_t *__restrict__ pleaf, int32_t *__restrict__ spos) {
    const int64_t i = (int64_t)blockIdx.x * T + threadIdx.x;
    if (i >= n) return;
    const uint64_t e = __ldcs(bp + i);
    const int64_t p = (i >> pb.w << pb.w) + pb.low(e);   // a window's list fills its place exactly
    if (p >= n) return;   // only after a sort that gave up
    pleaf[p] = pb.leaf(e);
    spos[p] = pb.pos(e);
}

// Boundary nodes, ordered by (face, owner): the blocks' counts scanned face
// by face, the leaves' order inside a block.  Also the face's adjacency.
__global__ void __launch_bounds__(T) k_boundary(const uint32_t *__restrict__ bcnt, const uint32_t *__restrict__ bpos,
                                                int nblk, int64_t n, int4 *__restrict__ ic,
                                                int32_t *__restrict__ owner, int8_t *__restrict__ face,
                                                int32_t *__restrict__ adj) {
    __shared__ uint32_t wc[T / 32];
    const int64_t j = (int64_t)blockIdx.x * T + threadIdx.x;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int4 q = j < n ? ic[j] : make_int4(0, 0, 0, 0);
    for (int f = 0; f < 6; ++f) {
        if (bcnt[(int64_t)f * nblk + blockIdx.x] == 0u) continue;   // the same for the whole block
        const bool on = j < n && on_face(q, f);
        const unsigned m = __ballot_sync(0xffffffffu, on);
        if (lane == 0) wc[w] = (uint32_t)__popc(m);
        __syncthreads();
        if (on) {
            uint32_t b = bpos[(int64_t)f * nblk + blockIdx.x] + __popc(m & ((1u << lane) - 1u));
            for (int v = 0; v < w; ++v) b += wc[v];
            int4 g = q;
            const int v = (f & 1) ? (1 << (KEY_DEPTH + 1)) : 0;
            if ((f >> 1) == 0) g.x = v; else if ((f >> 1) == 1) g.y = v; else g.z = v;
            ic[n + b] = g;
            owner[b] = (int32_t)j;
            face[b] = (int8_t)f;
            *reinterpret_cast<int4 *>(adj + j * 24 + f * 4) = make_int4((int)(n + b), -1, -1, -1);
        }
        __syncthreads();
    }
}

// Face adjacency (Section 4.3): per face of a leaf, the face neighbour when it
// is a leaf, else its 4 children touching the face (leaves by 2:1 balance),
// or the boundary node of that face (left in the face's slots by k_boundary).
// Eight lanes per leaf, one per face; the leaf's neighbours are packed to the
// front of its 24 slots, -1 after them.
__global__ void __launch_bounds__(T) k_adjacency(const uint64_t *__restrict__ anchor,
                                                 const int8_t *__restrict__ level, int64_t n, int L, int32_t *adj,
                                                 unsigned *err) {
    const int64_t j = ((int64_t)blockIdx.x * T + threadIdx.x) >> 3;
    const int f = threadIdx.x & 7, lane = threadIdx.x & 31;
    int kid[4] = {-1, -1, -1, -1}, cnt = 0;
    if (j < n && f < 6) {
        const int lev = level[j];
        const uint64_t aj = anchor[j], pre = (aj >> (3 * L)) << (3 * L);   // beam index bits
        uint32_t c[3];
        unmorton((aj ^ pre) >> (3 * (L - lev)), c[0], c[1], c[2]);
        const int d = f >> 1;
        const uint32_t cd = d == 0 ? c[0] : (d == 1 ? c[1] : c[2]);
        if (cd == ((f & 1) ? (1u << lev) - 1u : 0u)) {   // domain boundary
            kid[0] = adj[j * 24 + f * 4];
            cnt = 1;
        } else {
            const uint32_t nd = (f & 1) ? cd + 1 : cd - 1;
            const uint32_t x = d == 0 ? nd : c[0], y = d == 1 ? nd : c[1], z = d == 2 ? nd : c[2];
            const uint64_t a = pre | (morton(x, y, z) << (3 * (L - lev)));
            const int64_t k = leaf_of(anchor, n, a, j);
            if (k < 0) {
                atomicOr(err, ERR_BALANCE);
            } else if (level[k] <= lev) {
                kid[0] = (int)k;
                cnt = 1;
            } else {
                const int want = (f & 1) ? 0 : 1;
                cnt = 4;
                int64_t from = k;
#pragma unroll
                for (int q = 0; q < 4; ++q) {   // the four children on the face, in Morton order
                    const int o = d == 0 ? (want << 2 | q)
                                         : (d == 1 ? ((q >> 1) << 2 | want << 1 | (q & 1)) : (q << 1 | want));
                    const uint64_t ac = a | (uint64_t)o << (3 * (L - lev - 1));
                    const int64_t kk = leaf_of(anchor, n, ac, from);
                    if (kk < 0 || anchor[kk] != ac || level[kk] != lev + 1) {
                        atomicOr(err, ERR_BALANCE);
                        break;
                    }
                    kid[q] = (int)kk;
                    from = kk;
                }
            }
        }
    }
    // places of the faces' neighbours: a prefix sum over the leaf's lanes
    int inc = cnt;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, inc, o, 8);
        if ((lane & 7) >= o) inc += t;
    }
    const int tot = __shfl_sync(0xffffffffu, inc, 7, 8);
    __syncwarp();   // every boundary entry is read
    if (j >= n) return;
    int32_t *out = adj + j * 24;
    const int at = inc - cnt;
    if (cnt > 0) out[at] = kid[0];
    if (cnt == 4) {
        out[at + 1] = kid[1];
        out[at + 2] = kid[2];
        out[at + 3] = kid[3];
    }
    for (int t = tot + f; t < 24; t += 8) out[t] = -1;
}

// Different leaves among 32 particles side by side in the caller's order, summed
// over SPREAD_N such groups spread evenly over the set, a warp each (read by the
// choice of the gather's form)
constexpr int SPREAD_N = 128, SPREAD_MOST = 30, SPREAD_BLOCKS = SPREAD_N / (T / 32);
__device__ __forceinline__ void leaf_spread(const int32_t *pleaf, int64_t n, int group, unsigned *out) {
    const int lane = threadIdx.x & 31;
    const int32_t leaf = pleaf[(n - 32) * group / (SPREAD_N - 1) + lane];
    const unsigned peers = __match_any_sync(0xffffffffu, leaf);
    const unsigned firsts = __ballot_sync(0xffffffffu, lane == __ffs(peers) - 1);
    if (lane == 0) atomicAdd(out, (unsigned)__popc(firsts));
}

// Node ranges of every beam: interior nodes [r[b], r[b+1]) (the leaves are
// beam-sorted) and, per face f, boundary nodes [r[(1+f)(nb+1)+b], ...+1) (the
// boundary nodes are face-major, leaf-ordered within a face).
__global__ void k_beam_ranges(const int32_t *__restrict__ beam, int64_t n, int nb, const uint32_t *__restrict__ bpos,
                              int nblk, const uint32_t *__restrict__ nbnd, const int32_t *__restrict__ owner,
                              int64_t *__restrict__ r, int own, const int32_t *__restrict__ pleaf, int64_t npart,
                              unsigned *__restrict__ spread) {
    if ((int)blockIdx.x >= own) {   // blocks past those the ranges take
        leaf_spread(pleaf, npart, (blockIdx.x - own) * (T / 32) + (threadIdx.x >> 5), spread);
        return;
    }
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b > nb) return;
    int64_t lo = b == nb ? n : 0, hi = b == 0 ? 0 : n;   // the first and the last bound need no search
    while (lo < hi) {
        int64_t mid = (lo + hi) >> 1;
        if (beam[mid] < b) lo = mid + 1; else hi = mid;
    }
    r[b] = lo;
    for (int f = 0; f < 6; ++f) {   // the face's owners ascend
        int64_t p = bpos[(int64_t)f * nblk], e = f < 5 ? bpos[(int64_t)(f + 1) * nblk] : *nbnd;
        if (b == 0) e = p;
        if (b == nb) p = e;
        while (p < e) {
            const int64_t mid = (p + e) >> 1;
            if (owner[mid] < lo) p = mid + 1; else e = mid;
        }
        r[(int64_t)(1 + f) * (nb + 1) + b] = n + p;
    }
}

// beam index of every node (boundary nodes take their owner leaf's)
__global__ void k_node_beam(const int32_t *__restrict__ leaf_beam, const int32_t *__restrict__ owner, int64_t n,
                            int64_t nt, int32_t *__restrict__ out) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nt) return;
    out[i] = i < n ? leaf_beam[i] : leaf_beam[owner[i - n]];
}

}  // namespace

apcloud_status node_beams(apcloud_ctx *c, int32_t *out) {
    APC_LAUNCH(c, K_COPY, div_up(c->n_tot, T), T, 0, k_node_beam, ptr<int32_t>(c->leaf_beam),
               ptr<int32_t>(c->bowner), (int64_t)c->n_int, (int64_t)c->n_tot, out);
    return cuda_check(c, cudaGetLastError(), "node_beams");
}

namespace {

// Most opened cells the criterion alone can give: at level l no more than
// there are cells, nor than the particles fill with T_l each.
int64_t crit_bound(const Thresholds &th, int L, int64_t n, int nb) {
    double s = 0.0;
    for (int l = 0; l < L; ++l) {
        const double cells = std::ldexp((double)nb, 3 * l), full = (double)n / th.t[l];
        s += cells < full ? cells : full;
    }
    return (int64_t)s + nb;
}

constexpr int64_t CELLS_FIRST = 1ll << 27;

// units and guard of the integer keys; off where the domain does not allow them
KeyFix key_fix(const apcloud_params &P) {
    KeyFix k{};
    int e = 0;
    const double ext = P.hi[0] - P.lo[0];
    if (std::frexp(ext, &e) != 0.5) return k;   // ext = 2^(e - 1)
    double top = 0.0;
    for (int d = 0; d < 3; ++d) top = std::max(top, std::max(std::fabs(P.lo[d]), std::fabs(P.hi[d])));
    int et = 0;
    std::frexp(top, &et);                       // top < 2^et
    k.f = 62 - et;
    k.sh = k.f + e - 1 - KEY_DEPTH;
    const int g = k.f + e - 1 - 52;             // the rounding step of differences up to ext, in units
    // one lo for all axes (the kernel's units start there), whole numbers of units
    if (P.lo[0] != P.lo[1] || P.lo[0] != P.lo[2] || k.sh < 16 || k.sh > 60 || g > k.sh - 4 || k.f > 1000 ||
        k.f < -900)
        return k;
    const double lo = std::ldexp(P.lo[0], k.f), hi = std::ldexp(P.hi[0], k.f);
    if (lo != std::nearbyint(lo) || hi != std::nearbyint(hi) || std::fabs(lo) > 4.7e18 || std::fabs(hi) > 4.7e18)
        return k;
    k.lo = (int64_t)lo;
    k.ext = (uint64_t)((int64_t)hi - (int64_t)lo);
    k.guard = (g > 0 ? 1ull << g : 1ull) + 2;
    k.on = 1;
    return k;
}

// Bytes of the two arrays past which their random stores go window by window:
// 1e7 particles (80 MB, inside L2) take 0.19 ms straight and 0.20 ms in windows,
// 2e7 (160 MB) 1.03 ms straight and 0.31 ms in windows ordered in shared memory
constexpr int64_t PL_DIRECT_BYTES = 100ll << 20;

template <class K>
apcloud_status build_tree(apcloud_ctx *c, int64_t n, int nb, int bb) {
    const int L = c->L;
    unsigned *derr = ptr<unsigned>(c->derr);
    uint32_t *small = ptr<uint32_t>(c->dsmall);
    const int64_t nn = n > 0 ? n : 1;
    K *k0 = ensure<K>(c, c->key[0], nn), *k1 = ensure<K>(c, c->key[1], nn);
    uint32_t *v0 = ensure<uint32_t>(c, c->val[0], nn), *v1 = ensure<uint32_t>(c, c->val[1], nn);
    if (!k0 || !k1 || !v0 || !v1) return APCLOUD_E_NOMEM;
    const double ext = c->P.hi[0] - c->P.lo[0];
    const double s = ldexp(1.0, KEY_DEPTH) / ext;
    // K1 keys at depth L, K2 sort on the 3L key bits
    const RadixDigits dg = radix_digits(3 * L + bb);
    APC_TRY(clear_radix_counts(c, dg));
    const size_t hsm = (size_t)dg.passes * RS_BINS * sizeof(uint32_t);
    APC_LAUNCH(c, K_KEYS, std::min(div_up(n, 512), 608), 512, hsm, k_keys<K>, c->px, c->py, c->pz, n, c->P.lo[0],
               c->P.lo[1], c->P.lo[2], c->P.hi[0], c->P.hi[1], c->P.hi[2], s, KEY_DEPTH - L, key_fix(c->P),
               (const int64_t *)ptr<int64_t>(c->beam_off), nb, L, k0, dg, radix_counts(c), derr);
    account(c, K_KEYS, (24.0 + sizeof(K)) * n, 9.0 * n);   // positions in, keys out
    c->kbuf = 0;
    if (n > 0 && dg.passes > 0) APC_TRY(radix_sort_counted<K>(c, k0, v0, k1, v1, n, dg, &c->kbuf));
    else APC_LAUNCH(c, K_SORT, div_up(n, T), T, 0, k_iota, v0, n);   // depth 0, one beam: nothing to sort
    const K *skeys = c->kbuf ? k1 : k0;

    // opened cells: criterion, then the balance closure from the deepest level up
    Thresholds th{};
    const double c2 = c->P.c_refine * c->P.c_refine;
    for (int l = 0; l < L; ++l) {
        const double h = ldexp(ext, -l), h2 = h * h;
        // at most 4e9, more than there are particles: past 2^53 a step of one changes nothing
        double t = std::fmin(std::ceil(c2 / h2), 4e9);
        if (!(t >= 1.0)) t = 1.0;
        while (t > 1.0 && (t - 1.0) * h2 >= c2) t -= 1.0;
        while (t < 4e9 && t * h2 < c2) t += 1.0;
        th.t[l] = (uint32_t)t;
    }
    CellSet set{};
    uint32_t nopen = 0;
    // the bound counts particles level by level, whatever cells they share: a first
    // table of at most CELLS_FIRST (1.6 GB), larger ones where the cells outgrow it
    int64_t want = std::max<int64_t>(std::min(2 * crit_bound(th, L, n, nb), CELLS_FIRST), 2048);
    for (;;) {
        int lg = 11;
        while ((1ll << lg) < want) ++lg;
        const int64_t size = 1ll << lg;
        if (lg > 31) return fail(c, APCLOUD_E_NOMEM, "too many cells");
        uint64_t *mem = ensure<uint64_t>(c, c->opened, size + size / 2);
        if (!mem) return APCLOUD_E_NOMEM;
        set = CellSet{mem, mem + size, (uint32_t)(size - 1), (uint32_t)(size / 2), 64 - lg, derr + 3, derr};
        APC_CUDA(c, cudaMemsetAsync(mem, 0, sizeof(uint64_t) * (size + size / 2), c->s));
        if (n > 0 && L > 0) {
            APC_LAUNCH(c, K_TREE, div_up(n, T), T, 0, k_crit<K>, skeys, n, L, bb, th, set);
            const int grid = (int)std::min<int64_t>(div_up(size / 2 * 8, T), 608);
            for (int l1 = L - 1; l1 >= 1; --l1) APC_LAUNCH(c, K_TREE, grid, T, 0, k_close, set, l1, bb);
        }
        unsigned e[4];
        APC_TRY(read_back(c, e, derr, sizeof e));
        nopen = e[3];
        if (!(e[0] & ERR_CELLS)) break;
        // the balance opened more than the table holds: again with a larger one
        want = size * 4;
        const unsigned keep[4] = {e[0] & ~ERR_CELLS, e[1], e[2], 0u};
        APC_CUDA(c, cudaMemcpyAsync(derr, keep, sizeof keep, cudaMemcpyHostToDevice, c->s));
    }
    APC_CUDA(c, cudaMemsetAsync(derr + 3, 0, sizeof(unsigned), c->s));

    // leaves: every opened cell replaces one by eight
    const int64_t nleaf = nb + 7 * (int64_t)nopen;
    K *lk0 = ensure<K>(c, c->cand[0], nleaf), *lk1 = ensure<K>(c, c->cand[1], nleaf);
    uint32_t *lv0 = ensure<uint32_t>(c, c->cval[0], nleaf), *lv1 = ensure<uint32_t>(c, c->cval[1], nleaf);
    uint64_t *la = ensure<uint64_t>(c, c->leaf_anchor, nleaf);
    int8_t *ll = ensure<int8_t>(c, c->leaf_level, nleaf);
    int32_t *lb = ensure<int32_t>(c, c->leaf_beam, nleaf);
    int32_t *lf = ensure<int32_t>(c, c->leaf_first, nleaf);
    int32_t *lc = ensure<int32_t>(c, c->leaf_count, nleaf);
    const int nblk = div_up(nleaf, T);
    uint32_t *bcnt = ensure<uint32_t>(c, c->bidx, 12 * (int64_t)nblk);   // counts, then their scan
    // node coordinates and boundary records: at most 6 boundary nodes per leaf
    int4 *ic = ensure<int4>(c, c->node_ic, 7 * nleaf);
    int32_t *bo = ensure<int32_t>(c, c->bowner, 6 * nleaf);
    int8_t *bf = ensure<int8_t>(c, c->bface, 6 * nleaf);
    int32_t *adj = ensure<int32_t>(c, c->adj, 24 * nleaf);
    int32_t *pl = ensure<int32_t>(c, c->pleaf, nn), *sp = ensure<int32_t>(c, c->spos, nn);
    int64_t *rng = ensure<int64_t>(c, c->beam_rng, 7 * (nb + 1));
    if (!lk0 || !lk1 || !lv0 || !lv1 || !la || !ll || !lf || !lc || !bcnt || !lb || !ic || !bo || !bf || !adj || !pl ||
        !sp || !rng)
        return APCLOUD_E_NOMEM;
    APC_TRY(clear_radix_counts(c, dg));
    APC_LAUNCH(c, K_TREE, std::min(div_up(nleaf + nopen, 512), 608), 512, hsm, k_leaf_emit<K>, set, nopen, nb, L, bb,
               lk0, derr + 3, dg, radix_counts(c));
    int wl = 0;
    if (dg.passes > 0) APC_TRY(radix_sort_counted<K>(c, lk0, lv0, lk1, lv1, nleaf, dg, &wl));
    c->n_int = (int)nleaf;
    APC_LAUNCH(c, K_TREE, nblk, T, 0, k_leaf_geom<K>, (const K *)(wl ? lk1 : lk0), nleaf, L, nb, skeys, n, la, ll, lf,
               lc, ic, lb, bcnt, nblk);
    const uint32_t *perm = ptr<uint32_t>(c->val[c->kbuf]);
    if (n > 0) {
        int wbits = PL_WBITS;
        while ((n - 1) >> wbits >= PL_WIN) ++wbits;
        const PackBits pb{wbits, bits_of((uint64_t)nleaf - 1), bits_of((uint64_t)n - 1)};
        if (8 * n <= PL_DIRECT_BYTES || pb.w + pb.l + pb.s > 64) {
            APC_LAUNCH(c, K_TREE, div_up(n, PL_SMALL), PL_SMALL / 4, 0, k_particle_leaf<false>, (const int32_t *)lf,
                       (int)nleaf, perm, n, pl, sp, PL_SMALL, pb, (uint32_t *)nullptr, (uint64_t *)nullptr);
        } else {
            uint64_t *bp = ensure<uint64_t>(c, c->bkt, n + PL_WIN);
            if (!bp) return APCLOUD_E_NOMEM;
            uint32_t *cursor = reinterpret_cast<uint32_t *>(bp + n);
            const int smem = 2 * PL_WIN * 4 + PL_TILE * 10, wsm = 8 << PL_WBITS;
            APC_CUDA(c, cudaMemsetAsync(cursor, 0, PL_WIN * sizeof(uint32_t), c->s));
            APC_CUDA(c, cudaFuncSetAttribute(k_particle_leaf<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
            APC_CUDA(c, cudaFuncSetAttribute(k_particle_place, cudaFuncAttributeMaxDynamicSharedMemorySize, wsm));
            APC_LAUNCH(c, K_TREE, div_up(n, PL_TILE), PL_T, smem, k_particle_leaf<true>, (const int32_t *)lf,
                       (int)nleaf, perm, n, pl, sp, PL_TILE, pb, cursor, bp);
            if (wbits == PL_WBITS)
                APC_LAUNCH(c, K_TREE, div_up(n, 1 << PL_WBITS), 1024, wsm, k_particle_place, (const uint64_t *)bp, n, pb,
                           pl, sp);
            else
                APC_LAUNCH(c, K_TREE, div_up(n, T), T, 0, k_particle_place_l2, (const uint64_t *)bp, n, pb, pl, sp);
        }
    }
    uint32_t *bpos = bcnt + 6 * (int64_t)nblk;
    APC_TRY(scan_u32(c, bcnt, bpos, 6 * (int64_t)nblk, small + 4));
    APC_LAUNCH(c, K_TREE, nblk, T, 0, k_boundary, (const uint32_t *)bcnt, (const uint32_t *)bpos, nblk, nleaf, ic, bo,
               bf, adj);
    APC_LAUNCH(c, K_ADJ, div_up(8 * nleaf, T), T, 0, k_adjacency, la, ll, nleaf, L, adj, derr);
    const int rblk = div_up(nb + 1, T);
    const bool sample = nleaf >= STAGED_LEAVES && n >= 32;
    APC_LAUNCH(c, K_TREE, rblk + (sample ? SPREAD_BLOCKS : 0), T, 0, k_beam_ranges, lb, nleaf, nb,
               (const uint32_t *)bpos, nblk, (const uint32_t *)(small + 4), (const int32_t *)bo, rng, rblk,
               (const int32_t *)pl, n, derr + 1);
    APC_CUDA(c, cudaGetLastError());
    // the boundary count, the particles' spread and the error word in one read
    APC_CUDA(c, cudaMemcpyAsync(derr + 3, small + 4, sizeof(uint32_t), cudaMemcpyDeviceToDevice, c->s));
    unsigned e[4];
    APC_TRY(read_back(c, e, derr, sizeof e));
    c->n_bnd = (int)e[3];
    c->scattered = e[1] >= SPREAD_MOST * SPREAD_N;
    c->n_tot = c->n_int + c->n_bnd;
    return device_errors(c, e[0]);
}

}  // namespace

apcloud_status build_octree(apcloud_ctx *c, const double *x, const double *y, const double *z, int64_t n,
                            const int64_t *h_offsets, int nb) {
    const int L = c->P.max_depth;
    int bb = 0;  // bits of the beam index above the tree bits
    while ((1 << bb) < nb) ++bb;
    if (3 * L + bb > 63) return fail(c, APCLOUD_E_INVALID, "%d beams need %d key bits above depth %d", nb, bb, L);
    c->L = L;
    c->N = n;
    c->px = x; c->py = y; c->pz = z;
    c->nbeams = nb;
    c->beam_bits = bb;
    c->h_beam_off.assign(h_offsets, h_offsets + nb + 1);
    int64_t *doff = ensure<int64_t>(c, c->beam_off, nb + 1);
    if (!doff) return APCLOUD_E_NOMEM;
    APC_CUDA(c, cudaMemcpyAsync(doff, h_offsets, sizeof(int64_t) * (nb + 1), cudaMemcpyHostToDevice, c->s));
    APC_CUDA(c, cudaMemsetAsync(c->derr.p, 0, 4 * sizeof(unsigned), c->s));
    return 3 * L + bb <= 32 ? build_tree<uint32_t>(c, n, nb, bb) : build_tree<uint64_t>(c, n, nb, bb);
}

}  // namespace apc
