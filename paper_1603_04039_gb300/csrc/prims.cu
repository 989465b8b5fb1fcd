// prims.cu -- device-wide exclusive scan and stable LSD radix sort.
//
// The tree construction of Section 4 sorts particles by Morton key; these are
// the primitives it (and the node ordering) is built from.  Both are written
// for determinism: the scan is a fixed two-phase tree (integer sums, exact in
// any order), the sort is stable.
#include <algorithm>

#include "internal.cuh"

namespace apc {

namespace {

constexpr int SCAN_T = 256;
constexpr int SCAN_I = 8;
constexpr int SCAN_TILE = SCAN_T * SCAN_I;

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// exclusive block scan of one value per thread; returns the block total in *total
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t *sh, uint32_t *total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    uint32_t inc = warp_incl_scan(v);
    if (lane == 31) sh[wid] = inc;
    __syncthreads();
    if (wid == 0) {
        uint32_t w = (lane < nw) ? sh[lane] : 0u;
        uint32_t wi = warp_incl_scan(w);
        if (lane < nw) sh[lane] = wi - w;
        if (lane == nw - 1) sh[32] = wi;
    }
    __syncthreads();
    uint32_t r = inc - v + sh[wid];
    *total = sh[32];
    __syncthreads();
    return r;
}

__global__ void k_scan_reduce(const uint32_t *__restrict__ in, int64_t n, uint32_t *__restrict__ blk) {
    __shared__ uint32_t sh[33];
    int64_t base = (int64_t)blockIdx.x * SCAN_TILE;
    uint32_t s = 0;
#pragma unroll
    for (int i = 0; i < SCAN_I; ++i) {
        int64_t idx = base + (int64_t)i * SCAN_T + threadIdx.x;
        if (idx < n) s += in[idx];
    }
    uint32_t tot;
    block_excl_scan(s, sh, &tot);
    if (threadIdx.x == 0) blk[blockIdx.x] = tot;
}

// Block b scans its tile and adds the sum of the block totals before it (it
// sums blk[0 .. b) itself, so no pass scans the block totals); the last
// block writes the grand total.  blk == null: a single block.
__global__ void k_scan_down(const uint32_t *__restrict__ in, uint32_t *__restrict__ out, int64_t n,
                            const uint32_t *__restrict__ blk, uint32_t *__restrict__ d_total) {
    __shared__ uint32_t sh[33];
    uint32_t pre = 0;
    if (blk) {
        uint32_t ps = 0;
        for (int i = threadIdx.x; i < (int)blockIdx.x; i += blockDim.x) ps += blk[i];
        block_excl_scan(ps, sh, &pre);
    }
    int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_I;
    uint32_t v[SCAN_I];
    uint32_t s = 0;
#pragma unroll
    for (int i = 0; i < SCAN_I; ++i) {
        int64_t idx = base + i;
        v[i] = (idx < n) ? in[idx] : 0u;
        s += v[i];
    }
    uint32_t tot;
    uint32_t e = block_excl_scan(s, sh, &tot) + pre;
    if (d_total && threadIdx.x == 0 && blockIdx.x == gridDim.x - 1) *d_total = pre + tot;
#pragma unroll
    for (int i = 0; i < SCAN_I; ++i) {
        int64_t idx = base + i;
        if (idx < n) out[idx] = e;
        e += v[i];
    }
}

// ---------------------------------------------------------------- radix sort
// Stable LSD sort of (key, value) pairs, one kernel per digit after one pass
// that counts every digit at once (the counts of a digit do not depend on the
// order of the keys).  A block takes the next tile of the input, orders it by
// digit in shared memory and learns where each of its digits' runs goes from
// the tiles before it by decoupled look-back (Merrill and Garland, "Single-
// pass parallel prefix scan with decoupled look-back", 2016; Adinets and
// Merrill, "Onesweep", 2022): it publishes its own counts at once, adds up its
// predecessors' until it meets one that already knows its inclusive sum, and
// publishes its own.  Tiles are handed out by a counter, so the tiles a block
// waits for are always running.
//
// Against a histogram, a scan and a scatter kernel per digit (keys read twice,
// 256 x tiles counts written, scanned and read): 24 instead of 32 bytes per
// pair and digit, 16 with 32-bit keys, digits of up to 9 bits instead of 8
// and P + 2 launches instead of 4 P.
//
// What bounds it is the ranking of equal digits, not the stores: at 2e7 pairs of
// 32-bit keys the two passes over low, evenly spread digits take 207 and 200 us at
// 13 and 18% of the DRAM rate, a warp waiting 13 of the 25 cycles between two
// instructions for match.any and the counters in shared memory; the pass over the
// top digit, of few values, takes 116 us (31%).
constexpr int RS_T = 512;         // threads per block
// pairs per thread: 12 are the faster for many tiles, 8 for a few (two blocks
// per SM either way).  2e7 / 1e5 pairs, all passes: 585 / 84 us at 12, 647 / 67
// at 8; one block per SM (no register bound) 800 us.
constexpr int RS_I_FEW = 8, RS_I_MANY = 12;
constexpr int64_t RS_MANY = 4 << 20;
constexpr int RS_W = RS_T / 32;
constexpr int RS_LOOK = 8;        // predecessors polled at once
static_assert(RS_BINS == RS_T, "one digit per thread");
constexpr unsigned RS_SPIN = 1u << 22;   // polls of one predecessor before the sort is given up

// status word of (tile, digit): the pass's number and the kind of sum above
// the value; a number is never used twice with the same words
__device__ __forceinline__ uint64_t rs_word(uint32_t epoch, uint32_t inclusive, uint32_t v) {
    return (uint64_t)(epoch << 1 | inclusive) << 32 | v;
}
__device__ __forceinline__ void rs_put(uint64_t *p, uint64_t w) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}
__device__ __forceinline__ uint64_t rs_get(const uint64_t *p) {
    uint64_t w;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
    return w;
}

// exclusive sum over the block of one value per thread
__device__ __forceinline__ uint32_t rs_block_excl(uint32_t v, uint32_t *wtot) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t inc = warp_incl_scan(v);
    if (lane == 31) wtot[w] = inc;
    __syncthreads();
    uint32_t base = 0;
#pragma unroll
    for (int q = 0; q < RS_W; ++q)
        if (q < w) base += wtot[q];
    __syncthreads();
    return base + inc - v;
}

// every digit's counts, [pass][RS_BINS]
template <class K>
__global__ void __launch_bounds__(RS_T) k_rs_hist(const K *__restrict__ keys, int64_t n, RadixDigits dg,
                                                  uint32_t *__restrict__ hist) {
    __shared__ uint32_t h[RS_MAX_PASS * RS_BINS];
    for (int i = threadIdx.x; i < dg.passes * RS_BINS; i += RS_T) h[i] = 0;
    __syncthreads();
    for (int64_t i = (int64_t)blockIdx.x * RS_T + threadIdx.x; i < n; i += (int64_t)gridDim.x * RS_T)
        rs_count(keys[i], dg, h);
    __syncthreads();
    rs_flush(h, dg, hist);
}

template <class K, int RS_I>
struct RsShared {
    K sk[RS_T * RS_I];
    uint32_t sv[RS_T * RS_I];
    uint16_t cnt[RS_W][RS_BINS];
    uint32_t loc[RS_BINS], gof[RS_BINS], wtot[RS_W];
    uint32_t tile;
};

// One digit.  Warp w of the block owns the w-th part of the tile and walks it
// 32 pairs at a time in index order; equal digits inside a step are
// ranked by lane.  IOTA: the values are the pairs' positions.
template <class K, bool IOTA, int RS_I>
__global__ void __launch_bounds__(RS_T, 2) k_rs_pass(const K *__restrict__ kin, const uint32_t *__restrict__ vin,
                                                  K *__restrict__ kout, uint32_t *__restrict__ vout, int64_t n,
                                                  int shift, uint32_t mask, const uint32_t *__restrict__ hist,
                                                  uint32_t *__restrict__ ticket, uint64_t *__restrict__ status,
                                                  uint32_t epoch, unsigned *__restrict__ err) {
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int RS_TILE = RS_T * RS_I;
    RsShared<K, RS_I> &S = *reinterpret_cast<RsShared<K, RS_I> *>(smem);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, tid = threadIdx.x;
    if (tid == 0) S.tile = atomicAdd(ticket, 1u);
    for (int i = tid; i < RS_W * RS_BINS / 2; i += RS_T) reinterpret_cast<uint32_t *>(&S.cnt[0][0])[i] = 0u;
    // where the digit's keys start in the output
    const uint32_t first = rs_block_excl(hist[tid], S.wtot);   // ends with a barrier
    const int64_t tile = S.tile, tile0 = tile * RS_TILE;
    const int64_t base = tile0 + (int64_t)w * (32 * RS_I);
    const unsigned lt = (1u << lane) - 1u;
    K k[RS_I];
    uint32_t v[RS_I];
    uint32_t d[RS_I], r[RS_I];
#pragma unroll
    for (int i = 0; i < RS_I; ++i) {
        const int64_t idx = base + i * 32 + lane;
        const bool ok = idx < n;
        k[i] = ok ? kin[idx] : (K)0;
        v[i] = IOTA ? (uint32_t)idx : (ok ? vin[idx] : 0u);
        d[i] = ok ? ((uint32_t)(k[i] >> shift) & mask) : RS_BINS;   // RS_BINS: not a key
    }
#pragma unroll
    for (int i = 0; i < RS_I; ++i) {
        const bool ok = d[i] < RS_BINS;
        const unsigned peers = __match_any_sync(0xffffffffu, d[i]);
        uint32_t before = 0;
        if (ok) before = S.cnt[w][d[i]];
        __syncwarp();
        if (ok && lane == __ffs(peers) - 1) S.cnt[w][d[i]] = (uint16_t)(before + __popc(peers));
        __syncwarp();
        r[i] = before + __popc(peers & lt);
    }
    __syncthreads();
    // digit tid: prefix over the warps, the tile's count, published at once
    uint32_t tot = 0;
#pragma unroll
    for (int q = 0; q < RS_W; ++q) {
        const uint32_t t = S.cnt[q][tid];
        S.cnt[q][tid] = (uint16_t)tot;
        tot += t;
    }
    rs_put(status + tile * RS_BINS + tid, rs_word(epoch, tile == 0 ? 1u : 0u, tot));
    // where each digit's run starts in the staged tile
    S.loc[tid] = rs_block_excl(tot, S.wtot);   // ends with a barrier
    __syncthreads();
#pragma unroll
    for (int i = 0; i < RS_I; ++i) {
        if (d[i] < RS_BINS) {
            const uint32_t lp = S.loc[d[i]] + S.cnt[w][d[i]] + r[i];
            S.sk[lp] = k[i];
            S.sv[lp] = v[i];
        }
    }
    // look back: the counts of the digit in the tiles before this one, RS_LOOK
    // polls in flight (the tiles of the first wave all publish at once, and
    // the last of them has to pass half of them one by one)
    uint32_t excl = 0;
    if (tile > 0) {
        unsigned spins = 0;
        bool found = false;
        for (int64_t t = tile - 1; !found;) {
            uint64_t q[RS_LOOK];
#pragma unroll
            for (int u = 0; u < RS_LOOK; ++u) q[u] = t >= u ? rs_get(status + (t - u) * RS_BINS + tid) : 0ull;
            int used = 0;
#pragma unroll
            for (int u = 0; u < RS_LOOK; ++u) {
                const uint32_t tag = (uint32_t)(q[u] >> 32);
                if (!found && used == u && tag >> 1 == epoch) {
                    excl += (uint32_t)q[u];
                    found = tag & 1u;   // tile 0 publishes an inclusive sum
                    ++used;
                }
            }
            t -= used;
            if (used == 0 && ++spins > RS_SPIN) {   // the output stays in bounds whatever the offsets (see below)
                atomicOr(err, ERR_TIMEOUT);
                break;
            }
        }
        rs_put(status + tile * RS_BINS + tid, rs_word(epoch, 1u, excl + tot));
    }
    S.gof[tid] = first + excl;
    __syncthreads();
    const int m = (int)((n - tile0) < RS_TILE ? (n - tile0) : RS_TILE);
    for (int j = tid; j < m; j += RS_T) {
        const K kk = S.sk[j];
        const uint32_t dg = (uint32_t)(kk >> shift) & mask;
        const uint32_t dst = S.gof[dg] + (uint32_t)j - S.loc[dg];
        if (dst < n) {
            kout[dst] = kk;
            vout[dst] = S.sv[j];
        }
    }
}

template <class K, int RS_I>
apcloud_status sort_passes_of(apcloud_ctx *c, K *k0, uint32_t *v0, K *k1, uint32_t *v1, int64_t n, const RadixDigits &dg,
                           bool counted, bool iota, int *which) {
    *which = 0;
    const int ntile = div_up(n, RS_T * RS_I);
    uint32_t *hist = radix_counts(c);
    if (!hist) return APCLOUD_E_NOMEM;
    const size_t words = (size_t)ntile * RS_BINS;
    const bool fresh = !c->scan.p || c->scan.bytes < words * 8;
    uint64_t *status = ensure<uint64_t>(c, c->scan, words);
    if (!status) return APCLOUD_E_NOMEM;
    if (fresh || c->rs_epoch > 0x7FFFFF00u) {
        APC_CUDA(c, cudaMemsetAsync(status, 0, c->scan.bytes, c->s));
        c->rs_epoch = 0;
    }
    if (!counted) {
        APC_TRY(clear_radix_counts(c, dg));
        const int nb = std::min(div_up(n, RS_T * 4), 608);
        APC_LAUNCH(c, K_SORT, nb, RS_T, 0, k_rs_hist<K>, (const K *)k0, n, dg, hist);
        account(c, K_SORT, (double)sizeof(K) * n, 0.0);
    }
    uint32_t *ticket = hist + (size_t)dg.passes * RS_BINS;
    unsigned *derr = ptr<unsigned>(c->derr);
    const int smem = (int)sizeof(RsShared<K, RS_I>);
    APC_CUDA(c, cudaFuncSetAttribute(k_rs_pass<K, false, RS_I>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    APC_CUDA(c, cudaFuncSetAttribute(k_rs_pass<K, true, RS_I>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    K *ka = k0, *kb = k1;
    uint32_t *va = v0, *vb = v1;
    for (int p = 0; p < dg.passes; ++p) {
        const int sh = dg.shift[p];
        const uint32_t mask = (1u << dg.bits[p]) - 1u;
        const uint32_t *hp = hist + (size_t)p * RS_BINS;
        const uint32_t epoch = ++c->rs_epoch;
        if (iota && p == 0)
            APC_LAUNCH(c, K_SORT, ntile, RS_T, smem, (k_rs_pass<K, true, RS_I>), (const K *)ka, (const uint32_t *)va, kb, vb,
                       n, sh, mask, hp, ticket + p, status, epoch, derr);
        else
            APC_LAUNCH(c, K_SORT, ntile, RS_T, smem, (k_rs_pass<K, false, RS_I>), (const K *)ka, (const uint32_t *)va, kb,
                       vb, n, sh, mask, hp, ticket + p, status, epoch, derr);
        account(c, K_SORT, (2.0 * sizeof(K) + (iota && p == 0 ? 4.0 : 8.0)) * n, 0.0);
        std::swap(ka, kb);
        std::swap(va, vb);
    }
    *which = dg.passes & 1;
    return cuda_check(c, cudaGetLastError(), "radix_sort");
}

template <class K>
apcloud_status sort_passes(apcloud_ctx *c, K *k0, uint32_t *v0, K *k1, uint32_t *v1, int64_t n, const RadixDigits &dg,
                           bool counted, bool iota, int *which) {
    return n >= RS_MANY ? sort_passes_of<K, RS_I_MANY>(c, k0, v0, k1, v1, n, dg, counted, iota, which)
                        : sort_passes_of<K, RS_I_FEW>(c, k0, v0, k1, v1, n, dg, counted, iota, which);
}

}  // namespace

RadixDigits radix_digits(int nbits) {
    RadixDigits d{};
    d.passes = (nbits + RS_BITS - 1) / RS_BITS;
    for (int p = 0, at = 0; p < d.passes; ++p) {   // digits as equal as they get
        d.bits[p] = (nbits - at + d.passes - p - 1) / (d.passes - p);
        d.shift[p] = at;
        at += d.bits[p];
    }
    return d;
}

uint32_t *radix_counts(apcloud_ctx *c) {
    return ensure<uint32_t>(c, c->flags, RS_MAX_PASS * (RS_BINS + 1));
}

// zero counts, and the passes' tile counters behind them
apcloud_status clear_radix_counts(apcloud_ctx *c, const RadixDigits &dg) {
    uint32_t *h = radix_counts(c);
    if (!h) return APCLOUD_E_NOMEM;
    return cuda_check(c, cudaMemsetAsync(h, 0, sizeof(uint32_t) * dg.passes * (RS_BINS + 1), c->s), "radix_sort");
}

apcloud_status scan_u32(apcloud_ctx *c, const uint32_t *in, uint32_t *out, int64_t n, uint32_t *d_total) {
    if (n <= 0) {
        if (d_total) APC_CUDA(c, cudaMemsetAsync(d_total, 0, sizeof(uint32_t), c->s));
        return APCLOUD_OK;
    }
    int nb = div_up(n, SCAN_TILE);
    if (nb == 1) {
        APC_LAUNCH(c, K_TREE, 1, SCAN_T, 0, k_scan_down, in, out, n, (const uint32_t *)nullptr, d_total);
        return cuda_check(c, cudaGetLastError(), "scan");
    }
    uint32_t *blk = ensure<uint32_t>(c, c->scan_blk, nb);
    if (!blk) return APCLOUD_E_NOMEM;
    APC_LAUNCH(c, K_TREE, nb, SCAN_T, 0, k_scan_reduce, in, n, blk);
    APC_LAUNCH(c, K_TREE, nb, SCAN_T, 0, k_scan_down, in, out, n, (const uint32_t *)blk, d_total);
    return cuda_check(c, cudaGetLastError(), "scan");
}

apcloud_status radix_sort(apcloud_ctx *c, uint64_t *k0, uint32_t *v0, uint64_t *k1, uint32_t *v1, int64_t n,
                          int nbits, int *which) {
    *which = 0;
    if (n <= 1 || nbits <= 0) return APCLOUD_OK;
    return sort_passes<uint64_t>(c, k0, v0, k1, v1, n, radix_digits(nbits), false, false, which);
}

apcloud_status radix_sort(apcloud_ctx *c, uint32_t *k0, uint32_t *v0, uint32_t *k1, uint32_t *v1, int64_t n,
                          int nbits, int *which) {
    *which = 0;
    if (n <= 1 || nbits <= 0) return APCLOUD_OK;
    return sort_passes<uint32_t>(c, k0, v0, k1, v1, n, radix_digits(nbits), false, false, which);
}

// keys counted already (rs_count / rs_flush into radix_counts), values 0 .. n - 1
template <class K>
apcloud_status radix_sort_counted(apcloud_ctx *c, K *k0, uint32_t *v0, K *k1, uint32_t *v1, int64_t n,
                                  const RadixDigits &dg, int *which) {
    return sort_passes<K>(c, k0, v0, k1, v1, n, dg, true, true, which);
}
template apcloud_status radix_sort_counted<uint32_t>(apcloud_ctx *, uint32_t *, uint32_t *, uint32_t *, uint32_t *,
                                                     int64_t, const RadixDigits &, int *);
template apcloud_status radix_sort_counted<uint64_t>(apcloud_ctx *, uint64_t *, uint32_t *, uint64_t *, uint32_t *,
                                                     int64_t, const RadixDigits &, int *);

}  // namespace apc
