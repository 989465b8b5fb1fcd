// sweep.cu -- the preconditioner sweeps and Arnoldi products of systems too
// large for the resident solve (mixed polynomial form), on a block-local copy
// of the matrix.
//
// What bounds a sweep over a million rows on the ELL is not DRAM (the matrix is
// about as large as the L2, and the sweeps of one polynomial application follow
// one another) but the gathers of x: a warp's 32 entries touch 7 to 11
// different 128-byte lines, one L1 tag look-up each.  Here a block owns BL_ROWS
// consecutive rows.  They have some 3 BL_ROWS different columns (Morton order):
// the block loads those x once into shared memory, its own rows as they lie
// and the others through a sorted list, and the entries address them by 12-bit
// indices.  A gather from shared memory takes 2.4 passes over the banks, and an
// entry takes 3.5 bytes (index and FP16 value).
//
// Figures at 1.05e6 rows and 24.8e6 entries: with one chunk per thread ahead a
// sweep takes 30.7 us, with a whole row in registers before the wait for the
// sweep before, and the next row's chunks loaded as this one's are used up, 18.5
// us, with 12- instead of 16-bit indices 17.4 (26.2 us on a width-sorted copy
// with gathers from global memory, 41 us on the ELL).  There the load/store pipe
// is busy two thirds of the time; at 4.5e6 rows a sweep's 76 us are its bytes at
// DRAM rate.  Tried with 16-bit indices, for the solve of 120 steps: 512 rows
// in blocks of 256 threads 45.7 ms, 1024 rows of 512 threads 47, 1024 of 1024
// 62, 2048 of 512 58, 256 of 128 46.8, four rows a thread 61; index and value
// in two loads 47.1; five blocks per SM (registers spill) 57.
//
// Layout: 32-row slices in row order; the entries of a row in chunks of eight
// (chunk j of lane l at 32 j + l in its slice): 16 bytes of FP16 values, 8 and 4
// bytes of indices (the products load FP32 values instead).  Nine rows in ten
// have 17 to 24 entries, three chunks.  The diagonal, first in every row and 1
// after the scaling, is stored apart and read only where it is not.  Rows keep
// their entries in stored order: the results have the same bits as on the ELL.
// Lanes past their row's length load nothing.
#include <cuda_fp16.h>

#include <algorithm>
#include <climits>
#include <type_traits>

#include "internal.cuh"

namespace apc {

namespace {

constexpr int BL_ROWS = 512;               // rows per block
constexpr int BL_SL = BL_ROWS / 32;
constexpr int BL_HMAX = 4096 - BL_ROWS;    // other blocks' nodes a block can hold: indices of 12 bits
constexpr int BL_T = 256;                  // threads
constexpr int BL_RPT = BL_ROWS / BL_T;     // rows per thread
constexpr int BL_CE = 8, BL_CH = MMAX / BL_CE;   // entries of a chunk, chunks of a row at most
constexpr int BL_KEEP = 16;                // of so many blocks in turn, the first `keep` are kept in L2
static_assert(MMAX % BL_CE == 0, "whole chunks");
constexpr int BB_T = 512, BB_TAB = 8192, BB_LIST = 4096;   // threads, hash slots and list of the build
static_assert(BL_HMAX <= BB_LIST, "sorted in whole powers of two");

// One block's columns outside its rows, sorted, and its entries in the layout
// above.  A block with more than BL_HMAX such columns sets bit 0 of *bad: the
// system then stays on the ELL.  A diagonal that is not 1 (column-scaled systems)
// sets bit 1: the kernels then read the rows' diagonals from dg.
// 281 us at 1.05e6 rows, most of it latency (350 with one column and one chunk's
// values in flight per lane): three blocks per SM, a bitonic sort of some 1200
// nodes each.
__global__ void __launch_bounds__(BB_T) k_block_build(
    const uint32_t *__restrict__ sw, const uint32_t *__restrict__ soff, const int32_t *__restrict__ col,
    const __half *__restrict__ hA, const __half *__restrict__ hB, const float *__restrict__ fA,
    const float *__restrict__ fB, const int32_t *__restrict__ msz, int n_int, int n, int nsl,
    const uint32_t *__restrict__ off4, int32_t *__restrict__ hlist, int32_t *__restrict__ hcnt,
    uint8_t *__restrict__ len, uint2 *__restrict__ idx, uint32_t *__restrict__ idx4, uint4 *__restrict__ A2,
    uint4 *__restrict__ B2, float4 *__restrict__ A4, float4 *__restrict__ B4, float *__restrict__ dg, unsigned *bad) {
    extern __shared__ __align__(16) unsigned char smem[];
    int *key = reinterpret_cast<int *>(smem);                       // BB_TAB
    int *list = key + BB_TAB;                                       // BB_LIST
    uint16_t *loc = reinterpret_cast<uint16_t *>(list + BB_LIST);   // BB_TAB
    __shared__ int cnt;
    const int tid = threadIdx.x, blk = blockIdx.x;
    const int r0 = blk * BL_ROWS, r1 = min(r0 + BL_ROWS, n);
    const int s0 = blk * BL_SL, s1 = min(s0 + BL_SL, nsl);
    for (int i = tid; i < BB_TAB; i += BB_T) key[i] = -1;
    if (tid == 0) cnt = 0;
    __syncthreads();
    volatile int *vc = &cnt, *vkey = key;
    const int64_t e0 = (int64_t)soff[s0] * 32, e1 = ((int64_t)soff[s1 - 1] + sw[s1 - 1]) * 32;
    for (int64_t e = e0 + tid; e < e1; e += 8 * BB_T) {   // eight columns in flight
        int cc[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) cc[t] = e + t * BB_T < e1 ? col[e + t * BB_T] : r0;
#pragma unroll 1
        for (int t = 0; t < 8; ++t) {
            const int c = cc[0];
#pragma unroll
            for (int u = 0; u < 7; ++u) cc[u] = cc[u + 1];
            if ((c >= r0 && c < r1) || *vc > BL_HMAX) continue;   // the table never fills: at most BL_HMAX + BB_T entries
            unsigned h = (unsigned)c * 0x9E3779B1u >> 19;
            for (;;) {
                int old = vkey[h];   // most are there already
                if (old == -1) old = atomicCAS(key + h, -1, c);
                if (old == c) break;
                if (old == -1) {
                    const int p = atomicAdd(&cnt, 1);
                    if (p < BL_HMAX) list[p] = c;
                    break;
                }
                h = (h + 1) & (BB_TAB - 1);
            }
        }
    }
    __syncthreads();
    const int H = cnt;
    if (H > BL_HMAX) {
        if (tid == 0) {
            atomicOr(bad, 1u);
            hcnt[blk] = 0;
        }
        return;
    }
    int P = 1;
    while (P < H) P <<= 1;
    for (int i = H + tid; i < P; i += BB_T) list[i] = INT_MAX;
    __syncthreads();
    for (int k = 2; k <= P; k <<= 1) {   // bitonic sort
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = tid; i < P / 2; i += BB_T) {
                const int a = ((i & ~(j - 1)) << 1) | (i & (j - 1)), b = a | j;
                const int x = list[a], y = list[b];
                if ((x > y) == ((a & k) == 0)) {
                    list[a] = y;
                    list[b] = x;
                }
            }
            __syncthreads();
        }
    }
    for (int i = tid; i < H; i += BB_T) {
        const int c = list[i];
        hlist[(int64_t)blk * BL_HMAX + i] = c;
        unsigned h = (unsigned)c * 0x9E3779B1u >> 19;
        while (key[h] != c) h = (h + 1) & (BB_TAB - 1);
        loc[h] = (uint16_t)(BL_ROWS + i);
    }
    if (tid == 0) hcnt[blk] = H;
    __syncthreads();
    for (int s = s0 + (tid >> 5); s < s1; s += BB_T / 32) {   // a warp per slice
        const int lane = tid & 31, r = s * 32 + lane;
        const int m = r < n_int ? msz[r] : 0;
        const int w = (int)sw[s] - 1;
        const int64_t eb = (int64_t)soff[s] * 32 + lane + 32;   // past the diagonal
        if (r < n) {
            len[r] = (uint8_t)m;
            // of the sweeps (FP16 values), then of the products, B before A
            dg[r] = __half2float(hB[eb - 32]);
            dg[n + r] = __half2float(hA[eb - 32]);
            dg[2 * (int64_t)n + r] = fB[eb - 32];
            dg[3 * (int64_t)n + r] = fA[eb - 32];
            if (fA[eb - 32] != 1.f || fB[eb - 32] != 1.f) atomicOr(bad, 2u);
        }
        const int64_t ob = (int64_t)off4[s] * 32 + lane;
        for (int j = 0; j * BL_CE < w; ++j) {
            uint32_t ix[8], aw[4], bw[4];
            const int64_t o = ob + (int64_t)j * 32;
#pragma unroll
            for (int g = 0; g < 2; ++g) {   // four entries in flight
                int c[4];
                uint32_t a[4], b[4];
                float va[4], vb[4];
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const int k = BL_CE * j + 4 * g + t;
                    const int64_t e = eb + (int64_t)(k < m ? k : -1) * 32;   // past the row: the diagonal's place
                    c[t] = col[e];
                    a[t] = __half_as_ushort(hA[e]);
                    b[t] = __half_as_ushort(hB[e]);
                    va[t] = fA[e];
                    vb[t] = fB[e];
                }
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const bool in = BL_CE * j + 4 * g + t < m;
                    uint32_t i;
                    if (!in) {   // itself, times zero
                        a[t] = b[t] = 0u;
                        va[t] = vb[t] = 0.f;
                    }
                    if (!in || (c[t] >= r0 && c[t] < r1)) {
                        i = (uint32_t)(in ? c[t] - r0 : (r < n ? r - r0 : 0));
                    } else {
                        unsigned h = (unsigned)c[t] * 0x9E3779B1u >> 19;
                        while (key[h] != c[t]) h = (h + 1) & (BB_TAB - 1);
                        i = loc[h];
                    }
                    ix[4 * g + t] = i;
                }
                aw[2 * g] = a[0] | a[1] << 16;
                aw[2 * g + 1] = a[2] | a[3] << 16;
                bw[2 * g] = b[0] | b[1] << 16;
                bw[2 * g + 1] = b[2] | b[3] << 16;
                A4[2 * o - lane + 32 * g] = make_float4(va[0], va[1], va[2], va[3]);
                B4[2 * o - lane + 32 * g] = make_float4(vb[0], vb[1], vb[2], vb[3]);
            }
            idx[o] = make_uint2(ix[0] | ix[1] << 12 | ix[2] << 24, ix[2] >> 8 | ix[3] << 4 | ix[4] << 16 | ix[5] << 28);
            idx4[o] = ix[5] >> 4 | ix[6] << 8 | ix[7] << 20;
            A2[o] = make_uint4(aw[0], aw[1], aw[2], aw[3]);
            B2[o] = make_uint4(bw[0], bw[1], bw[2], bw[3]);
        }
    }
}

// Programmatic dependent launch: waits for the kernel before, then lets the
// next one start.  Released only after its own wait, so at most two are
// resident, and what ran before the one waited for has ended.
__device__ __forceinline__ void dep_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// matrix loads: not kept in L1 (read once), in L2 as the policy says
__device__ __forceinline__ uint32_t load(const uint32_t *p, uint64_t pol) {
    uint32_t v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.u32 %0, [%1], %2;" : "=r"(v) : "l"(p), "l"(pol));
    return v;
}
__device__ __forceinline__ uint2 load(const uint2 *p, uint64_t pol) {
    uint2 v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v2.u32 {%0, %1}, [%2], %3;"
                 : "=r"(v.x), "=r"(v.y)
                 : "l"(p), "l"(pol));
    return v;
}
__device__ __forceinline__ uint4 load(const uint4 *p, uint64_t pol) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p), "l"(pol));
    return v;
}
__device__ __forceinline__ float4 load(const float4 *p, uint64_t pol) {
    float4 v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "l"(p), "l"(pol));
    return v;
}

// eight 12-bit indices, and the x they stand for
struct Index8 {
    uint2 q;
    uint32_t p;
    __device__ __forceinline__ void get(const uint2 *idx, const uint32_t *idx4, int64_t o, uint64_t pol) {
        q = load(idx + o, pol);
        p = load(idx4 + o, pol);
    }
    __device__ __forceinline__ void gather(const float *xs, float (&x)[8]) const {
        const uint32_t at[8] = {q.x << 2, q.x >> 10, __funnelshift_r(q.x, q.y, 22), q.y >> 2,   // 4 times the index,
                                q.y >> 14, __funnelshift_r(q.y, p, 26), p >> 6, p >> 18};       // other bits around it
#pragma unroll
        for (int t = 0; t < 8; ++t)
            x[t] = *reinterpret_cast<const float *>(reinterpret_cast<const char *>(xs) + (at[t] & 0x3FFCu));
    }
};

// eight entries: indices, and FP16 values in one 16-byte load (sweeps) or FP32
// ones in two (products)
struct Chunk16 {
    Index8 i;
    uint4 v;
    __device__ __forceinline__ void get(const uint2 *idx, const uint32_t *idx4, const uint4 *val, int64_t o, int,
                                        uint64_t pol) {
        i.get(idx, idx4, o, pol);
        v = load(val + o, pol);
    }
    __device__ __forceinline__ float dot(float acc, const float *xs) const {
        float x[8];
        i.gather(xs, x);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&w[t]));
            acc = fmaf(f.x, x[2 * t], acc);
            acc = fmaf(f.y, x[2 * t + 1], acc);
        }
        return acc;
    }
};
struct Chunk32 {
    Index8 i;
    float4 a, b;
    __device__ __forceinline__ void get(const uint2 *idx, const uint32_t *idx4, const float4 *val, int64_t o, int lane,
                                        uint64_t pol) {
        i.get(idx, idx4, o, pol);
        a = load(val + 2 * o - lane, pol);
        b = load(val + 2 * o - lane + 32, pol);
    }
    __device__ __forceinline__ float dot(float acc, const float *xs) const {
        float x[8];
        i.gather(xs, x);
        acc = fmaf(a.x, x[0], acc);
        acc = fmaf(a.y, x[1], acc);
        acc = fmaf(a.z, x[2], acc);
        acc = fmaf(a.w, x[3], acc);
        acc = fmaf(b.x, x[4], acc);
        acc = fmaf(b.y, x[5], acc);
        acc = fmaf(b.z, x[6], acc);
        return fmaf(b.w, x[7], acc);
    }
};

// SWEEP: y = x + omega (b - Ahat x), damped Jacobi sweep of the polynomial
// (FP16 values); else y = Ahat x, the Arnoldi product (FP32 values).  Skipped
// once the cycle is done; rows of converged beams give 0.  The matrix is read
// as evict-first lines, but for the first `keep` of every BL_KEEP blocks: what
// stays in L2 from one sweep to the next is then read alongside what comes from
// DRAM (48.0 ms for the solve above, 49.6 ms with the kept blocks in a row).
// The product has no work before its loads to hide behind and takes a third
// more registers: three blocks per SM (38.3 us, 40.0 at four with half a row in
// flight).
// DIAG: a diagonal that is not 1, from dg.
template <bool SWEEP, class V, bool DIAG>
__global__ void __launch_bounds__(BL_T, SWEEP ? 4 : 3) k_block_rows(
    const uint32_t *__restrict__ off4, const uint8_t *__restrict__ len, const int32_t *__restrict__ hlist,
    const int32_t *__restrict__ hcnt, const uint2 *__restrict__ idx, const uint32_t *__restrict__ idx4,
    const V *__restrict__ val, const float *__restrict__ dg, int n, const float *x, float *__restrict__ y, const float *__restrict__ b, const GmresState *__restrict__ st,
    RowSkip skip, int keep) {
    __shared__ float xs[BL_ROWS + BL_HMAX];
    const int tid = threadIdx.x, blk = blockIdx.x, r0 = blk * BL_ROWS;
    uint64_t pol;
    if (blk % BL_KEEP < keep)
        asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(pol));
    else
        asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    // what no sweep writes is read before the wait: lengths, a row's chunks, b, the list
    int nch[BL_RPT];
    int64_t base[BL_RPT];
    bool act[BL_RPT], any = false;
    float br[BL_RPT];
#pragma unroll
    for (int q = 0; q < BL_RPT; ++q) {
        const int r = r0 + q * BL_T + tid;
        act[q] = r < n && !(skip.nbo && skip.bdone[skip.nbo[r]]);
        any |= act[q];
        nch[q] = act[q] ? (len[r] + BL_CE - 1) / BL_CE : 0;
        base[q] = r < n ? (int64_t)off4[r >> 5] * 32 + (r & 31) : 0;
        br[q] = SWEEP && act[q] ? b[r] : 0.f;
    }
    typename std::conditional<SWEEP, Chunk16, Chunk32>::type ch[BL_CH];
#pragma unroll
    for (int j = 0; j < BL_CH; ++j)
        if (j < nch[0]) ch[j].get(idx, idx4, val, base[0] + j * 32, tid & 31, pol);
    const int H = hcnt[blk];
    const int32_t *hl = hlist + (int64_t)blk * BL_HMAX;
    int32_t hi[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) hi[u] = tid + u * BL_T < H ? __ldg(hl + tid + u * BL_T) : -1;
    if (st->done) return;
    const float om = SWEEP ? (float)st->omega : 0.f;
    dep_wait();
    if (skip.nbo && !__syncthreads_or(any)) {   // every row's beam has converged
#pragma unroll
        for (int q = 0; q < BL_RPT; ++q) {
            const int r = r0 + q * BL_T + tid;
            if (r < n) y[r] = 0.f;
        }
        return;
    }
#pragma unroll
    for (int q = 0; q < BL_RPT; ++q) {
        const int r = r0 + q * BL_T + tid;
        xs[q * BL_T + tid] = r < n ? __ldcg(x + r) : 0.f;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
        if (hi[u] >= 0) xs[BL_ROWS + tid + u * BL_T] = __ldcg(x + hi[u]);
    for (int t = tid + 4 * BL_T; t < H; t += BL_T) xs[BL_ROWS + t] = __ldcg(x + __ldg(hl + t));
    __syncthreads();
#pragma unroll
    for (int q = 0; q < BL_RPT; ++q) {
        const int r = r0 + q * BL_T + tid, q1 = q + 1 < BL_RPT ? q + 1 : 0;
        const float own = xs[q * BL_T + tid];
        float acc = DIAG && act[q] ? fmaf(dg[r], own, 0.f) : own + 0.f;   // the diagonal's term
#pragma unroll
        for (int j = 0; j < BL_CH; ++j) {
            if (j < nch[q]) acc = ch[j].dot(acc, xs);
            if (q1 > q && j < nch[q1]) ch[j].get(idx, idx4, val, base[q1] + j * 32, tid & 31, pol);   // the next row's in its place
        }
        if (r < n) y[r] = act[q] ? (SWEEP ? fmaf(om, br[q] - acc, own) : acc) : 0.f;
    }
}

}  // namespace

// chunks per slice of the block-local copy
__global__ void k_chunks(const uint32_t *__restrict__ sw, int nsl, uint32_t *__restrict__ w4) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s < nsl) w4[s] = (sw[s] + BL_CE - 2) / BL_CE;   // the diagonal is not stored
}

apcloud_status count_blocks(apcloud_ctx *c, uint32_t *d_total) {
    c->bl_ok = c->bl_tried = false;
    const int nsl = c->n_slices;
    uint32_t *w4 = ensure<uint32_t>(c, c->bl_w4, nsl + 1), *o4 = ensure<uint32_t>(c, c->bl_off, nsl + 1);
    if (!w4 || !o4) return APCLOUD_E_NOMEM;
    APC_LAUNCH(c, K_ELL, div_up(nsl, 256), 256, 0, k_chunks, (const uint32_t *)ptr<uint32_t>(c->slice_w), nsl, w4);
    return scan_u32(c, w4, o4, nsl, d_total);
}

apcloud_status build_blocks(apcloud_ctx *c) {
    const int n = c->n_tot, nblk = div_up(n, BL_ROWS);
    const int64_t ch = c->bl_chunks * 32;
    int32_t *hl = ensure<int32_t>(c, c->bl_hlist, (int64_t)nblk * BL_HMAX), *hc = ensure<int32_t>(c, c->bl_hcnt, nblk + 1);
    uint8_t *len = ensure<uint8_t>(c, c->bl_len, n);
    uint32_t *ib = ensure<uint32_t>(c, c->bl_idx, 3 * ch + 2);
    uint2 *ix = reinterpret_cast<uint2 *>(ib);
    uint4 *A2 = ensure<uint4>(c, c->bl_A, ch + 1), *B2 = ensure<uint4>(c, c->bl_B, ch + 1);
    float4 *A4 = ensure<float4>(c, c->bl_A32, 2 * ch + 1), *B4 = ensure<float4>(c, c->bl_B32, 2 * ch + 1);
    float *dg = ensure<float>(c, c->bl_dg, 4 * (int64_t)n + 1);
    if (!hl || !hc || !len || !ib || !A2 || !B2 || !A4 || !B4 || !dg) return APCLOUD_E_NOMEM;
    const int smem = BB_TAB * 4 + BB_LIST * 4 + BB_TAB * 2;
    APC_CUDA(c, cudaFuncSetAttribute(k_block_build, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    unsigned *bad = ptr<uint32_t>(c->dsmall) + 14;
    APC_CUDA(c, cudaMemsetAsync(bad, 0, sizeof(unsigned), c->s));
    APC_LAUNCH(c, K_ELL, nblk, BB_T, smem, k_block_build, (const uint32_t *)ptr<uint32_t>(c->slice_w),
               (const uint32_t *)ptr<uint32_t>(c->slice_off), (const int32_t *)ptr<int32_t>(c->ell_col),
               (const __half *)ptr<__half>(c->ell_A16), (const __half *)ptr<__half>(c->ell_B16),
               (const float *)ptr<float>(c->ell_A32), (const float *)ptr<float>(c->ell_B32),
               (const int32_t *)ptr<int32_t>(c->msz), c->n_int, n, c->n_slices,
               (const uint32_t *)ptr<uint32_t>(c->bl_off), hl, hc, len, ix, ib + 2 * ch, A2, B2, A4, B4, dg, bad);
    APC_CUDA(c, cudaGetLastError());
    unsigned b = 0;
    APC_TRY(read_back(c, &b, bad, sizeof b));
    c->bl_ok = (b & 1u) == 0;
    c->bl_unit = (b & 2u) == 0;
    c->bl_tried = true;
    return APCLOUD_OK;
}

void block_sweep(apcloud_ctx *c, int which, const float *x, float *y, const float *b, const GmresState *st,
                 RowSkip skip, int keep, bool pdl) {
    const int nblk = div_up(c->n_tot, BL_ROWS);
    auto kern = c->bl_unit ? k_block_rows<true, uint4, false> : k_block_rows<true, uint4, true>;
    const uint4 *val = ptr<uint4>(which ? c->bl_A : c->bl_B);
    const float *dg = ptr<float>(c->bl_dg) + (int64_t)(which ? 1 : 0) * c->n_tot;
    if (pdl)
        APC_LAUNCH_PDL(c, K_SWEEP, nblk, BL_T, 0, kern, (const uint32_t *)ptr<uint32_t>(c->bl_off),
                       (const uint8_t *)ptr<uint8_t>(c->bl_len), (const int32_t *)ptr<int32_t>(c->bl_hlist),
                       (const int32_t *)ptr<int32_t>(c->bl_hcnt), (const uint2 *)ptr<uint2>(c->bl_idx),
                       (const uint32_t *)(ptr<uint32_t>(c->bl_idx) + 64 * c->bl_chunks), val, dg, c->n_tot, x,
                       y, b, st, skip, keep);
    else
        APC_LAUNCH(c, K_SWEEP, nblk, BL_T, 0, kern, (const uint32_t *)ptr<uint32_t>(c->bl_off),
                   (const uint8_t *)ptr<uint8_t>(c->bl_len), (const int32_t *)ptr<int32_t>(c->bl_hlist),
                   (const int32_t *)ptr<int32_t>(c->bl_hcnt), (const uint2 *)ptr<uint2>(c->bl_idx),
                       (const uint32_t *)(ptr<uint32_t>(c->bl_idx) + 64 * c->bl_chunks), val, dg, c->n_tot, x, y,
                   b, st, skip, keep);
}

void block_product(apcloud_ctx *c, int which, const float *x, float *y, const GmresState *st, RowSkip skip, bool pdl) {
    const int nblk = div_up(c->n_tot, BL_ROWS);
    auto kern = c->bl_unit ? k_block_rows<false, float4, false> : k_block_rows<false, float4, true>;
    const float4 *val = ptr<float4>(which ? c->bl_A32 : c->bl_B32);
    const float *dg = ptr<float>(c->bl_dg) + (int64_t)(which ? 3 : 2) * c->n_tot;
    if (pdl)
        APC_LAUNCH_PDL(c, K_SPMV, nblk, BL_T, 0, kern, (const uint32_t *)ptr<uint32_t>(c->bl_off),
                       (const uint8_t *)ptr<uint8_t>(c->bl_len), (const int32_t *)ptr<int32_t>(c->bl_hlist),
                       (const int32_t *)ptr<int32_t>(c->bl_hcnt), (const uint2 *)ptr<uint2>(c->bl_idx),
                       (const uint32_t *)(ptr<uint32_t>(c->bl_idx) + 64 * c->bl_chunks), val, dg, c->n_tot, x,
                       y, (const float *)nullptr, st, skip, 0);
    else
        APC_LAUNCH(c, K_SPMV, nblk, BL_T, 0, kern, (const uint32_t *)ptr<uint32_t>(c->bl_off),
                   (const uint8_t *)ptr<uint8_t>(c->bl_len), (const int32_t *)ptr<int32_t>(c->bl_hlist),
                   (const int32_t *)ptr<int32_t>(c->bl_hcnt), (const uint2 *)ptr<uint2>(c->bl_idx),
                       (const uint32_t *)(ptr<uint32_t>(c->bl_idx) + 64 * c->bl_chunks), val, dg, c->n_tot, x, y,
                   (const float *)nullptr, st, skip, 0);
}

int block_keep(double fraction) { return fraction >= 1.0 ? BL_KEEP : (int)(BL_KEEP * fraction); }

}  // namespace apc
