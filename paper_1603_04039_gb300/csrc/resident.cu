// resident.cu -- whole GMRES solves in one cooperative kernel, the matrix held
// in shared memory.
//
// For systems whose matrix fits the SMs' shared memory together (up to 2.2e5
// rows in the mixed polynomial form, 1.4e5 in the mixed Jacobi form, 8.8e4 in FP64:
// the largest seen to run) a solve made of one
// launch per product and reduction is bound by launches and by the latency of
// each grid-wide reduction, not by bytes: a 1.1e5-row matrix (16 MB as FP16
// values and 16-bit indices) streams in 2-3 us, a sweep took 5-7 us and a CGS2
// step ~60 us.  Here block c owns a contiguous range of 32-row slices for the
// whole solve and keeps in shared memory
//   * its slices of the sliced-ELL matrix, the columns renumbered to 16 bits:
//     own rows first, then the block's halo (the sorted distinct columns
//     outside its rows);
//   * the vector being multiplied, own rows and halo.
// A product needs only the halo from other blocks.  It travels as
// (value, tag) words: the owner stores every value together with the number
// of the exchange in one 64-bit word, the reader polls the word until the tag
// is the one it waits for, so neither a grid barrier nor a fence stands
// between two sweeps (~1 us from store to use instead of a kernel boundary).
// Grid sums travel the same way: each block stores its partial sums, block
// k mod G adds the partials of value k in block order, everybody reads the
// totals (small grids: everybody adds all partials).  Every block then keeps
// its own copy of the Hessenberg matrix and the rotations and runs the same
// scalar recurrences, so no block waits for a decision of another.
//
// The rows' sums run in stored order, as in the launched kernels; the sums of
// the reductions have a fixed order, so a solve is repeatable bit for bit.
//
// What bounds it: the latency of the exchanges (~1.3 us from the owner's
// store to the reader's barrier; a degree-16 step makes 16 and one sum, two
// more hops for more than ~20 blocks), the 16-bit gathers from shared memory
// once a block holds many rows (1.1e5 rows: 2.9 us per sweep, 1.4 of them
// exchange), and in FP64 the two lanes per clock of that pipe.
//
// Measured (GB300, beam with halo, one solve, launched kernels -> here):
//   FP64 Jacobi, rtol 1e-12:    1471 nodes, 71 steps    4.5 -> 1.0 ms
//                              15426 nodes, 657 steps  45.9 -> 10.2 ms
//                              86686 nodes              74 -> 32 us a step
//   mixed degree 16, 1e-11:    15426 nodes, 32 steps    3.4 -> 1.25 ms
//                             110059 nodes, 54 steps    6.4 -> 3.19 ms
//                             222416 nodes            165 -> 88 us a step
// 384 worker threads: 256 leave the solve of 1.1e5 rows at 3.48 ms, 512 make
// every barrier dearer (1.26 against 1.22 ms on 15426 nodes).  Counters of the
// 1.1e5-row solve: a warp waits 3.2 cycles at barriers and 3.4 for loads between
// two instructions, the schedulers issue in 31% of the cycles, the shared-memory
// pipe is 42% busy; of the 1.5e4-row FP64 solve: 18 of 28 at barriers.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>

#include "fpconv.cuh"
#include "internal.cuh"

namespace apc {

namespace {

constexpr int PT = 384;            // worker threads per block
constexpr int PW = PT / 32;
constexpr int PB = PT + 32;        // and a warp that runs the rotations beside them
constexpr int LPV = 8;             // lanes per basis vector of a dot product
constexpr int NGRP = PT / LPV;
constexpr int PM = RES_MAX_RESTART;   // longest restart (2 j + 4 sums per step fit 64 slots)
constexpr int PSL = 64;            // most slices per block
constexpr int RED_SLOTS = 64;     // values per reduction
// partials every block reads itself instead of the totals: one hop instead of
// two, but every block reads them all (54 steps of 1.1e5 rows: 3.25 ms at 800,
// 3.29 at 2048, 3.37 at 5000)
constexpr int DIRECT_MOST = 800;
constexpr unsigned SPIN_LIMIT = 1u << 20;   // polls of one wait (~1 s) before the solve is given up
constexpr int STEP_BUDGET = 8192;  // Arnoldi steps per launch
constexpr uint32_t TAGS_PER_LAUNCH = 1u << 16;   // >= 4 tags per step and cycle of a launch

// compensated FP32 pairs (TwoSum), as in the launched DCGS2 kernels
struct F2 {
    float s, e;
};
__device__ __forceinline__ F2 f2add(F2 a, F2 b) {
    const float s = a.s + b.s;
    const float bb = s - a.s;
    const float err = (a.s - (s - bb)) + (b.s - bb);
    return F2{s, (a.e + b.e) + err};
}

// a sum in flight: a double, or a pair for FP32 vectors
template <class T> struct Acc;
template <> struct Acc<double> {
    typedef double type;
    static __device__ __forceinline__ double zero() { return 0.0; }
    static __device__ __forceinline__ double of(double v) { return v; }
    static __device__ __forceinline__ double add(double a, double b) { return a + b; }
    static __device__ __forceinline__ double shfl(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
    static __device__ __forceinline__ uint2 bits(double v) {
        return make_uint2((uint32_t)__double2loint(v), (uint32_t)__double2hiint(v));
    }
    static __device__ __forceinline__ double from(uint2 b) { return __hiloint2double((int)b.y, (int)b.x); }
    static __device__ __forceinline__ double value(double v) { return v; }
};
template <> struct Acc<float> {
    typedef F2 type;
    static __device__ __forceinline__ F2 zero() { return F2{0.f, 0.f}; }
    static __device__ __forceinline__ F2 of(float v) { return F2{v, 0.f}; }
    static __device__ __forceinline__ F2 add(F2 a, F2 b) { return f2add(a, b); }
    static __device__ __forceinline__ F2 shfl(F2 v, int o) {
        return F2{__shfl_xor_sync(0xffffffffu, v.s, o), __shfl_xor_sync(0xffffffffu, v.e, o)};
    }
    static __device__ __forceinline__ uint2 bits(F2 v) { return make_uint2(__float_as_uint(v.s), __float_as_uint(v.e)); }
    static __device__ __forceinline__ F2 from(uint2 b) { return F2{__uint_as_float(b.x), __uint_as_float(b.y)}; }
    static __device__ __forceinline__ double value(F2 v) { return f32_to_f64_int(v.s) + f32_to_f64_int(v.e); }
};
template <class A>
__device__ __forceinline__ typename A::type warp_acc(typename A::type v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = A::add(v, A::shfl(v, o));
    return v;
}

// ---- tagged words: 32 bits of payload under 32 bits of tag, stored and
// loaded as one 64-bit access; payloads of 64 bits take two such words
__device__ __forceinline__ uint64_t pack(uint32_t v, uint32_t tag) { return (uint64_t)tag << 32 | v; }
__device__ __forceinline__ void put1(uint64_t *p, uint32_t v, uint32_t tag) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(pack(v, tag)) : "memory");
}
__device__ __forceinline__ uint64_t get1(const uint64_t *p) {
    uint64_t w;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
    return w;
}
__device__ __forceinline__ void put2(uint64_t *p, uint2 v, uint32_t tag) {
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(pack(v.x, tag)), "l"(pack(v.y, tag))
                 : "memory");
}
__device__ __forceinline__ void get2(const uint64_t *p, uint64_t &a, uint64_t &b) {
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}

// A wait that has polled `spins` times: false when it must end, because this
// block or another gave up (every wait of the solve then ends at once and the
// host reports a timeout).
__device__ __noinline__ bool keep_waiting(unsigned &spins, volatile int *s_abort, int *g_abort) {
    if (*s_abort) return false;
    if ((++spins & 255u) == 0u) {
        int ga;
        asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(ga) : "l"(g_abort) : "memory");
        if (ga || spins > SPIN_LIMIT) {
            atomicExch(g_abort, 1);
            *s_abort = 1;
            return false;
        }
    }
    return true;
}

struct Fixed {   // shared state of a block
    // The rotations' product, row by row: W[i] is row i once rotation i is
    // done; the row that is still open stays in the scalar warp's registers.
    // A column's carried entry is then one dot product (a chain of j rotations
    // took ~3 us at j = 30), and the triangular factor is formed at the cycle end.
    double W[PM * 32];
    double H[PM * (PM + 1) / 2];   // Hessenberg columns above the subdiagonal, packed
    double Rm[PM * (PM - 1) / 2];  // triangular factor above its diagonal, packed
    double rd[PM + 1], g[PM + 2], h1[PM + 2], h2[PM + 2], y[PM + 1], colp[PM + 2], colc[PM + 2];
    double res[RED_SLOTS];
    double nu, inu, nut, nut2, inv;
    uint2 val[RED_SLOTS];      // this block's partial sums
    uint2 part[2 * NGRP];
    uint32_t ssb[PSL], ssw[PSL];   // entry base and width of the block's slices
    uint32_t wtot[PW];
    // abort: a wait gave up (set at any time); stop: the same as the block saw
    // it at its last grid sum, so that all its threads decide alike
    int done, abort, stop, halo;
    float f1[PM + 2], f2[PM + 2], fy[PM + 1];   // h1, h2, y for FP32 vectors
};

struct Shape {   // what a block works on
    int r0, R, Rp, H;        // first row, rows, rows padded to slices, halo size
    int n;
    int64_t e0;              // first stored entry
};

// ---- grid sum of the nk values in S.val, in block order; totals in S.res.
// Ends with a block barrier.
template <class A>
__device__ void grid_sum(Fixed &S, int nk, uint64_t *red, uint32_t tag, int *g_abort) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, G = gridDim.x, c = blockIdx.x;
    uint64_t *P = red + (size_t)(tag & 1u) * RED_SLOTS * (G + 1) * 2;   // two sets: see below
    uint64_t *R = P + (size_t)RED_SLOTS * G * 2;
    // A set is written again two sums later: a block gets there only after
    // every block has stored its partials of the sum in between, which each
    // does after it has read the totals of this one.
    __syncthreads();
    if (tid < nk) put2(P + ((size_t)tid * G + c) * 2, S.val[tid], tag);
    volatile int *sa = &S.abort;
    const bool direct = G * nk <= DIRECT_MOST;
    // a value's partials are added by LS lanes, blocks l, l + LS, ... by lane
    // l with four polls in flight (fewer lanes per value for few blocks: the
    // shuffle tree of an FP64 sum costs a full-rate slot per level)
    const int LS = !direct || G > 64 ? 32 : (G > 32 ? 16 : (G > 16 ? 8 : 4)), per = 32 / LS;
    const int l = lane & (LS - 1), sub = lane / LS;
    for (int i = wid; wid < PW; i += PW) {
        if (direct ? i * per >= nk : c + i * G >= nk) break;
        const int k = direct ? i * per + sub : c + i * G;
        typename A::type s = A::zero();
        for (int q0 = l; k < nk && q0 < G; q0 += 4 * LS) {
            uint64_t w0[4], w1[4];
            unsigned pending = 0, spins = 0;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                w0[u] = w1[u] = 0;
                if (q0 + u * LS < G) pending |= 1u << u;
            }
            const unsigned have = pending;
            while (pending) {
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (pending >> u & 1u) get2(P + ((size_t)k * G + q0 + u * LS) * 2, w0[u], w1[u]);
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if ((uint32_t)(w0[u] >> 32) == tag && (uint32_t)(w1[u] >> 32) == tag) pending &= ~(1u << u);
                if (pending && !keep_waiting(spins, sa, g_abort)) break;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (have >> u & 1u) s = A::add(s, A::from(make_uint2((uint32_t)w0[u], (uint32_t)w1[u])));
        }
        __syncwarp();
        for (int o = LS >> 1; o > 0; o >>= 1) s = A::add(s, A::shfl(s, o));
        if (l == 0 && k < nk) {
            const double t = A::value(s);
            if (direct) S.res[k] = t;
            else put2(R + (size_t)k * 2, Acc<double>::bits(t), tag);
        }
    }
    if (!direct && tid < nk) {
        uint64_t a, b;
        unsigned spins = 0;
        for (;;) {
            get2(R + (size_t)tid * 2, a, b);
            if ((uint32_t)(a >> 32) == tag && (uint32_t)(b >> 32) == tag) break;
            if (!keep_waiting(spins, sa, g_abort)) break;
        }
        S.res[tid] = Acc<double>::from(make_uint2((uint32_t)a, (uint32_t)b));
    }
    __syncthreads();
    if (tid == 0) S.stop = *sa;
    __syncthreads();
}

// coefficients of the vector updates in the vectors' type
template <class T> __device__ __forceinline__ const T *coef_y(const Fixed &S);
template <> __device__ __forceinline__ const float *coef_y<float>(const Fixed &S) { return S.fy; }
template <> __device__ __forceinline__ const double *coef_y<double>(const Fixed &S) { return S.y; }

// the block's sum of one value per worker into S.val[k] (ends with a barrier)
template <class A>
__device__ __forceinline__ void block_sum(Fixed &S, typename A::type v, int k) {
    v = warp_acc<A>(v);
    if ((threadIdx.x & 31) == 0 && threadIdx.x < PT) S.part[threadIdx.x >> 5] = A::bits(v);
    __syncthreads();
    if (threadIdx.x == 0) {
        typename A::type s = A::zero();
        for (int q = 0; q < PW; ++q) s = A::add(s, A::from(S.part[q]));
        S.val[k] = A::bits(s);
    }
    __syncthreads();
}

// halo values of exchange `tag` from the owners' words into xh[0 .. H)
template <class T>
__device__ __forceinline__ void load_halo(Fixed &S, const Shape &h, const int32_t *hcol, const uint64_t *buf,
                                          uint32_t tag, T *xh, int *g_abort) {
    constexpr int U = 4;
    volatile int *sa = &S.abort;
    for (int b = threadIdx.x < PT ? (int)threadIdx.x : h.H; b < h.H; b += U * PT) {
        const uint64_t *p[U];
        unsigned pending = 0;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int q = b + u * PT;
            p[u] = buf;
            if (q < h.H) {
                p[u] = buf + (sizeof(T) == 4 ? (size_t)hcol[q] : (size_t)hcol[q] * 2);
                pending |= 1u << u;
            }
        }
        unsigned spins = 0;
        while (pending) {
            uint64_t a[U], c[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (pending >> u & 1u) {
                    if (sizeof(T) == 4) a[u] = c[u] = get1(p[u]);
                    else get2(p[u], a[u], c[u]);
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if ((pending >> u & 1u) && (uint32_t)(a[u] >> 32) == tag && (uint32_t)(c[u] >> 32) == tag) {
                    if constexpr (sizeof(T) == 4) xh[b + u * PT] = __uint_as_float((uint32_t)a[u]);
                    else xh[b + u * PT] = __hiloint2double((int)(uint32_t)c[u], (int)(uint32_t)a[u]);
                    pending &= ~(1u << u);
                }
            }
            if (pending && !keep_waiting(spins, sa, g_abort)) break;
        }
    }
}

__device__ __forceinline__ void publish(uint64_t *buf, int row, float v, uint32_t tag) {
    put1(buf + row, __float_as_uint(v), tag);
}
__device__ __forceinline__ void publish(uint64_t *buf, int row, double v, uint32_t tag) {
    put2(buf + (size_t)row * 2, Acc<double>::bits(v), tag);
}

// rotation that takes (a, b) to (r, 0), b2 = b^2: one reciprocal square root
__device__ __forceinline__ void rotation(double a, double b, double b2, double &c, double &s, double &r) {
    const double r2 = fma(a, a, b2);
    const double ir = r2 > 0.0 ? rsqrt(r2) : 0.0;
    r = r2 * ir;
    c = r2 > 0.0 ? a * ir : 1.0;
    s = b * ir;
}

// DCGS2 (see k_dcgs_dots of the launched form): S.res holds s (j), t (j),
// q.q, q.w, q.w, w.w.  What the next step's vectors need, by warp 0; the
// rotations follow in dcgs_rotate.
__device__ __forceinline__ void dcgs_scalars(Fixed &S, int j) {
    const int tid = threadIdx.x;
    if (tid < 32) {
        const double s = tid < j ? S.res[tid] : 0.0, t = tid < j ? S.res[j + 2 + tid] : 0.0;
        const double ss = warp_acc<Acc<double>>(s * s), st = warp_acc<Acc<double>>(s * t),
                     tt = warp_acc<Acc<double>>(t * t);
        const double alpha = S.res[j], beta = S.res[2 * j + 2], gamma = S.res[2 * j + 3];
        const double nu2 = j > 0 ? fmax(alpha - ss, 0.0) : 1.0;
        const double inu = nu2 > 0.0 ? rsqrt(nu2) : 0.0;
        const double tau = (beta - st) * inu;
        const double nut2 = fmax(gamma - tt - tau * tau, 0.0);
        const double inv = nut2 > 0.0 ? rsqrt(nut2) : 0.0;
        S.colp[tid] = fma(S.nut, s, S.h1[tid]);   // column j - 1 before its rotations
        S.colc[tid] = tid == j ? tau : t;
        __syncwarp();
        S.h1[tid] = tid == j ? tau : t;
        S.f1[tid] = (float)(tid == j ? tau : t);
        S.f2[tid] = (float)s;
        if (tid == 0) {
            S.colp[j] = S.nut * (nu2 * inu);
            S.nu = nu2 * inu;
            S.inu = inu;
            S.nut = nut2 * inv;
            S.nut2 = nut2;
            S.inv = inv;
        }
    }
    __syncthreads();
}

// State of the scalar warp over a cycle: lane k holds entry k of the open row
// of the rotations' product; g the open entry of the rotated right-hand side.
struct Rot {
    double t, g;
};

// the dot of the open row with a column, the rotation against the subdiagonal
// entry b (b2 = b^2), and the column's diagonal entry
__device__ __forceinline__ void rotate_column(Fixed &S, const Rot &q, int j, double colk, double b, double b2,
                                              double &c, double &s) {
    const double carry = warp_acc<Acc<double>>(q.t * colk);
    double r;
    rotation(carry, b, b2, c, s, r);
    const int lane = threadIdx.x & 31;
    if (lane <= j) S.H[j * (j + 1) / 2 + lane] = colk;
    if (lane == 0) {
        S.rd[j] = r;
        S.g[j] = c * q.g;
    }
}
__device__ __forceinline__ void close_row(Fixed &S, Rot &q, int j, double c, double s) {
    const int lane = threadIdx.x & 31;
    S.W[j * 32 + lane] = lane == j + 1 ? s : c * q.t;
    q.t = lane == j + 1 ? c : -s * q.t;
    q.g = -s * q.g;
}

// The rest of a DCGS2 step, by the scalar warp while the others go on: column
// j - 1 gets its rotation for good, column j a tentative one whose |g[j + 1]|
// is the stopping test.  S.done is read after the next exchange's barrier.
__device__ __noinline__ void dcgs_rotate(Fixed &S, Rot &q, int j, double thr) {
    const int lane = threadIdx.x & 31;
    double c, s;
    if (j > 0) {
        const double b = S.colp[j];
        rotate_column(S, q, j - 1, lane < j ? S.colp[lane] : 0.0, b, b * b, c, s);
        close_row(S, q, j - 1, c, s);
    }
    rotate_column(S, q, j, lane <= j ? S.colc[lane] : 0.0, S.nut, S.nut2, c, s);
    if (lane == 0) S.done = fabs(s * q.g) <= thr || S.nut2 == 0.0 || S.nu == 0.0 || S.stop;
}

// CGS2: h1 first projection, S.res = h2 (j + 1 values) and ||w'||^2
__device__ __forceinline__ void cgs_scalars(Fixed &S, int j) {
    const int tid = threadIdx.x;
    if (tid < 32) {
        const double h2 = tid <= j ? S.res[tid] : 0.0;
        const double hn2 = fmax(S.res[j + 1] - warp_acc<Acc<double>>(h2 * h2), 0.0);
        const double inv = hn2 > 0.0 ? rsqrt(hn2) : 0.0;
        S.h2[tid] = h2;
        S.colc[tid] = tid <= j ? S.h1[tid] + h2 : 0.0;
        if (tid == 0) {
            S.inv = inv;
            S.nut = hn2 * inv;
            S.nut2 = hn2;
        }
    }
    __syncthreads();
}

__device__ __noinline__ void cgs_rotate(Fixed &S, Rot &q, int j, double thr) {
    const int lane = threadIdx.x & 31;
    double c, s;
    rotate_column(S, q, j, lane <= j ? S.colc[lane] : 0.0, S.nut, S.nut2, c, s);
    close_row(S, q, j, c, s);
    if (lane == 0) S.done = fabs(q.g) <= thr || S.nut2 == 0.0 || S.stop;
}

// Dots of nv vectors (vec(k), k < nv) with x (and, Two, y): LPV lanes per
// vector, several parts of the rows per vector while there are groups left
// (a warp per vector would spend more FP64 instructions on its shuffle tree
// than on a small block's rows).  Results in S.val[k] and S.val[nv + k].
// FP32 terms are added RUN at a time before the run enters the pair (the
// launched kernels' chains: a lane has up to 256 terms here, and a plain chain of
// them carries an error that grows with it).
// Every thread of the block calls it; the caller's grid_sum is the barrier.
constexpr int RUN = 8;
template <class T, bool Two, class F>
__device__ __forceinline__ void block_dots(Fixed &S, int nv, int R, F vec, const T *x, const T *y) {
    typedef Acc<T> A;
    const int tid = threadIdx.x, lane = tid & 31, gl = lane & (LPV - 1), grp = tid / LPV;
    // FP64: no more parts than latency asks for, every part costs a shuffle tree
    int parts = (sizeof(T) == 8 ? NGRP / 4 : NGRP) / nv;
    if (parts > 8) parts = 8;
    if (parts < 1) parts = 1;
    for (int t0 = 0; t0 < nv * parts; t0 += NGRP) {
        const int t = t0 + grp;
        const bool on = tid < PT && t < nv * parts;
        typename A::type b0 = A::zero(), b1 = A::zero();
        if (on) {
            const int k = t % nv, part = t / nv;
            const T *vk = vec(k);
            const int step = LPV * parts;
            if constexpr (sizeof(T) == 4) {
                for (int r = gl + LPV * part; r < R; r += RUN * step) {
                    T x0 = (T)0, x1 = (T)0;
#pragma unroll
                    for (int u = 0; u < RUN; ++u) {
                        const int e = r + u * step;
                        const T v = e < R ? vk[e] : (T)0;
                        x0 = fma(v, x[e < R ? e : r], x0);
                        if (Two) x1 = fma(v, y[e < R ? e : r], x1);
                    }
                    b0 = A::add(b0, A::of(x0));
                    if (Two) b1 = A::add(b1, A::of(x1));
                }
            } else {
                T x0 = (T)0, x1 = (T)0;
#pragma unroll 8
                for (int r = gl + LPV * part; r < R; r += step) {
                    const T v = vk[r];
                    x0 = fma(v, x[r], x0);
                    if (Two) x1 = fma(v, y[r], x1);
                }
                b0 = A::of(x0);
                if (Two) b1 = A::of(x1);
            }
        }
        if (tid < PT) {
#pragma unroll
            for (int o = LPV / 2; o > 0; o >>= 1) {
                b0 = A::add(b0, A::shfl(b0, o));
                if (Two) b1 = A::add(b1, A::shfl(b1, o));
            }
        }
        if (on && gl == 0) {
            if (parts > 1) {
                S.part[t] = A::bits(b0);
                if (Two) S.part[NGRP + t] = A::bits(b1);
            } else {
                S.val[t] = A::bits(b0);
                if (Two) S.val[nv + t] = A::bits(b1);
            }
        }
    }
    if (parts > 1) {   // nv * parts <= NGRP here
        __syncthreads();
        if (tid < (Two ? 2 * nv : nv)) {
            const uint2 *q = tid < nv ? S.part + tid : S.part + NGRP + tid - nv;
            typename A::type s = A::zero();
            for (int i = 0; i < parts; ++i) s = A::add(s, A::from(q[nv * i]));
            S.val[tid] = A::bits(s);
        }
    }
}

// Matrix storage of a block: sweeps of the mixed polynomial form read a word
// of FP16 value and 16-bit index; the other forms a value and an index.
template <class T, bool POLY> struct Mat;
template <> struct Mat<float, true> {
    static constexpr int entry_bytes = 4;
    uint32_t *w;
    __device__ __forceinline__ void at(unsigned char *base, int64_t E) { w = reinterpret_cast<uint32_t *>(base); (void)E; }
    __device__ __forceinline__ void set(int64_t e, int64_t g, uint32_t ix, const ResidentArgs &a) {
        w[e] = (uint32_t)__half_as_ushort(a.val16[g]) << 16 | ix;
    }
    __device__ __forceinline__ int idx(int64_t e) const { return (int)(w[e] & 0xFFFFu); }
    __device__ __forceinline__ float sweep_val(int64_t e, int &ix) const {
        const uint32_t v = w[e];
        ix = (int)(v & 0xFFFFu);
        return __half2float(__ushort_as_half((unsigned short)(v >> 16)));
    }
    // products use the FP32 values, streamed from L2 once per step
    __device__ __forceinline__ float val(int64_t e, int64_t e0, const ResidentArgs &a) const { return __ldg(a.val32 + e0 + e); }
};
template <bool POLY> struct Mat<float, POLY> {
    static constexpr int entry_bytes = 6;
    float *v;
    uint16_t *ix_;
    __device__ __forceinline__ void at(unsigned char *base, int64_t E) {
        v = reinterpret_cast<float *>(base);
        ix_ = reinterpret_cast<uint16_t *>(base + E * 4);
    }
    __device__ __forceinline__ void set(int64_t e, int64_t g, uint32_t ix, const ResidentArgs &a) {
        v[e] = a.val32[g];
        ix_[e] = (uint16_t)ix;
    }
    __device__ __forceinline__ int idx(int64_t e) const { return ix_[e]; }
    __device__ __forceinline__ float sweep_val(int64_t e, int &ix) const { ix = ix_[e]; return v[e]; }
    __device__ __forceinline__ float val(int64_t e, int64_t, const ResidentArgs &) const { return v[e]; }
};
template <bool POLY> struct Mat<double, POLY> {
    static constexpr int entry_bytes = 10;
    double *v;
    uint16_t *ix_;
    __device__ __forceinline__ void at(unsigned char *base, int64_t E) {
        v = reinterpret_cast<double *>(base);
        ix_ = reinterpret_cast<uint16_t *>(base + E * 8);
    }
    __device__ __forceinline__ void set(int64_t e, int64_t g, uint32_t ix, const ResidentArgs &a) {
        v[e] = a.val64[g];
        ix_[e] = (uint16_t)ix;
    }
    __device__ __forceinline__ int idx(int64_t e) const { return ix_[e]; }
    __device__ __forceinline__ double sweep_val(int64_t e, int &ix) const { ix = ix_[e]; return v[e]; }
    __device__ __forceinline__ double val(int64_t e, int64_t, const ResidentArgs &) const { return v[e]; }
};

__device__ __forceinline__ unsigned char *carve(unsigned char *&p, size_t bytes) {
    unsigned char *q = p;
    p += (bytes + 15) & ~(size_t)15;
    return q;
}

// w -= V h over nv basis vectors, own rows
template <class T>
__device__ __forceinline__ void project(const T *h_, const Shape &h, int nv, const T *V, int64_t ldv, T *wv, int t0) {
    for (int r = t0; r < h.R; r += PT) {
        T b = wv[r];
#pragma unroll 8
        for (int k = 0; k < nv; ++k) b = fma(-V[(int64_t)k * ldv + r], h_[k], b);
        wv[r] = b;
    }
}

// Start of step j >= 1.  FP32 (DCGS2): v_{j-1} = (q_{j-1} - V s) inu finished
// in slot j - 1, the tentative q_j = (w - V h1) inv.  FP64 (CGS2):
// v_j = (w' - V h2) inv in slot j.  qv gets q_j (v_j).
template <class T>
__device__ __forceinline__ void update_vectors(Fixed &S, const Shape &h, int j, T *V, int64_t ldv, T *qv, T *wv,
                                               int t0) {
    if constexpr (sizeof(T) == 4) {
        const int pj = j - 1;
        const float inu = (float)S.inu, inut = (float)S.inv;
        for (int r = t0; r < h.R; r += PT) {
            float aq = qv[r], bw = wv[r];
#pragma unroll 8
            for (int k = 0; k < pj; ++k) {
                const float x = V[(int64_t)k * ldv + r];
                aq = fmaf(-x, S.f2[k], aq);
                bw = fmaf(-x, S.f1[k], bw);
            }
            if (pj > 0) {
                aq *= inu;
                V[(int64_t)pj * ldv + r] = aq;
            }
            bw = fmaf(-aq, S.f1[pj], bw);
            qv[r] = bw * inut;
        }
    } else {
        const double inv = S.inv;
        for (int r = t0; r < h.R; r += PT) {
            double bw = wv[r];
#pragma unroll 8
            for (int k = 0; k < j; ++k) bw = fma(-V[(int64_t)k * ldv + r], S.h2[k], bw);
            bw *= inv;
            qv[r] = bw;
            V[(int64_t)j * ldv + r] = bw;
        }
    }
}

// One solve (or the part of it that fits the step budget).  The exchanges and
// sums are numbered from a.in->tag0; no number is used twice with the same
// words.
template <class T, bool POLY>
__global__ void __launch_bounds__(PB, 1) k_gmres_resident(ResidentArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    Fixed &S = *reinterpret_cast<Fixed *>(smem);
    typedef Acc<T> A;
    typedef Acc<double> A64;
    const ResidentIn in = *a.in;
    int *g_abort = &a.out->abort;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int t0 = tid < PT ? tid : 1 << 30;   // first row (entry, word) of a worker; none for the scalar warp
    Shape h;
    const int s0 = blockIdx.x * a.spc, s1 = min(s0 + a.spc, a.nsl), ns = s1 - s0;
    h.n = a.n;
    h.r0 = s0 * 32;
    h.Rp = ns * 32;
    h.R = min(h.r0 + h.Rp, a.n) - h.r0;
    h.e0 = (int64_t)a.so[s0] * 32;
    const int64_t E = ((int64_t)a.so[s1 - 1] + a.sw[s1 - 1]) * 32 - h.e0;
    if (tid < ns) {
        S.ssb[tid] = (uint32_t)((int64_t)a.so[s0 + tid] * 32 - h.e0);
        S.ssw[tid] = a.sw[s0 + tid];
    }
    if (tid == 0) { S.abort = 0; S.stop = 0; S.done = 0; }
    unsigned char *mbase = smem + ((sizeof(Fixed) + 15) & ~(size_t)15);
    unsigned char *rest = mbase + (((size_t)E * Mat<T, POLY>::entry_bytes + 15) & ~(size_t)15);
    unsigned char *end = smem + a.smem;
    // ---- the halo: a bitmap of the columns outside the block's rows, ranked
    const int W = (a.n + 31) >> 5;
    uint32_t *bm = reinterpret_cast<uint32_t *>(end) - W;
    uint16_t *pre = reinterpret_cast<uint16_t *>(bm) - ((W + 1) & ~1);
    bool ok = rest + 64 <= reinterpret_cast<unsigned char *>(pre);
    h.H = 0;
    int32_t *hcol = reinterpret_cast<int32_t *>(rest);
    __syncthreads();
    if (ok) {
        for (int i = t0; i < W; i += PT) bm[i] = 0u;
        __syncthreads();
        for (int64_t e = t0; e < E; e += PT) {
            const int cidx = a.col[h.e0 + e];
            if (cidx < h.r0 || cidx >= h.r0 + h.R) atomicOr(&bm[cidx >> 5], 1u << (cidx & 31));
        }
        __syncthreads();
        const int per = (W + PT - 1) / PT, lo = tid < PT ? min(tid * per, W) : W, hi = min(lo + per, W);
        uint32_t cnt = 0;
        for (int i = lo; i < hi; ++i) cnt += __popc(bm[i]);
        uint32_t inc = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        if (lane == 31 && wid < PW) S.wtot[wid] = inc;
        __syncthreads();
        uint32_t base = inc - cnt;
        for (int q = 0; q < wid && q < PW; ++q) base += S.wtot[q];
        if (tid == PT - 1) S.halo = (int)(base + cnt);
        __syncthreads();
        h.H = S.halo;
        // room for the halo list beside the bitmap, and for the vectors after it
        const size_t xs = ((size_t)h.Rp + h.H + 3) & ~(size_t)3;
        ok = h.Rp + h.H <= 65535 && rest + ((size_t)h.H * 4 + 16) <= reinterpret_cast<unsigned char *>(pre) &&
             rest + ((size_t)h.H * 4 + 16) + (2 * xs + 2 * (size_t)h.Rp) * sizeof(T) + 64 <= end;
        if (ok) {
            uint32_t p = base;
            for (int i = lo; i < hi; ++i) {
                pre[i] = (uint16_t)p;
                uint32_t m = bm[i];
                while (m) {
                    hcol[p++] = i * 32 + __ffs(m) - 1;
                    m &= m - 1;
                }
            }
        }
        __syncthreads();
    }
    Mat<T, POLY> M;
    M.at(mbase, E);
    if (ok) {
        for (int64_t e = t0; e < E; e += PT) {
            const int cidx = a.col[h.e0 + e];
            uint32_t ix;
            if (cidx >= h.r0 && cidx < h.r0 + h.R) ix = (uint32_t)(cidx - h.r0);
            else ix = (uint32_t)(h.Rp + pre[cidx >> 5] + __popc(bm[cidx >> 5] & ((1u << (cidx & 31)) - 1u)));
            M.set(e, h.e0 + e, ix, a);
        }
    }
    __syncthreads();   // the bitmap's room is free now
    uint32_t rtag = in.tag0, xtag = in.tag0, utag = in.tag0;
    if (tid == 0) S.val[0] = A64::bits(ok ? 0.0 : 1.0);
    grid_sum<A64>(S, 1, a.red, ++rtag, g_abort);
    if (S.res[0] != 0.0 || S.stop) {   // some block does not fit: the same answer in every block
        if (blockIdx.x == 0 && tid == 0) a.out->status = S.stop ? RES_TIMEOUT : RES_UNFIT;
        return;
    }
    unsigned char *p = rest;
    carve(p, (size_t)h.H * 4);
    const size_t xs = ((size_t)h.Rp + h.H + 3) & ~(size_t)3;
    T *X = reinterpret_cast<T *>(carve(p, 2 * xs * sizeof(T)));
    T *qv = reinterpret_cast<T *>(carve(p, (size_t)h.Rp * sizeof(T)));
    T *wv = reinterpret_cast<T *>(carve(p, (size_t)h.Rp * sizeof(T)));
    double *ud = reinterpret_cast<double *>(X);   // the FP64 iterate, own rows and halo, in the residual phase
    // basis: in shared memory while there is room, else in global memory (own rows only, either way)
    T *V = reinterpret_cast<T *>(a.V) + h.r0, *Z = reinterpret_cast<T *>(a.Z) + h.r0;
    int64_t ldv = a.ldv, ldz = a.ldv;
    const bool zsep = a.Z != a.V;
    const int lds = h.Rp + 32 / (int)sizeof(T) * 2;   // 64 bytes past a multiple of 128: vectors start in other banks
    if (p + (size_t)(a.m + 1) * lds * sizeof(T) + 32 <= end) {
        V = reinterpret_cast<T *>(carve(p, (size_t)(a.m + 1) * lds * sizeof(T)));
        ldv = lds;
        if (!zsep) { Z = V; ldz = ldv; }
    }
    if (zsep && p + (size_t)a.m * lds * sizeof(T) + 32 <= end) {
        Z = reinterpret_cast<T *>(carve(p, (size_t)a.m * lds * sizeof(T)));
        ldz = lds;
    }
    for (int r = h.R + min(t0, h.Rp); r < h.Rp; r += PT) { qv[r] = (T)0; wv[r] = (T)0; X[r] = (T)0; X[xs + r] = (T)0; }

    const bool timed = a.timing && blockIdx.x == 0 && tid == 0;
    unsigned long long last = 0, ns_[RES_KINDS];
    unsigned cn_[RES_KINDS];
#pragma unroll
    for (int i = 0; i < RES_KINDS; ++i) { ns_[i] = 0; cn_[i] = 0; }
#define RES_MARK(kind)                                                     \
    do {                                                                   \
        if (timed) {                                                       \
            unsigned long long now_;                                       \
            asm volatile("mov.u64 %0, %globaltimer;" : "=l"(now_));        \
            if ((kind) >= 0) { ns_[(kind) < 0 ? 0 : (kind)] += now_ - last; cn_[(kind) < 0 ? 0 : (kind)]++; } \
            last = now_;                                                   \
        }                                                                  \
    } while (0)

    double *u = a.u + h.r0;
    double bb = 0.0;
    for (int r = t0; r < h.R; r += PT) {
        u[r] = in.resume ? u[r] : in.x[h.r0 + r] * a.d[h.r0 + r];
        const double bv = in.b[h.r0 + r];
        bb = fma(bv, bv, bb);
    }
    block_sum<A64>(S, bb, 1);
    int iters = 0, cycles = 0, status = RES_MAXITER;
    long long sumj = 0;
    double bnorm = 0.0, beta = 0.0;
    RES_MARK(-1);
    for (;;) {
        // ---- r = b - Ahat u in FP64
        ++utag;
        for (int r = t0; r < h.R; r += PT) {
            const double v = u[r];
            ud[r] = v;
            publish(a.ull, h.r0 + r, v, utag);
        }
        load_halo<double>(S, h, hcol, a.ull, utag, ud + h.Rp, g_abort);
        __syncthreads();
        double rr = 0.0;
        for (int r = t0; r < h.R; r += PT) {
            const int w = (int)S.ssw[r >> 5];
            const int64_t eb = S.ssb[r >> 5] + (r & 31);
            double acc = 0.0;
#pragma unroll 4
            for (int k = 0; k < w; ++k) {
                const int64_t e = eb + (int64_t)k * 32;
                const double v = sizeof(T) == 8 ? (double)M.val(e, h.e0, a) : __ldg(a.val64 + h.e0 + e);
                acc = fma(v, ud[M.idx(e)], acc);
            }
            const double res = in.b[h.r0 + r] - acc;
            rr = fma(res, res, rr);
            if constexpr (sizeof(T) == 8) wv[r] = res;
            else u[a.ldv + r] = res;   // kept in FP64 until beta is known (second row of the iterate's buffer)
        }
        block_sum<A64>(S, rr, 0);
        grid_sum<A64>(S, cycles == 0 ? 2 : 1, a.red, ++rtag, g_abort);
        if (cycles == 0) bnorm = sqrt(S.res[1]);
        beta = sqrt(S.res[0]);
        RES_MARK(RES_SPMV);
        if (S.stop) { status = RES_TIMEOUT; break; }
        if (bnorm == 0.0 || beta <= in.rtol * bnorm) { status = RES_OK; break; }
        if (iters >= in.max_iter) break;
        if (iters >= STEP_BUDGET) { status = RES_MORE; break; }
        double thr = in.rtol * bnorm;
        if (sizeof(T) == 4) {
            // FP32 cycle: to what the outer tolerance still needs, at most four digits
            double inner = 0.5 * in.rtol * bnorm / beta;
            if (inner < 1e-4) inner = 1e-4;
            thr = inner * beta;
        }
        const int jmax = min(a.m, in.max_iter - iters);
        const double ib = 1.0 / beta;
        if (tid == 0) S.done = 0;
        Rot rot{lane == 0 ? 1.0 : 0.0, beta};
        for (int r = t0; r < h.R; r += PT) {
            T q;
            if constexpr (sizeof(T) == 8) q = wv[r] * ib;
            else q = (float)u[a.ldv + r] * (float)ib;
            qv[r] = q;
            V[r] = q;
        }
        int je = 0;
        for (int j = 0; j < jmax; ++j) {
            // ---- q_j (tentative, FP32) or v_j (FP64), own rows in qv
            if (j > 0) update_vectors<T>(S, h, j, V, ldv, qv, wv, t0);
            RES_MARK(j > 0 ? RES_UPDNORM : -1);
            // ---- z = p(Ahat) q_j, w = Ahat z
            ++xtag;
            T *xa = X, *xb = X + xs;
            const size_t bstride = (size_t)a.n * (sizeof(T) / 4);
            const T om = (T)in.omega;
            T *Zj = Z + (int64_t)j * ldz;
            for (int r = t0; r < h.R; r += PT) {
                const T z = POLY ? om * qv[r] : qv[r];
                xa[r] = z;
                publish(a.xll, h.r0 + r, z, xtag);
                if (!POLY && zsep) Zj[r] = z;
            }
            load_halo<T>(S, h, hcol, a.xll, xtag, xa + h.Rp, g_abort);
            __syncthreads();
            if (S.done) break;   // the test of step j - 1, decided meanwhile by the scalar warp
            if (POLY) {
                for (int i = 1; i < a.pdeg; ++i) {
                    for (int r = t0; r < h.R; r += PT) {
                        const int w = (int)S.ssw[r >> 5];
                        const int eb = (int)S.ssb[r >> 5] + (r & 31);
                        T acc = (T)0;
#pragma unroll 8
                        for (int k = 0; k < w; ++k) {
                            int ix;
                            const T v = M.sweep_val(eb + k * 32, ix);
                            acc = fma(v, xa[ix], acc);
                        }
                        const T y = fma(om, qv[r] - acc, xa[r]);
                        xb[r] = y;
                        publish(a.xll + i * bstride, h.r0 + r, y, xtag);
                        if (i + 1 == a.pdeg) Zj[r] = y;
                    }
                    T *t = xa; xa = xb; xb = t;
                    load_halo<T>(S, h, hcol, a.xll + i * bstride, xtag, xa + h.Rp, g_abort);
                    __syncthreads();
                }
                RES_MARK(RES_SWEEP);
            }
            for (int r = t0; r < h.R; r += PT) {
                const int w = (int)S.ssw[r >> 5];
                const int eb = (int)S.ssb[r >> 5] + (r & 31);
                T acc = (T)0;
#pragma unroll 8
                for (int k = 0; k < w; ++k) {
                    const int e = eb + k * 32;
                    acc = fma(M.val(e, h.e0, a), xa[M.idx(e)], acc);
                }
                wv[r] = acc;
            }
            __syncthreads();
            RES_MARK(RES_SPMV);
            // ---- Gram-Schmidt
            if constexpr (sizeof(T) == 4) {
                // s = V^T q, t = V^T w and, as two more vectors, q and w themselves
                block_dots<T, true>(S, j + 2, h.R, [&](int k) -> const T * {
                    return k < j ? V + (int64_t)k * ldv : (k == j ? qv : wv);
                }, qv, wv);
                grid_sum<A>(S, 2 * j + 4, a.red, ++rtag, g_abort);
                dcgs_scalars(S, j);
                if (wid == PW) dcgs_rotate(S, rot, j, thr);
                RES_MARK(RES_DOT);
            } else {
                block_dots<T, false>(S, j + 1, h.R, [&](int k) -> const T * { return V + (int64_t)k * ldv; }, wv, wv);
                grid_sum<A>(S, j + 1, a.red, ++rtag, g_abort);
                if (tid <= j) S.h1[tid] = S.res[tid];
                __syncthreads();
                RES_MARK(RES_DOT);
                project<T>(S.h1, h, j + 1, V, ldv, wv, t0);   // w -= V h1
                __syncthreads();
                block_dots<T, false>(S, j + 2, h.R, [&](int k) -> const T * {
                    return k <= j ? V + (int64_t)k * ldv : wv;
                }, wv, wv);
                grid_sum<A>(S, j + 2, a.red, ++rtag, g_abort);
                cgs_scalars(S, j);
                if (wid == PW) cgs_rotate(S, rot, j, thr);
                RES_MARK(RES_UPDDOT);
            }
            sumj += j;
            je = j + 1;
        }
        __syncthreads();   // the scalar warp's last rotation
        // ---- cycle end: the triangular factor R = W H, R y = g by one warp, u += Z y
        for (int t = tid; t < je * (je - 1) / 2; t += PB) {
            int k = (int)((1.0f + sqrtf(8.0f * t + 1.0f)) * 0.5f);   // column k holds entries k (k - 1) / 2 ..
            while (k * (k - 1) / 2 > t) --k;
            while (k * (k + 1) / 2 <= t) ++k;
            const int i = t - k * (k - 1) / 2;
            const double *hk = S.H + k * (k + 1) / 2, *wi = S.W + i * 32;
            double v = 0.0;
            for (int e = 0; e <= i + 1; ++e) v = fma(wi[e], hk[e], v);
            S.Rm[t] = v;
        }
        __syncthreads();
        if (wid == 0) {
            double gi = lane < je ? S.g[lane] : 0.0;   // je <= 31
            for (int k = je - 1; k >= 0; --k) {
                const double yk = __shfl_sync(0xffffffffu, gi, k) / S.rd[k];
                if (lane == k) {
                    S.y[k] = yk;
                    S.fy[k] = (float)yk;
                }
                if (lane < k) gi = fma(-S.Rm[k * (k - 1) / 2 + lane], yk, gi);
            }
        }
        __syncthreads();
        for (int r = t0; r < h.R; r += PT) {
            T s = (T)0;
#pragma unroll 8
            for (int k = 0; k < je; ++k) s = fma(Z[(int64_t)k * ldz + r], coef_y<T>(S)[k], s);
            u[r] += (double)s;
        }
        iters += je;
        ++cycles;
        RES_MARK(RES_CYCLE);
    }
    for (int r = t0; r < h.R; r += PT) in.x[h.r0 + r] = u[r] / a.d[h.r0 + r];
    if (blockIdx.x == 0 && tid == 0) {
        ResidentOut *o = a.out;
        o->status = status;
        o->iters = iters;
        o->cycles = cycles;
        o->relres = bnorm > 0.0 ? beta / bnorm : 0.0;
        o->sumj = sumj;
        for (int i = 0; i < RES_KINDS; ++i) { o->ns[i] = ns_[i]; o->count[i] = cn_[i]; }
    }
#undef RES_MARK
}

template <class T, bool POLY>
const void *kernel_of() { return reinterpret_cast<const void *>(&k_gmres_resident<T, POLY>); }

const void *pick_kernel(bool mixed, bool poly) {
    if (mixed) return poly ? kernel_of<float, true>() : kernel_of<float, false>();
    return poly ? kernel_of<double, true>() : kernel_of<double, false>();
}


}  // namespace

// Fewest rows of a block: more blocks shorten the FP64 arithmetic of a block
// (two FP64 lanes per clock and SM), but lengthen the sums over blocks.  1471
// nodes, FP64 Jacobi: 1.08-1.12 ms at 32, 64 or 128 rows; mixed: 0.49 ms at 64
// and 128, 0.51 at 256.
constexpr int MIN_ROWS_F64 = 32, MIN_ROWS_F32 = 128;

// slices per block and grid of a resident solve of n rows on this device
void resident_grid(const apcloud_ctx *c, int *spc, int *grid) {
    const int n = c->n_tot;
    int sms = 0, dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms < 1) sms = 1;
    const int nsl = div_up(n, 32);
    int s = div_up(nsl, sms);
    s = std::max(s, (c->P.precision == 0 ? MIN_ROWS_F64 : MIN_ROWS_F32) / 32);
    *spc = s;
    *grid = div_up(nsl, s);
}

int64_t resident_red_words(int grid) { return (int64_t)2 * RED_SLOTS * (grid + 1) * 2; }

bool resident_ok(const apcloud_ctx *c, int which) {
    if (c->nbeams > 1 || c->P.restart > PM || c->ilu_which == which || c->n_tot < 1 || c->res_unfit) return false;
    int spc = 0, grid = 0, lim = 0, coop = 0, dev = 0;
    resident_grid(c, &spc, &grid);
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&lim, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (!coop || spc > PSL) return false;
    // the average block has to fit with room for its vectors; the kernel checks the exact sizes
    const int eb = c->P.precision == 0 ? 10 : (c->P.poly_degree > 1 ? 4 : 6);
    const double mat = (double)c->ell_entries / c->n_slices * spc * eb;
    return sizeof(Fixed) + mat + 6.0 * ((c->n_tot + 31) / 32) + 128.0 <= (double)lim;
}

// Launches the solve on prepared buffers and waits for it; *out receives what
// it reports.  graph: replay as a CUDA graph (one kernel node), keyed by the
// buffers.
static apcloud_status run_resident(apcloud_ctx *c, ResidentArgs a, const ResidentIn &in, int grid, bool graph,
                                   ResidentOut *out) {
    const bool mixed = c->P.precision == 1, poly = a.pdeg > 1;
    const void *kern = pick_kernel(mixed, poly);
    int lim = 0, dev = 0;
    APC_CUDA(c, cudaGetDevice(&dev));
    APC_CUDA(c, cudaDeviceGetAttribute(&lim, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    APC_CUDA(c, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, lim));
    a.smem = lim;
    APC_CUDA(c, cudaMemcpyAsync(const_cast<ResidentIn *>(a.in), &in, sizeof in, cudaMemcpyHostToDevice, c->s));
    APC_CUDA(c, cudaMemsetAsync(a.out, 0, sizeof(ResidentOut), c->s));
    timer_close(c);
    bool unfit = false;
    auto launch = [&]() -> apcloud_status {
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeCooperative;
        at[0].val.cooperative = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)grid);
        cfg.blockDim = dim3(PB);
        cfg.dynamicSmemBytes = (size_t)lim;
        cfg.stream = c->s;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        void *args[1] = {&a};
        const cudaError_t e = cudaLaunchKernelExC(&cfg, kern, args);
        if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported) {
            // fewer SMs than the device reports (a partition of it): the launched kernels take over
            cudaGetLastError();
            unfit = true;
            return c->capturing ? APCLOUD_E_CUDA : APCLOUD_OK;   // an empty capture is discarded
        }
        APC_CUDA(c, e);
        if (c->capturing) count_captured(c);
        else c->launches++;
        return APCLOUD_OK;
    };
    bool launched = false;
    if (graph && c->graphs_on && c->timer.mask == 0) {
        GraphKey key;
        memset(&key, 0, sizeof key);
        key.tsize = mixed ? 4 : 8;
        key.n = a.n;
        key.pdeg = a.pdeg;
        key.nblk = grid;
        key.ldv = a.ldv;
        key.spmv_bs = a.m;
        key.skeep = a.spc;
        const void *p[] = {kern, a.sw, a.so, a.col, a.val64, a.val32, a.val16, a.d, a.u, a.V, a.Z, a.xll, a.ull,
                           a.red, a.in, a.out};
        for (size_t i = 0; i < sizeof p / sizeof p[0]; ++i) key.p[i] = p[i];
        GraphEntry *g = find_graph(c, key);
        if (!g) {
            g = begin_capture(c, key);
            if (g) {
                const apcloud_status st = launch();
                g = end_capture(c, g, st);
            }
        }
        if (g) {
            APC_TRY(launch_graph(c, g));
            c->last_stepped = nullptr;
            launched = true;
        }
    }
    if (!launched) APC_TRY(launch());
    if (unfit) {
        out->status = RES_UNFIT;
        return APCLOUD_OK;
    }
    APC_TRY(read_back(c, out, a.out, sizeof *out));
    if (c->timer.mask) {
        static const int kinds[RES_KINDS] = {K_SPMV, K_SWEEP, K_DOT, K_UPDDOT, K_UPDNORM, K_CYCLE};
        for (int i = 0; i < RES_KINDS; ++i) {
            if (!(c->timer.mask >> kinds[i] & 1u)) continue;
            c->timer.ms[kinds[i]] += (double)out->ns[i] * 1e-6;
            c->timer.launches[kinds[i]] += out->count[i];
        }
        // algorithmic traffic, as for the launched kernels
        const double vb = mixed ? 4.0 : 8.0, dn = a.n, it = out->iters, cy = out->cycles,
                     nnz = (double)c->sum_m + c->n_int + c->n_bnd, sj = (double)out->sumj;
        account(c, K_SPMV, ((vb + 2.0) * nnz + 2.0 * vb * dn) * it + (10.0 * nnz + 16.0 * dn) * (cy + 1.0),
                2.0 * nnz * (it + cy + 1.0));
        if (poly) {
            const double sw = (a.pdeg - 1.0) * it;
            account(c, K_SWEEP, ((mixed ? 4.0 : 10.0) * nnz + 3.0 * vb * dn) * sw, 2.0 * nnz * sw);
        }
        if (mixed) {
            account(c, K_DOT, vb * dn * (sj + 2.0 * it), dn * (4.0 * sj + 6.0 * it));
            account(c, K_UPDNORM, vb * dn * (sj + 3.0 * (it - cy)), 4.0 * dn * sj);
        } else {
            account(c, K_DOT, vb * dn * (sj + 2.0 * it), 2.0 * dn * (sj + it));
            account(c, K_UPDDOT, vb * dn * (sj + 3.0 * it), dn * (4.0 * (sj + it) + 2.0 * it));
            account(c, K_UPDNORM, vb * dn * (sj + 3.0 * (it - cy)), 2.0 * dn * (sj + it));
        }
        account(c, K_CYCLE, vb * dn * (it + 2.0 * cy), 2.0 * dn * it);
    }
    return APCLOUD_OK;
}

// The solve loop around the kernel (a launch ends after its step budget).
// *ran is false, and nothing has changed, when a block's share does not fit.
apcloud_status resident_run(apcloud_ctx *c, ResidentArgs a, const double *b, double *x, double rtol, int max_iter,
                            uint32_t *tag, int grid, bool graph, apcloud_solve_info *info, bool *ran) {
    *ran = false;
    int iters = 0, cycles = 0;
    ResidentOut o{};
    for (;;) {
        ResidentIn in{};
        in.b = b;
        in.x = x;
        in.rtol = rtol;
        in.omega = a.pdeg > 1 ? c->P.poly_omega : 1.0;
        in.max_iter = max_iter - iters;
        in.tag0 = *tag;
        in.resume = iters > 0;
        *tag += TAGS_PER_LAUNCH;
        APC_TRY(run_resident(c, a, in, grid, graph, &o));
        if (o.status == RES_UNFIT && iters == 0) {
            c->res_unfit = true;   // not asked again for these operators
            return APCLOUD_OK;
        }
        if (o.status == RES_TIMEOUT || o.abort)
            return fail(c, APCLOUD_E_TIMEOUT, "a block gave up waiting for another's part of a vector");
        iters += o.iters;
        cycles += o.cycles;
        if (o.status != RES_MORE) break;
    }
    *ran = true;
    if (info) {
        info->iters = iters;
        info->restarts = cycles;
        info->relres = o.relres;
    }
    return o.status == RES_OK ? APCLOUD_OK : APCLOUD_W_NOT_CONVERGED;
}

apcloud_status resident_solve(apcloud_ctx *c, int which, const double *b, double *x, double rtol, int max_iter,
                              apcloud_solve_info *info, bool *ran) {
    *ran = false;
    if (!resident_ok(c, which)) return APCLOUD_OK;
    const bool mixed = c->P.precision == 1;
    const int n = c->n_tot, m = c->P.restart, pdeg = c->P.poly_degree;
    const int64_t ldv = ((int64_t)n + 31) / 32 * 32;
    int spc = 0, grid = 0;
    resident_grid(c, &spc, &grid);
    ResidentArgs a{};
    a.sw = ptr<uint32_t>(c->slice_w);
    a.so = ptr<uint32_t>(c->slice_off);
    a.col = ptr<int32_t>(c->ell_col);
    a.val64 = ptr<double>(which ? c->ell_A : c->ell_B);
    a.val32 = mixed ? ptr<float>(which ? c->ell_A32 : c->ell_B32) : nullptr;
    a.val16 = mixed ? ptr<__half>(which ? c->ell_A16 : c->ell_B16) : nullptr;
    a.d = ptr<double>(which ? c->dA : c->dB);
    a.n = n;
    a.nsl = c->n_slices;
    a.spc = spc;
    a.ldv = ldv;
    a.m = m;
    a.pdeg = pdeg;
    a.timing = c->timer.mask ? 1 : 0;
    a.u = ensure<double>(c, c->u, 2 * ldv + 1);
    if (mixed) a.V = ensure<float>(c, c->V32, (int64_t)(m + 1) * ldv);
    else a.V = ensure<double>(c, c->V, (int64_t)(m + 1) * ldv);
    a.Z = a.V;
    if (pdeg > 1 || mixed) {
        if (mixed) a.Z = ensure<float>(c, c->zbasis, (int64_t)m * ldv);
        else a.Z = ensure<double>(c, c->zbasis, (int64_t)m * ldv);
    }
    // the tagged words: one exchange buffer per sweep, the FP64 iterate's, the
    // sums' two sets; fresh memory is cleared, and so is old memory once the
    // 32-bit numbers are used up
    const int64_t xw = (int64_t)pdeg * n * (mixed ? 1 : 2), uw = 2 * (int64_t)n, rw = resident_red_words(grid);
    const size_t need = (size_t)(xw + uw + rw) * 8 + 64;
    const bool fresh = !c->res_words.p || c->res_words.bytes < need;
    if (fresh && !ensure_bytes(c, c->res_words, need)) return APCLOUD_E_NOMEM;
    ResidentState *st = ensure<ResidentState>(c, c->res_state, 1);
    if (!a.u || !a.V || !a.Z || !st) return APCLOUD_E_NOMEM;
    if (fresh || c->res_tag > 0xF0000000u) {
        APC_CUDA(c, cudaMemsetAsync(c->res_words.p, 0, c->res_words.bytes, c->s));
        c->res_tag = 1;
    }
    // 16-byte words first; every part starts on 16 bytes
    uint64_t *w = ptr<uint64_t>(c->res_words);
    a.ull = w;
    a.red = w + uw;
    a.xll = w + uw + rw;
    a.in = &st->in;
    a.out = &st->out;
    return resident_run(c, a, b, x, rtol, max_iter, &c->res_tag, grid, true, info, ran);
}

}  // namespace apc
