// stencil.cu -- Section 3.1 (WLS GFD operators) with the k-ring neighbour
// search of Section 4.3, and assembly of the density matrix B and the
// Poisson matrix A of Section 3.2 in sliced ELL.
//
// One warp per node grows the k-ring (k = 2..ring_max) by BFS over
// the face adjacency with the candidate set in shared memory, sorts the
// candidates once by (exact integer squared distance, node index) and takes the
// octant picks, the nearest fill and the ties as prefix counts (ballots) along
// that order.  The least-squares operator P = (W V0)^+ W of the weighted scaled
// Vandermonde W V0 (a row per neighbour, m <= 32) is formed by Cholesky QR
// applied twice (CholeskyQR2): two 9x9 Gram matrices, their factorisations, and
// triangular solves row by row, column j of P being R^-1 q_j^T W_j.  In FP64 the
// same warp goes on with it, one lane per neighbour; in the mixed form a second
// kernel does, four nodes per warp (k_wls32), and the few nodes that its FP32
// factorisation cannot certify start again in a third (the list kernel).
#include <cuda_fp16.h>

#include <cmath>
#include <type_traits>

#include "fpconv.cuh"
#include "fprecip.cuh"
#include "internal.cuh"

namespace apc {

namespace {

constexpr int ASTR = NCOL;      // row stride of the staged Vandermonde

// MC candidate slots: MAXC_FAST in the kernel over all nodes, MAXC in the one
// that redoes the nodes whose rings outgrew them
template <int MC>
struct __align__(16) SelectSmemT {
    int32_t cand[MC];
    long long d2[MC];   // hash set of the candidates (2 MC ints), then their rank keys, then squared distances
    uint16_t srt[MC];   // candidate slots in (d2, index) order
    uint8_t oct[MC];
    uint8_t pick[MC];   // octant picks, by sorted position
    int32_t sel[MMAX];
    long long seld2[MMAX];
};
template <int MC>
struct __align__(16) WarpSmemT : SelectSmemT<MC> {
    double A[MMAX * ASTR];
    double G[48];
    double R1[NCOL * NCOL];
    double R2[NCOL * NCOL];
    double Ri1[NCOL], Ri2[NCOL];   // reciprocal diagonals of R1, R2
};

__device__ __forceinline__ bool key_less(long long da, int ia, long long db, int ib) {
    return da < db || (da == db && ia < ib);
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Packed upper storage of the symmetric 9x9 Gram matrix: entry (a, b), a <= b,
// sits at a * 9 - a (a - 1) / 2 + (b - a), 45 entries in all.  Lane l owns
// entries l and l + 32 (the second only for l < 13).
__device__ __forceinline__ int pk_idx(int a, int b) { return a * NCOL - a * (a - 1) / 2 + (b - a); }

struct GramOwn {
    int a1, b1, a2, b2;
    bool two;
};

__device__ __forceinline__ void pk_rowcol(int e, int &a, int &b) {
    int e0 = 0;
    a = 0;
    while (e - e0 >= NCOL - a) { e0 += NCOL - a; ++a; }
    b = a + (e - e0);
}

__device__ __forceinline__ GramOwn gram_own(int lane) {
    GramOwn o;
    o.two = lane + 32 < NCOL * (NCOL + 1) / 2;
    pk_rowcol(lane, o.a1, o.b1);
    pk_rowcol(o.two ? lane + 32 : 0, o.a2, o.b2);
    return o;
}

// Cholesky G = R^T R of the packed Gram matrix by the whole warp: right-looking,
// each lane updating the trailing entries it owns after the pivot row k is
// scaled.  R is row-major upper (the strict lower part is not written), Ri the
// reciprocals of its diagonal.  G is overwritten.  Returns false on a
// non-positive pivot, the same decision in every lane.
template <class T>
__device__ bool cholesky_warp(T *G, T *R, T *Ri, const GramOwn &o, int lane) {
    for (int k = 0; k < NCOL; ++k) {
        const T gkk = G[pk_idx(k, k)];
        if (!(gkk > (T)0)) return false;
        const T d = sqrt(gkk), rd = (T)1 / d;
        if (o.a1 == k) R[k * NCOL + o.b1] = (o.b1 == k) ? d : G[lane] * rd;
        else if (o.a1 > k) G[lane] -= (G[pk_idx(k, o.a1)] * rd) * (G[pk_idx(k, o.b1)] * rd);
        if (o.two) {
            if (o.a2 == k) R[k * NCOL + o.b2] = (o.b2 == k) ? d : G[lane + 32] * rd;
            else if (o.a2 > k) G[lane + 32] -= (G[pk_idx(k, o.a2)] * rd) * (G[pk_idx(k, o.b2)] * rd);
        }
        if (lane == 0) Ri[k] = rd;
        __syncwarp();
    }
    return true;
}

// FP32 Cholesky G = R^T R of the packed Gram matrix, computed by every lane at
// once in registers (the 45 entries are broadcast from shared memory, the nine
// pivot steps run without any exchange between lanes): g becomes R, rd the
// reciprocals of its diagonal.  The reciprocal square root of each pivot gives
// both R_kk = g * rsqrt(g) and 1 / R_kk.  Returns false on a non-positive pivot,
// the same decision in every lane.
__device__ __forceinline__ bool cholesky_regs(const float *G, float (&g)[48], float (&rd)[NCOL]) {
#pragma unroll
    for (int e = 0; e < 12; ++e) {
        const float4 v = reinterpret_cast<const float4 *>(G)[e];
        g[4 * e] = v.x;
        g[4 * e + 1] = v.y;
        g[4 * e + 2] = v.z;
        g[4 * e + 3] = v.w;
    }
    bool ok = true;
#pragma unroll
    for (int k = 0; k < NCOL; ++k) {
        const float gkk = g[pk_idx(k, k)];
        ok = ok && gkk > 0.f;
        const float r = rsqrtf(ok ? gkk : 1.f);
        rd[k] = r;
        g[pk_idx(k, k)] = gkk * r;
#pragma unroll
        for (int j = k + 1; j < NCOL; ++j) g[pk_idx(k, j)] *= r;
#pragma unroll
        for (int i = k + 1; i < NCOL; ++i)
#pragma unroll
            for (int j = i; j < NCOL; ++j) g[pk_idx(i, j)] = fmaf(-g[pk_idx(k, i)], g[pk_idx(k, j)], g[pk_idx(i, j)]);
    }
    return ok;
}

// solve q R = a for the row vector q (R upper), in place on v
template <class T>
__device__ __forceinline__ void row_solve_upper(const T *R, const T *Ri, T *v) {
#pragma unroll
    for (int c = 0; c < NCOL; ++c) {
        T s = v[c];
#pragma unroll
        for (int k = 0; k < c; ++k) s -= v[k] * R[k * NCOL + c];
        v[c] = s * Ri[c];
    }
}

// solve R z = v for the column vector z (R upper), in place
template <class T>
__device__ __forceinline__ void col_solve_upper(const T *R, const T *Ri, T *v) {
#pragma unroll
    for (int c = NCOL - 1; c >= 0; --c) {
        T s = v[c];
#pragma unroll
        for (int k = c + 1; k < NCOL; ++k) s -= R[c * NCOL + k] * v[k];
        v[c] = s * Ri[c];
    }
}

// solve q R = a for the row vector q (R upper, packed), in place on v
__device__ __forceinline__ void row_solve_upper(const float (&R)[48], const float (&Ri)[NCOL], float *v) {
#pragma unroll
    for (int c = 0; c < NCOL; ++c) {
        float s = v[c];
#pragma unroll
        for (int k = 0; k < c; ++k) s -= v[k] * R[pk_idx(k, c)];
        v[c] = s * Ri[c];
    }
}

// solve R z = v for the column vector z (R upper, packed), in place
__device__ __forceinline__ void col_solve_upper(const float (&R)[48], const float (&Ri)[NCOL], float *v) {
#pragma unroll
    for (int c = NCOL - 1; c >= 0; --c) {
        float s = v[c];
#pragma unroll
        for (int k = c + 1; k < NCOL; ++k) s -= R[pk_idx(c, k)] * v[k];
        v[c] = s * Ri[c];
    }
}

// col_solve_upper in the place of the first (open) and the second (tail) of two
// solves one after another, with a stop between them: the first entry is handed
// over before its division by R_00 (rd00 its reciprocal), which the second
// rounds together with the first term, as the compiler contracts the two
// written in one piece (wls_column_f32).
__device__ __forceinline__ void col_solve_rows(const float (&R)[48], const float (&Ri)[NCOL], float *v) {
#pragma unroll
    for (int c = NCOL - 1; c > 0; --c) {
        float s = v[c];
#pragma unroll
        for (int k = c + 1; k < NCOL; ++k) s -= R[pk_idx(c, k)] * v[k];
        v[c] = s * Ri[c];
    }
}
__device__ __forceinline__ void col_solve_open(const float (&R)[48], const float (&Ri)[NCOL], float *v) {
    col_solve_rows(R, Ri, v);
#pragma unroll
    for (int k = 1; k < NCOL; ++k) v[0] -= R[pk_idx(0, k)] * v[k];
}
__device__ __forceinline__ void col_solve_tail(const float (&R)[48], const float (&Ri)[NCOL], float *v, float rd00) {
    col_solve_rows(R, Ri, v);
    float s = __fmaf_rn(v[0], rd00, -__fmul_rn(R[pk_idx(0, 1)], v[1]));
#pragma unroll
    for (int k = 2; k < NCOL; ++k) s -= R[pk_idx(0, k)] * v[k];
    v[0] = s * Ri[0];
}

// Gram matrix of the m rows staged by columns (entry e of row j at e * FSTR + j,
// zeros in rows m to 31), the lane's two owned entries accumulated side by side
// in row order, four rows to a load
constexpr int FSTR = 36;
__device__ __forceinline__ void gram_f32(const float *A, int m, float *G, const GramOwn &o, int lane) {
    float s1 = 0.f, s2 = 0.f;
    const float *a1 = A + o.a1 * FSTR, *b1 = A + o.b1 * FSTR, *a2 = A + o.a2 * FSTR, *b2 = A + o.b2 * FSTR;
    for (int j = 0; j < m; j += 4) {
        const float4 p = *reinterpret_cast<const float4 *>(a1 + j), q = *reinterpret_cast<const float4 *>(b1 + j);
        const float4 r = *reinterpret_cast<const float4 *>(a2 + j), t = *reinterpret_cast<const float4 *>(b2 + j);
        s1 = fmaf(p.x, q.x, s1);
        s2 = fmaf(r.x, t.x, s2);
        s1 = fmaf(p.y, q.y, s1);
        s2 = fmaf(r.y, t.y, s2);
        s1 = fmaf(p.z, q.z, s1);
        s2 = fmaf(r.z, t.z, s2);
        s1 = fmaf(p.w, q.w, s1);
        s2 = fmaf(r.w, t.w, s2);
    }
    G[lane] = s1;
    if (o.two) G[lane + 32] = s2;
}

// The FP32 column's constants: the weight's, and the least condition estimates
// (min / max of |R_ii|) that it takes and that any column needs, each the least
// FP32 number not below the FP64 one (r < the one exactly when r < the other).
struct Fp32Args {
    float ec, inv_1mec, rcond_min, rank_min;
};
float fp32_not_below(double v) {
    const float f = (float)v;
    return (double)f < v ? std::nextafter(f, INFINITY) : f;
}

// Weighted least-squares operator (Section 3.1) of the stencil staged in
// W.sel / W.seld2, in FP32: rows of W V0 (Eq. regfd with the
// normalized Gaussian weight), CholeskyQR2, and column `lane` of
// P = (W V0)^+ W unscaled by h and h^2.  Returns false when
// a Cholesky pivot fails; rratio = min |R_ii| / max |R_ii|.
// Conversions to and from 64-bit types run on the narrow FP64 pipe: offsets
// are 32-bit integers here, the squared distances too (in half cells of the
// deepest level, unless they need more), and h takes the one FP64 product.
template <class WS>
__device__ bool wls_column_f32(WS &W, int m, int lane, const GramOwn &own, int4 c0, const int4 *__restrict__ ic,
                               double unit, const Fp32Args &fa, int d2_shift, float (&qout)[NCOL],
                               float &lapj, float &rratio) {
    typedef float T;
    T *A = reinterpret_cast<T *>(W.A);
    T *G = reinterpret_cast<T *>(W.G);
    T *R1 = reinterpret_cast<T *>(W.R1);
    int off[3] = {0, 0, 0};
    int amax = 0;
    unsigned long long mydist = 0;
    if (lane < m) {
        int4 q = ic[W.sel[lane]];
        off[0] = q.x - c0.x; off[1] = q.y - c0.y; off[2] = q.z - c0.z;
        mydist = (unsigned long long)W.seld2[lane] >> d2_shift;
        for (int d = 0; d < 3; ++d) amax = max(amax, abs(off[d]));
    }
    const int hint = __reduce_max_sync(0xffffffffu, amax);
    const unsigned long long r2max = (unsigned long long)W.seld2[m - 1] >> d2_shift;
    T wj = (T)0;
    {
        T row[NCOL];
#pragma unroll
        for (int e = 0; e < NCOL; ++e) row[e] = (T)0;
        if (lane < m) {
            // xi = dy / h with h = max |dy_d| (Section 3.1): exact integers, one rounding in T
            T xi0 = (T)off[0] / (T)hint, xi1 = (T)off[1] / (T)hint, xi2 = (T)off[2] / (T)hint;
            T ratio = (r2max >> 32) ? (T)mydist / (T)r2max : (T)(unsigned)mydist / (T)(unsigned)r2max;
            wj = (expf(-ratio) - fa.ec) * fa.inv_1mec;
            const T half = (T)0.5;
            row[0] = xi0; row[1] = xi1; row[2] = xi2;
            row[3] = (half * xi0) * xi0;
            row[4] = xi0 * xi1;
            row[5] = xi0 * xi2;
            row[6] = (half * xi1) * xi1;
            row[7] = xi1 * xi2;
            row[8] = (half * xi2) * xi2;
#pragma unroll
            for (int e = 0; e < NCOL; ++e) row[e] = wj * row[e];
        }
#pragma unroll
        for (int e = 0; e < NCOL; ++e) A[e * FSTR + lane] = row[e];
    }
    __syncwarp();
    gram_f32(A, m, G, own, lane);
    __syncwarp();
    // the factors stay in registers for the solves that follow them; the first,
    // needed again at the end, waits in shared memory
    T R[48], Ri[NCOL];
    bool ok = cholesky_regs(G, R, Ri);
    T q[NCOL];
    T dr[NCOL];   // diagonal of R1, then of R1 R2
#pragma unroll
    for (int e = 0; e < NCOL; ++e) dr[e] = R[pk_idx(e, e)];
    if (ok) {
        if (lane == 0) {
#pragma unroll
            for (int e = 0; e < 12; ++e)
                reinterpret_cast<float4 *>(R1)[e] = make_float4(R[4 * e], R[4 * e + 1], R[4 * e + 2], R[4 * e + 3]);
#pragma unroll
            for (int e = 0; e < NCOL; ++e) R1[48 + e] = Ri[e];
        }
#pragma unroll
        for (int e = 0; e < NCOL; ++e) q[e] = A[e * FSTR + lane];   // zeros past the rows
        row_solve_upper(R, Ri, q);
#pragma unroll
        for (int e = 0; e < NCOL; ++e) A[e * FSTR + lane] = q[e];
        __syncwarp();
        gram_f32(A, m, G, own, lane);
        __syncwarp();
        ok = cholesky_regs(G, R, Ri);
    }
    rratio = 0.f;
    lapj = 0.f;
    if (!ok) return false;
    T dmin = (T)1e30, dmax = (T)0;
#pragma unroll
    for (int e = 0; e < NCOL; ++e) {
        T r = fabs(dr[e] * R[pk_idx(e, e)]);
        dmin = fmin(dmin, r);
        dmax = fmax(dmax, r);
    }
    rratio = dmin / dmax;
    // unscale rows by 1/h and 1/h^2 (h = max |dy_d|), in T
    const T h = (T)((double)hint * unit);   // hint < 2^23: exact in FP32
    const T ih = (T)1 / h, ih2 = ih * ih;
    if (lane < m) {
#pragma unroll
        for (int e = 0; e < NCOL; ++e) q[e] = A[e * FSTR + lane];
        row_solve_upper(R, Ri, q);
        col_solve_upper(R, Ri, q);
#pragma unroll
        for (int e = 0; e < 12; ++e) {
            const float4 v = reinterpret_cast<const float4 *>(R1)[e];
            R[4 * e] = v.x;
            R[4 * e + 1] = v.y;
            R[4 * e + 2] = v.z;
            R[4 * e + 3] = v.w;
        }
#pragma unroll
        for (int e = 0; e < NCOL; ++e) Ri[e] = R1[48 + e];
        col_solve_upper(R, Ri, q);
        T lj = (T)0;
#pragma unroll
        for (int e = 0; e < NCOL; ++e) {
            const T v = (q[e] * wj) * (e < 3 ? ih : ih2);
            qout[e] = v;
            if (e == 3 || e == 6 || e == 8) lj += v;
        }
        lapj = lj;
    } else {
#pragma unroll
        for (int e = 0; e < NCOL; ++e) qout[e] = 0.f;
    }
    return true;
}

// Gram matrix of m staged FP64 rows: lane l sums entry l over all rows; the 13
// entries past 32 are shared by two lanes each (lanes 0-12 the even rows, lanes
// 16-28 the odd ones), so they cost m / 2 issue slots of the FP64 pipe, not m.
__device__ __forceinline__ void gram_f64(const double *A, int m, const GramOwn &o, int a2, int b2, int lane,
                                         double &s1, double &s2) {
    s1 = 0.0;
    s2 = 0.0;
    for (int j = 0; j < m; ++j) s1 = fma(A[j * ASTR + o.a1], A[j * ASTR + o.b1], s1);
    for (int j = lane >> 4; j < m; j += 2) s2 = fma(A[j * ASTR + a2], A[j * ASTR + b2], s2);
    s2 += __shfl_xor_sync(0xffffffffu, s2, 16);
}

// wls_column_f32 in FP64, counted by the FP64 pipe's issue slots (16 cycles per
// warp instruction and SM, whatever the number of active lanes): the two
// serial factorisations with a square root and a division per pivot were more
// than half of the ~940 a node took.  Here the pivots are reciprocal square
// roots, and the second Cholesky QR pass is a correction: with Q1 = A R1^-1 and
// G2 = Q1^T Q1 = I + E, P = R1^-1 G2^-1 Q1^T and G2^-1 = I - E + O(E^2); E is
// the rounding of the first pass (kappa^2 eps), and below 1e-9 its square is
// below 1e-18 and the FP32 rounding of the correction E q below 1e-15 of q.
// A block with a larger E goes through the full second pass.
// ~335 slots: 2.8e5 nodes 12.76 -> 5.13 ms, the FP64 pipe's own time for them
// (fewer resident warps change nothing).  Against QR in extended precision the
// operator's rows are off by 1.9e-16 to 2.6e-16 of their norm on average (the full
// second pass: 2.4e-16 to 3.5e-16) from condition estimates of 0.02 up, by 2.0e-14
// (2.1e-14) where they fall to 3e-4; the estimate itself by 6e-16 to 1.9e-15.
template <class WS>
__device__ bool wls_column_f64(WS &W, int m, int lane, const GramOwn &own, int4 c0, const int4 *__restrict__ ic,
                               double inv_unit, double ec, double inv_1mec, double (&q)[NCOL], double &lapj,
                               double &rratio) {
    double *A = W.A, *G = W.G, *R = W.R1, *Ri = W.Ri1;
    const unsigned FULL = 0xffffffffu;
    int off[3] = {0, 0, 0};
    long long mydist = 0;
    if (lane < m) {
        const int4 p = ic[W.sel[lane]];
        off[0] = p.x - c0.x;
        off[1] = p.y - c0.y;
        off[2] = p.z - c0.z;
        mydist = W.seld2[lane];
    }
    const int hint = __reduce_max_sync(FULL, max(abs(off[0]), max(abs(off[1]), abs(off[2]))));
    // offsets are below 2^24: exact in FP32; squared distances below 2^48
    const double rh = recip_f64(f32_to_f64_int((float)hint));
    const double rr = recip_f64((double)W.seld2[m - 1]);
    double wj = 0.0;
    rratio = 0.0;
    lapj = 0.0;
    {
        // xi = dy / h with h = max |dy_d| (Section 3.1)
        const double x0 = f32_to_f64_int((float)off[0]) * rh, x1 = f32_to_f64_int((float)off[1]) * rh,
                     x2 = f32_to_f64_int((float)off[2]) * rh;
        const double dist = __hiloint2double(0x43300000 | (int)(mydist >> 32), (int)mydist) - 4503599627370496.0;
        const double w = (exp(-(dist * rr)) - ec) * inv_1mec;
        if (lane < m) wj = w;
        const double w0 = wj * x0, w1 = wj * x1, w2 = wj * x2;
        const double h0 = 0.5 * x0;
        double *a = A + lane * ASTR;
        a[0] = w0;
        a[1] = w1;
        a[2] = w2;
        a[3] = w0 * h0;
        a[4] = w0 * x1;
        a[5] = w0 * x2;
        a[6] = w1 * (0.5 * x1);
        a[7] = w1 * x2;
        a[8] = w2 * (0.5 * x2);
    }
    int a2, b2;
    const int e2 = 32 + (lane & 15);
    const bool two = (lane & 15) < 13;
    pk_rowcol(two ? e2 : 32, a2, b2);
    __syncwarp();
    double g1, g2;
    gram_f64(A, m, own, a2, b2, lane, g1, g2);
    // Cholesky G = R^T R, right-looking: entries stay with their lanes, the pivot
    // row goes through shared memory.  A pivot below 1e-30 (the entries are O(1))
    // is a rank deficiency either way.
    for (int k = 0; k < NCOL; ++k) {
        if (own.a1 == k) R[k * NCOL + own.b1] = g1;
        if (two && a2 == k && lane < 16) R[k * NCOL + b2] = g2;
        __syncwarp();
        const double gkk = R[k * NCOL + k];
        if (!(gkk > 1e-30)) return false;   // the same in every lane
        const double rd = rsqrt_f64(gkk);
        const double mine = (lane >= k && lane < NCOL ? R[k * NCOL + lane] : 0.0) * rd;
        __syncwarp();
        if (lane >= k && lane < NCOL) R[k * NCOL + lane] = mine;
        if (lane == 0) Ri[k] = rd;
        __syncwarp();
        if (k < 4 && own.a1 > k) g1 = fma(-R[k * NCOL + own.a1], R[k * NCOL + own.b1], g1);
        if (k < 8 && a2 > k) g2 = fma(-R[k * NCOL + a2], R[k * NCOL + b2], g2);
    }
#pragma unroll
    for (int e = 0; e < NCOL; ++e) q[e] = A[lane * ASTR + e];
    row_solve_upper<double>(R, Ri, q);
#pragma unroll
    for (int e = 0; e < NCOL; ++e) A[lane * ASTR + e] = q[e];
    __syncwarp();
    gram_f64(A, m, own, a2, b2, lane, g1, g2);
    const double e1 = own.a1 == own.b1 ? g1 - 1.0 : g1, ee = a2 == b2 ? g2 - 1.0 : g2;
    const float f1 = f64_to_f32_int(e1), f2 = f64_to_f32_int(ee);
    const bool small = __all_sync(FULL, fabsf(f1) < 1e-9f && fabsf(f2) < 1e-9f);
    double *R2 = W.R2, *Ri2 = W.Ri2;
    if (small) {
        float *E = reinterpret_cast<float *>(G);
        E[lane] = f1;
        if (two && lane < 16) E[e2] = f2;
        __syncwarp();
        float qf[NCOL], z[NCOL];
#pragma unroll
        for (int r = 0; r < NCOL; ++r) {
            qf[r] = f64_to_f32_int(q[r]);
            z[r] = 0.f;
        }
#pragma unroll
        for (int r = 0; r < NCOL; ++r)
#pragma unroll
            for (int k = r; k < NCOL; ++k) {
                const float v = E[pk_idx(r, k)];
                z[r] = fmaf(v, qf[k], z[r]);
                if (k != r) z[k] = fmaf(v, qf[r], z[k]);
            }
#pragma unroll
        for (int r = 0; r < NCOL; ++r) q[r] -= f32_to_f64_int(z[r]);
    } else {
        G[lane] = g1;
        if (two && lane < 16) G[e2] = g2;
        __syncwarp();
        if (!cholesky_warp<double>(G, R2, Ri2, own, lane)) return false;
        row_solve_upper<double>(R2, Ri2, q);
        col_solve_upper<double>(R2, Ri2, q);
    }
    col_solve_upper<double>(R, Ri, q);
    // condition estimate min / max of |R_ii|, an entry per lane (R_ii > 0: ordered
    // like its encoding); below 1e-9 the diagonal of G2's factor is 1 + E_ii / 2
    double rii = 1.0;
    if (lane < NCOL) {
        rii = R[lane * NCOL + lane];
        if (small) rii = fma(0.5 * rii, f32_to_f64_int(reinterpret_cast<const float *>(G)[pk_idx(lane, lane)]), rii);
        else rii *= R2[lane * NCOL + lane];
    }
    const unsigned dh = (unsigned)__double2hiint(rii), dl = (unsigned)__double2loint(rii);
    const bool mine = lane < NCOL;
    const unsigned lh = __reduce_min_sync(FULL, mine ? dh : ~0u), hh = __reduce_max_sync(FULL, mine ? dh : 0u);
    const unsigned ll = __reduce_min_sync(FULL, mine && dh == lh ? dl : ~0u),
                   hl = __reduce_max_sync(FULL, mine && dh == hh ? dl : 0u);
    rratio = __hiloint2double((int)lh, (int)ll) * recip_f64(__hiloint2double((int)hh, (int)hl));
    const double ih = rh * inv_unit, s1 = wj * ih, s2 = s1 * ih;
#pragma unroll
    for (int e = 0; e < NCOL; ++e) q[e] *= e < 3 ? s1 : s2;   // wj = 0 past the stencil
    lapj = q[3] + q[6] + q[8];
    return true;
}

// The rows of the derivative operator D (row-of-operator major, nodes
// fastest) of a block's SW nodes.  Each warp stages its node's 9 x MMAX block
// in its W.A as [e * MMAX + lane] (free once the WLS is done); the last warp
// of the block to finish writes every row as SW consecutive nodes, one
// 8 x SW-byte run per row, where each warp writing its own node would store
// 288 lone 8-byte words, each in a sector of its own.  Warps without a node
// (past n_int) only arrive.
template <int SW, class WS>
__device__ __forceinline__ void write_block_d(const unsigned char *smem_raw, unsigned *arrived, int lane, int y_base,
                                              int n_int, double *__restrict__ D_out, int64_t dstride) {
    __threadfence_block();
    __syncwarp();
    unsigned last = 0u;
    if (lane == 0) last = (atomicAdd(arrived, 1u) == SW - 1) ? 1u : 0u;
    last = __shfl_sync(0xffffffffu, last, 0);
    if (!last) return;
    __threadfence_block();
    const WS *Ws = reinterpret_cast<const WS *>(smem_raw);
    for (int t = lane; t < NCOL * MMAX * SW; t += 32) {
        const int row = t / SW, w = t - row * SW;
        const int y = y_base + w;
        if (y < n_int) D_out[(int64_t)row * dstride + y] = Ws[w].A[row];
    }
}

// Inserts node v into the warp's hash set of 2 MC slots (at most half full);
// true for the lane that brought it in.
template <int MC>
__device__ __forceinline__ bool ring_insert(int *tab, int v) {
    constexpr unsigned M = 2 * MC - 1;
    unsigned h = ((unsigned)v * 0x9E3779B1u >> 16) & M;
    for (;;) {   // ends: the table never fills
        const int old = atomicCAS(tab + h, -1, v);
        if (old == -1) return true;
        if (old == v) return false;
        h = (h + 1) & M;
    }
}

// SW warps (nodes) per block, one WarpSmemT<MC> each (and the block's
// arrival count after them); the autotuner picks SW.  Three forms:
//   FP64, every node (MC = MAXC_FAST): 6.6 KB of shared memory per warp and 32
//     warps per SM; a node whose ring outgrows MC candidates goes to ovf_list
//     instead of failing (against 512 slots at 16 warps a fifth faster);
//   SELECT, every node of the mixed form: ring and selection only, 2.4 KB and
//     40 registers, 48 warps per SM (0.29 ms for 2.8e5 nodes, bound by
//     instructions: 91% of the issue slots);
//   LIST (MC = MAXC): the n_list nodes of list, each warp writing its own D
//     columns.
// One kernel for the mixed form's every node took 1.22 ms at 2.8e5 nodes and
// 5.13 at 1.05e6, SELECT, k_wls32 and LIST 0.66 and 2.57.  slots <= MC is the
// capacity in force (the context's stencil_slots in the first kernel).
template <int SW, int MC, bool LIST, bool MIXED, bool SELECT>
__global__ void __launch_bounds__(SW * 32, SELECT ? 48 / SW : (MC < MAXC ? 32 : 16) / SW) k_stencil(
    const int4 *__restrict__ ic, const int32_t *__restrict__ adj, const int32_t *__restrict__ bowner, int n_int,
    int m_target, int ring_max, double unit, double inv_unit, double ec, double inv_1mec, int32_t *__restrict__ nbr_out,
    int32_t *__restrict__ m_out, int32_t *__restrict__ ring_out, double *__restrict__ lap_out,
    double *__restrict__ lapd_out, double *__restrict__ D_out, int64_t dstride, double *__restrict__ rcond_out,
    double fp32_rcond_min, int *__restrict__ fp64_count, unsigned *err,
    const int32_t *__restrict__ list, int n_list, unsigned *__restrict__ ovf_count, int32_t *__restrict__ ovf_list,
    int slots, int idx_bits, int d2_shift, Fp32Args fa) {
    typedef typename std::conditional<SELECT, SelectSmemT<MC>, WarpSmemT<MC>>::type WarpSmem;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    WarpSmem &W = reinterpret_cast<WarpSmem *>(smem_raw)[wid];
    const int li = blockIdx.x * SW + wid;
    const int y0 = LIST ? (li < n_list ? list[li] : n_int) : li;
    const unsigned FULL = 0xffffffffu;
    const unsigned lt = (1u << lane) - 1u;
    unsigned *arrived = reinterpret_cast<unsigned *>(reinterpret_cast<WarpSmem *>(smem_raw) + SW);
    (void)arrived;
    if (!LIST && !SELECT) {
        if (threadIdx.x == 0) *arrived = 0u;
        __syncthreads();
    }
    if (y0 >= n_int) {
        if constexpr (!LIST && !SELECT) write_block_d<SW, WarpSmem>(smem_raw, arrived, lane, blockIdx.x * SW, n_int, D_out, dstride);
        return;
    }

    const int4 c0 = ic[y0];
    int nc = 1;
    if (lane == 0) W.cand[0] = y0;
    __syncwarp();
    int head = 0, tail = 1;
    bool done = false, overflow = false;
    int m = 0, ring = 0;
    double rmin_over_rmax = 0.0;

    const GramOwn own = gram_own(lane);
    int *tab = reinterpret_cast<int *>(W.d2);   // 2 MC slots
    bool hashed = false;

    for (int k = 1; k <= ring_max && !done; ++k) {
        // ---- grow the ring by one layer (Section 4.3: (k+1)-ring = k-ring
        // plus the face neighbours of its nodes).  Eight lanes per frontier
        // node read its neighbours (packed first in its 24 slots; nearly all
        // nodes have at most eight), sixteen nodes' loads in flight.  A hash set
        // of the candidates, in the d2 area until they are ranked, tells the new
        // ones (a scan of all candidates for each took as long as the search).
        if (!hashed) {
            int4 *t4 = reinterpret_cast<int4 *>(tab);
            for (int t = lane; t < MC / 2; t += 32) t4[t] = make_int4(-1, -1, -1, -1);
            __syncwarp();
            for (int t = lane; t < nc; t += 32) ring_insert<MC>(tab, W.cand[t]);
            __syncwarp();
            hashed = true;
        }
        for (int g0 = head; g0 < tail && !overflow; g0 += 16) {
            int vb[4], ub[4];
            const int sub = lane & 7;
#pragma unroll
            for (int bt = 0; bt < 4; ++bt) {
                const int t = g0 + bt * 4 + (lane >> 3);
                ub[bt] = t < tail ? W.cand[t] : -1;
            }
#pragma unroll
            for (int bt = 0; bt < 4; ++bt) {
                const int u = ub[bt];
                vb[bt] = u < 0 ? -1 : (u < n_int ? adj[(int64_t)u * 24 + sub] : (sub == 0 ? bowner[u - n_int] : -1));
            }
#pragma unroll 1
            for (int bt = 0; bt < 4 && g0 + bt * 4 < tail && !overflow; ++bt) {
                int v = vb[0];
                const int u = ub[0];
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    vb[q] = vb[q + 1];
                    ub[q] = ub[q + 1];
                }
                for (int more = 0; more < 24; more += 8) {
                    if (more > 0) {   // a node with its eight slots full may have more
                        const bool ask = u >= 0 && u < n_int;
                        if (!__any_sync(FULL, ask && sub == 7 && v >= 0)) break;
                        v = ask ? adj[(int64_t)u * 24 + more + sub] : -1;
                    }
                    const bool fresh = v >= 0 && ring_insert<MC>(tab, v);
                    const unsigned bal = __ballot_sync(FULL, fresh);
                    const int p = nc + __popc(bal & lt);
                    if (fresh && p < slots) W.cand[p] = v;
                    nc += __popc(bal);
                    if (nc > slots) {
                        overflow = true;   // the same in every lane
                        break;
                    }
                    __syncwarp();
                }
            }
        }
        if (overflow) break;
        head = tail;
        tail = nc;
        if (k < 2) continue;
        const int ncand = nc - 1;
        if (ncand < m_target && k < ring_max) continue;
        if (ncand < NCOL) continue;

        // ---- order the candidates by (exact integer squared distance, node
        // index): every later choice is a prefix of this order
        // (two candidates per lane and pass over the others).  Offsets are
        // whole half cells of the deepest level, 2^(d2_shift / 2) units, so
        // distance and index fit one 64-bit key unless the tree is very deep
        // and large (idx_bits 0).
        hashed = false;
        for (int t0 = 1; t0 < nc; t0 += 64) {   // d2 area: keys of all candidates
            for (int t = t0 + lane; t < nc && t < t0 + 64; t += 32) {
                const int id = W.cand[t];
                int4 q = ic[id];
                long long dx = (long long)q.x - c0.x, dy = (long long)q.y - c0.y, dz = (long long)q.z - c0.z;
                const long long dd = dx * dx + dy * dy + dz * dz;
                W.d2[t] = idx_bits ? (dd >> d2_shift) << idx_bits | id : dd;
                W.oct[t] = (uint8_t)(((dx >= 0) << 2) | ((dy >= 0) << 1) | (dz >= 0));
            }
        }
        __syncwarp();
        if (idx_bits) {
            for (int t0 = 1; t0 < nc; t0 += 64) {
                const int ta = t0 + lane, tb = ta + 32;
                const unsigned long long ka = ta < nc ? W.d2[ta] : ~0ull, kb = tb < nc ? W.d2[tb] : ~0ull;
                int ra = 0, rb = 0;
#pragma unroll 4
                for (int u = 1; u < nc; ++u) {
                    const unsigned long long ku = W.d2[u];
                    ra += ku < ka;
                    rb += ku < kb;
                }
                if (ta < nc) W.srt[ra] = (uint16_t)ta;
                if (tb < nc) W.srt[rb] = (uint16_t)tb;
            }
            __syncwarp();
            for (int t = 1 + lane; t < nc; t += 32) W.d2[t] = (W.d2[t] >> idx_bits) << d2_shift;
        } else {
            for (int t = 1 + lane; t < nc; t += 32) {
                const long long dt = W.d2[t];
                const int it = W.cand[t];
                int r = 0;
                for (int u = 1; u < nc; ++u) r += key_less(W.d2[u], W.cand[u], dt, it) ? 1 : 0;
                W.srt[r] = (uint16_t)t;
            }
        }
        __syncwarp();
        // ---- Section 3.1 quadrant criterion, octants in 3-D: the two nearest
        // in each octant, counted along the order 32 positions at a time
        int nA = 0;
        {
            unsigned seen_lo = 0u, seen_hi = 0u;   // counts of octants 0-3 and 4-7, a byte each (capped at 2)
            for (int p0 = 0; p0 < ncand; p0 += 32) {
                const int pos = p0 + lane;
                const int o = (pos < ncand) ? (int)W.oct[W.srt[pos]] : 8;
                const unsigned peers = __match_any_sync(FULL, o);
                const unsigned word = o < 4 ? seen_lo : seen_hi;
                const int sh = (o & 3) * 8, rank = __popc(peers & lt);
                const bool pk = o < 8 && (int)(word >> sh & 255u) + rank < 2;
                if (pos < ncand) W.pick[pos] = pk ? 1 : 0;
                nA += __popc(__ballot_sync(FULL, pk));
                if (p0 + 32 < ncand) {   // picks are what counts towards two per octant
                    seen_lo += __reduce_add_sync(FULL, pk && o < 4 ? 1u << sh : 0u);
                    seen_hi += __reduce_add_sync(FULL, pk && o >= 4 ? 1u << sh : 0u);
                }
            }
        }
        __syncwarp();
        // target sizes m_target, m_target + 2, ... (a rank-deficient stencil or
        // one whose Laplacian diagonal is not negative is not used).  One pass
        // along the order: the picks, then the nearest non-picked up to the
        // target (the last of them sets the cut distance), then every further
        // candidate tied at the cut while the stencil has room, in index order;
        // the stencil is written in (d2, index) order.
        for (int mt = m_target; mt <= MMAX && !done; mt += 2) {
        const int need = mt - nA;
        const int room = MMAX - nA - (need > 0 ? need : 0);
        int nsel = 0, nnp = 0, ntie = 0;
        bool cut_found = false;
        long long cut = 0;
        for (int p0 = 0; p0 < ncand; p0 += 32) {
            const int pos = p0 + lane;
            const bool valid = pos < ncand;
            int t = 0;
            long long d = 0;
            bool pk = false;
            if (valid) { t = W.srt[pos]; d = W.d2[t]; pk = W.pick[pos] != 0; }
            const bool np = valid && !pk;
            const unsigned bnp = __ballot_sync(FULL, np);
            const int npr = nnp + __popc(bnp & lt);
            const bool fill = np && npr < need;
            if (!cut_found) {
                const unsigned bc = __ballot_sync(FULL, np && npr == need - 1);
                if (bc) {
                    cut = __shfl_sync(FULL, d, __ffs(bc) - 1);
                    cut_found = true;
                }
            }
            const bool te = np && !fill && cut_found && d == cut;
            const unsigned bte = __ballot_sync(FULL, te);
            const bool tie = te && ntie + __popc(bte & lt) < room;
            ntie += __popc(__ballot_sync(FULL, tie));
            const bool sl = pk || fill || tie;
            const unsigned bs = __ballot_sync(FULL, sl);
            if (sl) {
                const int r = nsel + __popc(bs & lt);
                W.sel[r] = W.cand[t];
                W.seld2[r] = d;
            }
            nsel += __popc(bs);
            nnp += __popc(bnp);
        }
        __syncwarp();
        m = nsel;

        if constexpr (SELECT) {   // the operators are the next kernel's
            nbr_out[(int64_t)y0 * MMAX + lane] = (lane < m) ? W.sel[lane] : -1;
            if (lane == 0) {
                m_out[y0] = m;
                ring_out[y0] = k;
            }
            done = true;
        } else {
        // ---- weighted least squares: FP32 first when asked, FP64 for blocks the
        // FP32 factorisation cannot certify (Cholesky failure or condition
        // estimate min|R_ii|/max|R_ii| below fp32_rcond_min, by default 1e-3,
        // where FP32 Cholesky QR loses its accuracy)
        double q[NCOL], lapj = 0.0;
        bool ok = false;
        if constexpr (MIXED) {
            float qf[NCOL], lf, rf;
            ok = wls_column_f32(W, m, lane, own, c0, ic, unit, fa, d2_shift, qf, lf, rf) && !(rf < fa.rcond_min);
            if (!ok && lane == 0) atomicAdd(fp64_count, 1);
            if (ok) {
                rmin_over_rmax = (double)rf;
                lapj = (double)lf;
#pragma unroll
                for (int e = 0; e < NCOL; ++e) q[e] = (double)qf[e];
            }
        }
        if (!ok) ok = wls_column_f64(W, m, lane, own, c0, ic, inv_unit, ec, inv_1mec, q, lapj, rmin_over_rmax);
        if (ok) ok = rmin_over_rmax >= RANK_TOL;
        if (!ok) lapj = 0.0;
        const double lsum = warp_sum_d(lapj);
        if (!ok || !(-lsum < 0.0)) {       // unusable: more neighbours, then a wider ring
            if (m >= nc - 1) break;
            continue;
        }

        nbr_out[(int64_t)y0 * MMAX + lane] = (lane < m) ? W.sel[lane] : -1;
        lap_out[(int64_t)y0 * MMAX + lane] = lapj;
        if (lane == 0) {
            lapd_out[y0] = -lsum;
            m_out[y0] = m;
            ring_out[y0] = k;
            rcond_out[y0] = rmin_over_rmax;
        }
        __syncwarp();
        // derivative operator, staged for write_block_d (the list kernel's
        // nodes are not consecutive: each warp writes its own columns)
        __syncwarp();
        if (LIST) {
#pragma unroll
            for (int e = 0; e < NCOL; ++e) D_out[((int64_t)e * MMAX + lane) * dstride + y0] = (lane < m) ? q[e] : 0.0;
        } else {
#pragma unroll
            for (int e = 0; e < NCOL; ++e) W.A[e * MMAX + lane] = (lane < m) ? q[e] : 0.0;
        }
        ring = k;
        done = true;
        }
        }   // target sizes
    }
    if (!done) {
        const bool ovf = overflow;
        if (lane == 0) {
            if (ovf && !LIST) ovf_list[atomicAdd(ovf_count, 1u)] = y0;   // redone with MAXC slots
            else atomicOr(err, ovf ? (ERR_STENCIL | ERR_OVERFLOW) : ERR_STENCIL);
            m_out[y0] = 0;
            ring_out[y0] = -1;
            lapd_out[y0] = 0.0;
            rcond_out[y0] = 0.0;
        }
        nbr_out[(int64_t)y0 * MMAX + lane] = -1;
        lap_out[(int64_t)y0 * MMAX + lane] = 0.0;
        __syncwarp();
        if constexpr (LIST) {
#pragma unroll
            for (int e = 0; e < NCOL; ++e) D_out[((int64_t)e * MMAX + lane) * dstride + y0] = 0.0;
        } else if constexpr (!SELECT) {
#pragma unroll
            for (int e = 0; e < NCOL; ++e) W.A[e * MMAX + lane] = 0.0;
        }
    }
    (void)ring;
    if constexpr (!LIST && !SELECT) write_block_d<SW, WarpSmem>(smem_raw, arrived, lane, blockIdx.x * SW, n_int, D_out, dstride);
}

// The mixed form's operators of the selected stencils: wls_column_f32, four
// nodes per warp.  With a warp per node, both 9x9 factorisations run in every
// lane at once, 450 of 1700 instructions 32 times over; the loads of their
// operands keep the shared-memory pipe busy; and the kernel that also selects
// outgrows the instruction cache (1.9 of 10 cycles between instructions waited
// for the next one).  Here a lane builds the rows of its neighbour for the four
// nodes; then eight lanes have one node each: 3 x 3 blocks of its Gram matrix, the
// factor in registers, every eighth row in the solves.  The same operations in
// the same order: the same bits.  0.35 ms for 2.8e5 nodes, of which the operator's
// 663 MB take 0.1 (with an entry of the Gram matrix per lane and the factors read
// back from shared memory for every node 0.48: the load/store pipe 88% busy).
// Conversions stay on the FP64 pipe: it is a third busy, and the integer ones
// cost more issue slots than it has to spare.  Nodes the FP32
// factorisation cannot certify, and those that need more neighbours, go to the
// list kernel, which starts them again.
constexpr int WN = 4;   // nodes per warp
constexpr int WLS_SW = 4;                      // warps per block
struct __align__(16) Wls32Smem {
    float A[WN][(NCOL + 1) * FSTR];   // rows by columns, then the weights; at the end the operator, [e * MMAX + lane]
    unsigned good, pad[3];
    float G[WN][48], R1[WN][60];      // Gram matrix, then R2; R1: 45 packed entries, from 48 on the reciprocal diagonal
};

__device__ __forceinline__ void load_factor(const float *F, float (&R)[48], float (&Ri)[NCOL]) {
#pragma unroll
    for (int e = 0; e < 12; ++e) {
        const float4 v = reinterpret_cast<const float4 *>(F)[e];
        R[4 * e] = v.x;
        R[4 * e + 1] = v.y;
        R[4 * e + 2] = v.z;
        R[4 * e + 3] = v.w;
    }
#pragma unroll
    for (int e = 0; e < NCOL; ++e) Ri[e] = F[48 + e];
}
__device__ __forceinline__ void store_factor(float *F, const float (&R)[48], const float (&Ri)[NCOL]) {
#pragma unroll
    for (int e = 0; e < 12; ++e)
        reinterpret_cast<float4 *>(F)[e] = make_float4(R[4 * e], R[4 * e + 1], R[4 * e + 2], R[4 * e + 3]);
#pragma unroll
    for (int e = 0; e < NCOL; ++e) F[48 + e] = Ri[e];
}

// Gram matrix of one node's rows by eight lanes, six of them a 3 x 3 block each
// (what falls below the diagonal is not stored): six loads of four rows for 36
// multiply-adds, where an entry per lane takes four for eight.  Rows m to
// mmax (below 32) are zeros; every entry is summed in row order.
__device__ __forceinline__ void gram_blocks(const float *A, int mmax, float *G, int blk) {
    const int br = blk < 3 ? 0 : (blk < 5 ? 1 : 2), bc = blk < 3 ? blk : (blk < 5 ? blk - 2 : 2);
    const float *pa = A + 3 * br * FSTR, *pb = A + 3 * bc * FSTR;
    float s[3][3] = {};
#pragma unroll 1
    for (int j = 0; j < mmax; j += 4) {
        float4 a[3], b[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            a[i] = *reinterpret_cast<const float4 *>(pa + i * FSTR + j);
            b[i] = *reinterpret_cast<const float4 *>(pb + i * FSTR + j);
        }
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                float t = s[i][k];
                t = fmaf(a[i].x, b[k].x, t);
                t = fmaf(a[i].y, b[k].y, t);
                t = fmaf(a[i].z, b[k].z, t);
                s[i][k] = fmaf(a[i].w, b[k].w, t);
            }
    }
    if (blk < 6) {
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int k = 0; k < 3; ++k)
                if (br < bc || i <= k) G[pk_idx(3 * br + i, 3 * bc + k)] = s[i][k];
    }
}

template <int SW>
__global__ void __launch_bounds__(SW * 32, 24 / SW) k_wls32(
    const int4 *__restrict__ ic, int n_int, double unit, Fp32Args fa, int d2_shift, const int32_t *__restrict__ nbr,
    const int32_t *__restrict__ msz, double *__restrict__ lap_out, double *__restrict__ lapd_out,
    double *__restrict__ D_out, int64_t dstride, double *__restrict__ rcond_out, unsigned *__restrict__ list_count,
    int32_t *__restrict__ list) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    Wls32Smem &W = reinterpret_cast<Wls32Smem *>(smem_raw)[wid];
    const int w0 = (blockIdx.x * SW + wid) * WN;   // past the last node: empty stencils
    const unsigned FULL = 0xffffffffu;
    // ---- rows, a lane per neighbour; lane q < WN keeps node q's size and h in units
    const int my_m = lane < WN && w0 + lane < n_int ? msz[w0 + lane] : 0;
    float my_hint = 1.f;
    int4 p[WN], c0[WN];
#pragma unroll
    for (int q = 0; q < WN; ++q) {
        const int m = __shfl_sync(FULL, my_m, q);
        const int id = lane < m ? nbr[(int64_t)(w0 + q) * MMAX + lane] : -1;
        c0[q] = m > 0 ? ic[w0 + q] : make_int4(0, 0, 0, 0);
        p[q] = id >= 0 ? ic[id] : c0[q];
    }
#pragma unroll
    for (int q = 0; q < WN; ++q) {
        const int m = __shfl_sync(FULL, my_m, q);
        const int o0 = p[q].x - c0[q].x, o1 = p[q].y - c0[q].y, o2 = p[q].z - c0[q].z;
        const int hint = __reduce_max_sync(FULL, max(abs(o0), max(abs(o1), abs(o2))));
        // offsets are whole multiples of 2^(d2_shift / 2), half cells of the deepest level
        const int h0 = o0 >> (d2_shift >> 1), h1 = o1 >> (d2_shift >> 1), h2 = o2 >> (d2_shift >> 1);
        const unsigned long long d = (unsigned long long)((long long)h0 * h0 + (long long)h1 * h1 + (long long)h2 * h2);
        const unsigned long long r2max = __shfl_sync(FULL, d, m - 1);   // the last is the farthest
        if (lane == q) my_hint = (float)hint;
        float row[NCOL], wj = 0.f;
#pragma unroll
        for (int e = 0; e < NCOL; ++e) row[e] = 0.f;
        if (lane < m) {
            const float fh = (float)hint;
            const float xi0 = (float)o0 / fh, xi1 = (float)o1 / fh, xi2 = (float)o2 / fh;
            const float ratio = (r2max >> 32) ? (float)d / (float)r2max : (float)(unsigned)d / (float)(unsigned)r2max;
            wj = (expf(-ratio) - fa.ec) * fa.inv_1mec;
            row[0] = xi0; row[1] = xi1; row[2] = xi2;
            row[3] = (0.5f * xi0) * xi0;
            row[4] = xi0 * xi1;
            row[5] = xi0 * xi2;
            row[6] = (0.5f * xi1) * xi1;
            row[7] = xi1 * xi2;
            row[8] = (0.5f * xi2) * xi2;
#pragma unroll
            for (int e = 0; e < NCOL; ++e) row[e] = wj * row[e];
        }
#pragma unroll
        for (int e = 0; e < NCOL; ++e) W.A[q][e * FSTR + lane] = row[e];
        W.A[q][NCOL * FSTR + lane] = wj;
    }
    __syncwarp();
    // ---- from here on lanes 8 q to 8 q + 7 have node q: a 3 x 3 block of its Gram
    // matrix each, its factor in the registers of all eight, every eighth row
    const int sub = lane >> 3, r0 = lane & 7, mmax = __reduce_max_sync(FULL, my_m), m = __shfl_sync(FULL, my_m, sub);
    float *A = W.A[sub] + r0;
    gram_blocks(W.A[sub], mmax, W.G[sub], r0);
    __syncwarp();
    float R[48], Ri[NCOL];
    bool ok = cholesky_regs(W.G[sub], R, Ri);
    if (r0 == 0) store_factor(W.R1[sub], R, Ri);
#pragma unroll 1
    for (int i = 0; i < MMAX; i += 8) {
        float v[NCOL];
#pragma unroll
        for (int e = 0; e < NCOL; ++e) v[e] = A[e * FSTR + i];
        row_solve_upper(R, Ri, v);
#pragma unroll
        for (int e = 0; e < NCOL; ++e) A[e * FSTR + i] = v[e];
    }
    __syncwarp();
    gram_blocks(W.A[sub], mmax, W.G[sub], r0);
    __syncwarp();
    ok = cholesky_regs(W.G[sub], R, Ri) && ok;
    float rf;
    {
        float dmin = 1e30f, dmax = 0.f;
#pragma unroll
        for (int e = 0; e < NCOL; ++e) {
            const float r = fabsf(W.R1[sub][pk_idx(e, e)] * R[pk_idx(e, e)]);
            dmin = fminf(dmin, r);
            dmax = fmaxf(dmax, r);
        }
        rf = dmin / dmax;
    }
    ok = ok && !(rf < fa.rcond_min) && rf >= fa.rank_min;
#pragma unroll 1
    for (int i = 0; i < MMAX; i += 8) {
        float v[NCOL];
#pragma unroll
        for (int e = 0; e < NCOL; ++e) v[e] = A[e * FSTR + i];
        row_solve_upper(R, Ri, v);
        col_solve_open(R, Ri, v);
#pragma unroll
        for (int e = 0; e < NCOL; ++e) A[e * FSTR + i] = v[e];
    }
    const float rd20 = Ri[0];
    // columns of P, unscaled by 1/h and 1/h^2, and the Laplacian's in place of the weights
    load_factor(W.R1[sub], R, Ri);
    const float h = (float)((double)__shfl_sync(FULL, my_hint, sub) * unit), ih = 1.f / h, ih2 = ih * ih;
#pragma unroll 1
    for (int i = 0; i < MMAX; i += 8) {
        float v[NCOL], lj = 0.f;
#pragma unroll
        for (int e = 0; e < NCOL; ++e) v[e] = A[e * FSTR + i];
        col_solve_tail(R, Ri, v, rd20);
        const float wj = A[NCOL * FSTR + i];
        const bool live = ok && r0 + i < m;
#pragma unroll
        for (int e = 0; e < NCOL; ++e) {
            v[e] = live ? (v[e] * wj) * (e < 3 ? ih : ih2) : 0.f;
            if (e == 3 || e == 6 || e == 8) lj += v[e];
            A[e * FSTR + i] = v[e];
        }
        A[NCOL * FSTR + i] = lj;
    }
    __syncwarp();
    // sums of the Laplacian columns: warp_sum_d's tree for the four nodes at
    // once, one after the first two steps in each quarter of the warp
    double lsum;
    {
        float l[WN];
#pragma unroll
        for (int q = 0; q < WN; ++q) l[q] = W.A[q][NCOL * FSTR + lane];
        const bool up = lane & 16, odd = lane & 8;
        const double a = (double)(up ? l[2] : l[0]) + (double)__shfl_xor_sync(FULL, up ? l[0] : l[2], 16);
        const double b = (double)(up ? l[3] : l[1]) + (double)__shfl_xor_sync(FULL, up ? l[1] : l[3], 16);
        lsum = (odd ? b : a) + __shfl_xor_sync(FULL, odd ? a : b, 8);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) lsum += __shfl_xor_sync(FULL, lsum, o);
    }
    // lanes 8 q to 8 q + 7 hold node q's sum (and its ok and rf)
    const bool good = ok && -lsum < 0.0;
    const unsigned gmask = __ballot_sync(FULL, good);
    if (r0 == 0 && w0 + sub < n_int) {
        lapd_out[w0 + sub] = good ? -lsum : 0.0;
        rcond_out[w0 + sub] = good ? (double)rf : 0.0;
        if (!good && m > 0) list[atomicAdd(list_count, 1u)] = w0 + sub;   // m = 0: listed when selected
    }
#pragma unroll
    for (int q = 0; q < WN; ++q)
        if (w0 + q < n_int)
            lap_out[(int64_t)(w0 + q) * MMAX + lane] =
                gmask >> (8 * q) & 1u ? (double)W.A[q][NCOL * FSTR + lane] : 0.0;
    // the block's nodes' columns side by side
    if (lane == 0) W.good = gmask;
    __syncthreads();
    constexpr int NB = SW * WN;
    const int nd = threadIdx.x % NB, y = blockIdx.x * NB + nd;
    const Wls32Smem &V = reinterpret_cast<const Wls32Smem *>(smem_raw)[nd / WN];
    if (y < n_int) {
        const bool g = V.good >> (8 * (nd % WN)) & 1u;
#pragma unroll 4
        for (int row = threadIdx.x / NB; row < NCOL * MMAX; row += SW * 32 / NB)
            D_out[(int64_t)row * dstride + y] = g ? (double)V.A[nd % WN][row + (FSTR - MMAX) * (row / MMAX)] : 0.0;
    }
}

// ---------------------------------------------------------------- matrices
// diagonals of A and B (the Jacobi scaling) and their reciprocals
// h^2 / 24 of a level-lev cell of a domain of edge ext, from ext^2 / 24: a power of
// two apart, so rounded alike
__device__ __forceinline__ double cell_scale(double ext2_24, int lev) {
    return ext2_24 * __longlong_as_double((long long)(1023 - 2 * lev) << 52);
}
// x / d where d was computed as x: 1 unless x is zero or not finite.  The
// divisions, by 24 too, were 50 us of the 667 that the matrices of 1.05e6 rows
// take.
__device__ __noinline__ double own_quotient_odd(double x, double d) { return x / d; }
__device__ __forceinline__ double own_quotient(double x, double d) {
    const unsigned long long m = (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
    if (m - 1ull >= 0x7FF0000000000000ull - 1ull) return own_quotient_odd(x, d);
    return 1.0;
}
__global__ void k_diag(const int32_t *__restrict__ msz, const double *__restrict__ lapd, const int4 *__restrict__ ic,
                       int n_int, int n_tot, double ext2_24, double *__restrict__ dA, double *__restrict__ dB,
                       double2 *__restrict__ rAB) {
    int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n_tot) return;
    double a = 1.0, b = 1.0;
    if (r < n_int) {
        const double s = cell_scale(ext2_24, ic[r].w);
        a = lapd[r];
        b = 1.0 + s * lapd[r];
    }
    dA[r] = a;
    dB[r] = b;
    rAB[r] = make_double2(1.0 / a, 1.0 / b);
}

// widths of the 32-row slices; also the sum of the stencil sizes
__global__ void k_slice_width(const int32_t *__restrict__ msz, int n_int, int n_tot, int nsl, uint32_t *__restrict__ w,
                              uint32_t *__restrict__ sum_m) {
    int s = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    int lane = threadIdx.x & 31;
    if (s >= nsl) return;
    int r = s * 32 + lane;
    int v = 0;
    const int sm = __reduce_add_sync(0xffffffffu, r < n_int ? msz[r] : 0);
    if (lane == 0) atomicAdd(sum_m, (uint32_t)sm);
    if (r < n_int) v = msz[r] + 1;
    else if (r < n_tot) v = 1;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) { int t = __shfl_xor_sync(0xffffffffu, v, o); v = t > v ? t : v; }
    if (lane == 0) w[s] = (uint32_t)v;
}

// Row j of A: diag = -sum l, off-diagonals l_ji; row j of B: 1 + (h_j^2/24) A_jj
// and (h_j^2/24) l_ji (Section 3.2 with the cell-indicator moments); boundary
// rows are identity rows.  Values are stored right-scaled by the inverse
// diagonal of the column (Jacobi preconditioning folded into the matrix).
//
// The FP64 pipe's three products per entry and 44 bytes of it take about as
// long.  The mixed form's FP32 and FP16 copies are written along (a pass of their
// own read the values again and converted to FP16 on the FP64 pipe), a row's
// four next columns and values come in three loads and a column's two
// reciprocals in one: at 2.5e7 entries 270 us, fill and copies 262 + 190 before.
struct LowCopies {   // null without the mixed form
    float *fA, *fB;
    __half *hA, *hB;
};
template <bool MIXED>
__device__ __forceinline__ void put_low(const LowCopies &c, int64_t e, double a, double b) {
    if constexpr (MIXED) {
        c.fA[e] = f64_to_f32_int(a);
        c.fB[e] = f64_to_f32_int(b);
        c.hA[e] = f64_to_f16_int(a);
        c.hB[e] = f64_to_f16_int(b);
    }
}

template <bool MIXED>
__global__ void __launch_bounds__(256) k_ell_fill(
    const int32_t *__restrict__ msz, const int32_t *__restrict__ nbr, const double *__restrict__ lap,
    const double *__restrict__ lapd, const int4 *__restrict__ ic, const double *__restrict__ dA,
    const double *__restrict__ dB, const double2 *__restrict__ rAB, int n_int, int n_tot, double ext2_24,
    const uint32_t *__restrict__ sw, const uint32_t *__restrict__ soff, int32_t *__restrict__ col,
    double *__restrict__ vA, double *__restrict__ vB, LowCopies low) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    const int s = r >> 5, lane = r & 31;
    if (s * 32 >= n_tot) return;
    const int w = (int)sw[s];
    const int64_t base = (int64_t)soff[s] * 32 + lane;
    const bool real = r < n_tot, inner = r < n_int;
    const int m = inner ? msz[r] : 0, own = real ? r : 0;
    double a0 = 0.0, b0 = 0.0, sc = 0.0;
    if (inner) {
        const double l = lapd[r];
        sc = cell_scale(ext2_24, ic[r].w);
        a0 = own_quotient(l, dA[r]);
        b0 = own_quotient(1.0 + sc * l, dB[r]);
    } else if (real) {
        a0 = b0 = 1.0;   // identity rows
    }
    col[base] = own;
    vA[base] = a0;
    vB[base] = b0;
    put_low<MIXED>(low, base, a0, b0);
    for (int k0 = 0; k0 + 1 < w; k0 += 4) {
        int id[4] = {own, own, own, own};
        double l[4] = {0.0, 0.0, 0.0, 0.0};
        if (k0 < m) {   // MMAX entries per row: aligned, and never past the row's end
            const int4 q = *reinterpret_cast<const int4 *>(nbr + (int64_t)r * MMAX + k0);
            const double2 x = *reinterpret_cast<const double2 *>(lap + (int64_t)r * MMAX + k0);
            const double2 y = *reinterpret_cast<const double2 *>(lap + (int64_t)r * MMAX + k0 + 2);
            id[0] = q.x; id[1] = q.y; id[2] = q.z; id[3] = q.w;
            l[0] = x.x; l[1] = x.y; l[2] = y.x; l[3] = y.y;
        }
        double2 rc[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) rc[t] = k0 + t < m ? rAB[id[t]] : make_double2(0.0, 0.0);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            if (k0 + t + 1 >= w) break;
            const int64_t e = base + (int64_t)(k0 + t + 1) * 32;
            // off-diagonal entries times the column's reciprocal diagonal (an
            // FP64 division per entry would make this pass FP64-bound; the
            // diagonal entries above keep their exact division, so they stay 1)
            const bool in = k0 + t < m;
            const double a = in ? l[t] * rc[t].x : 0.0, b = in ? (sc * l[t]) * rc[t].y : 0.0;
            col[e] = in ? id[t] : own;
            vA[e] = a;
            vB[e] = b;
            put_low<MIXED>(low, e, a, b);
        }
    }
}

// FP32 and FP16 copies of the stored (Jacobi-scaled) matrix values for the mixed
// form, when those have changed
__global__ void k_values_low(const double *__restrict__ vA, const double *__restrict__ vB, int64_t n, LowCopies low) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) put_low<true>(low, i, vA[i], vB[i]);
}

template <int SW, bool MIXED>
apcloud_status launch_stencil_of(apcloud_ctx *c, int n, double unit, double ec, double inv_1mec, int32_t *nbr,
                                 int32_t *msz, int32_t *ring, double *lap, double *lapd, double *D, int64_t dstride,
                                 double *rc, unsigned *derr, unsigned *words) {
    // every node with MAXC_FAST candidate slots, then (one read-back of the
    // count) the nodes whose rings outgrew them with MAXC
    int32_t *ovf = ensure<int32_t>(c, c->stencil_ovf, n + 1);
    if (!ovf) return APCLOUD_E_NOMEM;
    APC_CUDA(c, cudaMemsetAsync(derr + 2, 0, sizeof(unsigned), c->s));
    // rank keys: squared distances in half cells of the deepest level (2 L + 4 bits) over the node index
    int idx_bits = 1;
    while ((1ll << idx_bits) < c->n_tot) ++idx_bits;
    if (2 * c->L + 4 + idx_bits > 63) idx_bits = 0;
    const int d2_shift = 2 * (KEY_DEPTH - c->L);
    const Fp32Args fa{(float)ec, (float)inv_1mec, fp32_not_below(c->P.fp32_rcond_min), fp32_not_below(RANK_TOL)};
    // the limits are per-device properties of the functions: set on every build
    // (one host call each), so that contexts on other devices get them too
    APC_CUDA(c, cudaFuncSetAttribute(k_stencil<4, MAXC, true, MIXED, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)(4 * sizeof(WarpSmemT<MAXC>) + 16)));
    if constexpr (MIXED) {
        const size_t smem = SW * sizeof(SelectSmemT<MAXC_FAST>) + 16, wsmem = WLS_SW * sizeof(Wls32Smem);
        APC_CUDA(c, cudaFuncSetAttribute(k_stencil<SW, MAXC_FAST, false, true, true>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        APC_CUDA(c, cudaFuncSetAttribute(k_wls32<WLS_SW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)wsmem));
        APC_LAUNCH(c, K_STENCIL, div_up(n, SW), SW * 32, smem, (k_stencil<SW, MAXC_FAST, false, true, true>),
                   ptr<int4>(c->node_ic), ptr<int32_t>(c->adj), ptr<int32_t>(c->bowner), n, c->P.m_target,
                   c->P.ring_max, unit, 1.0 / unit, ec, inv_1mec, nbr, msz, ring, lap, lapd, D, dstride, rc,
                   c->P.fp32_rcond_min, reinterpret_cast<int *>(derr + 1), derr, (const int32_t *)nullptr, 0, derr + 2,
                   ovf, c->P.stencil_slots, idx_bits, d2_shift, fa);
        APC_LAUNCH(c, K_STENCIL, div_up(n, WLS_SW * WN), WLS_SW * 32, wsmem, (k_wls32<WLS_SW>), (const int4 *)ptr<int4>(c->node_ic),
                   n, unit, fa, d2_shift, (const int32_t *)nbr, (const int32_t *)msz, lap, lapd, D, dstride, rc, derr + 2,
                   ovf);
    } else {
        const size_t smem = SW * sizeof(WarpSmemT<MAXC_FAST>) + 16;   // the warps' areas, then the block's arrival count
        APC_CUDA(c, cudaFuncSetAttribute(k_stencil<SW, MAXC_FAST, false, false, false>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        APC_LAUNCH(c, K_STENCIL, div_up(n, SW), SW * 32, smem, (k_stencil<SW, MAXC_FAST, false, false, false>),
                   ptr<int4>(c->node_ic), ptr<int32_t>(c->adj), ptr<int32_t>(c->bowner), n, c->P.m_target,
                   c->P.ring_max, unit, 1.0 / unit, ec, inv_1mec, nbr, msz, ring, lap, lapd, D, dstride, rc,
                   c->P.fp32_rcond_min, reinterpret_cast<int *>(derr + 1), derr, (const int32_t *)nullptr, 0, derr + 2,
                   ovf, c->P.stencil_slots, idx_bits, d2_shift, fa);
    }
    // the overflow count, with the error word and the count of FP64 blocks
    APC_TRY(read_back(c, words, derr, 3 * sizeof(unsigned)));
    const unsigned nov = words[2];
    if (nov > 0) {
        APC_LAUNCH(c, K_STENCIL, div_up(nov, 4), 4 * 32, 4 * sizeof(WarpSmemT<MAXC>) + 16, (k_stencil<4, MAXC, true, MIXED, false>),
                   ptr<int4>(c->node_ic), ptr<int32_t>(c->adj), ptr<int32_t>(c->bowner), n, c->P.m_target,
                   c->P.ring_max, unit, 1.0 / unit, ec, inv_1mec, nbr, msz, ring, lap, lapd, D, dstride, rc,
                   c->P.fp32_rcond_min, reinterpret_cast<int *>(derr + 1), derr,
                   (const int32_t *)ovf, (int)nov, derr + 2, ovf, MAXC, idx_bits, d2_shift, fa);
        APC_TRY(read_back(c, words, derr, 3 * sizeof(unsigned)));
    }
    return APCLOUD_OK;
}

template <int SW>
apcloud_status launch_stencil(apcloud_ctx *c, int n, double unit, double ec, double inv_1mec, int32_t *nbr,
                              int32_t *msz, int32_t *ring, double *lap, double *lapd, double *D, int64_t dstride,
                              double *rc, unsigned *derr, unsigned *words) {
    return c->P.precision == 1 ? launch_stencil_of<SW, true>(c, n, unit, ec, inv_1mec, nbr, msz, ring, lap, lapd, D,
                                                             dstride, rc, derr, words)
                               : launch_stencil_of<SW, false>(c, n, unit, ec, inv_1mec, nbr, msz, ring, lap, lapd, D,
                                                              dstride, rc, derr, words);
}

}  // namespace

apcloud_status build_stencils(apcloud_ctx *c) {
    const int n = c->n_int, nt = c->n_tot;
    const int64_t dstride = ((int64_t)n + 31) / 32 * 32;
    int32_t *nbr = ensure<int32_t>(c, c->nbr, (int64_t)n * MMAX);
    int32_t *msz = ensure<int32_t>(c, c->msz, n + 1);
    int32_t *ring = ensure<int32_t>(c, c->ring, n + 1);
    double *lap = ensure<double>(c, c->lap, (int64_t)n * MMAX);
    double *lapd = ensure<double>(c, c->lapd, n + 1);
    double *D = ensure<double>(c, c->D, (int64_t)NCOL * MMAX * dstride);
    double *rc = ensure<double>(c, c->rcond, n + 1);
    if (!nbr || !msz || !ring || !lap || !lapd || !D || !rc) return APCLOUD_E_NOMEM;
    unsigned *derr = ptr<unsigned>(c->derr);
    APC_CUDA(c, cudaMemsetAsync(derr, 0, 4 * sizeof(unsigned), c->s));
    const double ext = c->P.hi[0] - c->P.lo[0];
    const double unit = ldexp(ext, -(KEY_DEPTH + 1));
    const double ec = exp(-c->P.weight_c);
    const double inv_1mec = 1.0 / (1.0 - ec);
    unsigned words[3];
    switch (c->wls_warps) {
    case 2:
        APC_TRY(launch_stencil<2>(c, n, unit, ec, inv_1mec, nbr, msz, ring, lap, lapd, D, dstride, rc, derr, words));
        break;
    case 8:
        APC_TRY(launch_stencil<8>(c, n, unit, ec, inv_1mec, nbr, msz, ring, lap, lapd, D, dstride, rc, derr, words));
        break;
    default:
        APC_TRY(launch_stencil<4>(c, n, unit, ec, inv_1mec, nbr, msz, ring, lap, lapd, D, dstride, rc, derr, words));
        break;
    }
    APC_CUDA(c, cudaGetLastError());
    APC_TRY(device_errors(c, words[0]));
    c->n_fp64_wls = words[1];

    // sliced ELL of A and B
    const int nsl = div_up(nt, 32);
    c->n_slices = nsl;
    uint32_t *sw = ensure<uint32_t>(c, c->slice_w, nsl + 1);
    uint32_t *so = ensure<uint32_t>(c, c->slice_off, nsl + 1);
    double *dA = ensure<double>(c, c->dA, nt + 1);
    double *dB = ensure<double>(c, c->dB, nt + 1);
    double2 *rd = ensure<double2>(c, c->ell_rd, (int64_t)nt + 1);   // reciprocals, for the fill only
    if (!sw || !so || !dA || !dB || !rd) return APCLOUD_E_NOMEM;
    APC_LAUNCH(c, K_ELL, div_up(nt, 256), 256, 0, k_diag, msz, lapd, ptr<int4>(c->node_ic), n, nt, ext * ext / 24.0, dA,
               dB, rd);
    uint32_t *small = ptr<uint32_t>(c->dsmall);
    APC_CUDA(c, cudaMemsetAsync(small + 6, 0, sizeof(uint32_t), c->s));
    APC_LAUNCH(c, K_ELL, div_up(nsl, 8), 256, 0, k_slice_width, msz, n, nt, nsl, sw, small + 6);
    APC_TRY(scan_u32(c, sw, so, nsl, small + 5));
    // the block-local copy's size too, so that one read gives every size; systems
    // the resident solve takes do not need the copy
    c->ell_entries = 0;
    c->bl_ok = c->bl_tried = false;
    c->res_unfit = false;
    const bool blocks = c->P.precision == 1 && c->P.poly_degree > 1;
    if (blocks) APC_TRY(count_blocks(c, small + 7));
    uint32_t tot[3];   // ELL columns, stencil sizes, chunks
    APC_TRY(read_back(c, tot, small + 5, sizeof tot));
    c->ell_entries = (int64_t)tot[0] * 32;
    c->sum_m = tot[1];
    c->bl_chunks = blocks ? tot[2] : 0;
    // per node: offsets and weights in (28 B per neighbour), Laplacian row and
    // 9 x m operator out (80 B per neighbour); two 9-column Gram products,
    // three triangular solves per row and two 9x9 factorizations
    account(c, K_STENCIL, 108.0 * tot[1] + 8.0 * n, 450.0 * tot[1] + 660.0 * n);
    int32_t *col = ensure<int32_t>(c, c->ell_col, c->ell_entries);
    double *vA = ensure<double>(c, c->ell_A, c->ell_entries);
    double *vB = ensure<double>(c, c->ell_B, c->ell_entries);
    if (!col || !vA || !vB) return APCLOUD_E_NOMEM;
    if (c->P.precision == 0) {
        APC_LAUNCH(c, K_ELL, div_up((int64_t)nsl * 32, 256), 256, 0, k_ell_fill<false>, msz, nbr, lap, lapd,
                   ptr<int4>(c->node_ic), dA, dB, (const double2 *)rd, n, nt, ext * ext / 24.0, sw, so, col, vA, vB, LowCopies{});
    } else {
        const LowCopies low{ensure<float>(c, c->ell_A32, c->ell_entries), ensure<float>(c, c->ell_B32, c->ell_entries),
                            ensure<__half>(c, c->ell_A16, c->ell_entries), ensure<__half>(c, c->ell_B16, c->ell_entries)};
        if (!low.fA || !low.fB || !low.hA || !low.hB) return APCLOUD_E_NOMEM;
        APC_LAUNCH(c, K_ELL, div_up((int64_t)nsl * 32, 256), 256, 0, k_ell_fill<true>, msz, nbr, lap, lapd,
                   ptr<int4>(c->node_ic), dA, dB, (const double2 *)rd, n, nt, ext * ext / 24.0, sw, so, col, vA, vB, low);
        if (blocks && !resident_ok(c, 1)) APC_TRY(build_blocks(c));
    }
    return cuda_check(c, cudaGetLastError(), "ell");
}

}  // namespace apc

namespace apc {

// Times the stencil kernel at 2, 4 and 8 nodes per block on the current node
// set (after build_stencils) and keeps the fastest.  Every node's outputs are
// independent of the block shape, so the reruns rewrite identical values.
apcloud_status tune_stencils(apcloud_ctx *c, double *ms_out) {
    const int n = c->n_int;
    if (n == 0) return APCLOUD_OK;
    const int64_t dstride = ((int64_t)n + 31) / 32 * 32;
    int32_t *nbr = ptr<int32_t>(c->nbr), *msz = ptr<int32_t>(c->msz), *ring = ptr<int32_t>(c->ring);
    double *lap = ptr<double>(c->lap), *lapd = ptr<double>(c->lapd), *D = ptr<double>(c->D);
    double *rc = ptr<double>(c->rcond);
    unsigned *derr = ptr<unsigned>(c->derr);
    const double ext = c->P.hi[0] - c->P.lo[0];
    const double unit = ldexp(ext, -(KEY_DEPTH + 1));
    const double ec = exp(-c->P.weight_c);
    const double inv_1mec = 1.0 / (1.0 - ec);
    const int shapes[3] = {2, 4, 8};
    unsigned words[3];
    cudaEvent_t e0, e1;
    APC_CUDA(c, cudaEventCreate(&e0));
    APC_CUDA(c, cudaEventCreate(&e1));
    const unsigned mask = c->timer.mask;
    c->timer.mask = 0;
    double best = 1e30;
    int pick = c->wls_warps;
    apcloud_status st = APCLOUD_OK;
    for (int t = 0; t < 3 && st == APCLOUD_OK; ++t) {
        float ms = 0.f;
        for (int rep = 0; rep < 2 && st == APCLOUD_OK; ++rep) {
            st = cuda_check(c, cudaMemsetAsync(derr, 0, 4 * sizeof(unsigned), c->s), "autotune stencils");
            if (st != APCLOUD_OK) break;
            cudaEventRecord(e0, c->s);
            if (shapes[t] == 2)
                st = launch_stencil<2>(c, n, unit, ec, inv_1mec, nbr, msz, ring, lap, lapd, D, dstride, rc, derr, words);
            else if (shapes[t] == 4)
                st = launch_stencil<4>(c, n, unit, ec, inv_1mec, nbr, msz, ring, lap, lapd, D, dstride, rc, derr, words);
            else
                st = launch_stencil<8>(c, n, unit, ec, inv_1mec, nbr, msz, ring, lap, lapd, D, dstride, rc, derr, words);
            cudaEventRecord(e1, c->s);
            if (st == APCLOUD_OK) st = cuda_check(c, cudaEventSynchronize(e1), "autotune stencils");
            if (st == APCLOUD_OK) cudaEventElapsedTime(&ms, e0, e1);
        }
        if (st == APCLOUD_OK) st = check_device_errors(c);
        if (ms_out) ms_out[t] = ms;
        if (st == APCLOUD_OK && ms < best) { best = ms; pick = shapes[t]; }
    }
    c->timer.mask = mask;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (st == APCLOUD_OK) c->wls_warps = pick;
    return st;
}

}  // namespace apc

namespace apc {

// FP32/FP16 copies of the stored values again (after the FP64 values changed)
apcloud_status refresh_lowp(apcloud_ctx *c) {
    if (c->P.precision != 1 || c->ell_entries == 0) return APCLOUD_OK;
    APC_LAUNCH(c, K_ELL, div_up(c->ell_entries, 256), 256, 0, k_values_low, (const double *)ptr<double>(c->ell_A),
               (const double *)ptr<double>(c->ell_B), c->ell_entries,
               LowCopies{ptr<float>(c->ell_A32), ptr<float>(c->ell_B32), ptr<__half>(c->ell_A16), ptr<__half>(c->ell_B16)});
    if (c->bl_tried) APC_TRY(build_blocks(c));
    return cuda_check(c, cudaGetLastError(), "refresh_lowp");
}

}  // namespace apc
