// gather.cu -- Section 3.2 step 3: GFD gradient and Hessian of phi at every
// interior node, and second-order Taylor interpolation of phi and E = grad phi
// (Section 2) from the centre of each particle's own leaf.
//
// Node pass: one thread per node walks its ELL row (the stencil neighbours in
// order) and the derivative operator stored with nodes fastest, so the loads
// of a warp are contiguous.  Particle pass: one thread per particle in the
// caller's order reads the particle's leaf (recorded when the tree was
// built), its position, the leaf's centre and its record (potential and
// derivatives), and writes phi and E coalesced; the particle streams bypass L2
// retention so the node records stay cached.  Interpolation at arbitrary
// points (no recorded leaf) recomputes the point's Morton key and finds its
// leaf by binary search over the Morton-ordered leaf anchors (the leaves
// partition the key space).
#include <cmath>

#include "fpconv.cuh"
#include "internal.cuh"

namespace apc {

namespace {

// per-node record: phi, 9 derivatives, the node's centre, 1 pad.  A centre
// computed per particle from the integer coordinates cost 9 of the 33 FP64
// instructions of the FP64 particle pass, which the FP64 pipe bounds (824 us for
// 2e7 particles, 1183 before); here each node computes it once, the same way.
constexpr int NF = NODE_RECORD;
// compact per-node record of the mixed form's particle pass, 80 bytes in 4-byte
// words: phi and the node centre (FP64, words 0-7), gradient and Hessian
// fx fy fz fxx fxy fxz fyy fyz fzz (FP32, words 8-16), pad
constexpr int NF32 = 20;
constexpr int GT = 256;  // threads of the mixed form's particle pass

// Ten FP64 instructions per stencil entry keep the FP64 pipe busy four fifths of
// the time; the operator's 72 bytes per entry take about as long as it leaves.
// Two entries per step put the second's loads behind the first's arithmetic:
// 141 us for 265186 nodes (150 one at a time, 183 with four: registers).
__global__ void k_derivs(const uint32_t *__restrict__ sw, const uint32_t *__restrict__ soff,
                         const int32_t *__restrict__ col, const double *__restrict__ D, int64_t dstride,
                         const double *__restrict__ phi, int n_int, double *__restrict__ nf,
                         const int4 *__restrict__ ic, double lo0, double lo1, double lo2, double unit,
                         float *__restrict__ nf32) {
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n_int) return;
    const int sl = j >> 5, lane = j & 31;
    const int w = (int)sw[sl];
    const int64_t base = (int64_t)soff[sl] * 32 + lane;
    const double p0 = phi[j];
    double acc[NCOL];
#pragma unroll
    for (int r = 0; r < NCOL; ++r) acc[r] = 0.0;
#pragma unroll 2
    for (int k = 1; k < w; ++k) {
        const int cj = col[base + (int64_t)k * 32];
        const double diff = phi[cj] - p0;
#pragma unroll
        for (int r = 0; r < NCOL; ++r) acc[r] = fma(D[((int64_t)r * MMAX + (k - 1)) * dstride + j], diff, acc[r]);
    }
    double *o = nf + (int64_t)j * NF;
    o[0] = p0;
#pragma unroll
    for (int r = 0; r < NCOL; ++r) o[1 + r] = acc[r];
    const int4 q = ic[j];
    const double c0 = __dadd_rn(lo0, __dmul_rn((double)q.x, unit)), c1 = __dadd_rn(lo1, __dmul_rn((double)q.y, unit)),
                 c2d = __dadd_rn(lo2, __dmul_rn((double)q.z, unit));
    o[10] = c0;
    o[11] = c1;
    o[12] = c2d;
    o[13] = 0.0;
    if (nf32) {
        double2 *c2 = reinterpret_cast<double2 *>(nf32 + (int64_t)j * NF32);
        c2[0] = make_double2(p0, c0);
        c2[1] = make_double2(c1, c2d);
        float4 *f4 = reinterpret_cast<float4 *>(nf32 + (int64_t)j * NF32 + 8);
        f4[0] = make_float4((float)acc[0], (float)acc[1], (float)acc[2], (float)acc[3]);
        f4[1] = make_float4((float)acc[4], (float)acc[5], (float)acc[6], (float)acc[7]);
        f4[2] = make_float4((float)acc[8], 0.f, 0.f, 0.f);
    }
}

__device__ __forceinline__ int leaf_of(const uint64_t *anchor, int n, uint64_t v) {
    int lo = 0, hi = n;
    while (lo < hi) {
        int mid = (lo + hi) >> 1;
        if (__ldg(anchor + mid) <= v) lo = mid + 1; else hi = mid;
    }
    return lo - 1;
}

// Second-order Taylor expansion about the leaf centre (Section 3.2 step 3):
// phi_p = phi + g.r + r.H.r / 2, E_p = g + H r (E = grad phi, Section 2).
__device__ __forceinline__ void taylor(const double *__restrict__ nf, int j, double x0, double x1, double x2,
                                       double &php, double &ex, double &ey, double &ez) {
    const double2 *f2 = reinterpret_cast<const double2 *>(nf + (int64_t)j * NF);
    const double2 a = f2[0], b = f2[1], c = f2[2], d = f2[3], e = f2[4], ctr = f2[5];
    const double r0 = x0 - ctr.x, r1 = x1 - ctr.y, r2 = x2 - f2[6].x;
    // a = (phi, fx), b = (fy, fz), c = (fxx, fxy), d = (fxz, fyy), e = (fyz, fzz)
    const double hr0 = c.x * r0 + c.y * r1 + d.x * r2;
    const double hr1 = c.y * r0 + d.y * r1 + e.x * r2;
    const double hr2 = d.x * r0 + e.x * r1 + e.y * r2;
    const double g0 = a.y, g1 = b.x, g2 = b.y;
    php = a.x + (g0 * r0 + g1 * r1 + g2 * r2) + 0.5 * (r0 * hr0 + r1 * hr1 + r2 * hr2);
    ex = g0 + hr0;
    ey = g1 + hr1;
    ez = g2 + hr2;
}

__global__ void __launch_bounds__(256) k_gather_leaf(
    const double *__restrict__ x, const double *__restrict__ y, const double *__restrict__ z, int64_t n,
    const int32_t *__restrict__ pleaf, const double *__restrict__ nf, double *__restrict__ php, double *__restrict__ ex, double *__restrict__ ey,
    double *__restrict__ ez) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int j = __ldcs(pleaf + i);
    const double p0 = __ldcs(x + i), p1 = __ldcs(y + i), p2 = __ldcs(z + i);
    double v, gx, gy, gz;
    taylor(nf, j, p0, p1, p2, v, gx, gy, gz);
    if (php) __stcs(php + i, v);
    if (ex) __stcs(ex + i, gx);
    if (ey) __stcs(ey + i, gy);
    if (ez) __stcs(ez + i, gz);
}

// the two doubles of a 16-byte part of a record
__device__ __forceinline__ double f4_lo(const float4 &v) {
    return __hiloint2double(__float_as_int(v.y), __float_as_int(v.x));
}
__device__ __forceinline__ double f4_hi(const float4 &v) {
    return __hiloint2double(__float_as_int(v.w), __float_as_int(v.z));
}

// The mixed form: corrections (g.r, H r, r.H.r) in FP32 around the FP64 node
// potential, from the compact record; its node derivatives carry FP32 accuracy
// already (FP32 stencils).  The pass stays off the slow FP64 pipe but for the
// offsets from the centre and the potential's add: the seven double/float
// conversions run on the integer pipe.
//
// A record per lane costs five loads of as many lines as the warp has different
// leaves.  With few leaves (their records in L1) or with particles in cell order
// that is little.  Particles in any order on many leaves take 160 L1 look-ups a
// warp; there (STAGED) a warp fetches its 32 records together, the five 16-byte
// parts of a record by neighbouring lanes (a third of the look-ups), and hands
// them over through shared memory (rows of 80 bytes: no bank conflicts), which
// costs the same whatever the leaves.  2e7 particles, a record per lane / staged:
//     leaves               1128       5104       26202      36807      215111     320804
//     in any order      241 / 293  251 / 304  292 / 295  301 / 294  312 / 295  313 / 297 us
//     pairs in a leaf   238 / 287  246 / 289  250 / 289  250 / 288  252 / 288  254 / 291
//     in cell order     235 / 280  235 / 279  236 / 280  235 / 280  243 / 292  245 / 297
// Hence STAGED_LEAVES, and staged only where the warps of a sample taken with the
// tree hold nearly as many leaves as particles (c->scattered).  A choice by each warp
// keeps the shared memory out of L1 in either case: 272 in place of 243 us in cell
// order.  Records of 96 or 128 bytes change nothing; loads past L1 (358 us) and
// asynchronous copies into shared memory (310 us) lose.
template <bool STAGED>
__global__ void __launch_bounds__(GT) k_gather_leaf32(
    const double *__restrict__ x, const double *__restrict__ y, const double *__restrict__ z, int64_t n,
    const int32_t *__restrict__ pleaf, const float *__restrict__ nf32, double *__restrict__ php,
    double *__restrict__ ex, double *__restrict__ ey, double *__restrict__ ez) {
    const int64_t i = (int64_t)blockIdx.x * GT + threadIdx.x;
    const bool live = i < n;
    if (!STAGED && !live) return;
    const int j = live ? __ldcs(pleaf + i) : 0;
    const double p0 = live ? __ldcs(x + i) : 0.0, p1 = live ? __ldcs(y + i) : 0.0, p2 = live ? __ldcs(z + i) : 0.0;
    float4 f[5];
    if constexpr (STAGED) {
        __shared__ float4 rec[GT * 5];
        const int lane = threadIdx.x & 31;
        float4 *mine = rec + (threadIdx.x - lane) * 5;
#pragma unroll
        for (int t = 0; t < 5; ++t) {
            const int e = t * 32 + lane, o = e / 5;
            const int jo = __shfl_sync(0xFFFFFFFFu, j, o);
            f[t] = __ldg(reinterpret_cast<const float4 *>(nf32 + (int64_t)jo * NF32) + (e - o * 5));
        }
#pragma unroll
        for (int t = 0; t < 5; ++t) mine[t * 32 + lane] = f[t];
        __syncwarp();
        if (!live) return;
#pragma unroll
        for (int t = 0; t < 5; ++t) f[t] = mine[lane * 5 + t];
    } else {
        const float4 *r = reinterpret_cast<const float4 *>(nf32 + (int64_t)j * NF32);
#pragma unroll
        for (int t = 0; t < 5; ++t) f[t] = __ldg(r + t);
    }
    const double pc = f4_lo(f[0]), cx = f4_hi(f[0]), cy = f4_lo(f[1]), cz = f4_hi(f[1]);
    const float4 u = f[2], w = f[3];
    const float fzz = f[4].x;
    const float r0 = f64_to_f32_int(p0 - cx), r1 = f64_to_f32_int(p1 - cy), r2 = f64_to_f32_int(p2 - cz);
    // u = (fx, fy, fz, fxx), w = (fxy, fxz, fyy, fyz)
    const float hr0 = fmaf(w.y, r2, fmaf(w.x, r1, u.w * r0));
    const float hr1 = fmaf(w.w, r2, fmaf(w.z, r1, w.x * r0));
    const float hr2 = fmaf(fzz, r2, fmaf(w.w, r1, w.y * r0));
    const float corr = fmaf(u.z, r2, fmaf(u.y, r1, u.x * r0)) + 0.5f * fmaf(r2, hr2, fmaf(r1, hr1, r0 * hr0));
    if (php) __stcs(php + i, pc + f32_to_f64_int(corr));
    if (ex) __stcs(ex + i, f32_to_f64_int(u.x + hr0));
    if (ey) __stcs(ey + i, f32_to_f64_int(u.y + hr1));
    if (ez) __stcs(ez + i, f32_to_f64_int(u.z + hr2));
}

__global__ void k_gather(const double *__restrict__ x, const double *__restrict__ y, const double *__restrict__ z,
                         int64_t n, double lo0, double lo1, double lo2, double s, int shift,
                         const int64_t *__restrict__ offs, int nb, int L, const uint64_t *__restrict__ anchor, int n_int,
                         const double *__restrict__ nf, double *__restrict__ php, double *__restrict__ ex,
                         double *__restrict__ ey, double *__restrict__ ez) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double p[3] = {x[i], y[i], z[i]};
    const double lo[3] = {lo0, lo1, lo2};
    uint32_t cc[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        double t = floor(__dmul_rn(__dsub_rn(p[d], lo[d]), s));
        t = fmin(fmax(t, 0.0), (double)((1u << KEY_DEPTH) - 1u));
        cc[d] = (uint32_t)t >> shift;
    }
    uint64_t pre = 0;
    if (nb > 1) {   // beam of particle i from the batch offsets
        int lo = 0, hi = nb;
        while (hi - lo > 1) {
            int mid = (lo + hi) >> 1;
            if (offs[mid] <= i) lo = mid; else hi = mid;
        }
        pre = (uint64_t)lo << (3 * L);
    }
    const int j = leaf_of(anchor, n_int, pre | morton(cc[0], cc[1], cc[2]));
    double v, gx, gy, gz;
    taylor(nf, j, p[0], p[1], p[2], v, gx, gy, gz);
    if (php) php[i] = v;
    if (ex) ex[i] = gx;
    if (ey) ey[i] = gy;
    if (ez) ez[i] = gz;
}

}  // namespace

apcloud_status gather_field(apcloud_ctx *c, double *phi_p, double *ex, double *ey, double *ez) {
    const int n = c->n_int;
    const bool mixed = c->P.precision == 1;
    double *nf = ensure<double>(c, c->nodefield, (int64_t)n * NF);
    float *nf32 = mixed ? ensure<float>(c, c->nodefield32, (int64_t)n * NF32 + 4) : nullptr;
    if (!nf || (mixed && !nf32)) return APCLOUD_E_NOMEM;
    const int64_t dstride = ((int64_t)n + 31) / 32 * 32;
    const double ext = c->P.hi[0] - c->P.lo[0];
    const double unit = ldexp(ext, -(KEY_DEPTH + 1));
    // few nodes: single warps, so that their FP64 work spreads over the SMs (1500
    // nodes in blocks of 128 are 12 SMs' work: 43 us)
    const int db = n < 128 * 4 * sm_count() ? 32 : 128;
    APC_LAUNCH(c, K_DERIV, div_up(n, db), db, 0, k_derivs, ptr<uint32_t>(c->slice_w), ptr<uint32_t>(c->slice_off),
               ptr<int32_t>(c->ell_col), ptr<double>(c->D), dstride, ptr<double>(c->phi), n, nf,
               ptr<int4>(c->node_ic), c->P.lo[0], c->P.lo[1], c->P.lo[2], unit, nf32);
    if (mixed && c->scattered)
        APC_LAUNCH(c, K_GATHER, div_up(c->N, GT), GT, 0, k_gather_leaf32<true>, c->px, c->py, c->pz, c->N,
                   (const int32_t *)ptr<int32_t>(c->pleaf), (const float *)nf32, phi_p, ex, ey, ez);
    else if (mixed)
        APC_LAUNCH(c, K_GATHER, div_up(c->N, GT), GT, 0, k_gather_leaf32<false>, c->px, c->py, c->pz, c->N,
                   (const int32_t *)ptr<int32_t>(c->pleaf), (const float *)nf32, phi_p, ex, ey, ez);
    else
        APC_LAUNCH(c, K_GATHER, div_up(c->N, 256), 256, 0, k_gather_leaf, c->px, c->py, c->pz, c->N,
                   (const int32_t *)ptr<int32_t>(c->pleaf), (const double *)nf, phi_p, ex, ey, ez);
    // node pass: operator (72 B), column (4 B) and neighbour value (8 B) per
    // stencil entry plus the 112 B record (and the 80 B compact record of the
    // mixed form); particle pass: leaf index and position in (28 B), phi and E
    // out (32 B), and each leaf's record once (FP64: 112 B; mixed: the 80 B
    // compact record)
    account(c, K_DERIV, 84.0 * c->sum_m + (mixed ? 216.0 : 136.0) * n, 19.0 * c->sum_m);
    account(c, K_GATHER, 60.0 * c->N + (mixed ? 80.0 : 112.0) * n, 29.0 * c->N);
    return cuda_check(c, cudaGetLastError(), "gather");
}

}  // namespace apc

// ---------------------------------------------------------------- time stepping support
namespace apc {
namespace {

// Leapfrog half steps for particles with charge-to-mass ratio qm in the field
// E = grad phi (Section 2): v += qm dt_kick E, then x += dt_drift v, with
// specular reflection at the walls of the cubic domain.
//
// The tests and clamps were half of the FP64 instructions that bound the pass:
// 66 us for 1e6 particles.  A position strictly inside takes none, told apart on
// the integer pipe: 22 us (64 with every particle past a wall).
__device__ __noinline__ void push_wall(double &p, double &v, double lo, double hi, int64_t klo, int64_t khi) {
    const bool nan = (__double_as_longlong(p) & 0x7FFFFFFFFFFFFFFFll) > 0x7FF0000000000000ll;
    if (!nan && f64_order_key(p) > khi) { p = 2.0 * hi - p; v = -v; }
    if (!nan && f64_order_key(p) < klo) { p = 2.0 * lo - p; v = -v; }
    p = fmin(fmax(p, lo), hi);
}
__global__ void k_push(double *__restrict__ x, double *__restrict__ y, double *__restrict__ z,
                       double *__restrict__ vx, double *__restrict__ vy, double *__restrict__ vz, int64_t n,
                       const double *__restrict__ ex, const double *__restrict__ ey, const double *__restrict__ ez,
                       double qm_dt, double dt, double lo, double hi) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double p[3] = {x[i], y[i], z[i]}, v[3] = {vx[i], vy[i], vz[i]};
    const int64_t klo = f64_order_key(lo), khi = f64_order_key(hi);
    if (ex) { v[0] += qm_dt * ex[i]; v[1] += qm_dt * ey[i]; v[2] += qm_dt * ez[i]; }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        p[d] += dt * v[d];
        const int64_t k = f64_order_key(p[d]);   // NaN: beyond either end
        if (!(k > klo && k < khi)) push_wall(p[d], v[d], lo, hi, klo, khi);
    }
    x[i] = p[0]; y[i] = p[1]; z[i] = p[2];
    vx[i] = v[0]; vy[i] = v[1]; vz[i] = v[2];
}

// W = 1/2 sum over leaves of |grad phi|^2 h^3 (node derivatives times cell volume),
// one block, fixed summation order
__global__ void k_field_energy(const double *__restrict__ nf, const int4 *__restrict__ ic, int n, double ext,
                               double *__restrict__ out) {
    __shared__ double sh[1024];
    double s = 0.0;
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        const double *f = nf + (int64_t)j * NF;
        double h = ldexp(ext, -ic[j].w);
        s += (f[1] * f[1] + f[2] * f[2] + f[3] * f[3]) * (h * h * h);
    }
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = 0.5 * sh[0];
}

}  // namespace

apcloud_status interpolate_phi(apcloud_ctx *c, const double *x, const double *y, const double *z, int64_t n,
                               double *phi) {
    const double ext = c->P.hi[0] - c->P.lo[0];
    const double s = ldexp(1.0, KEY_DEPTH) / ext;
    APC_LAUNCH(c, K_GATHER, div_up(n, 256), 256, 0, k_gather, x, y, z, n, c->P.lo[0], c->P.lo[1], c->P.lo[2], s,
               KEY_DEPTH - c->L, (const int64_t *)nullptr, 1, c->L, ptr<uint64_t>(c->leaf_anchor), c->n_int,
               ptr<double>(c->nodefield), phi, (double *)nullptr, (double *)nullptr, (double *)nullptr);
    return cuda_check(c, cudaGetLastError(), "interpolate");
}

apcloud_status push(apcloud_ctx *c, double *x, double *y, double *z, double *vx, double *vy, double *vz, int64_t n,
                    const double *ex, const double *ey, const double *ez, double qm_dt, double dt) {
    APC_LAUNCH(c, K_VEC, div_up(n, 256), 256, 0, k_push, x, y, z, vx, vy, vz, n, ex, ey, ez, qm_dt, dt, c->P.lo[0],
               c->P.hi[0]);
    return cuda_check(c, cudaGetLastError(), "push");
}

apcloud_status field_energy(apcloud_ctx *c, double *h_out) {
    double *tmp = ensure<double>(c, c->tmp, 2);
    if (!tmp) return APCLOUD_E_NOMEM;
    APC_LAUNCH(c, K_VEC, 1, 1024, 0, k_field_energy, ptr<double>(c->nodefield), ptr<int4>(c->node_ic), c->n_int,
               c->P.hi[0] - c->P.lo[0], tmp);
    return read_back(c, h_out, tmp, sizeof(double));
}

}  // namespace apc
