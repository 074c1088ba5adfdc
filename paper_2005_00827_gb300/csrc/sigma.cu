// Real-frequency two-loop self-energy and the quasi-particle weight Z.
//
// Sigma(k_j, w) = sum_{p,q} w_p w_q Z_a Z_b Z_c W F / (w + i eta - E)
//   r = k_j + p - q,  E = x_q + x_r - x_p,
//   F = f_p (1-f_q)(1-f_r) + (1-f_p) f_q f_r,
//   W = 2 V(k_j,p,q)^2 - V(k_j,p,q) V(k_j,p,r),
// a, b, c the patches of p, q, r (the two-loop term of Sec. A.2/A.3 with the
// static vertex and Z-weighted lines).  Z_j = (1 - slope)^-1, Eq.
// (definition_Z), with the slope the chord of Re Sigma over xi_j +- 2T
// ("from outside", Sec. 3.1.1).
//
// Wedge grid: sigma_fast_kernel (FP32) and sigma64_kernel evaluate Re Sigma
// exactly at the two chord frequencies; sigma_hist_kernel (FP32) and
// sigma64_kernel<HIST> bin W F by pole energy E with moments 0..4 for the
// frequency grid, which sigma_resum_kernel resums and sigma_spread_kernel copies
// to the images.  Lattice and shell modes: sigma_kernel<R,HIST>.  Each CTA
// stages the points of one patch a of p (k_j + p, cos/sin, Fermi factors) and
// the vertex row V[j][a][:] in shared memory and loops over them with its q.
// In the mixed flow the C4v-irreducible patches 0..N/8 are evaluated (the vertex
// and Z keep the lattice symmetry), of a given vertex the targets that a C4v
// test on the device admits; their sums are copied to the images, which decide the
// pairs on a boundary between patches themselves (sigma_fix_kernel).
#include <algorithm>
#include <cstdlib>

#include "atan_poly.h"
#include "qpfrg_internal.h"

namespace qpfrg {

__device__ __forceinline__ float sexp(float x) { return __expf(x); }
__device__ __forceinline__ double sexp(double x) { return exp(x); }
// typed absolute value: plain sabs() on a float would promote to FP64
__device__ __forceinline__ float sabs(float x) { return fabsf(x); }
__device__ __forceinline__ double sabs(double x) { return fabs(x); }
__device__ __forceinline__ float sdiv(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double sdiv(double a, double b) { return a / b; }
__device__ __forceinline__ float srint(float x) { return rintf(x); }
__device__ __forceinline__ double srint(double x) { return rint(x); }
__device__ __forceinline__ float satan2(float y, float x) { return atan2f(y, x); }
__device__ __forceinline__ double satan2(double y, double x) { return atan2(y, x); }
__device__ __forceinline__ float sfloor(float x) { return floorf(x); }
__device__ __forceinline__ double sfloor(double x) { return floor(x); }

// f(x) and 1 - f(x) without cancellation: with e = exp(-|x|/T) they are
// e/(1+e) and 1/(1+e), one reciprocal.
template <typename R>
__device__ __forceinline__ void sfermi(R x, R invT, R &f, R &fc)
{
    const R e = sexp(-sabs(x) * invT);
    const R hi = sdiv(R(1), R(1) + e), lo = e * hi;
    f = x > R(0) ? lo : hi;
    fc = x > R(0) ? hi : lo;
}

// atan2 in FP32 from the odd polynomial t P(t^2), t = min/max on [0, 1], a
// Remez minimax fit of atan(t) (degree 11; coefficients and the error bound
// kAtanErr = 1.75e-6 rad of the FP32 evaluation generated by atan_fit.py into
// atan_poly.h), then octant reflections.  Caller guarantees (x, y) != (0, 0).
__device__ __forceinline__ float atan2_poly(float y, float x)
{
    const float ax = fabsf(x), ay = fabsf(y);
    const float t = __fdividef(fminf(ax, ay), fmaxf(ax, ay));
    const float s = t * t;
    float p = fmaf(s, kAtanC5, kAtanC4);
    p = fmaf(s, p, kAtanC3);
    p = fmaf(s, p, kAtanC2);
    p = fmaf(s, p, kAtanC1);
    p = fmaf(s, p, kAtanC0);
    float a = t * p;
    if (ay > ax) a = 1.57079633f - a;
    if (x < 0.f) a = 3.14159265f - a;
    return copysignf(a, y);
}

// Round to nearest even without a conversion instruction (|x| < 2^22): the
// float sum with 1.5 * 2^23 keeps rint(x) in its low mantissa bits.
__device__ __forceinline__ float rint_add(float x, int &as_int)
{
    const float s = x + 12582912.f;
    as_int = __float_as_int(s) - 0x4B400000;
    return s - 12582912.f;
}

// FP32 wedge projection with a guard band: the FP32 momentum carries an
// absolute error below 1.4e-6 per component (FP32 rounding of k+p, q, their
// difference and the fold) and atan2_poly below 2.3e-6 rad (kAtanErr, the
// approximate quotient t and the rounding of the octant reflections), so the angle is
// trusted only when it lies more than 8e-6 + 8e-6/|r| rad from a wedge
// boundary and the point is more than 4e-6 from the zone edge.  Returns -1
// near a wedge boundary, -2 near the zone edge or the origin; jc gets the
// nearest-centre estimate.
__device__ __forceinline__ void fold32(float rx, float ry, float &x, float &y)
{
    const float tp = 6.28318531f;
    int ix;
    x = rx - tp * rint_add(rx * 0.159154943f, ix);
    y = ry - tp * rint_add(ry * 0.159154943f, ix);
}

// (x, y) already folded.
__device__ __forceinline__ int project32_guarded(float x, float y, int N, float inv_dth, float dth, int &jc)
{
    const float r2 = x * x + y * y;
    const float u = atan2_poly(y, x) * inv_dth;      // angle in units of the wedge width
    int j;
    const float fj = rint_add(u, j);                 // nearest centre
    jc = j;
    if (fabsf(x) > 3.14159265f - 4e-6f || fabsf(y) > 3.14159265f - 4e-6f || r2 < 1e-8f) return -2;
    const float m = (0.5f - fabsf(u - fj)) * dth;    // distance to the nearest boundary, rad
    if (m < 8e-6f || m * m * r2 < 6.4e-11f) return -1;
    if (j < 0) j += N;
    if (j >= N) j -= N;
    return j;
}

// Error-free transformations on the FP32 pipes (float-float arithmetic).
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// sign of cross(b, x) = b_c x_y - b_s x_x with b and x as float-float pairs;
// accurate to ~1e-14 of |b||x|
__device__ __forceinline__ float cross_ff(float4 b, float xh, float xl, float yh, float yl)
{
    const float p1 = b.x * yh, e1 = fmaf(b.x, yh, -p1);
    const float p2 = b.z * xh, e2 = fmaf(b.z, xh, -p2);
    float s, es;
    two_sum(p1, -p2, s, es);
    const float t = es + e1 - e2 + b.x * yl + b.y * yh - b.z * xl - b.w * xh;
    return s + t;
}

// Wedge of a folded momentum (float-float) from ray tests: the estimated wedge jc
// and its neighbours.  bnd[m] = (cos hi, cos lo, sin hi, sin lo) of the ray
// between wedges m-1 and m, at angle (m - 1/2) 2 pi / N.  margin: |r| times the
// distance to the nearer of the wedge's rays.
__device__ __forceinline__ int rays_ff(float xh, float xl, float yh, float yl, int jc, int N, const float4 *bnd,
                                       float &margin)
{
    int j = jc;
    for (int it = 0; it < 3; ++it) {
        const int jj = j < 0 ? j + N : (j >= N ? j - N : j);
        const int jn = jj + 1 == N ? 0 : jj + 1;
        const float lo = cross_ff(bnd[jj], xh, xl, yh, yl), hi = cross_ff(bnd[jn], xh, xl, yh, yl);
        const bool ccw_lo = lo >= 0.f;   // on or after the lower ray
        const bool cw_hi = hi < 0.f;     // before the upper ray
        margin = fminf(fabsf(lo), fabsf(hi));
        if (ccw_lo && cw_hi) return jj;
        j = ccw_lo ? jj + 1 : jj - 1;
    }
    return j < 0 ? j + N : (j >= N ? j - N : j);
}

// Guarded cases away from the zone edge: r = (k+p) - q in float-float, folded
// (|r| < 3 pi; the fold decision is safe away from the zone edge), then the ray
// tests.
__device__ __forceinline__ int project_ff(float kph, float kpl, float kqh, float kql, float qxh, float qxl,
                                          float qyh, float qyl, int jc, int N, const float4 *bnd, float &margin)
{
    const float C1 = 6.28318548f, C2 = -1.7484555e-7f;   // 2 pi = C1 + C2 (float-float)
    float xh, xl, yh, yl, e;
    two_sum(kph, -qxh, xh, e);
    xl = e + (kpl - qxl);
    two_sum(kqh, -qyh, yh, e);
    yl = e + (kql - qyl);
    const float kx_ = xh > 3.14159265f ? 1.f : (xh < -3.14159265f ? -1.f : 0.f);
    const float ky_ = yh > 3.14159265f ? 1.f : (yh < -3.14159265f ? -1.f : 0.f);
    two_sum(xh, -kx_ * C1, xh, e);
    xl = xl + e - kx_ * C2;
    two_sum(yh, -ky_ * C1, yh, e);
    yl = yl + e - ky_ * C2;
    return rays_ff(xh, xl, yh, yl, jc, N, bnd, margin);
}

// Per target j and loop point, once per self-energy call: k_j + p as FP32
// hi/lo pairs (from the FP64 sum, the same sum as the FP64 path) and in fixed
// point, and, per target, cos/sin of k_j's components.  The pair kernels convert
// nothing in FP64 (a conversion per record and loop point in every CTA took a
// tenth of the chord kernel at 256 points per patch, 40 % at 64).
__global__ void kp_table_kernel(const double *kf, const int *jlist, int nj, const double *kx64, const double *ky64,
                                int M, float4 *kp, int2 *kfx, float4 *kcs)
{
    const long total = (long)nj * M;
    for (long idx = blockIdx.x * (long)blockDim.x + threadIdx.x; idx < total; idx += (long)gridDim.x * blockDim.x) {
        const int ji = (int)(idx / M), p = (int)(idx - (long)ji * M);
        const int j = jlist ? jlist[ji] : ji;
        const double x = kf[2 * j] + kx64[p], y = kf[2 * j + 1] + ky64[p];
        const float xh = (float)x, yh = (float)y;
        const float xl = (float)(x - xh), yl = (float)(y - yh);
        kp[(long)j * M + p] = make_float4(xh, xl, yh, yl);
        if (kfx) kfx[(long)j * M + p] = make_int2(angle_fx((double)xh + (double)xl), angle_fx((double)yh + (double)yl));
        if (p == 0) {
            double sx, cx, sy, cy;
            sincos(kf[2 * j], &sx, &cx);
            sincos(kf[2 * j + 1], &sy, &cy);
            kcs[j] = make_float4((float)cx, (float)sx, (float)cy, (float)sy);
        }
    }
}

template <typename R>
struct SigmaArgs {
    Problem pb;
    FineTable<R> fine;
    const double *kf;    // N x 2
    const double *V;     // N^3 FP64
    const double *Z;     // N
    // interaction flow with the self-energy ODE: Katanin factors per patch
    // (NULL otherwise); the lines then carry the weights of a G, an S and an
    // inner K S line averaged over their assignments (see gflow.cu)
    const double *K;
    double *sig;         // [target]: chord slope of Re Sigma over xi_j +- 2T
    double T;
    int nj;
    const int *jlist;    // targets (may be NULL: j = blockIdx.z)
    const double *kx64, *ky64;  // FP64 fine momenta (guarded FP32 projection)
    const double *xij;          // xi(k_F(j)), FP64
    const float4 *bnd;          // boundary rays of the wedges, float-float (FP32 projection fallback)
    const float4 *kp;           // [patch j][p]: k_j + p as (x hi, x lo, y hi, y lo)
    const float4 *kcs;          // [patch j]: cos, sin of k_j's components
    const float *qxl, *qyl;     // FP32 residuals of the fine momenta
    // scalars of the inner loop in R (a double scalar re-read inside the loop
    // would cost a conversion on the FP64 pipe per use)
    R t_r, tp_r, mu_r, eta_r, invT_r, twoT_r;
    const R *xij_r;             // xi(k_F(j)) in R
    // frequency-grid histogram (sigma_hist_kernel)
    double *hist;        // [j][moment 0..4][bin]
    double e_min, inv_h;
    int nbins;
};

// Shared-memory record of one loop point p of patch a, for target k_j:
// k+p (x, y), cos/sin of its components, line energy x_p, f_p, 1-f_p, w_p.
constexpr int REC = 12;

__device__ __forceinline__ void load_rec(const float *base, int i, float (&r)[REC])
{
    const float4 *p = reinterpret_cast<const float4 *>(base + REC * i);
    const float4 a = p[0], b = p[1], c = p[2];
    r[0] = a.x; r[1] = a.y; r[2] = a.z; r[3] = a.w;
    r[4] = b.x; r[5] = b.y; r[6] = b.z; r[7] = b.w;
    r[8] = c.x; r[9] = c.y; r[10] = c.z; r[11] = c.w;
}

__device__ __forceinline__ void load_rec(const double *base, int i, double (&r)[REC])
{
    const double2 *p = reinterpret_cast<const double2 *>(base + REC * i);
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const double2 v = p[k];
        r[2 * k] = v.x;
        r[2 * k + 1] = v.y;
    }
    r[10] = r[11] = 0.0;
}

template <typename R, bool HIST>
__global__ void __launch_bounds__(256) sigma_kernel(SigmaArgs<R> A)
{
    const int N = A.pb.N, P = A.pb.P, M = A.pb.M;
    const int a = blockIdx.y;
    const int jidx = blockIdx.z;
    const int j = A.jlist ? A.jlist[jidx] : jidx;
    const int tid = threadIdx.x;
    const bool qp = A.pb.propagator == QPFRG_PROP_QP;
    // wedge and shell modes: the FP32 path decides the wedge by guarded ray
    // tests (and the shell by the FP32 line energy, guarded)
    const bool angular = A.pb.mode == QPFRG_GRID_WEDGE || A.pb.mode == QPFRG_GRID_SHELL;
    const int ns = A.pb.n_shell, Na = N / ns;
    const R invT = A.invT_r, eta = A.eta_r;
    const R t = A.t_r, tp = A.tp_r, mu = A.mu_r;
    constexpr bool f32 = sizeof(R) == 4;

    extern __shared__ __align__(16) unsigned char smem_raw[];
    R *s_rec = reinterpret_cast<R *>(smem_raw);          // P x REC
    R *s_VZ = s_rec + (size_t)REC * P;                   // N x {V[j][a][c], Z_c}
    float4 *s_bnd = reinterpret_cast<float4 *>(s_VZ + 2 * N + (2 * N * sizeof(R)) % 16 / sizeof(R));
    R *s_K = reinterpret_cast<R *>(s_bnd + N);           // N Katanin factors (interaction-flow lines)

    const double kx = A.kf[2 * j], ky = A.kf[2 * j + 1];
    for (int i = tid; i < N; i += blockDim.x) {
        s_VZ[2 * i] = (R)A.V[((long)j * N + a) * N + i];
        s_VZ[2 * i + 1] = A.Z ? (R)A.Z[i] : R(1);
        if (f32 && angular) s_bnd[i] = A.bnd[i];
        if (A.K) s_K[i] = (R)A.K[i];
    }
    __shared__ R s_k[4];
    if (tid == 0) {
        if (f32) {
            const float4 k4 = A.kcs[j];
            s_k[0] = (R)k4.x; s_k[1] = (R)k4.y; s_k[2] = (R)k4.z; s_k[3] = (R)k4.w;
        } else {
            double sx, cx, sy, cy;
            sincos(kx, &sx, &cx);
            sincos(ky, &sy, &cy);
            s_k[0] = (R)cx; s_k[1] = (R)sx; s_k[2] = (R)cy; s_k[3] = (R)sy;
        }
    }
    __syncthreads();
    const R Za = s_VZ[2 * a + 1];
    const R ckx = s_k[0], skx = s_k[1], cky = s_k[2], sky = s_k[3];
    // records in angular-minor order: storage index s * n_theta + t for the
    // point (t, s), so consecutive records are angular neighbours
    const int nt = A.pb.n_theta, nr = A.pb.n_r;
    for (int i = tid; i < P; i += blockDim.x) {
        const int p = a * P + (i % nt) * nr + i / nt;
        R *rec = s_rec + (size_t)REC * i;
        if (f32) {
            // k_j + p as FP32 hi/lo pairs from the per-call table
            const float4 k4 = A.kp[(long)j * M + p];
            rec[0] = (R)k4.x;
            rec[10] = (R)k4.y;
            rec[1] = (R)k4.z;
            rec[11] = (R)k4.w;
        } else {
            rec[0] = (R)(kx + A.kx64[p]);
            rec[1] = (R)(ky + A.ky64[p]);
            rec[10] = rec[11] = R(0);
        }
        const R cpx = A.fine.cx[p], spx = A.fine.sx[p], cpy = A.fine.cy[p], spy = A.fine.sy[p];
        rec[2] = ckx * cpx - skx * spx;
        rec[3] = skx * cpx + ckx * spx;
        rec[4] = cky * cpy - sky * spy;
        rec[5] = sky * cpy + cky * spy;
        const R xp = qp ? Za * A.fine.xi[p] : A.fine.xi[p];
        rec[6] = xp;
        R f, fc;
        sfermi(xp, invT, f, fc);
        rec[7] = f;
        rec[8] = fc;
        rec[9] = A.fine.w[p];
    }
    __syncthreads();

    const int q = blockIdx.x * blockDim.x + tid;
    R acc = R(0);
    if (q < M) {
        const int b = q / P;
        const R qx = A.fine.kx[q], qy = A.fine.ky[q];
        const double qxd = A.kx64[q], qyd = A.ky64[q];
        const float qxl = f32 ? A.qxl[q] : 0.f, qyl = f32 ? A.qyl[q] : 0.f;
        const R cqx = A.fine.cx[q], sqx = A.fine.sx[q], cqy = A.fine.cy[q], sqy = A.fine.sy[q];
        const R Zb = s_VZ[2 * b + 1];
        const R xq = qp ? Zb * A.fine.xi[q] : A.fine.xi[q];
        R fq, fcq;
        sfermi(xq, invT, fq, fcq);
        const R vab = s_VZ[2 * b];
        const R pref = Za * Zb * A.fine.w[q];
        const bool glines = A.K != nullptr;
        const R uab = glines ? s_K[a] * Za * Zb + s_K[b] * Zb * Za : R(0);   // K_a Z_a Z_b + K_b Z_b Z_a
        const R kza = glines ? s_K[a] * Za : R(0), kzb = glines ? s_K[b] * Zb : R(0);
        const R d0shift = A.xij_r[j], twoT = A.twoT_r;
        const R eta2 = eta * eta;
        const float inv_dth = (float)(Na / kTwoPi), dth = (float)(kTwoPi / Na);
        const float invD = ns > 1 ? (float)(1.0 / A.pb.shell_D) : 0.f, half_ns = 0.5f * ns;
        // guard band of the shell decision in units of the shell width: ten
        // times the error bound of the FP32 line energy (products of FP32-rounded
        // cosines: 1.2e-6 per unit of 2|t| + 4|t'|, 1.2e-7 |mu|) plus the
        // rounding of u itself
        const float gu = 10.f * (1.2e-6f * (2.f * fabsf((float)A.pb.t) + 4.f * fabsf((float)A.pb.tp)) +
                                 1.2e-7f * fabsf((float)A.pb.mu)) * invD + 1e-6f;
        // wedge of the previous pair and its two boundary rays (FP32)
        int cprev = -1;
        float blx = 0.f, bly = 0.f, bhx = 0.f, bhy = 0.f;
        for (int i = 0; i < P; ++i) {
            R r[REC];
            load_rec(s_rec, i, r);
            // cos(k+p-q) by angle addition, and the bare line energy of r
            const R crx = r[2] * cqx + r[3] * sqx;
            const R cry = r[4] * cqy + r[5] * sqy;
            R xr = R(-2) * t * (crx + cry) - R(4) * tp * crx * cry - mu;
            int c = -1;
            if (f32 && angular) {
                float x, y;
                fold32((float)(r[0] - qx), (float)(r[1] - qy), x, y);
                // inside the previous pair's wedge by more than the FP32 error
                // of (x, y) (2.1e-6) plus that of the rays: same wedge
                const bool edge = fabsf(x) > 3.14159265f - 4e-6f || fabsf(y) > 3.14159265f - 4e-6f;
                int cw;
                if (!edge && cprev >= 0 && blx * y - bly * x >= 4e-6f && bhx * y - bhy * x <= -4e-6f) {
                    cw = cprev;
                } else {
                    int jc;
                    cw = project32_guarded(x, y, Na, inv_dth, dth, jc);
                    if (cw == -1) {
                        // near a wedge boundary: float-float decision on the FP32 pipes
                        float margin;
                        cw = project_ff((float)r[0], (float)r[10], (float)r[1], (float)r[11], (float)qx, qxl,
                                        (float)qy, qyl, jc, Na, s_bnd, margin);
                    } else if (cw == -2) {
                        // zone edge or origin: the exact FP64 projection
                        const int p = a * P + (i % nt) * nr + i / nt;
                        c = project_fp64((kx + A.kx64[p]) - qxd, (ky + A.ky64[p]) - qyd, A.pb);
                        cw = c / ns;
                    }
                    cprev = cw;
                    const float4 lo = s_bnd[cw], hi = s_bnd[cw + 1 == Na ? 0 : cw + 1];
                    blx = lo.x; bly = lo.z; bhx = hi.x; bhy = hi.z;
                }
                if (c < 0) {
                    if (ns == 1) {
                        c = cw;
                    } else {
                        // shell of the FP32 line energy; within the guard band of
                        // a shell edge the exact FP64 projection decides
                        const float u = (float)xr * invD + half_ns;
                        const float ur = rintf(u);
                        if (fabsf(u - ur) < gu && ur >= 1.f && ur <= (float)(ns - 1)) {
                            const int p = a * P + (i % nt) * nr + i / nt;
                            c = project_fp64((kx + A.kx64[p]) - qxd, (ky + A.ky64[p]) - qyd, A.pb);
                        } else {
                            int sh = (int)floorf(u);
                            sh = sh < 0 ? 0 : (sh > ns - 1 ? ns - 1 : sh);
                            c = cw * ns + sh;
                        }
                    }
                }
            } else {
                const int p = a * P + (i % nt) * nr + i / nt;
                c = project_fp64((kx + A.kx64[p]) - qxd, (ky + A.ky64[p]) - qyd, A.pb);
            }
            const R vac = s_VZ[2 * c], Zc = s_VZ[2 * c + 1];
            if (qp) xr *= Zc;
            R fr, fcr;
            sfermi(xr, invT, fr, fcr);
            const R F = r[7] * fcq * fcr + r[8] * fq * fr;
            R amp = r[9] * pref * Zc * (R(2) * vab * vab - vab * vac) * F;
            if (glines)   // (1/6)[K_a Z_a (Z_b + Z_c) + K_b Z_b (Z_a + Z_c) + K_c Z_c (Z_a + Z_b)]
                amp *= (uab + Zc * (kza + kzb) + s_K[c] * Zc * (Za + Zb)) * R(1.0 / 6.0);
            const R E = xq + xr - r[6];
            if (HIST) {
                const double eb = ((double)E - A.e_min) * A.inv_h;
                int bin = (int)floor(eb);
                bin = bin < 0 ? 0 : (bin >= A.nbins ? A.nbins - 1 : bin);
                const double d = (double)E - (A.e_min + (bin + 0.5) / A.inv_h);
                double *h = A.hist + ((long)jidx * 5) * A.nbins + bin;
                double m = (double)amp;
#pragma unroll
                for (int mo = 0; mo < 5; ++mo) {
                    atomicAdd(h + (long)mo * A.nbins, m);
                    m *= d;
                }
            } else {
                // chord slope of Re 1/(w - E + i eta) over w = xi_j +- 2T:
                // [d+/(d+^2+eta^2) - d-/(d-^2+eta^2)] / 4T
                //   = (eta^2 - d+ d-) / ((d+^2 + eta^2)(d-^2 + eta^2))
                const R d0 = d0shift - E;
                const R dp = d0 + twoT, dm = d0 - twoT;
                acc += amp * sdiv(eta2 - dp * dm, (dp * dp + eta2) * (dm * dm + eta2));
            }
        }
    }
    if (HIST) return;
    // block reduction of the partial slopes
    __shared__ double red[32];
    double v = (double)acc;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    const int lane = tid & 31, warp = tid >> 5;
    if (lane == 0) red[warp] = v;
    __syncthreads();
    if (warp == 0) {
        const int nw = blockDim.x >> 5;
        v = lane < nw ? red[lane] : 0.0;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
        if (lane == 0) atomicAdd(&A.sig[jidx], v);
    }
}

// ---------------------------------------------------------------------------
// FP32 chord-slope kernel of the wedge grid (the flow's self-energy).
//
// Same sum as sigma_kernel<float,false>, arranged for instruction count:
// * momenta are fixed-point turns (angle_fx), so r = k_j + p - q folds by
//   integer wrap-around; the patch c of r comes from a shared-memory cell
//   table over the folded zone indexed by the top bytes (one byte per cell:
//   the lower of the at most two wedges the cell touches) and one FP32 test
//   against the ray between them; cells near the origin, points within 4e-6
//   of a ray and points within 4e-6 of the zone edge take the guarded paths
//   of sigma_kernel (float-float rays, exact FP64 projection), so every patch
//   decision equals the FP64 one;
// * f_r enters only through F = A + f_r (B - A) with A = w_p f_p (1 - f_q),
//   B = w_p (1 - f_p) f_q (times Z_a Z_b w_q), so one exp2 and one
//   reciprocal give it;
// * per patch c the table cz holds (Z_c, Z_c V[j][a][c], -2t l_c, -mu l_c)
//   times (1, 1, log2(e)/T, log2(e)/T), l_c = Z_c for quasi-particle lines
//   (else 1), so the line energy of r (Z-scaled, in units of T/log2(e)) is one
//   FMA from cos(r_x) + cos(r_y) and feeds exp2 directly;
// * with d0 = xi_j - E the chord term is -u / (u^2 + 4 eta^2 d0^2),
//   u = d0^2 - 4T^2 - eta^2 (the product of the two Lorentzian denominators
//   written out);
// * each thread owns SF_QPT = 2 loop points q, so a record of p read from
//   shared memory serves two pairs, whose arithmetic runs as the two lanes of
//   packed FP32x2 instructions (Fermi factor, weight, chord term, sum), and
//   cos r_x, cos r_y of one pair form one packed FMA pair; the lanes of a warp own angular neighbours at
//   one radius (angular-minor order), so their r lie on a short arc and their
//   table cells, rays and patch slots mostly coincide (few bank conflicts,
//   rare divergence into the guarded paths).
// Launch: grid (ceil(M / (256 SF_QPT qb)), N patches a, targets), 256 threads,
// two CTAs per SM.
constexpr int SF_QPT = 2;
constexpr int SF_QB = 4;        // default blocks of 256 SF_QPT loop points q per CTA
constexpr int SF_PCH = 1024;    // loop points p staged per pass
constexpr int SF_QCAP = 896;    // guarded pairs queued per pass (two CTAs per SM, see sf_smem_layout)
constexpr int SF_SLOTS = 257;   // per-patch slots: c in 0..N (c = N is patch 0 again), padded to 257

struct SigmaFastArgs {
    Problem pb;
    FineTable<float> fine;
    const double *V, *Z, *kx64, *ky64, *kf;
    const float *xij_f, *qxl, *qyl;
    const double *xi64, *w64, *xij64;   // dispersion and weight of the fine points, xi(k_F(j))
    double T64;
    double fold0, fold1;    // last doubles k with rint(k / 2 pi) = 0 and < 2
    double dth64;           // 2 pi / N
    int sub0;               // records of a pass's first chunk (queue of guarded pairs)
    int qcap;               // guarded pairs that the queue holds
    const float4 *kp, *kcs, *bnd;
    const int2 *kfx, *pfx;  // k_j + p and the fine points in fixed point
    const uint8_t *ptab;
    const uint8_t *rtab;    // patch of r per (target, p, q) (RT launches; rtab_build_kernel)
    const int *jlist;
    // sym.mode == 2: jlist holds every patch, its first n_list the targets that a
    // C4v-symmetric (V, Z) needs (the other slots then return); own[j]: slot of j
    SymMode sym;
    int n_list;
    const int *own;
    const double *K;        // Katanin factors (interaction-flow lines; the GL kernels)
    double *sig;
    // pairs on a boundary between patches met by a reduced launch, and per patch
    // its own slope less its representative's (sigma_fix_kernel; the frequency grid:
    // its own histogram less its representative's, in its slot); nevents[0] their
    // number, nevents[1] the corrections made; only_full: run only when there were
    // more pairs than the record holds
    int4 *events;
    unsigned *nevents, max_events;
    bool only_full;
    double *corr;
    float t, tp, mu, invT, cT;                      // cT = log2(e) / T
    float tln2, kchord, eta2x4;                     // T ln 2, 4 T^2 + eta^2, 4 eta^2
    float inv_dth, dth;                             // N / 2 pi, 2 pi / N
    int mirror;     // n_theta even and symmetric targets: halve the mirror-line targets
    int qb;         // blocks of 256 SF_QPT loop points q per CTA
    // grid mode: pole energies E binned from e_min in bins of h, moments 0..4
    // of the offset from the bin centre, hist[target][moment][bin] (FP64)
    double *hist;
    float h;
    // bin of E: c_int + rint(x), x = E / h + c_frac (1 / h = inv_h + inv_h_lo, so
    // that the offset x - rint(x) keeps FP32 accuracy at every bin)
    float inv_h, inv_h_lo, c_frac;
    int nbins, c_int;
    double e_min, h64;
    float w_max;            // largest quadrature weight
};

// Target of slot z; false where the slot has none.
__device__ __forceinline__ bool sigma_target(const SigmaFastArgs &A, int z, int &j, bool &sym)
{
    sym = A.sym.mode == 2 ? sym_compact(A.sym) : A.jlist != nullptr;
    if (sym && A.sym.mode == 2 && z >= A.n_list) return false;
    j = A.jlist ? A.jlist[z] : z;
    return true;
}

// A target on a mirror line of the zone (the line through k_j, j a multiple of
// N/8, which reflects patch a to 2j - a) has a sum symmetric under that mirror:
// keep the patches a on one side of it with weight fac = 2 and half of each patch
// the mirror maps onto itself (P loop points: angular index t < n_theta / 2).
// fac = 0: the mirror patch carries this one.
__device__ __forceinline__ void mirror_part(int mirror, int N, int j, int a, int &fac, int &P)
{
    fac = 1;
    if (!mirror || (8 * j) % N != 0) return;
    const int ma = ((2 * j - a) % N + N) % N;
    if (ma == a) {
        fac = 2;
        P /= 2;
    } else {
        const int rel = ((a - j) % N + N) % N;
        fac = (rel > 0 && 2 * rel < N) ? 2 : 0;
    }
}

__device__ __forceinline__ float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float rcp_approx(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Table patch of r = (k+p) - q from fixed-point components: the lower wedge e
// of the cell and the side of the ray between e and e + 1 (c = e or e + 1).
// slow: within the guard band of that ray, of the zone edge, or in a cell of
// three or more wedges (e = 255 reads the zero ray 256, cr = 0).  tabc points
// at the cell of the origin; x, y come back in fixed-point units.
__device__ __forceinline__ int fx_patch(int kpx, int kpy, int qx, int qy, const unsigned char *tabc,
                                        const float2 *ray, float &x, float &y, bool &slow)
{
    const int X = (int)((unsigned)kpx - (unsigned)qx);
    const int Y = (int)((unsigned)kpy - (unsigned)qy);
    x = __int2float_rn(X);
    y = __int2float_rn(Y);
    const int e = tabc[(Y >> 24) * kProjStride + (X >> 24)];
    const float2 rr = ray[e + 1];
    const float cr = rr.x * y - rr.y * x;
    slow = fmaxf(fabsf(x), fabsf(y)) > kFxEdge || fabsf(cr) < kFxGuard;
    return e + (cr >= 0.f ? 1 : 0);
}

// The same for a pair that fx_patch left undecided, where r lies near the origin
// (cells of three or more wedges, 1 % of all pairs at 48 patches and 4 % at 96):
// the wedges are cones, so the table's cell of 2^s r decides as well, s <= 6
// keeping the scaled position error below the cells' margin.
__device__ __forceinline__ int fx_zoom(int kpx, int kpy, int qx, int qy, const unsigned char *tabc, const float2 *ray,
                                       bool &slow)
{
    const int X = (int)((unsigned)kpx - (unsigned)qx);
    const int Y = (int)((unsigned)kpy - (unsigned)qy);
    const int s = min(max(__clz(max(abs(X), abs(Y))) - 1, 0), 6);
    const float x = __int2float_rn(X), y = __int2float_rn(Y);
    const int e = tabc[((Y << s) >> 24) * kProjStride + ((X << s) >> 24)];
    const float2 rr = ray[e + 1];
    const float cr = rr.x * y - rr.y * x;
    slow = fmaxf(fabsf(x), fabsf(y)) > kFxEdge || fabsf(cr) < kFxGuard;
    return e + (cr >= 0.f ? 1 : 0);
}

struct SfSmem {
    size_t rA, rB, cz, ray, cd, ck, rC, tab, queue, total;
};

// (a launch that reads the patch table has no use for the queue)
__host__ __device__ constexpr SfSmem sf_smem_layout(int pch, bool rt)
{
    SfSmem L{};
    L.rA = 0;                                  // pch + 1 records: room for a pad record
    L.rB = L.rA + (size_t)16 * (pch + 1);
    L.cz = L.rB + (size_t)16 * (pch + 1);
    L.ray = L.cz + (size_t)16 * SF_SLOTS;
    L.cd = L.ray + (size_t)8 * SF_SLOTS;
    L.rC = (L.cd + (size_t)4 * SF_SLOTS + 15) / 16 * 16;
    L.tab = (L.rC + (size_t)4 * (pch + 1) + 15) / 16 * 16;
    L.queue = L.tab + ((size_t)kProjW * kProjStride + 15) / 16 * 16;
    L.ck = L.queue + (size_t)4 * (1 + SF_QCAP);
    L.total = rt ? L.queue : L.ck + (size_t)4 * SF_SLOTS;
    return L;
}
// Two CTAs per SM at the longest pass (32 x 32 points): each takes its layout, 256
// bytes of static shared memory and the 1 KB that the SM reserves.  A queue of 1024
// pairs left one CTA: Z of an unsymmetric vertex, np48, 32 x 32, 149 -> 197 ms.
static_assert(2 * (sf_smem_layout(SF_PCH, false).total + 256 + 1024) <= 228 * 1024, "two CTAs per SM");

// Patch of r for a lane that left the table path: near a ray or the origin
// (float-float ray tests) or near the zone edge.  There the FP64 fold decides: its
// count rint(k / 2 pi) changes where k passes fold0 (pi) and fold1 (3 pi), the
// last doubles of the lower count, so two FP64 additions and comparisons per
// component give the folded momentum of project_fp64, and the wedge follows from
// FP32 and float-float ray tests; only within 1e-11 of a ray (where the FP64
// rounding decides), or of the origin, does the FP64 projection run (its atan2 and divisions, 170 instructions at 64
// clocks each per warp, made the CTAs of coinciding p and q the tail of the launch:
// np48, Z of a symmetric vertex 4.5 -> 3.9 ms).  flags: 1 near the zone edge, 2
// record a pair within 1e-9 of a ray or of the zone edge in A.events (correcting
// its image targets on the spot cost the pair loop 600 bytes of spills).
__device__ __noinline__ int sf_slow_patch(const SigmaFastArgs &A, int j, int p, int q, float x, float y, int flags,
                                          const float4 *bnd)
{
    const int N = A.pb.N;
    float margin = 0.f;
    auto record = [&](int c) {
        if (!(flags & 2)) return;
        const unsigned n = atomicAdd(A.nevents, 1u);
        if (n < A.max_events) A.events[n] = make_int4(j, p, q, c);
    };
    if (!(flags & 1)) {
        int jc;
        const int c = project32_guarded(x, y, N, A.inv_dth, A.dth, jc);
        if (c >= 0) return c;
        if (c == -1) {
            const float4 k4 = A.kp[(long)j * A.pb.M + p];
            const int r = project_ff(k4.x, k4.y, k4.z, k4.w, A.fine.kx[q], A.qxl[q], A.fine.ky[q], A.qyl[q], jc, N, bnd,
                                     margin);
            if (margin >= 1e-11f) {
                if (margin < 1e-9f) record(r);
                return r;
            }
        }
    }
    const double kx = (A.kf[2 * j] + A.kx64[p]) - A.kx64[q], ky = (A.kf[2 * j + 1] + A.ky64[p]) - A.ky64[q];
    const double nx = kx > A.fold0 ? -kTwoPi : (kx < -A.fold0 ? kTwoPi : 0.0);
    const double ny = ky > A.fold0 ? -kTwoPi : (ky < -A.fold0 ? kTwoPi : 0.0);
    const double fx = kx + nx, fy = ky + ny;
    const float xh = (float)fx, yh = (float)fy, xl = (float)(fx - (double)xh), yl = (float)(fy - (double)yh);
    const float r2 = xh * xh + yh * yh;
    if (kx > A.fold1 || kx < -A.fold1 || ky > A.fold1 || ky < -A.fold1 || r2 < 1e-8f) {
        const int c = project_fp64(kx, ky, A.pb);
        record(c);
        return c;
    }
    // distance to the zone edge: pi = 3.14159274f - 8.7422777e-8f
    const float ex = (3.14159274f - fabsf(xh)) - (copysignf(xl, xh * xl) + 8.7422777e-8f);
    const float ey = (3.14159274f - fabsf(yh)) - (copysignf(yl, yh * yl) + 8.7422777e-8f);
    int jc;
    rint_add(atan2_poly(yh, xh) * A.inv_dth, jc);
    int c = rays_ff(xh, xl, yh, yl, jc, N, bnd, margin);
    if (margin < 1e-11f) {       // project_fp64 of the folded momentum
        c = (int)floor(atan2(fy, fx) / A.dth64 + 0.5);
        c = c < 0 ? c + N : (c >= N ? c - N : c);
    }
    if (fminf(fminf(fabsf(ex), fabsf(ey)), margin) < 1e-9f) record(c);
    return c;
}

// Weight W F and pole energy E of one pair with r in patch c, in FP64 from the
// tables (rare).
__device__ __noinline__ double sf_pair_weight(const SigmaFastArgs &A, int j, int p, int q, int c, double &E)
{
    const int N = A.pb.N, PP = A.pb.P, a = p / PP, b = q / PP;
    auto z = [&](int k) { return A.Z ? A.Z[k] : 1.0; };
    const bool qp = A.pb.propagator == QPFRG_PROP_QP;
    const double Za = z(a), Zb = z(b), Zc = z(c), invT = 1.0 / A.T64;
    const double cx = cos(A.kf[2 * j] + A.kx64[p] - A.kx64[q]), cy = cos(A.kf[2 * j + 1] + A.ky64[p] - A.ky64[q]);
    const double xp = (qp ? Za : 1.0) * A.xi64[p], xq = (qp ? Zb : 1.0) * A.xi64[q];
    const double xr = (qp ? Zc : 1.0) * (-2.0 * A.pb.t * (cx + cy) - 4.0 * A.pb.tp * cx * cy - A.pb.mu);
    auto f = [&](double x) { return 1.0 / (1.0 + exp(x * invT)); };
    const double F = f(xp) * f(-xq) * f(-xr) + f(-xp) * f(xq) * f(xr);
    const double *V = A.V + ((long)j * N + a) * N;
    double amp = A.w64[p] * A.w64[q] * Za * Zb * Zc * (2.0 * V[b] * V[b] - V[b] * V[c]) * F;
    if (A.K)
        amp *= (A.K[a] * Za * (Zb + Zc) + A.K[b] * Zb * (Za + Zc) + A.K[c] * Zc * (Za + Zb)) * (1.0 / 6.0);
    E = xq + xr - xp;
    return amp;
}

// A recorded pair (p, q) of target j, patch c, lies on a boundary: every image
// target that copies j's sum is corrected where its own pair is decided
// otherwise, so that each patch keeps its own sum.  hist: the difference goes into
// the image's own slot of the frequency grid's histogram, else into its slope.
__global__ void __launch_bounds__(128) sigma_fix_kernel(SigmaFastArgs A, double *hist)
{
    if (*A.nevents > A.max_events) return;      // every patch is summed
    const int N = A.pb.N, PP = A.pb.P, nt = A.pb.n_theta, nr = A.pb.n_r;
    const unsigned n = *A.nevents;
    auto image = [&](int g, int k) {
        const int a = k / PP, l = k - a * PP, t = l / nr, s = l - t * nr;
        return c4v_apply(g, a, N, 1) * PP + ((g & 4) ? nt - 1 - t : t) * nr + s;
    };
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < 7u * n; i += gridDim.x * blockDim.x) {
        const int4 e = A.events[i / 7u];
        const int g = 1 + (int)(i % 7u), j = e.x, jg = c4v_apply(g, j, N, 1);
        bool seen = jg == j;       // one element per image target
        for (int k = 1; k < g; ++k) seen |= c4v_apply(k, j, N, 1) == jg;
        if (seen) continue;
        const int pg = image(g, e.y), qg = image(g, e.z);
        const int own = sf_slow_patch(A, jg, pg, qg, 0.f, 0.f, 1, A.bnd), copied = c4v_apply(g, e.w, N, 1);
        if (own == copied) continue;
        atomicAdd(A.nevents + 1, 1u);
        for (int u = 0; u < 2; ++u) {
            double E, amp = sf_pair_weight(A, jg, pg, qg, u ? copied : own, E);
            if (u) amp = -amp;
            if (hist) {
                const int bin = (int)fmin(fmax(floor((E - A.e_min) / A.h64), 0.0), A.nbins - 1.0);
                const double d = E - (A.e_min + (bin + 0.5) * A.h64);
                double *H = hist + (long)A.own[jg] * 5 * A.nbins + bin;
                for (int mo = 0; mo < 5; ++mo, amp *= d) atomicAdd(H + (long)mo * A.nbins, amp);
            } else {
                const double eta2 = A.pb.eta * A.pb.eta;
                const double d0 = A.xij64[jg] - E, dp = d0 + 2.0 * A.T64, dm = d0 - 2.0 * A.T64;
                atomicAdd(&A.corr[jg], amp * (eta2 - dp * dm) / ((dp * dp + eta2) * (dm * dm + eta2)));
            }
        }
    }
}

// Number of boundary pairs among n pairs of the list's targets, every pair
// (stride 1) or a sample: *A.nevents (sigma_plan).
__global__ void boundary_count_kernel(const SigmaFastArgs A, unsigned n, unsigned long long stride)
{
    const unsigned long long M = A.pb.M, all = M * M * A.n_list;
    const unsigned char *tabc = A.ptab + (kProjW / 2) * (kProjStride + 1);   // the cell of the origin
    __shared__ float2 ray[SF_SLOTS];
    for (int i = threadIdx.x; i < SF_SLOTS; i += blockDim.x) {
        const float4 bd = A.bnd[i < A.pb.N ? i : 0];
        ray[i] = i <= A.pb.N ? make_float2(bd.x, bd.z) : make_float2(0.f, 0.f);
    }
    __syncthreads();
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const unsigned long long k = i * stride % all;
        const int q = (int)(k % M), p = (int)(k / M % M), j = A.jlist[k / M / M];
        if ((4 * j) % A.pb.N == 0) continue;
        const int2 kp = A.kfx[(long)j * A.pb.M + p], kq = A.pfx[q];
        float x, y;
        bool slow;
        fx_patch(kp.x, kp.y, kq.x, kq.y, tabc, ray, x, y, slow);
        if (slow) fx_zoom(kp.x, kp.y, kq.x, kq.y, tabc, ray, slow);
        const bool edge = fmaxf(fabsf(x), fabsf(y)) > kFxEdge;
        if (slow) sf_slow_patch(A, j, p, q, x * kRadPerFx, y * kRadPerFx, edge ? 3 : 2, A.bnd);
    }
}

// The patch of r = k_j + p - q for every target of the list (position jidx),
// every loop point p = a P + i and every loop point q (angular-minor index iq,
// the order in which sigma_fast_kernel walks them), one byte each at
// rtab[(((jidx N + a) P/8 + i/8) M + iq) 8 + i % 8]: a thread reads the bytes
// of eight records as one 8-byte word, and the words of a warp's 32 loop
// points q are contiguous (256 B): the same decisions as the kernel's table
// path and its guarded slow path, so a launch that reads them gives the same
// sums.  They depend on the geometry only (targets, fine grid), so one build
// serves every later call.  Grid (ceil(M / 256), N, targets), 256 threads.
constexpr size_t kRtabTabBytes = ((size_t)kProjW * kProjStride + 15) / 16 * 16;
constexpr size_t kRtabSmem = kRtabTabBytes + (size_t)SF_SLOTS * sizeof(float2);   // + P int2 records

__global__ void __launch_bounds__(256) rtab_build_kernel(SigmaFastArgs A, uint8_t *__restrict__ rtab)
{
    const int N = A.pb.N, M = A.pb.M, PP = A.pb.P;
    const int a = blockIdx.y, jidx = blockIdx.z;
    const int j = A.jlist ? A.jlist[jidx] : jidx;
    const int tid = threadIdx.x;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char *tab = smem_raw;                                      // the cell table
    float2 *ray = reinterpret_cast<float2 *>(smem_raw + kRtabTabBytes); // rays between wedges
    int2 *rec = reinterpret_cast<int2 *>(ray + SF_SLOTS);               // k_j + p of the patch (fixed point)
    {
        const uint4 *src = reinterpret_cast<const uint4 *>(A.ptab);
        uint4 *dst = reinterpret_cast<uint4 *>(tab);
        const int n16 = (kProjW * kProjStride + 15) / 16;
        for (int i = tid; i < n16; i += blockDim.x) dst[i] = src[i];
        for (int i = tid; i < SF_SLOTS; i += blockDim.x) {
            const float4 bd = A.bnd[i == N ? 0 : (i < N ? i : 0)];
            ray[i] = i <= N ? make_float2(bd.x, bd.z) : make_float2(0.f, 0.f);
        }
        for (int i = tid; i < PP; i += blockDim.x) {
            rec[i] = A.kfx[(long)j * M + a * PP + i];
        }
    }
    __syncthreads();
    const unsigned char *tabc = tab + (kProjW / 2) * (kProjStride + 1);   // the cell of the origin
    const int iq = blockIdx.x * 256 + tid;
    if (iq >= M) return;
    const int b = iq / PP, rem = iq - b * PP;
    const int qq = b * PP + (rem % A.pb.n_theta) * A.pb.n_r + rem / A.pb.n_theta;
    const int qx = A.pfx[qq].x, qy = A.pfx[qq].y;
    // the thread's P bytes, as P/8 words of eight records (P a multiple of 16)
    uint2 *out = reinterpret_cast<uint2 *>(rtab) + ((long)jidx * N + a) * (long)(PP / 8) * M + iq;
    for (int i0 = 0; i0 < PP; i0 += 8) {
        unsigned w[2] = {0u, 0u};
        for (int i = i0; i < i0 + 8; ++i) {
            const int p = a * PP + i;
            const int2 kr = rec[i];
            float x, y;
            bool slow;
            int c = fx_patch(kr.x, kr.y, qx, qy, tabc, ray, x, y, slow);
            if (slow) c = fx_zoom(kr.x, kr.y, qx, qy, tabc, ray, slow);
            if (slow) {
                const bool edge = fmaxf(fabsf(x), fabsf(y)) > kFxEdge;
                c = sf_slow_patch(A, j, p, qq, x * kRadPerFx, y * kRadPerFx, edge ? 1 : 0, A.bnd);
            }
            w[(i - i0) >> 2] |= (unsigned)c << (8 * ((i - i0) & 3));
        }
        out[(long)(i0 >> 3) * M] = make_uint2(w[0], w[1]);
    }
}

// UNIB: every block of 256 SF_QPT loop points q lies in one patch b (P a
// multiple of 256 SF_QPT), so the vertex weight is a per-patch table:
// cz[c] = (Z_c (2 V_jab^2 - V_jab V_jac), -, -2t l_c, -mu l_c); otherwise
// cz[c] = (Z_c, Z_c V_jac, -2t l_c, -mu l_c) and the weight is formed per pair.
// GL: the interaction flow's line weights, (1/6)[K_a Z_a (Z_b + Z_c) + K_b Z_b
// (Z_a + Z_c) + K_c Z_c (Z_a + Z_b)] times Z_a Z_b Z_c.
template <bool TP0, bool UNIB, bool RT, bool GL>
__global__ void __launch_bounds__(256, 2) sigma_fast_kernel(SigmaFastArgs A)
{
    const int N = A.pb.N, M = A.pb.M;
    const int a = blockIdx.y, jidx = blockIdx.z;
    int j;
    bool sym = true;
    if (RT) {                   // the table's targets
        j = A.jlist[jidx];
    } else {
        if (A.only_full && *A.nevents <= A.max_events) return;
        if (!sigma_target(A, jidx, j, sym)) return;      // uniform over the CTA
    }
    const int tid = threadIdx.x;
    const bool qp = A.pb.propagator == QPFRG_PROP_QP;
    int fac, P = A.pb.P;
    mirror_part(sym ? A.mirror : 0, N, j, a, fac, P);
    if (fac == 0) return;       // the mirror patch carries this one (uniform over the CTA)
    const int PP = A.pb.P;      // points per patch (record and loop-point indexing)
    const int pch = P < SF_PCH ? P : SF_PCH;
    const SfSmem L = sf_smem_layout(pch, RT);

    extern __shared__ __align__(16) unsigned char smem_raw[];
    float4 *rA = reinterpret_cast<float4 *>(smem_raw + L.rA);   // (k+p)_x, (k+p)_y (fixed point), cos of both
    float4 *rB = reinterpret_cast<float4 *>(smem_raw + L.rB);   // sin of both, w_p f_p, w_p (1 - f_p)
    float4 *cz = reinterpret_cast<float4 *>(smem_raw + L.cz);
    float2 *ray = reinterpret_cast<float2 *>(smem_raw + L.ray);
    float *cd = reinterpret_cast<float *>(smem_raw + L.cd);     // -4 t' l_c
    float *rC = reinterpret_cast<float *>(smem_raw + L.rC);     // x_j + x_p + 2T
    float *ck = reinterpret_cast<float *>(smem_raw + L.ck);     // K_c Z_c (GL)
    unsigned char *tab = smem_raw + L.tab;
    int &s_nq = *reinterpret_cast<int *>(smem_raw + L.queue);              // guarded pairs of a pass
    unsigned *queue = reinterpret_cast<unsigned *>(smem_raw + L.queue) + 1;

    if (!RT) {
        if (tid == 0) s_nq = 0;
        const uint4 *src = reinterpret_cast<const uint4 *>(A.ptab);
        uint4 *dst = reinterpret_cast<uint4 *>(tab);
        const int n16 = (kProjW * kProjStride + 15) / 16;
        for (int i = tid; i < n16; i += blockDim.x) dst[i] = src[i];
    }
    const double *Vja = A.V + ((long)j * N + a) * N;
    // per-patch slots; with UNIB the weight column is filled per q block (b)
    const float Za = A.Z ? (float)A.Z[a] : 1.f;
    const float kza = GL ? (float)A.K[a] * Za : 0.f;
    auto fill_slots = [&](int b) {
        const float vb = UNIB ? (float)Vja[b] : 0.f;
        const float Zb = UNIB && GL ? (A.Z ? (float)A.Z[b] : 1.f) : 0.f, kzb = UNIB && GL ? (float)A.K[b] * Zb : 0.f;
        for (int i = tid; i < SF_SLOTS; i += blockDim.x) {
            if (i <= N) {
                const int cc = i == N ? 0 : i;
                const float Zc = A.Z ? (float)A.Z[cc] : 1.f;
                const float lz = qp ? Zc : 1.f;
                const float vc = (float)Vja[cc];
                const float lzc = lz * A.cT;     // energies of r in units of T / log2(e)
                const float kzc = GL ? (float)A.K[cc] * Zc : 0.f;
                if (GL) ck[i] = kzc;
                const float gl = UNIB && GL ? (kza * (Zb + Zc) + kzb * (Za + Zc) + kzc * (Za + Zb)) * (1.f / 6.f) : 1.f;
                cz[i] = UNIB ? make_float4(gl * Zc * (2.f * vb * vb - vb * vc), 0.f, -2.f * A.t * lzc, -A.mu * lzc)
                             : make_float4(Zc, Zc * vc, -2.f * A.t * lzc, -A.mu * lzc);
                cd[i] = -4.f * A.tp * lzc;
                const float4 bd = A.bnd[cc];
                ray[i] = make_float2(bd.x, bd.z);
            } else {
                cz[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                cd[i] = 0.f;
                if (GL) ck[i] = 0.f;
                ray[i] = make_float2(0.f, 0.f);
            }
        }
    };
    int b_slots = UNIB ? (blockIdx.x * A.qb * 256 * SF_QPT) / PP : 0;
    fill_slots(b_slots);
    const float lza = qp ? Za : 1.f;
    const float4 kcs = A.kcs[j];
    const float xj = A.xij_f[j];

    const unsigned char *tabc = tab + (kProjW / 2) * (kProjStride + 1);   // the cell of the origin
    // records of the loop points p0 .. p0 + cnt - 1 of patch a
    auto stage = [&](int p0, int cnt) {
        for (int i = tid; i < cnt; i += blockDim.x) {
            const int p = a * PP + p0 + i;
            const int2 kf = RT ? make_int2(0, 0) : A.kfx[(long)j * M + p];   // (the table needs no momenta)
            const float cpx = A.fine.cx[p], spx = A.fine.sx[p], cpy = A.fine.cy[p], spy = A.fine.sy[p];
            const float xp = lza * A.fine.xi[p];
            float fp, fcp;
            sfermi(xp, A.invT, fp, fcp);
            const float wp = A.fine.w[p];
            rA[i] = make_float4(__int_as_float(kf.x), __int_as_float(kf.y), kcs.x * cpx - kcs.y * spx,
                                kcs.z * cpy - kcs.w * spy);
            rB[i] = make_float4(kcs.y * cpx + kcs.x * spx, kcs.w * cpy + kcs.z * spy, wp * fp, wp * fcp);
            rC[i] = xj + xp;
            if (i == cnt - 1 && (cnt & 1)) {   // pad: the same point with weight 0
                rA[i + 1] = rA[i];
                rB[i + 1] = make_float4(rB[i].x, rB[i].y, 0.f, 0.f);
                rC[i + 1] = rC[i];
            }
        }
    };
    const bool one_pass = P <= pch;
    if (one_pass) stage(0, P);
    __syncthreads();   // tables (and the records of a single pass) written

    static_assert(SF_QPT == 2, "the loop points of a thread are the two lanes of the packed arithmetic");
    const float2 one2 = make_float2(1.f, 1.f), ntln2 = make_float2(-A.tln2, -A.tln2);
    const float2 nkchord = make_float2(-A.kchord, -A.kchord), eta2x4 = make_float2(A.eta2x4, A.eta2x4);
    double vsum = 0.0;
    // A.qb blocks of 256 SF_QPT loop points q per CTA reuse the staged tables
    for (int qb = 0; qb < A.qb; ++qb) {
        const int blk = blockIdx.x * A.qb + qb;
        if (blk * (256 * SF_QPT) >= M) break;   // uniform over the CTA
        if (UNIB && blk * (256 * SF_QPT) / PP != b_slots) {
            b_slots = blk * (256 * SF_QPT) / PP;
            __syncthreads();   // every warp is done with the previous weights
            fill_slots(b_slots);
            __syncthreads();
        }
        // the SF_QPT loop points q of this thread (an index past M gets weight 0)
        // (cos, sin) of (q_x, q_y) as pairs: cos r_x and cos r_y in one packed FMA
        float2 cq[SF_QPT], sq[SF_QPT];
        float fqp[SF_QPT], fcqp[SF_QPT], v2[SF_QPT], vab[SF_QPT], mxq[SF_QPT];
        float2 acc = make_float2(0.f, 0.f);     // the SF_QPT = 2 loop points as the two lanes
        float ga[SF_QPT], gb[SF_QPT], gc[SF_QPT];   // GL: bracket = ga + gb Z_c + gc K_c Z_c
        int qx[SF_QPT], qy[SF_QPT];
        const uint8_t *rq[SF_QPT];   // RT: the patch-of-r rows of this thread's loop points q
#pragma unroll
        for (int k = 0; k < SF_QPT; ++k) {
            const int iq = blk * (256 * SF_QPT) + k * 256 + tid;   // angular-minor index
            const bool valid = iq < M;
            const int ii = valid ? iq : M - 1;
            rq[k] = RT ? A.rtab + (((long)jidx * N + a) * (long)(PP / 8) * M + ii) * 8 : nullptr;
            const int b = ii / PP, rem = ii - b * PP;
            const int qq = b * PP + (rem % A.pb.n_theta) * A.pb.n_r + rem / A.pb.n_theta;
            const float Zb = A.Z ? (float)A.Z[b] : 1.f;
            qx[k] = A.pfx[qq].x;
            qy[k] = A.pfx[qq].y;
            cq[k] = make_float2(A.fine.cx[qq], A.fine.cy[qq]);
            sq[k] = make_float2(A.fine.sx[qq], A.fine.sy[qq]);
            const float xq = (qp ? Zb : 1.f) * A.fine.xi[qq];
            float fq, fcq;
            sfermi(xq, A.invT, fq, fcq);
            const float pref = valid ? Za * Zb * A.fine.w[qq] : 0.f;
            fqp[k] = fq * pref;
            fcqp[k] = fcq * pref;
            if (GL && !UNIB) {
                const float kzb = (float)A.K[b] * Zb;
                ga[k] = (kza * Zb + kzb * Za) * (1.f / 6.f);
                gb[k] = (kza + kzb) * (1.f / 6.f);
                gc[k] = (Za + Zb) * (1.f / 6.f);
            }
            vab[k] = (float)Vja[b];
            v2[k] = 2.f * vab[k] * vab[k];
            mxq[k] = -xq;
        }

        for (int p0 = 0; p0 < P; p0 += pch) {
            const int cnt = P - p0 < pch ? P - p0 : pch;
            if (!one_pass) {
                __syncthreads();   // previous pass done with the records
                stage(p0, cnt);
                __syncthreads();
            }
            // the arithmetic of two records (ra, rb, upp) and their 2 x SF_QPT
            // patches c: the two loop points q of a record as the lanes of
            // packed FP32x2 operations where the operands pair up
            auto pair_math = [&](const float4 (&ra)[2], const float4 (&rb)[2], const float (&upp)[2],
                                 const int (&c)[2][SF_QPT]) {
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    float2 xr, amp, sum;
                    float2 fr, aq, dq;
#pragma unroll
                    for (int k = 0; k < SF_QPT; ++k) {
                        const float4 z = cz[c[r][k]];
                        // (cos r_x, cos r_y) by angle addition
                        const float2 cr2 = __ffma2_rn(make_float2(ra[r].z, ra[r].w), cq[k],
                                                      __fmul2_rn(make_float2(rb[r].x, rb[r].y), sq[k]));
                        float x = fmaf(cr2.x + cr2.y, z.z, z.w);       // Z-scaled line energy of r / (T ln 2)
                        if (!TP0) x = fmaf(cr2.x * cr2.y, cd[c[r][k]], x);
                        const float ex = ex2_approx(x);
                        const float a = rb[r].z * fcqp[k];
                        const float d = fmaf(rb[r].w, fqp[k], -a);
                        float w = UNIB ? z.x : fmaf(-vab[k], z.y, z.x * v2[k]);
                        if (GL && !UNIB) w *= fmaf(gc[k], ck[c[r][k]], fmaf(gb[k], z.x, ga[k]));
                        const float sm = upp[r] + mxq[k];
                        if (k == 0) { xr.x = x; fr.x = ex; aq.x = a; dq.x = d; amp.x = w; sum.x = sm; }
                        else        { xr.y = x; fr.y = ex; aq.y = a; dq.y = d; amp.y = w; sum.y = sm; }
                    }
                    const float2 g = __fadd2_rn(fr, one2);
                    fr = make_float2(rcp_approx(g.x), rcp_approx(g.y));
                    const float2 F = __ffma2_rn(fr, dq, aq);           // A + f_r (B - A)
                    amp = __fmul2_rn(amp, F);
                    // d0 = xi_j - E, E = x_q + x_r - x_p
                    const float2 d0 = __ffma2_rn(xr, ntln2, sum);
                    const float2 u = __ffma2_rn(d0, d0, nkchord);
                    const float2 den = __ffma2_rn(__fmul2_rn(eta2x4, d0), d0, __fmul2_rn(u, u));
                    acc = __ffma2_rn(__fmul2_rn(amp, u), make_float2(rcp_approx(den.x), rcp_approx(den.y)), acc);
                }
            };
            if (RT) {
                // eight records per trip: their patches for each loop point q
                // are one 8-byte word of the table, loaded one trip ahead
                // (word of records i .. i+7 at rq + i M)
                uint2 wn[SF_QPT];
#pragma unroll
                for (int k = 0; k < SF_QPT; ++k) wn[k] = __ldcs(reinterpret_cast<const uint2 *>(rq[k] + (long)p0 * M));
                for (int i = 0; i < cnt; i += 8) {
                    uint2 w[SF_QPT];
#pragma unroll
                    for (int k = 0; k < SF_QPT; ++k) {
                        w[k] = wn[k];
                        if (i + 8 < cnt) wn[k] = __ldcs(reinterpret_cast<const uint2 *>(rq[k] + (long)(p0 + i + 8) * M));
                    }
#pragma unroll 2
                    for (int s2 = 0; s2 < 4; ++s2) {
                        float4 ra[2], rb[2];
                        float upp[2];
                        int c[2][SF_QPT];
#pragma unroll
                        for (int r = 0; r < 2; ++r) {
                            ra[r] = rA[i + 2 * s2 + r];
                            rb[r] = rB[i + 2 * s2 + r];
                            upp[r] = rC[i + 2 * s2 + r];
#pragma unroll
                            for (int k = 0; k < SF_QPT; ++k) {
                                const int byte = 2 * s2 + r;
                                const unsigned word = byte < 4 ? w[k].x : w[k].y;
                                c[r][k] = (int)((word >> (8 * (byte & 3))) & 255u);
                            }
                        }
                        pair_math(ra, rb, upp, c);
                    }
                }
            } else {
            // two records per iteration: the patches of all 2 x SF_QPT pairs
            // first, one rarely taken branch that queues the guarded ones, then the
            // arithmetic of all of them with the table's patch (one large block for
            // the scheduler; a call for the exact patch here spilled registers in
            // every iteration, 40 % of the time);
            // an odd count reads the zero-weight pad record after the last one;
            // the loop is unrolled four times (eight records per trip, 122
            // registers: the loop overhead amortised, more independent work).
            // The queue is settled after a chunk of records that leaves it a quarter
            // full, and at the end of the pass.  The first chunk is 16 records, or 256
            // where boundary pairs are known to be few (sigma_plan), the next four times
            // the last while few pairs are queued: where the lattice's mirror lies on a
            // boundary (N = 4 mod 8) up to 6 % of the pairs are exact ties, which a queue
            // per pass could not hold: N = 60, 10 x 14 points, 55 ms against 8.5 without.
            int sub = A.sub0, kept = 0, settled = 0;
            for (int i0 = 0; i0 < cnt;) {
            const int i1 = min(cnt, i0 + sub);
#pragma unroll 4
            for (int i = i0; i < i1; i += 2) {
                float4 ra[2], rb[2];
                float upp[2];
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    ra[r] = rA[i + r];
                    rb[r] = rB[i + r];
                    upp[r] = rC[i + r];
                }
                int c[2][SF_QPT];
                unsigned slow_mask = 0;
#pragma unroll
                for (int r = 0; r < 2; ++r)
#pragma unroll
                    for (int k = 0; k < SF_QPT; ++k) {
                        float x, y;
                        bool slow;
                        c[r][k] = fx_patch(__float_as_int(ra[r].x), __float_as_int(ra[r].y), qx[k], qy[k], tabc, ray,
                                           x, y, slow);
                        slow_mask |= slow ? 1u << (2 * r + k) : 0u;
                    }
                if (__any_sync(0xffffffffu, slow_mask != 0)) {
                    // taken by the whole warp (a branch per lane left the lanes apart
                    // for the rest of the unrolled trip: 84 instead of 40 issue slots
                    // per pair); one copy of the code for the four pairs
                    unsigned todo = __reduce_or_sync(0xffffffffu, slow_mask);
#pragma unroll 1
                    for (; todo; todo &= todo - 1) {
                        const int e = __ffs(todo) - 1;
                        const bool r1 = e >= SF_QPT, k1 = (e & 1) != 0;
                        bool slow;
                        const int cc = fx_zoom(__float_as_int(r1 ? ra[1].x : ra[0].x), __float_as_int(r1 ? ra[1].y : ra[0].y),
                                               k1 ? qx[1] : qx[0], k1 ? qy[1] : qy[0], tabc, ray, slow);
                        const bool mine = (slow_mask >> e & 1u) != 0;
                        const int rec = i + (r1 ? 1 : 0);
                        if (mine && slow && rec < cnt) {     // (the pad record has weight 0)
                            const int at = atomicAdd(&s_nq, 1);
                            if (at < A.qcap) queue[at] = (unsigned)rec | (unsigned)((k1 ? 256 : 0) + tid) << 12;
                        }
                        __syncwarp();
                        if (mine && !r1 && !k1) c[0][0] = cc;
                        if (mine && !r1 && k1) c[0][1] = cc;
                        if (mine && r1 && !k1) c[1][0] = cc;
                        if (mine && r1 && k1) c[1][1] = cc;
                    }
                }
                pair_math(ra, rb, upp, c);
            }
            // the guarded pairs: where the exact patch differs from the table's, the
            // difference of the two chord terms
            __syncthreads();
            const int nq = s_nq;
            __syncthreads();
            const int added = nq - kept, nrec = i1 - settled;
            sub = added > A.qcap / 4 ? max(16, sub / 4) : (added < 16 ? min(SF_PCH, 4 * sub) : sub);
            kept = nq;
            i0 = i1;
            if (i1 < cnt && nq <= A.qcap / 4) continue;     // uniform over the CTA
            if (tid == 0) s_nq = 0;
            const bool over = nq > A.qcap;      // more than the queue holds: look at every pair again
            const int ntot = over ? nrec * (256 * SF_QPT) : nq;
            for (int e = tid; e < ntot; e += 256) {
                const unsigned en = over ? (unsigned)(settled + e % nrec) | (unsigned)(e / nrec) << 12 : queue[e];
                const int i = en & 4095u, iq = blk * (256 * SF_QPT) + (int)(en >> 12);
                if (iq >= M) continue;
                const int b = iq / PP, rem = iq - b * PP;
                const int qq = b * PP + (rem % A.pb.n_theta) * A.pb.n_r + rem / A.pb.n_theta;
                const float4 ra = rA[i], rb = rB[i];
                // the patch the loop used
                float x, y;
                bool slow;
                fx_patch(__float_as_int(ra.x), __float_as_int(ra.y), A.pfx[qq].x, A.pfx[qq].y, tabc, ray, x, y, slow);
                if (!slow) continue;
                const int c0 = fx_zoom(__float_as_int(ra.x), __float_as_int(ra.y), A.pfx[qq].x, A.pfx[qq].y, tabc, ray, slow);
                if (!slow) continue;
                const bool edge = fmaxf(fabsf(x), fabsf(y)) > kFxEdge;
                const bool fix = A.sym.mode == 2 && sym && (4 * j) % N != 0;   // the zone-edge targets have no images
                const int c1 = sf_slow_patch(A, j, a * PP + p0 + i, qq, x * kRadPerFx, y * kRadPerFx,
                                             (edge ? 1 : 0) | (fix ? 2 : 0), A.bnd);
                if (c1 == c0) continue;
                const float Zb = A.Z ? (float)A.Z[b] : 1.f, vb = (float)Vja[b];
                const float xq = (qp ? Zb : 1.f) * A.fine.xi[qq];
                float fq, fcq;
                sfermi(xq, A.invT, fq, fcq);
                const float pref = Za * Zb * A.fine.w[qq];
                const float2 cr = __ffma2_rn(make_float2(ra.z, ra.w), make_float2(A.fine.cx[qq], A.fine.cy[qq]),
                                             __fmul2_rn(make_float2(rb.x, rb.y),
                                                        make_float2(A.fine.sx[qq], A.fine.sy[qq])));
                const float aq = rb.z * (fcq * pref), dq = fmaf(rb.w, fq * pref, -aq);
#pragma unroll 1
                for (int u = 0; u < 2; ++u) {
                    const int cc = u ? c0 : c1;
                    const float4 z = cz[cc];
                    float xr = fmaf(cr.x + cr.y, z.z, z.w);
                    if (!TP0) xr = fmaf(cr.x * cr.y, cd[cc], xr);
                    float w = UNIB ? z.x : fmaf(-vb, z.y, z.x * (2.f * vb * vb));
                    if (GL && !UNIB) {
                        const float kzb = (float)A.K[b] * Zb;
                        w *= ((kza * Zb + kzb * Za) + (kza + kzb) * z.x + (Za + Zb) * ck[cc]) * (1.f / 6.f);
                    }
                    const float F = fmaf(rcp_approx(1.f + ex2_approx(xr)), dq, aq);
                    const float d0 = fmaf(xr, -A.tln2, rC[i] - xq);
                    const float uu = fmaf(d0, d0, -A.kchord);
                    const float t = w * F * uu * rcp_approx(fmaf(A.eta2x4 * d0, d0, uu * uu));
                    acc.x += u ? -t : t;
                }
            }
            __syncthreads();
            kept = 0;
            settled = i1;
            }
            }
        }
        vsum -= (double)acc.x + (double)acc.y;   // the chord term is -u / den
    }
    vsum *= fac;
    __shared__ double red[32];
    double v = vsum;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    const int lane = tid & 31, warp = tid >> 5;
    if (lane == 0) red[warp] = v;
    __syncthreads();
    if (warp == 0) {
        const int nw = blockDim.x >> 5;
        v = lane < nw ? red[lane] : 0.0;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
        if (lane == 0) atomicAdd(&A.sig[jidx], v);
    }
}

// Frequency-grid variant of sigma_fast_kernel: instead of the chord slope, W F
// binned by pole energy E = x_q + x_r - x_p (moments 0..4 of E about the bin
// centre in units of half a bin) in a shared-memory histogram per CTA, flushed
// to the FP64 histogram after every block of loop points q.
//
// What bounds it: the shared-memory adds, five or six per pair.  A float add on
// shared memory is a compare-and-swap loop, so the histogram is 32-bit fixed
// point with native integer reductions.  The lanes of a warp own neighbouring
// radii of q, whose energies lie many bins apart (angular neighbours share
// bins, and equal addresses serialise).  The scale of a flush period (1024
// loop points q times the patch's points p) follows from a bound on the sum of
// all its |W F| <= W_b max(f_p (1 - f_q), (1 - f_p) f_q), W_b the largest weight
// over c, so no bin leaves +-2^30 (a pair is then hundreds of units), and one
// addend stays below 2^21 units (rounded by adding 1.5 * 2^23, no conversion).
// What moment 0 rounds off goes into a second word (LO) in units 2^30 / pairs
// finer; the higher moments enter Sigma with (h/2|z - E|)^n <= 8^-n, which
// carries their rounding below that of the FP32 pairs.  np48, 16 x 16 points, 10
// targets, 512 frequencies: 26.0 -> 7.0 ms (58 -> 216 Gpair/s).
//
// Launch: grid (q splits, N patches a, targets), 512 threads, one CTA per SM
// (the histogram).  NBS: words per moment (a constant, so that the moments are
// immediate offsets), nbins <= NBS.  HALF: nbins <= 2 NBS, each half of the bins by
// CTAs of its own that walk every pair (even and odd blockIdx.x).
constexpr int HF_THR = 512;
constexpr int HF_QPT = 2;
constexpr int HF_REC = 256;     // loop points p staged per pass
constexpr int HF_QCAP = 1024;   // guarded pairs queued per pass

struct HfSmem {
    size_t rA, rB, cz, ray, cd, ck, wb, rC, queue, tab, hist, total;
};

__host__ __device__ constexpr HfSmem hf_smem_layout(int nbs, bool lo)
{
    HfSmem L{};
    L.rA = 0;
    L.rB = L.rA + (size_t)16 * HF_REC;
    L.cz = L.rB + (size_t)16 * HF_REC;
    L.ray = L.cz + (size_t)16 * SF_SLOTS;
    L.cd = L.ray + (size_t)8 * SF_SLOTS;
    L.ck = L.cd + (size_t)4 * SF_SLOTS;
    L.wb = L.ck + (size_t)4 * SF_SLOTS;
    L.rC = (L.wb + (size_t)4 * SF_SLOTS + 15) / 16 * 16;
    L.queue = L.rC + (size_t)4 * HF_REC;
    L.tab = L.queue + (size_t)4 * HF_QCAP;
    L.hist = L.tab + ((size_t)kProjW * kProjStride + 15) / 16 * 16;
    L.total = L.hist + (size_t)4 * nbs * (lo ? 6 : 5);
    return L;
}

__device__ __forceinline__ void red_shared(unsigned addr, int v)
{
    asm volatile("red.shared.add.s32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// A pole outside the bins (quasi-particle lines with a weight above z_max): the
// moments about the edge bin, which are far from one half bin (rare).
__device__ __noinline__ void hist_outside(const SigmaFastArgs &A, double *H, double m, float E)
{
    const int bin = E < A.e_min + 0.5 * A.nbins * A.h64 ? 0 : A.nbins - 1;
    const double d = (double)E - (A.e_min + (bin + 0.5) * A.h64);
    for (int mo = 0; mo < 5; ++mo, m *= d) atomicAdd(H + (long)mo * A.nbins + bin, m);
}

template <int NBS, bool LO, bool GL, bool HALF>
__global__ void __launch_bounds__(HF_THR, 1) sigma_hist_kernel(const SigmaFastArgs A)
{
    const int N = A.pb.N, M = A.pb.M, PP = A.pb.P;
    const int a = blockIdx.y, jidx = blockIdx.z;
    int j;
    bool sym;
    if (A.only_full && *A.nevents <= A.max_events) return;
    if (!sigma_target(A, jidx, j, sym)) return;      // uniform over the CTA
    const int P = PP;
    const int tid = threadIdx.x;
    const bool qp = A.pb.propagator == QPFRG_PROP_QP;
    const HfSmem L = hf_smem_layout(NBS, LO);

    extern __shared__ __align__(16) unsigned char smem_raw[];
    float4 *rA = reinterpret_cast<float4 *>(smem_raw + L.rA);   // (k+p)_x, (k+p)_y (fixed point), cos of both
    float4 *rB = reinterpret_cast<float4 *>(smem_raw + L.rB);   // sin of both, w_p f_p, w_p (1 - f_p)
    float4 *cz = reinterpret_cast<float4 *>(smem_raw + L.cz);   // Z_c, Z_c V_jac, -2t l_c, -mu l_c
    float2 *ray = reinterpret_cast<float2 *>(smem_raw + L.ray);
    float *cd = reinterpret_cast<float *>(smem_raw + L.cd);     // -4 t' l_c
    float *ck = reinterpret_cast<float *>(smem_raw + L.ck);     // K_c Z_c (GL)
    float *rC = reinterpret_cast<float *>(smem_raw + L.rC);     // x_p
    unsigned char *tab = smem_raw + L.tab;
    unsigned *queue = reinterpret_cast<unsigned *>(smem_raw + L.queue);   // guarded pairs of a pass
    __shared__ int s_nq;
    int *hs = reinterpret_cast<int *>(smem_raw + L.hist);       // [moment 0..4, rest of moment 0][NBS]
    float *wb = reinterpret_cast<float *>(smem_raw + L.wb);     // max over c of a pair's vertex and line weight
    __shared__ float s_max[2];                                  // max |Z|, |K Z|
    __shared__ float s_sum[2], s_blk[3];                        // sums of w_p f_p, w_p (1 - f_p); of a block of q
    __shared__ int s_bad;

    for (int i = tid; i < NBS * (LO ? 6 : 5); i += HF_THR) hs[i] = 0;
    if (tid < 2) s_max[tid] = s_sum[tid] = 0.f;
    if (tid == 2) s_bad = s_nq = 0;
    {
        const uint4 *src = reinterpret_cast<const uint4 *>(A.ptab);
        uint4 *dst = reinterpret_cast<uint4 *>(tab);
        const int n16 = (kProjW * kProjStride + 15) / 16;
        for (int i = tid; i < n16; i += HF_THR) dst[i] = src[i];
    }
    __syncthreads();
    const double *Vja = A.V + ((long)j * N + a) * N;
    const float Za = A.Z ? (float)A.Z[a] : 1.f;
    const float kza = GL ? (float)A.K[a] * Za : 0.f;
    const float lza = qp ? Za : 1.f;
    for (int i = tid; i < SF_SLOTS; i += HF_THR) {
        if (i <= N) {
            const int cc = i == N ? 0 : i;
            const float Zc = A.Z ? (float)A.Z[cc] : 1.f;
            const float lz = qp ? Zc : 1.f;
            const float vc = (float)Vja[cc];
            const float kzc = GL ? (float)A.K[cc] * Zc : 1.f;
            cz[i] = make_float4(Zc, Zc * vc, -2.f * A.t * lz, -A.mu * lz);
            cd[i] = -4.f * A.tp * lz;
            if (GL) ck[i] = kzc;
            const float4 bd = A.bnd[cc];
            ray[i] = make_float2(bd.x, bd.z);
            // non-negative floats order like their bits
            atomicMax(reinterpret_cast<int *>(&s_max[0]), __float_as_int(fabsf(Zc)));
            atomicMax(reinterpret_cast<int *>(&s_max[1]), __float_as_int(fabsf(kzc)));
            if (!isfinite(vc) || !isfinite(Zc) || !isfinite(kzc)) s_bad = 1;
        } else {
            cz[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            cd[i] = 0.f;
            if (GL) ck[i] = 0.f;
            ray[i] = make_float2(0.f, 0.f);
        }
    }
    __syncthreads();
    double *H = A.hist + (long)jidx * 5 * A.nbins;
    // the bins bin0 .. bin0 + nb - 1 of this CTA
    const bool upper = HALF && (blockIdx.x & 1);
    const int bin0 = upper ? NBS : 0, nb = HALF ? (upper ? A.nbins - NBS : NBS) : A.nbins;
    if (s_bad) {       // a non-finite vertex or weight: as in the sums, every frequency of this target
        if (tid == 0) atomicAdd(&H[0], __longlong_as_double(0x7ff8000000000000LL));
        return;
    }
    const float4 kcs = A.kcs[j];
    const unsigned char *tabc = tab + (kProjW / 2) * (kProjStride + 1);   // the cell of the origin
    // bounds of the fixed-point scale (see above): the largest weight of patch b,
    // and the sums over the patch's points p
    const float gl_max = GL ? s_max[1] * s_max[0] : 1.f;
    for (int b = tid; b < N; b += HF_THR) {
        const float vb = (float)Vja[b];
        float m = 0.f;
        bool fin = true;         // (fmaxf drops a NaN)
        for (int c = 0; c < N; ++c) {
            const float w = fabsf(fmaf(-vb, cz[c].y, cz[c].x * 2.f * vb * vb));
            m = fmaxf(m, w);
            fin = fin && w <= 3e38f;
        }
        wb[b] = fin ? m * gl_max : __int_as_float(0x7f800000);
    }
    for (int i = tid; i < P; i += HF_THR) {
        float fp, fcp;
        sfermi(lza * A.fine.xi[a * PP + i], A.invT, fp, fcp);
        const float w = A.fine.w[a * PP + i];
        atomicAdd(&s_sum[0], w * fp);
        atomicAdd(&s_sum[1], w * fcp);
    }
    const float pairs = (float)(HF_THR * HF_QPT) * (float)P;
    const float lo_scale = 1073741824.f / pairs;
    constexpr float kMagic = 12582912.f;
    const unsigned hbase = (unsigned)__cvta_generic_to_shared(hs);

    // one pair of weight amp and pole energy E: its bin, the offset from the
    // bin's centre in half bins, and the moments
    auto deposit = [&](float amp, float E, float scale, float lift) {
        const float u = amp * scale;                     // in units of the histogram
        int r;                                           // (past +-2^22: no bin either)
        const float rr = rint_add(fmaf(E, A.inv_h, A.c_frac), r);
        const float d = 2.f * (fmaf(E, A.inv_h, -rr) + fmaf(E, A.inv_h_lo, A.c_frac));
        const int bin = r + A.c_int - bin0;
        if ((unsigned)bin >= (unsigned)nb) {
            if (!HALF || (!upper && (unsigned)bin >= (unsigned)A.nbins)) hist_outside(A, H, (double)amp / lift, E);
            return;
        }
        const unsigned h = hbase + 4u * (unsigned)bin;
        const float u0 = u + kMagic;
        red_shared(h, __float_as_int(u0) - 0x4B400000);
        if (LO) {
            const float rest = fmaf(amp, scale, -(u0 - kMagic)) * lo_scale;
            red_shared(h + 20u * NBS, __float_as_int(rest + kMagic) - 0x4B400000);
        }
        float m = u;
#pragma unroll
        for (int mo = 1; mo < 5; ++mo) {
            m *= d;
            red_shared(h + 4u * NBS * mo, __float_as_int(m + kMagic) - 0x4B400000);
        }
    };
    const bool one_pass = P <= HF_REC;
    auto stage = [&](int p0, int cnt) {
        for (int i = tid; i < cnt; i += HF_THR) {
            const int p = a * PP + p0 + i;
            const int2 kf = A.kfx[(long)j * M + p];
            const float cpx = A.fine.cx[p], spx = A.fine.sx[p], cpy = A.fine.cy[p], spy = A.fine.sy[p];
            const float xp = lza * A.fine.xi[p];
            float fp, fcp;
            sfermi(xp, A.invT, fp, fcp);
            const float wp = A.fine.w[p];
            rA[i] = make_float4(__int_as_float(kf.x), __int_as_float(kf.y), kcs.x * cpx - kcs.y * spx,
                                kcs.z * cpy - kcs.w * spy);
            rB[i] = make_float4(kcs.y * cpx + kcs.x * spx, kcs.w * cpy + kcs.z * spy, wp * fp, wp * fcp);
            rC[i] = xp;
        }
    };
    if (one_pass) stage(0, P);

    const int nblk = (M + HF_THR * HF_QPT - 1) / (HF_THR * HF_QPT);
    for (int blk = HALF ? blockIdx.x >> 1 : blockIdx.x; blk < nblk; blk += HALF ? gridDim.x >> 1 : gridDim.x) {
        float2 cq[HF_QPT], sq[HF_QPT];
        float fqp[HF_QPT], fcqp[HF_QPT], v2[HF_QPT], vab[HF_QPT], xqk[HF_QPT], ga[HF_QPT], gb[HF_QPT], gc[HF_QPT];
        int qx[HF_QPT], qy[HF_QPT];
        if (tid < 3) s_blk[tid] = 0.f;
        __syncthreads();
        float t1 = 0.f, t2 = 0.f, t3 = 0.f;      // sums and maximum of the weights of this thread's q
#pragma unroll
        for (int k = 0; k < HF_QPT; ++k) {
            const int iq = blk * (HF_THR * HF_QPT) + k * HF_THR + tid;   // radial-minor: the storage order
            const bool valid = iq < M;
            const int qq = valid ? iq : M - 1;
            const int b = qq / PP;
            const float Zb = A.Z ? (float)A.Z[b] : 1.f;
            qx[k] = A.pfx[qq].x;
            qy[k] = A.pfx[qq].y;
            cq[k] = make_float2(A.fine.cx[qq], A.fine.cy[qq]);
            sq[k] = make_float2(A.fine.sx[qq], A.fine.sy[qq]);
            const float xq = (qp ? Zb : 1.f) * A.fine.xi[qq];
            float fq, fcq;
            sfermi(xq, A.invT, fq, fcq);
            const float pref = valid ? Za * Zb * A.fine.w[qq] : 0.f;
            fqp[k] = fq * pref;
            fcqp[k] = fcq * pref;
            vab[k] = (float)Vja[b];
            v2[k] = 2.f * vab[k] * vab[k];
            xqk[k] = xq;
            if (GL) {
                const float kzb = (float)A.K[b] * Zb;
                ga[k] = (kza * Zb + kzb * Za) * (1.f / 6.f);
                gb[k] = (kza + kzb) * (1.f / 6.f);
                gc[k] = (Za + Zb) * (1.f / 6.f);
            }
            t1 += fabsf(fcqp[k]) * wb[b];
            t2 += fabsf(fqp[k]) * wb[b];
            t3 = fmaxf(t3, fabsf(pref) * wb[b]);
        }
        for (int off = 16; off > 0; off >>= 1) {
            t1 += __shfl_down_sync(0xffffffffu, t1, off);
            t2 += __shfl_down_sync(0xffffffffu, t2, off);
            t3 = fmaxf(t3, __shfl_down_sync(0xffffffffu, t3, off));
        }
        if ((tid & 31) == 0) {
            atomicAdd(&s_blk[0], t1);
            atomicAdd(&s_blk[1], t2);
            atomicMax(reinterpret_cast<int *>(&s_blk[2]), __float_as_int(t3));
        }
        __syncthreads();
        // |W F| <= W max(f_p (1 - f_q), (1 - f_p) f_q) summed over the block
        float total = s_sum[0] * s_blk[0] + s_sum[1] * s_blk[1], single = A.w_max * s_blk[2];
        if (!(total <= 3e38f && single <= 3e38f)) {      // a weight overflows: as non-finite ones
            if (tid == 0) atomicAdd(&H[0], __longlong_as_double(0x7ff8000000000000LL));
            return;
        }
        // a small block is raised by a power of two, so that the scale stays finite
        const float lift = total < 1e-20f ? 1.2089258e24f : 1.f;
        total *= lift;
        single *= lift;
#pragma unroll
        for (int k = 0; k < HF_QPT; ++k) {
            fqp[k] *= lift;
            fcqp[k] *= lift;
        }
        const float scale = total > 0.f ? fminf(1073741824.f / total, 2097152.f / single) : 0.f;
        const double unit = scale > 0.f ? 1.0 / ((double)scale * (double)lift) : 0.0, unit_lo = unit / (double)lo_scale;
        for (int p0 = 0; p0 < P; p0 += HF_REC) {
            const int cnt = min(HF_REC, P - p0);
            if (!one_pass) {
                __syncthreads();   // previous pass done with the records
                stage(p0, cnt);
                __syncthreads();
            }
            // the queue is settled in chunks, as in sigma_fast_kernel
            int sub = A.sub0 / 2, kept = 0, settled = 0;
            for (int i0 = 0; i0 < cnt;) {
            const int i1 = min(cnt, i0 + sub);
#pragma unroll 2
            for (int i = i0; i < i1; ++i) {
                const float4 ra = rA[i], rb = rB[i];
                const float xp = rC[i];
                int c[HF_QPT];
                bool slow[HF_QPT];
#pragma unroll
                for (int k = 0; k < HF_QPT; ++k) {
                    float x, y;
                    c[k] = fx_patch(__float_as_int(ra.x), __float_as_int(ra.y), qx[k], qy[k], tabc, ray, x, y, slow[k]);
                }
                if (__any_sync(0xffffffffu, slow[0] || slow[1])) {      // taken by the whole warp
#pragma unroll
                    for (int k = 0; k < HF_QPT; ++k) {
                        bool still;
                        const int cc = fx_zoom(__float_as_int(ra.x), __float_as_int(ra.y), qx[k], qy[k], tabc, ray, still);
                        if (slow[k]) c[k] = cc;
                        if (slow[k] && still) {       // queued; the table's patch until the pass ends
                            const int at = atomicAdd(&s_nq, 1);
                            if (at < A.qcap) queue[at] = (unsigned)i | (unsigned)(k * HF_THR + tid) << 12;
                        }
                        __syncwarp();
                    }
                }
#pragma unroll
                for (int k = 0; k < HF_QPT; ++k) {
                    const float4 z = cz[c[k]];
                    const float2 cr = __ffma2_rn(make_float2(ra.z, ra.w), cq[k],
                                                 __fmul2_rn(make_float2(rb.x, rb.y), sq[k]));
                    float xr = fmaf(cr.x + cr.y, z.z, z.w);          // Z-scaled line energy of r
                    xr = fmaf(cr.x * cr.y, cd[c[k]], xr);
                    const float Aq = rb.z * fcqp[k], Bq = rb.w * fqp[k];
                    const float F = fmaf(rcp_approx(1.f + ex2_approx(xr * A.cT)), Bq - Aq, Aq);
                    float w = fmaf(-vab[k], z.y, z.x * v2[k]);
                    if (GL) w *= fmaf(gc[k], ck[c[k]], fmaf(gb[k], z.x, ga[k]));
                    deposit(w * F, (xr + xqk[k]) - xp, scale, lift);
                }
            }
            // the guarded pairs: where the exact patch differs from the table's, its
            // contribution is taken out (the same rounded addends) and the right one
            // put in
            __syncthreads();
            const int nq = s_nq;
            __syncthreads();
            const int added = nq - kept, nrec = i1 - settled;
            sub = added > A.qcap / 4 ? max(8, sub / 4) : (added < 16 ? 4 * sub : sub);
            kept = nq;
            i0 = i1;
            if (i1 < cnt && nq <= A.qcap / 4) continue;     // uniform over the CTA
            if (tid == 0) s_nq = 0;
            const bool over = nq > A.qcap;      // more than the queue holds: look at every pair again
            const int ntot = over ? nrec * (HF_THR * HF_QPT) : nq;
            for (int e = tid; e < ntot; e += HF_THR) {
                const unsigned en = over ? (unsigned)(settled + e % nrec) | (unsigned)(e / nrec) << 12 : queue[e];
                const int i = en & 4095u, qq = blk * (HF_THR * HF_QPT) + (int)(en >> 12);
                if (qq >= M) continue;
                const float4 ra = rA[i], rb = rB[i];
                // the patch the loop used
                float x, y;
                bool slow;
                fx_patch(__float_as_int(ra.x), __float_as_int(ra.y), A.pfx[qq].x, A.pfx[qq].y, tabc, ray, x, y, slow);
                if (!slow) continue;
                const int c0 = fx_zoom(__float_as_int(ra.x), __float_as_int(ra.y), A.pfx[qq].x, A.pfx[qq].y, tabc, ray, slow);
                if (!slow) continue;
                const bool edge = fmaxf(fabsf(x), fabsf(y)) > kFxEdge;
                const bool fix = A.sym.mode == 2 && sym && (4 * j) % N != 0;   // the zone-edge targets have no images
                const int c1 = sf_slow_patch(A, j, a * PP + p0 + i, qq, x * kRadPerFx, y * kRadPerFx,
                                             (edge ? 1 : 0) | (fix ? 2 : 0), A.bnd);
                if (c1 == c0) continue;
                const int b = qq / PP;
                const float Zb = A.Z ? (float)A.Z[b] : 1.f, vb = (float)Vja[b];
                const float xq = (qp ? Zb : 1.f) * A.fine.xi[qq];
                float fq, fcq;
                sfermi(xq, A.invT, fq, fcq);
                const float pref = Za * Zb * A.fine.w[qq] * lift;
                const float2 cr = __ffma2_rn(make_float2(ra.z, ra.w), make_float2(A.fine.cx[qq], A.fine.cy[qq]),
                                             __fmul2_rn(make_float2(rb.x, rb.y),
                                                        make_float2(A.fine.sx[qq], A.fine.sy[qq])));
                const float Aq = rb.z * (fcq * pref), Bq = rb.w * (fq * pref);
#pragma unroll 1
                for (int u = 0; u < 2; ++u) {
                    const int cc = u ? c0 : c1;
                    const float4 z = cz[cc];
                    float xr = fmaf(cr.x + cr.y, z.z, z.w);
                    xr = fmaf(cr.x * cr.y, cd[cc], xr);
                    const float F = fmaf(rcp_approx(1.f + ex2_approx(xr * A.cT)), Bq - Aq, Aq);
                    float w = fmaf(-vb, z.y, z.x * (2.f * vb * vb));
                    if (GL) {
                        const float kzb = (float)A.K[b] * Zb;
                        w *= fmaf((Za + Zb) * (1.f / 6.f), ck[cc],
                                  fmaf((kza + kzb) * (1.f / 6.f), z.x, (kza * Zb + kzb * Za) * (1.f / 6.f)));
                    }
                    deposit(u ? -(w * F) : w * F, (xr + xq) - rC[i], scale, lift);
                }
            }
            __syncthreads();
            kept = 0;
            settled = i1;
            }
            // without the second word the rounding of moment 0 is kept small by
            // flushing after every pass
            if (!LO || p0 + HF_REC >= P) {
                for (int i = tid; i < nb; i += HF_THR) {
                    const int v = hs[i], lo = LO ? hs[5 * NBS + i] : 0;
                    if (v == 0 && lo == 0) continue;
                    hs[i] = 0;
                    if (LO) hs[5 * NBS + i] = 0;
                    atomicAdd(&H[bin0 + i], unit * (double)v + unit_lo * (double)lo);
                }
                float mom = scale > 0.f ? 1.f / scale : 0.f;     // (h/2)^moment per lifted unit
                for (int mo = 1; mo < 5; ++mo) {
                    mom *= 0.5f * A.h;
                    for (int i = tid; i < nb; i += HF_THR) {
                        const int v = hs[mo * NBS + i];
                        if (v == 0) continue;
                        hs[mo * NBS + i] = 0;
                        const double x = (double)((float)v * mom);
                        atomicAdd(&H[(long)mo * A.nbins + bin0 + i], lift == 1.f ? x : x / (double)lift);
                    }
                }
                __syncthreads();
            }
        }
    }
}

// FP64 self-energy of the wedge grid: the sum of sigma_kernel<double>, with the
// patches of r decided as in the FP32 kernels (fixed-point table, exact near the
// boundaries) and, for the chord, the targets that a symmetric (V, Z) needs.
//
// What bounds it: FP64 instructions, 64 clocks each per warp and scheduler.
// sigma_kernel<double> issued about 180 per pair, 100 of them for the projection
// (atan2 and three divisions); here about 55: the projection runs on the integer
// and FP32 pipes, and F and the chord term share one division,
//   F = (A + B e) / (1 + e) for x_r > 0, (A e + B) / (1 + e) otherwise, e = exp(-|x_r|/T),
//   A = w_p f_p (1 - f_q), B = w_p (1 - f_p) f_q.
// np16, 8 x 8 points, Z of a symmetric vertex (6 of 16 targets): 4.82 -> 0.83 ms.
// Launch: grid (ceil(M / 256), N patches a, target slots), 256 threads, one q each.
// GL: the interaction flow's line weights.  HIST: binned pole weights (every patch).
struct Sigma64Args {
    SigmaFastArgs a;
    FineTable<double> f;
    double *hist;
    double e_min, inv_h;
    int nbins;
};
constexpr int S64_REC = 128;    // loop points p staged per pass
struct S64Rec {
    double cx, sx, cy, sy, x, wf, wfc;   // cos, sin of k + p, x_p, w_p f_p, w_p (1 - f_p)
    int kx, ky;                          // k + p in fixed point
};

template <bool TP0, bool GL, bool HIST>
__global__ void __launch_bounds__(256) sigma64_kernel(const Sigma64Args S)
{
    const SigmaFastArgs &A = S.a;
    const int N = A.pb.N, M = A.pb.M, PP = A.pb.P;
    const int a = blockIdx.y, jidx = blockIdx.z, tid = threadIdx.x;
    int j;
    bool sym;
    if (A.only_full && *A.nevents <= A.max_events) return;
    if (!sigma_target(A, jidx, j, sym)) return;      // uniform over the CTA
    const bool qp = A.pb.propagator == QPFRG_PROP_QP;
    const double T = A.T64, invT = 1.0 / T, eta2 = A.pb.eta * A.pb.eta;

    extern __shared__ __align__(16) unsigned char smem_raw[];
    S64Rec *rec = reinterpret_cast<S64Rec *>(smem_raw);
    double2 *zv = reinterpret_cast<double2 *>(rec + S64_REC);          // Z_c, Z_c V_jac
    double *kz = reinterpret_cast<double *>(zv + SF_SLOTS);            // K_c Z_c (GL)
    float2 *ray = reinterpret_cast<float2 *>(kz + (GL ? SF_SLOTS : 0));
    const unsigned char *tabc = A.ptab + (kProjW / 2) * (kProjStride + 1);   // the cell of the origin
    const double *Vja = A.V + ((long)j * N + a) * N;
    for (int i = tid; i < SF_SLOTS; i += 256) {
        const int c = i < N ? i : 0;
        const bool ok = i <= N;
        const double Zc = A.Z ? A.Z[c] : 1.0;
        zv[i] = ok ? make_double2(Zc, Zc * Vja[c]) : make_double2(0.0, 0.0);
        if (GL) kz[i] = ok ? A.K[c] * Zc : 0.0;
        const float4 bd = A.bnd[c];
        ray[i] = ok ? make_float2(bd.x, bd.z) : make_float2(0.f, 0.f);
    }
    const double Za = A.Z ? A.Z[a] : 1.0;
    double skx, ckx, sky, cky;
    sincos(A.kf[2 * j], &skx, &ckx);
    sincos(A.kf[2 * j + 1], &sky, &cky);
    auto fermi = [&](double x, double &f, double &fc) {
        const double e = exp(-fabs(x) * invT), hi = 1.0 / (1.0 + e), lo = e * hi;
        f = x > 0.0 ? lo : hi;
        fc = x > 0.0 ? hi : lo;
    };

    const int q = blockIdx.x * 256 + tid;
    const bool valid = q < M;
    const int qq = valid ? q : M - 1, b = qq / PP;
    const int qx = A.pfx[qq].x, qy = A.pfx[qq].y;
    const double cqx = S.f.cx[qq], sqx = S.f.sx[qq], cqy = S.f.cy[qq], sqy = S.f.sy[qq];
    const double Zb = A.Z ? A.Z[b] : 1.0;
    const double xq = (qp ? Zb : 1.0) * S.f.xi[qq];
    double fq, fcq;
    fermi(xq, fq, fcq);
    const double pref = valid ? Za * Zb * S.f.w[qq] : 0.0;
    fq *= pref;
    fcq *= pref;
    const double vab = Vja[b], v2 = 2.0 * vab * vab, dq = A.xij64[j] - xq, twoT = 2.0 * T;
    double ga = 0.0, gb = 0.0, gc = 0.0;     // GL: bracket = ga + gb Z_c + gc K_c Z_c
    if (GL) {
        const double kza = A.K[a] * Za, kzb = A.K[b] * Zb;
        ga = (kza * Zb + kzb * Za) * (1.0 / 6.0);
        gb = (kza + kzb) * (1.0 / 6.0);
        gc = (Za + Zb) * (1.0 / 6.0);
    }
    double acc = 0.0;
    for (int p0 = 0; p0 < PP; p0 += S64_REC) {
        const int cnt = min(S64_REC, PP - p0);
        __syncthreads();         // the slots written, the previous pass done
        for (int i = tid; i < cnt; i += 256) {
            const int p = a * PP + p0 + i;
            S64Rec r;
            const double cpx = S.f.cx[p], spx = S.f.sx[p], cpy = S.f.cy[p], spy = S.f.sy[p];
            r.cx = ckx * cpx - skx * spx;
            r.sx = skx * cpx + ckx * spx;
            r.cy = cky * cpy - sky * spy;
            r.sy = sky * cpy + cky * spy;
            r.x = (qp ? Za : 1.0) * S.f.xi[p];
            double f, fc;
            fermi(r.x, f, fc);
            r.wf = S.f.w[p] * f;
            r.wfc = S.f.w[p] * fc;
            const int2 k = A.kfx[(long)j * M + p];
            r.kx = k.x;
            r.ky = k.y;
            rec[i] = r;
        }
        __syncthreads();
        for (int i = 0; i < cnt; ++i) {
            const S64Rec &r = rec[i];
            float x, y;
            bool slow;
            int c = fx_patch(r.kx, r.ky, qx, qy, tabc, ray, x, y, slow);
            if (__any_sync(0xffffffffu, slow)) {          // taken by the whole warp
                bool still;
                const int cc = fx_zoom(r.kx, r.ky, qx, qy, tabc, ray, still);
                if (slow) c = cc;
                if (slow && still) {
                    const bool edge = fmaxf(fabsf(x), fabsf(y)) > kFxEdge;
                    // (the zone-edge targets have no images)
                    const bool fix = !HIST && A.sym.mode == 2 && sym && (4 * j) % N != 0 && valid;
                    c = sf_slow_patch(A, j, a * PP + p0 + i, qq, x * kRadPerFx, y * kRadPerFx,
                                      (edge ? 1 : 0) | (fix ? 2 : 0), A.bnd);
                }
                __syncwarp();
            }
            const double crx = r.cx * cqx + r.sx * sqx, cry = r.cy * cqy + r.sy * sqy;
            double xr = -2.0 * A.pb.t * (crx + cry) - A.pb.mu;
            if (!TP0) xr -= 4.0 * A.pb.tp * crx * cry;
            const double2 z = zv[c];
            if (qp) xr *= z.x;
            const double e = exp(-fabs(xr) * invT), An = r.wf * fcq, Bn = r.wfc * fq;
            double w = fma(-vab, z.y, z.x * v2) * (xr > 0.0 ? fma(Bn, e, An) : fma(An, e, Bn));
            if (GL) w *= fma(gc, kz[c], fma(gb, z.x, ga));
            if (HIST) {
                const double E = xq + xr - r.x, amp = w / (1.0 + e);
                int bin = (int)floor((E - S.e_min) * S.inv_h);
                bin = bin < 0 ? 0 : (bin >= S.nbins ? S.nbins - 1 : bin);
                const double d = E - (S.e_min + (bin + 0.5) / S.inv_h);
                double *h = S.hist + (long)jidx * 5 * S.nbins + bin;
                double m = amp;
                if (valid) {
#pragma unroll
                    for (int mo = 0; mo < 5; ++mo) {
                        atomicAdd(h + (long)mo * S.nbins, m);
                        m *= d;
                    }
                }
            } else {
                // chord slope of Re 1/(w - E + i eta) over w = xi_j +- 2T:
                // (eta^2 - d+ d-) / ((d+^2 + eta^2)(d-^2 + eta^2))
                const double d0 = dq - xr + r.x, dp = d0 + twoT, dm = d0 - twoT;
                acc += w * fma(-dp, dm, eta2) / ((1.0 + e) * (fma(dp, dp, eta2) * fma(dm, dm, eta2)));
            }
        }
    }
    if constexpr (!HIST) {
        __shared__ double red[8];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, off);
        if ((tid & 31) == 0) red[tid >> 5] = acc;
        __syncthreads();
        if (tid == 0) {
            double v = 0.0;
            for (int i = 0; i < 8; ++i) v += red[i];
            atomicAdd(&A.sig[jidx], v);
        }
    }
}

// Z_j = 1/(1 - slope) with the chord slope accumulated per target slot, or the
// slopes themselves (slopes_out).  rep[j] (may be NULL) is the slot of j's C4v
// representative among the targets, own[j] its own (NULL: j); sym.mode == 2: where the C4v test holds, with
// the patch's own correction corr[j], or from the sums of every patch (full) when
// the record of boundary pairs ran over.
__global__ void z_update_kernel(const double *slope, const double *corr, const double *full, const unsigned *nevents,
                                unsigned max_events, const int *rep, const int *own, SymMode sym, double *Zout,
                                double *slopes_out, int N)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= N) return;
    const bool use = rep && (sym.mode != 2 || sym_compact(sym));
    double s = slope[use ? rep[j] : (own ? own[j] : j)];
    if (sym.mode == 2 && use) s = *nevents > max_events ? full[j] : s + corr[j];
    if (slopes_out) slopes_out[j] = s;
    if (Zout) Zout[j] = 1.0 / (1.0 - s);
}

// Sigma on the grid from the binned moments: sum_b sum_n H_n[b] / (z - E_b)^(n+1),
// z = w_m + i eta (Taylor expansion of 1/(z - E_b - d) in the offset d), for the
// target slots of the histogram, accumulated into acc[slot][re, im][m].
//
// What bounds it: FP64 FMAs (2 per clock and SM).  The powers of u = 1/(z - E_b)
// do not depend on the target, so a thread (one frequency) computes them once
// for RG_T targets (32 FP64 operations, then 10 per target), empty bins cost one
// read, only the targets of a symmetric vertex are resummed, and the bins are
// split over the grid.  np48, 512 frequencies, 4 801 bins: 15.7 -> 1.5 ms.
constexpr int RG_T = 8;         // targets per thread
constexpr int RG_BINS = 64;     // bins per CTA

__global__ void __launch_bounds__(128) sigma_resum_kernel(const double *__restrict__ hist, int nbins, double e_min,
                                                          double h, int n_omega, double w0, double dw, double eta,
                                                          double *__restrict__ acc, int ntarget, int n_list, SymMode sym,
                                                          const unsigned *nevents, unsigned max_events)
{
    // the slots past the list hold the corrections of the images, or their own sums
    const bool more = sym.mode == 2 && (nevents[1] != 0 || nevents[0] > max_events);
    const int nt = sym.mode == 2 && !more && sym_compact(sym) ? n_list : ntarget;
    const int t0 = blockIdx.z * RG_T;
    if (t0 >= nt) return;
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    const double w = w0 + dw * min(m, n_omega - 1);
    const int b0 = blockIdx.y * RG_BINS, b1 = min(nbins, b0 + RG_BINS);
    const double eta2 = eta * eta;
    double sr[RG_T] = {}, si[RG_T] = {};
    for (int b = b0; b < b1; ++b) {
        double hv[RG_T][5];
        bool any = false;
#pragma unroll
        for (int t = 0; t < RG_T; ++t) {
            const double *H = hist + (long)(t0 + t) * 5 * nbins + b;
#pragma unroll
            for (int mo = 0; mo < 5; ++mo) hv[t][mo] = t0 + t < nt ? __ldg(H + (long)mo * nbins) : 0.0;
#pragma unroll
            for (int mo = 0; mo < 5; ++mo) any = any || hv[t][mo] != 0.0;
        }
        if (!any) continue;                      // uniform over the warp
        const double Eb = e_min + (b + 0.5) * h;
        const double dx = w - Eb, inv = 1.0 / fma(dx, dx, eta2);
        const double ur = dx * inv, ui = -eta * inv;
        double pr = ur, pi = ui;                 // u^(n+1)
#pragma unroll
        for (int mo = 0; mo < 5; ++mo) {
#pragma unroll
            for (int t = 0; t < RG_T; ++t) {
                sr[t] = fma(hv[t][mo], pr, sr[t]);
                si[t] = fma(hv[t][mo], pi, si[t]);
            }
            const double nr = pr * ur - pi * ui;
            pi = pr * ui + pi * ur;
            pr = nr;
        }
    }
    if (m >= n_omega) return;
#pragma unroll
    for (int t = 0; t < RG_T; ++t) {
        if (t0 + t >= nt || (sr[t] == 0.0 && si[t] == 0.0)) continue;
        atomicAdd(&acc[(2L * (t0 + t)) * n_omega + m], sr[t]);
        atomicAdd(&acc[(2L * (t0 + t) + 1) * n_omega + m], si[t]);
    }
}

// Sigma of every patch from its target slot; an image adds the correction in its
// own slot, which holds its whole sum when the record of boundary pairs ran over.
__global__ void sigma_spread_kernel(const double *__restrict__ acc, const int *rep, const int *own, SymMode sym,
                                    const unsigned *nevents, unsigned max_events, int n_omega, double *__restrict__ re,
                                    double *__restrict__ im)
{
    const int m = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
    if (m >= n_omega) return;
    const bool use = rep && (sym.mode != 2 || sym_compact(sym));
    const int so = own ? own[j] : j, sr = use ? rep[j] : so;
    const bool full = use && own && *nevents > max_events;
    const double *a = acc + 2L * (full ? so : sr) * n_omega + m;
    double x = a[0], y = a[n_omega];
    if (use && own && so != sr && !full) {
        a = acc + 2L * so * n_omega + m;
        x += a[0];
        y += a[n_omega];
    }
    re[(long)j * n_omega + m] = x;
    im[(long)j * n_omega + m] = y;
}

static qpfrg_status launch_kp_table(qpfrg_ctx *c, const int *jlist, int nj, bool fixed = true)
{
    const long total = (long)nj * c->pb.M;
    prof_begin(c);
    kp_table_kernel<<<(int)std::min<long>((total + 255) / 256, 152L * 8), 256, 0, c->stream>>>(
        c->d_kf, jlist, nj, c->f64.kx, c->f64.ky, c->pb.M, c->d_kp, fixed ? c->d_kfx : nullptr, c->d_kcs);
    prof_end(c, K_KP_TABLE);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? QPFRG_OK : cuda_fail(c, e, "kp_table_kernel");
}

template <typename R>
static qpfrg_status launch_sigma(qpfrg_ctx *c, bool hist, SigmaArgs<R> &A, int kid)
{
    const int P = c->pb.P, N = c->pb.N;
    const size_t smem = (size_t)(REC * P + 2 * N) * sizeof(R) + 16 + (size_t)N * sizeof(float4) + (size_t)N * sizeof(R);
    if (sizeof(R) == 4) {
        const qpfrg_status s = launch_kp_table(c, A.jlist, A.nj);
        if (s != QPFRG_OK) return s;
    }
    auto kern = hist ? sigma_kernel<R, true> : sigma_kernel<R, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_fail(c, e, "sigma smem attribute");
    dim3 grid(div_up(c->pb.M, 256), N, A.nj);
    prof_begin(c);
    kern<<<grid, 256, smem, c->stream>>>(A);
    prof_end(c, kid);
    e = cudaGetLastError();
    return e == cudaSuccess ? QPFRG_OK : cuda_fail(c, e, "sigma_kernel");
}

// Target slots of a self-energy call: a fixed list (mode 0; jlist NULL: every
// patch) or the list where the C4v test of (V, Z) holds and every patch where it
// does not, decided on the device (mode 2).
struct SigmaTargets {
    const int *jlist = nullptr;
    int n = 0;              // targets of the list
    SymMode sym;
    const int *rep = nullptr;   // slot of each patch under the list
    const int *own = nullptr;   // slot of each patch where every patch is evaluated (mode 2)
    int mirror = 0;             // mirror_part of the list's targets
    int slots(int N) const { return sym.mode == 2 || !jlist ? N : n; }
};

// Targets of a given (V, Z): with the symmetry that the device finds (red), the
// irreducible patches and the zone-edge patches, unhalved (every boundary pair is
// met); images copy the sum of their representative and correct it.
static SigmaTargets device_targets(const qpfrg_ctx *c, double tol, const unsigned long long *red)
{
    SigmaTargets t;
    t.n = c->pb.N;
    if (!c->max_events) return t;
    t.jlist = c->d_jgrid;
    t.n = c->n_grid;
    t.rep = c->d_repgrid;
    t.own = c->d_owngrid;
    t.sym.mode = 2;
    t.sym.red = red;
    t.sym.tol = tol / 3.0;
    return t;
}

// The last double k > 0 with rint(k / 2 pi) <= n (round to even at the half: 0.5
// folds to 0, 1.5 to 2), the comparisons of the FP64 fold.
static double fold_limit(int n)
{
    double k = (2 * n + 1) * kPi;
    while (std::rint(k / kTwoPi) > n) k = std::nextafter(k, 0.0);
    while (std::rint(std::nextafter(k, 1e9) / kTwoPi) <= n) k = std::nextafter(k, 1e9);
    return k;
}

// A smaller capacity for tests of what happens when it is exceeded.
static int test_limit(const char *name, int given)
{
    const char *s = std::getenv(name);
    return s ? std::min(given, std::max(0, std::atoi(s))) : given;
}

static SigmaFastArgs fast_args(qpfrg_ctx *c, double T, const double *d_V, const double *d_Z, const double *d_K,
                               const SigmaTargets &tg)
{
    SigmaFastArgs A{};
    A.pb = c->pb;
    A.fine = c->f32;
    A.V = d_V;
    A.Z = d_Z;
    A.K = d_K;
    A.kx64 = c->f64.kx;
    A.ky64 = c->f64.ky;
    A.kf = c->d_kf;
    A.xij_f = c->d_xij_f;
    A.qxl = c->d_qxl;
    A.qyl = c->d_qyl;
    A.kp = c->d_kp;
    A.kfx = c->d_kfx;
    A.pfx = c->d_pfx;
    A.kcs = c->d_kcs;
    A.bnd = c->d_bnd;
    A.ptab = c->d_ptab;
    A.jlist = tg.jlist;
    A.sym = tg.sym;
    A.n_list = tg.n;
    A.own = tg.own;
    A.mirror = tg.mirror;
    A.sig = c->d_sig;
    A.corr = c->d_sig + 2 * c->pb.N;
    A.events = c->d_events;
    A.nevents = reinterpret_cast<unsigned *>(c->d_sig + 4 * c->pb.N);
    A.max_events = c->max_events;
    A.t = (float)c->pb.t;
    A.tp = (float)c->pb.tp;
    A.mu = (float)c->pb.mu;
    A.invT = (float)(1.0 / T);
    A.cT = (float)(1.4426950408889634 / T);
    A.tln2 = (float)(0.6931471805599453 * T);
    A.kchord = (float)(4.0 * T * T + c->pb.eta * c->pb.eta);
    A.eta2x4 = (float)(4.0 * c->pb.eta * c->pb.eta);
    A.inv_dth = (float)(c->pb.N / kTwoPi);
    A.dth = (float)(kTwoPi / c->pb.N);
    A.w_max = (float)c->fw_max;
    A.xi64 = c->f64.xi;
    A.w64 = c->f64.w;
    A.xij64 = c->d_xij;
    A.T64 = T;
    static const double fold0 = fold_limit(0), fold1 = fold_limit(1);
    A.fold0 = fold0;
    A.fold1 = fold1;
    A.dth64 = kTwoPi / c->pb.N;
    A.sub0 = c->max_events > 0 ? 256 : 16;
    A.qcap = test_limit("QPFRG_TEST_QUEUE", 1 << 20);
    return A;
}

// Once per context: whether the reduced targets pay.  A boundary pair costs
// corrections of up to seven images in FP64 (7.5 ns, as long as the sums of 1800 FP32 or
// 85 FP64 pairs), so the list is used where the pairs that it saves cost twice that;
// the record of pairs is sized for them.  Generic grids have few; with N = 4 mod 8, mu
// and t' = 0 the lattice's mirror is a boundary between wedges and up to 6 % of the
// pairs lie on it: every patch is summed.  Counted where there are at most 2^22 pairs,
// else estimated from a sample.
qpfrg_status sigma_plan(qpfrg_ctx *c)
{
    c->max_events = 0;
    if (!c->d_ptab || !c->d_jgrid) return QPFRG_OK;
    qpfrg_status s = launch_kp_table(c, nullptr, c->pb.N);
    if (s != QPFRG_OK) return s;
    SigmaTargets tg;
    tg.jlist = c->d_jgrid;
    tg.n = c->n_grid;
    SigmaFastArgs A = fast_args(c, 1.0, nullptr, nullptr, nullptr, tg);
    const double M = c->pb.M, all = M * M * c->n_grid;
    const double n = std::fmin(all, 4194304.0);
    // an odd stride near the golden section of all pairs spreads the sample evenly
    const unsigned long long stride = n < all ? (unsigned long long)(0.6180339887498949 * all) | 1ull : 1ull;
    cudaError_t e = cudaMemsetAsync(A.nevents, 0, sizeof(unsigned), c->stream);
    if (e != cudaSuccess) return cuda_fail(c, e, "memset boundary pairs");
    boundary_count_kernel<<<152 * 4, 256, 0, c->stream>>>(A, (unsigned)n, stride);
    unsigned found = 0;
    if ((e = cudaGetLastError()) != cudaSuccess ||
        (e = cudaMemcpyAsync(&found, A.nevents, sizeof(found), cudaMemcpyDeviceToHost, c->stream)) != cudaSuccess ||
        (e = cudaStreamSynchronize(c->stream)) != cudaSuccess)
        return cuda_fail(c, e, "boundary pairs");
    const double pairs = found * (all / n), worth = c->opt.precision == QPFRG_FP64 ? 170.0 : 3600.0;
    // room for them, and for what a sample may have missed (np96, 32 x 32 points: some
    // 1e6 of 1.5e11 pairs are some 30 of the sample): at most 512 MB
    const double cap = n < all ? (found + 6.0 * std::sqrt((double)found) + 36.0) * (all / n) : pairs + 64.0;
    if (pairs * worth > (c->pb.N - c->n_grid) * M * M || cap > 33554432.0) return QPFRG_OK;
    if ((e = cudaMalloc((void **)&c->d_events, (size_t)cap * sizeof(int4))) != cudaSuccess)
        return cuda_fail(c, e, "cudaMalloc(boundary pairs)");
    c->max_events = (unsigned)std::max(1, test_limit("QPFRG_TEST_BOUNDARY_PAIRS", (int)cap));
    return QPFRG_OK;
}

// Chord slopes of the target slots into d_sig (FP32, wedge grid).
static qpfrg_status launch_sigma_fast(qpfrg_ctx *c, double T, const double *d_V, const double *d_Z, const double *d_K,
                                      const SigmaTargets &tg)
{
    const int nj = tg.slots(c->pb.N);
    // a list decided on the device may be any patch: k + p of all of them; a
    // launch that reads the patch table needs no fixed-point momenta
    const bool listed = !d_K && tg.sym.mode == 0 && tg.jlist != nullptr && tg.jlist == c->d_jirr;
    qpfrg_status s = launch_kp_table(c, tg.sym.mode == 2 ? nullptr : tg.jlist, nj, !(listed && c->d_rtab));
    if (s != QPFRG_OK) return s;
    SigmaFastArgs A = fast_args(c, T, d_V, d_Z, d_K, tg);
    A.qcap = std::min(A.qcap, SF_QCAP);
    const bool unib = c->pb.P % (256 * SF_QPT) == 0;
    // The flow's Z on the C4v-irreducible targets reads the patches of r from
    // a table built on first use (one byte per target, p and q: N_irr M^2
    // bytes, 126 GB at np96_n32), when it fits in 60 % of the free device
    // memory and options.sigma_table >= 0; otherwise it decides them per pair.
    // (record passes of a multiple of 8 records: P a multiple of 16, mirror halves included)
    const bool rt_list = listed && nj == c->n_irr && c->pb.P % 16 == 0 && c->pb.P <= SF_PCH;
    if (rt_list && !c->rtab_tried && c->opt.sigma_table >= 0) {
        c->rtab_tried = true;
        const size_t bytes = (size_t)nj * c->pb.N * (size_t)c->pb.P * (size_t)c->pb.M;
        size_t fr = 0, tot = 0;
        if (cudaMemGetInfo(&fr, &tot) == cudaSuccess && bytes <= fr / 10 * 6) {
            if (cudaMalloc((void **)&c->d_rtab, bytes) == cudaSuccess) {
                const size_t smem_b = kRtabSmem + (size_t)c->pb.P * sizeof(int2);
                cudaError_t e = cudaFuncSetAttribute(rtab_build_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                     (int)smem_b);
                if (e != cudaSuccess) return cuda_fail(c, e, "rtab smem attribute");
                prof_begin(c);
                rtab_build_kernel<<<dim3(div_up(c->pb.M, 256), c->pb.N, nj), 256, smem_b, c->stream>>>(A,
                                                                                                      c->d_rtab);
                prof_end(c, K_RTAB);
                if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(c, e, "rtab_build_kernel");
            } else {
                c->d_rtab = nullptr;
                cudaGetLastError();   // not enough memory: decide per pair
            }
        }
    }
    const bool rt = rt_list && c->d_rtab != nullptr;
    const size_t smem = sf_smem_layout(c->pb.P < SF_PCH ? c->pb.P : SF_PCH, rt).total;
    A.rtab = rt ? c->d_rtab : nullptr;
    using Kern = void (*)(SigmaFastArgs);
    static const Kern plain[2][2][2] = {   // [t' = 0][uniform blocks][table]
        {{sigma_fast_kernel<false, false, false, false>, sigma_fast_kernel<false, false, true, false>},
         {sigma_fast_kernel<false, true, false, false>, sigma_fast_kernel<false, true, true, false>}},
        {{sigma_fast_kernel<true, false, false, false>, sigma_fast_kernel<true, false, true, false>},
         {sigma_fast_kernel<true, true, false, false>, sigma_fast_kernel<true, true, true, false>}}};
    static const Kern lines[2][2] = {
        {sigma_fast_kernel<false, false, false, true>, sigma_fast_kernel<false, true, false, true>},
        {sigma_fast_kernel<true, false, false, true>, sigma_fast_kernel<true, true, false, true>}};
    const int tp0 = c->pb.tp == 0.0;
    const Kern kern = d_K ? lines[tp0][unib] : plain[tp0][unib][rt];
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_fail(c, e, "sigma_fast smem attribute");
    const int nqb = div_up(c->pb.M, 256 * SF_QPT);
    // equal shares of at most SF_QB blocks (4 + 2 of 6 blocks left the GPU to the
    // larger half)
    A.qb = c->tune.sigma_qblocks > 0 ? c->tune.sigma_qblocks : div_up(nqb, div_up(nqb, SF_QB));
    prof_begin(c);
    kern<<<dim3(div_up(nqb, A.qb), c->pb.N, nj), 256, smem, c->stream>>>(A);
    if (tg.sym.mode == 2) {
        sigma_fix_kernel<<<152, 128, 0, c->stream>>>(A, nullptr);
        // every patch, should the record have run over
        SigmaFastArgs F = A;
        F.only_full = true;
        F.jlist = nullptr;
        F.sym = SymMode();
        F.sig = c->d_sig + 3 * c->pb.N;
        kern<<<dim3(div_up(nqb, A.qb), c->pb.N, c->pb.N), 256, smem, c->stream>>>(F);
    }
    prof_end(c, K_SIGMA_Z);
    e = cudaGetLastError();
    return e == cudaSuccess ? QPFRG_OK : cuda_fail(c, e, "sigma_fast_kernel");
}

// Words per moment of the frequency-grid histogram: 227 KB of shared memory hold,
// beside the projection table, 6 x 5952 (a second word of moment 0) or 5 x 7136.
// More bins than that: two halves of 6 words each, which walk the pairs twice.
constexpr int kHfBins = 5952, kHfBinsOne = 7136;
static_assert(hf_smem_layout(kHfBins, true).total + 64 <= 227 * 1024 &&
                  hf_smem_layout(kHfBinsOne, false).total + 64 <= 227 * 1024, "shared memory of the histogram");

static int hist_variant(int nbins)
{
    return nbins <= kHfBins ? 0 : (nbins <= kHfBinsOne ? 1 : (nbins <= 2 * kHfBins ? 2 : -1));
}

// Binned pole density of the target slots into hist (FP32, wedge grid).
static qpfrg_status launch_sigma_hist(qpfrg_ctx *c, double T, const double *d_V, const double *d_Z, const double *d_K,
                                      const SigmaTargets &tg, double *hist, double e_min, double h, int nbins)
{
    const int nj = tg.slots(c->pb.N), N = c->pb.N, v = hist_variant(nbins);
    qpfrg_status s = launch_kp_table(c, tg.sym.mode == 2 ? nullptr : tg.jlist, nj);
    if (s != QPFRG_OK) return s;
    SigmaFastArgs A = fast_args(c, T, d_V, d_Z, d_K, tg);
    A.qcap = std::min(A.qcap, HF_QCAP);
    A.hist = hist;
    const double c0 = -e_min / h - 0.5;      // bin centre b at e_min + (b + 1/2) h
    A.c_int = (int)std::rint(c0);
    A.c_frac = (float)(c0 - A.c_int);
    A.inv_h = (float)(1.0 / h);
    A.inv_h_lo = (float)(1.0 / h - (double)A.inv_h);
    A.h = (float)h;
    A.nbins = nbins;
    A.e_min = e_min;
    A.h64 = h;
    using Kern = void (*)(SigmaFastArgs);
    static const Kern table[3][2] = {
        {sigma_hist_kernel<kHfBins, true, false, false>, sigma_hist_kernel<kHfBins, true, true, false>},
        {sigma_hist_kernel<kHfBinsOne, false, false, false>, sigma_hist_kernel<kHfBinsOne, false, true, false>},
        {sigma_hist_kernel<kHfBins, true, false, true>, sigma_hist_kernel<kHfBins, true, true, true>}};
    const Kern kern = table[v][d_K ? 1 : 0];
    const size_t smem = v == 1 ? hf_smem_layout(kHfBinsOne, false).total : hf_smem_layout(kHfBins, true).total;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_fail(c, e, "sigma_hist smem attribute");
    // one CTA per SM: split the q blocks until there are eight waves of the
    // listed targets (a flush follows every block either way)
    const int nqb = div_up(c->pb.M, HF_THR * HF_QPT);
    const long per = (long)N * (tg.jlist ? tg.n : nj);
    const int split = (int)std::max<long>(1, std::min<long>(nqb, (8 * 152 + per - 1) / per));
    prof_begin(c);
    const int halves = v == 2 ? 2 : 1;
    kern<<<dim3(split * halves, N, nj), HF_THR, smem, c->stream>>>(A);
    if (tg.sym.mode == 2) {
        sigma_fix_kernel<<<152, 128, 0, c->stream>>>(A, hist);
        // the images' own sums, should the record have run over
        SigmaFastArgs F = A;
        F.only_full = true;
        F.jlist = tg.jlist + tg.n;
        F.hist = hist + (long)tg.n * 5 * nbins;
        F.sym = SymMode();
        if (N > tg.n) kern<<<dim3(halves, N, N - tg.n), HF_THR, smem, c->stream>>>(F);
    }
    prof_end(c, K_SIGMA_HIST);
    e = cudaGetLastError();
    return e == cudaSuccess ? QPFRG_OK : cuda_fail(c, e, "sigma_hist_kernel");
}

// FP64 chord slopes of the target slots into d_sig or, with nbins, the binned
// pole weights of every patch into hist.
static qpfrg_status launch_sigma64(qpfrg_ctx *c, double T, const double *d_V, const double *d_Z, const double *d_K,
                                   const SigmaTargets &tg, double *hist = nullptr, double e_min = 0.0, double h = 1.0,
                                   int nbins = 0)
{
    const int N = c->pb.N, nj = tg.slots(N);
    qpfrg_status s = launch_kp_table(c, nullptr, N);
    if (s != QPFRG_OK) return s;
    Sigma64Args S{};
    S.a = fast_args(c, T, d_V, d_Z, d_K, tg);
    S.f = c->f64;
    S.hist = hist;
    S.e_min = e_min;
    S.inv_h = 1.0 / h;
    S.nbins = nbins;
    using Kern = void (*)(const Sigma64Args);
    static const Kern table[2][2][2] = {   // [t' = 0][lines][histogram]
        {{sigma64_kernel<false, false, false>, sigma64_kernel<false, false, true>},
         {sigma64_kernel<false, true, false>, sigma64_kernel<false, true, true>}},
        {{sigma64_kernel<true, false, false>, sigma64_kernel<true, false, true>},
         {sigma64_kernel<true, true, false>, sigma64_kernel<true, true, true>}}};
    const Kern kern = table[c->pb.tp == 0.0][d_K ? 1 : 0][nbins > 0 ? 1 : 0];
    const size_t smem = S64_REC * sizeof(S64Rec) + SF_SLOTS * (sizeof(double2) + (d_K ? sizeof(double) : 0) + sizeof(float2));
    const dim3 grid(div_up(c->pb.M, 256), N, nj);
    prof_begin(c);
    kern<<<grid, 256, smem, c->stream>>>(S);
    if (tg.sym.mode == 2 && nbins == 0) {
        sigma_fix_kernel<<<152, 128, 0, c->stream>>>(S.a, nullptr);
        Sigma64Args F = S;       // every patch, should the record have run over
        F.a.only_full = true;
        F.a.jlist = nullptr;
        F.a.sym = SymMode();
        F.a.sig = c->d_sig + 3 * N;
        kern<<<dim3(grid.x, N, N), 256, smem, c->stream>>>(F);
    }
    prof_end(c, nbins > 0 ? K_SIGMA_HIST : K_SIGMA_Z);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? QPFRG_OK : cuda_fail(c, e, "sigma64_kernel");
}

template <typename R>
static void fill_args(qpfrg_ctx *c, SigmaArgs<R> &A, const FineTable<R> &fine, double T, const double *d_V,
                      const double *d_Z)
{
    A.pb = c->pb;
    A.fine = fine;
    A.kf = c->d_kf;
    A.V = d_V;
    A.Z = d_Z;
    A.K = nullptr;
    A.sig = c->d_sig;
    A.T = T;
    A.nj = c->pb.N;
    A.jlist = nullptr;
    A.kx64 = c->f64.kx;
    A.ky64 = c->f64.ky;
    A.xij = c->d_xij;
    A.t_r = (R)c->pb.t;
    A.tp_r = (R)c->pb.tp;
    A.mu_r = (R)c->pb.mu;
    A.eta_r = (R)c->pb.eta;
    A.invT_r = (R)(1.0 / T);
    A.twoT_r = (R)(2.0 * T);
    A.xij_r = sizeof(R) == 4 ? reinterpret_cast<const R *>(c->d_xij_f) : reinterpret_cast<const R *>(c->d_xij);
    A.bnd = c->d_bnd;
    A.kp = c->d_kp;
    A.kcs = c->d_kcs;
    A.qxl = c->d_qxl;
    A.qyl = c->d_qyl;
    A.hist = c->d_hist;
    A.e_min = 0.0;
    A.inv_h = 1.0;
    A.nbins = 0;
}

// Z or slopes of every patch from the target slots' sums in d_sig
static qpfrg_status launch_z_update(qpfrg_ctx *c, const SigmaTargets &tg, double *Z, double *slopes)
{
    const int N = c->pb.N;
    prof_begin(c);
    z_update_kernel<<<div_up(N, 128), 128, 0, c->stream>>>(c->d_sig, c->d_sig + 2 * N, c->d_sig + 3 * N,
                                                              reinterpret_cast<unsigned *>(c->d_sig + 4 * N),
                                                              c->max_events, tg.rep, tg.own, tg.sym, Z, slopes, N);
    prof_end(c, K_Z_UPDATE);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? QPFRG_OK : cuda_fail(c, e, "z_update_kernel");
}

// Tolerance, relative to the largest magnitudes, of the C4v test that admits the
// reduced targets of the temperature flow's frequency grid, whose own accuracy is
// 3e-5 (Z, the slopes and the interaction flow's grid, which is integrated: rows_tol,
// so that no difference of an input above rounding is dropped).
constexpr double kTolGrid = 1e-5;

// state_symmetric: (V, Z) is the flow's state, symmetric by construction
// (irreducible targets, halved on the mirror lines).
qpfrg_status launch_sigma_z(qpfrg_ctx *c, double T, const double *d_V, const double *d_Z, double *d_Zout,
                            bool state_symmetric)
{
    const int N = c->pb.N;
    cudaError_t e = cudaMemsetAsync(c->d_sig, 0, (4 * (size_t)N + 1) * sizeof(double), c->stream);
    if (e != cudaSuccess) return cuda_fail(c, e, "memset sigma");
    qpfrg_status s;
    SigmaTargets tg;
    tg.n = N;
    // The zone edge breaks the C4v covariance of the angular projection at
    // the rounding level (mirror pairs land on |k_x| = pi exactly), which
    // moves Z on symmetric patches by ~1e-6: the state's reduction in mixed
    // precision only.
    if (state_symmetric && c->d_jirr != nullptr && c->opt.precision != QPFRG_FP64) {
        tg.jlist = c->d_jirr;
        tg.n = c->n_irr;
        tg.rep = c->d_rep;
        tg.mirror = c->pb.n_theta % 2 == 0 ? 1 : 0;
    }
    if (c->d_ptab) {
        const bool fp64 = c->opt.precision == QPFRG_FP64;
        if (!tg.jlist) {
            tg = device_targets(c, rows_tol(c), c->d_sym_v);
            if (tg.sym.mode == 2 && (s = launch_sym_test(c, d_V, d_Z, 1, c->d_sym_v)) != QPFRG_OK) return s;
        }
        s = fp64 ? launch_sigma64(c, T, d_V, d_Z, nullptr, tg) : launch_sigma_fast(c, T, d_V, d_Z, nullptr, tg);
    } else if (c->opt.precision == QPFRG_FP64) {
        SigmaArgs<double> A;
        fill_args(c, A, c->f64, T, d_V, d_Z);
        s = launch_sigma(c, false, A, K_SIGMA_Z);
    } else {
        SigmaArgs<float> A;
        fill_args(c, A, c->f32, T, d_V, d_Z);
        A.nj = tg.n;
        A.jlist = tg.jlist;
        s = launch_sigma(c, false, A, K_SIGMA_Z);
    }
    if (s != QPFRG_OK) return s;
    return launch_z_update(c, tg, d_Zout, nullptr);
}

// Chord slopes of the two-loop term with the interaction flow's line weights
// (Katanin factors d_K, ones without the correction) for every patch, into
// d_slopes.  FP32 wedge grid: the targets that the C4v test of (V, Z, K) in
// c->d_sym admits; otherwise the generic kernel for every patch.
qpfrg_status launch_sigma_lines(qpfrg_ctx *c, double T, const double *d_V, const double *d_Z, const double *d_K,
                                double *d_slopes)
{
    cudaError_t e = cudaMemsetAsync(c->d_sig, 0, (4 * (size_t)c->pb.N + 1) * sizeof(double), c->stream);
    if (e != cudaSuccess) return cuda_fail(c, e, "memset sigma");
    SigmaTargets tg;
    tg.n = c->pb.N;
    qpfrg_status s;
    if (c->d_ptab) {
        const bool fp64 = c->opt.precision == QPFRG_FP64;
        tg = device_targets(c, rows_tol(c), c->d_sym);
        s = fp64 ? launch_sigma64(c, T, d_V, d_Z, d_K, tg) : launch_sigma_fast(c, T, d_V, d_Z, d_K, tg);
    } else if (c->opt.precision == QPFRG_FP64) {
        SigmaArgs<double> A;
        fill_args(c, A, c->f64, T, d_V, d_Z);
        A.K = d_K;
        s = launch_sigma(c, false, A, K_SIGMA_Z);
    } else {
        SigmaArgs<float> A;
        fill_args(c, A, c->f32, T, d_V, d_Z);
        A.K = d_K;
        s = launch_sigma(c, false, A, K_SIGMA_Z);
    }
    if (s != QPFRG_OK) return s;
    return launch_z_update(c, tg, nullptr, d_slopes);
}

// d_K (interaction flow): the C4v test of (V, Z, K) is already in c->d_sym
qpfrg_status launch_sigma_grid(qpfrg_ctx *c, double T, const double *d_V, const double *d_Z, double *d_re,
                               double *d_im, const double *d_K)
{
    const int N = c->pb.N, n_omega = c->opt.n_omega;
    // pole energies E = x_q + x_r - x_p lie in [2 min x - max x, 2 max x - min x];
    // r = k + p - q is not a fine point: bound its dispersion by the band
    double xmin = c->fx_min, xmax = c->fx_max;
    const double band_lo = -4.0 * std::fabs(c->pb.t) - 4.0 * std::fabs(c->pb.tp) - c->pb.mu;
    const double band_hi = 4.0 * std::fabs(c->pb.t) + 4.0 * std::fabs(c->pb.tp) - c->pb.mu;
    xmin = std::fmin(xmin, band_lo);
    xmax = std::fmax(xmax, band_hi);
    if (c->pb.propagator == QPFRG_PROP_QP) {   // Z in (0, z_max] rescales the poles
        xmin *= c->opt.z_max;
        xmax *= c->opt.z_max;
    }
    // Bins of width h <= eta / 4: the offset of a pole from its bin centre is at
    // most |z - E_b| / 8, so the moment expansion truncated after moment 4 is
    // accurate to 8^-5 = 3e-5 relative per pole.
    const double e_min = 2.0 * xmin - xmax - 1e-9, e_max = 2.0 * xmax - xmin + 1e-9;
    const int nbins = (int)std::fmin(std::fmax(std::ceil((e_max - e_min) / (0.25 * c->opt.eta)), 64.0), 65536.0);
    const double h = (e_max - e_min) / nbins;
    // histogram, then the sums per target slot
    const size_t hist_n = (size_t)N * 5 * nbins, need = hist_n + 2 * (size_t)N * n_omega;
    if (need > c->hist_elems) {
        if (c->d_hist) cudaFree(c->d_hist);
        c->d_hist = nullptr;
        cudaError_t e = cudaMalloc((void **)&c->d_hist, need * sizeof(double));
        if (e != cudaSuccess) {
            c->hist_elems = 0;
            return cuda_fail(c, e, "cudaMalloc(sigma histogram)");
        }
        c->hist_elems = need;
    }
    cudaError_t e = cudaMemsetAsync(c->d_hist, 0, need * sizeof(double), c->stream);
    if (e != cudaSuccess) return cuda_fail(c, e, "memset histogram");
    double *acc = c->d_hist + hist_n;
    unsigned *nevents = reinterpret_cast<unsigned *>(c->d_sig + 4 * N);
    if ((e = cudaMemsetAsync(nevents, 0, 2 * sizeof(unsigned), c->stream)) != cudaSuccess)
        return cuda_fail(c, e, "memset boundary pairs");
    qpfrg_status s;
    SigmaTargets tg;
    tg.n = N;
    if (c->opt.precision != QPFRG_FP64 && c->d_ptab && hist_variant(nbins) >= 0) {
        // FP32 wedge grid: table projection, histogram in shared memory; a
        // C4v-symmetric (V, Z) needs only the irreducible and zone-edge targets
        tg = device_targets(c, d_K ? rows_tol(c) : kTolGrid, d_K ? c->d_sym : c->d_sym_v);
        if (tg.sym.mode == 2 && !d_K && (s = launch_sym_test(c, d_V, d_Z, 1, c->d_sym_v)) != QPFRG_OK) return s;
        s = launch_sigma_hist(c, T, d_V, d_Z, d_K, tg, c->d_hist, e_min, h, nbins);
    } else if (c->opt.precision == QPFRG_FP64 && c->d_ptab) {
        s = launch_sigma64(c, T, d_V, d_Z, d_K, tg, c->d_hist, e_min, h, nbins);
    } else if (c->opt.precision == QPFRG_FP64) {
        SigmaArgs<double> A;
        fill_args(c, A, c->f64, T, d_V, d_Z);
        A.K = d_K;
        A.e_min = e_min;
        A.inv_h = 1.0 / h;
        A.nbins = nbins;
        s = launch_sigma(c, true, A, K_SIGMA_HIST);
    } else {
        SigmaArgs<float> A;
        fill_args(c, A, c->f32, T, d_V, d_Z);
        A.K = d_K;
        A.e_min = e_min;
        A.inv_h = 1.0 / h;
        A.nbins = nbins;
        s = launch_sigma(c, true, A, K_SIGMA_HIST);
    }
    if (s != QPFRG_OK) return s;
    const double w0 = c->opt.omega_min;
    const double dw = n_omega > 1 ? (c->opt.omega_max - c->opt.omega_min) / (n_omega - 1) : 0.0;
    const int nslot = tg.slots(N);
    prof_begin(c);
    sigma_resum_kernel<<<dim3(div_up(n_omega, 128), div_up(nbins, RG_BINS), div_up(nslot, RG_T)), 128, 0, c->stream>>>(
        c->d_hist, nbins, e_min, h, n_omega, w0, dw, c->pb.eta, acc, nslot, tg.n, tg.sym, nevents, c->max_events);
    sigma_spread_kernel<<<dim3(div_up(n_omega, 128), N), 128, 0, c->stream>>>(acc, tg.rep, tg.own, tg.sym, nevents,
                                                                             c->max_events, n_omega, d_re, d_im);
    prof_end(c, K_SIGMA_GRID);
    e = cudaGetLastError();
    return e == cudaSuccess ? QPFRG_OK : cuda_fail(c, e, "sigma_resum_kernel");
}

}  // namespace qpfrg

namespace qpfrg {

// Spectral function of patch j on the frequency grid, A = -(1/pi) Im G with
// G = 1/(w - xi_j - Sigma), and its Fermi-liquid (Gaussian) approximation: a
// Gaussian of weight Z_j centred on xi_j, equal to A there (linear
// interpolation on the grid): A_FL = A0 exp(-pi A0^2 (w - xi_j)^2 / Z_j^2).
// One CTA per patch; A at the grid points, then A0 and A_FL.
__global__ void spectral_kernel(const double *re, const double *im, const double *Z, const double *xij, int n_omega,
                                double w0, double dw, double *A, double *Afl)
{
    const int j = blockIdx.x;
    const double x0 = xij[j];
    const double *sr = re + (long)j * n_omega, *si = im + (long)j * n_omega;
    double *a = A + (long)j * n_omega;
    for (int m = threadIdx.x; m < n_omega; m += blockDim.x) {
        const double x = w0 + dw * m - x0 - sr[m], y = si[m];
        const double d = x * x + y * y;
        a[m] = d > 0.0 ? -y / (kPi * d) : 0.0;    // Sigma = 0 exactly at w = xi: no grid value
    }
    __syncthreads();
    __shared__ double A0;
    if (threadIdx.x == 0) {
        double v = 0.0;
        if (n_omega > 1 && dw > 0.0) {
            const double t = (x0 - w0) / dw;
            long m0 = (long)floor(t);
            if (m0 == n_omega - 1 && t == (double)m0) m0 -= 1;   // xi on the last grid point
            if (m0 >= 0 && m0 + 1 < n_omega) {
                const double u = t - (double)m0;
                v = (1.0 - u) * a[m0] + u * a[m0 + 1];
            }
        }
        A0 = v;
    }
    __syncthreads();
    if (!Afl) return;
    const double zj = Z ? Z[j] : 1.0;
    const double k = kPi * A0 * A0 / (zj * zj);
    for (int m = threadIdx.x; m < n_omega; m += blockDim.x) {
        const double d = w0 + dw * m - x0;
        Afl[(long)j * n_omega + m] = A0 * exp(-k * d * d);
    }
}

}  // namespace qpfrg

extern "C" qpfrg_status qpfrg_spectral(qpfrg_t c, const double *d_sigma_re, const double *d_sigma_im, const double *d_Z,
                                       double *d_A, double *d_A_fl)
{
    using namespace qpfrg;
    if (!c) return QPFRG_ERR_INVALID;
    if (c->opt.n_omega < 1 || !d_sigma_re || !d_sigma_im || !d_A) {
        c->err = "qpfrg_spectral needs the frequency grid (n_omega > 0), Sigma and an output";
        return QPFRG_ERR_INVALID;
    }
    const int n = c->opt.n_omega;
    const double w0 = c->opt.omega_min, dw = n > 1 ? (c->opt.omega_max - c->opt.omega_min) / (n - 1) : 0.0;
    spectral_kernel<<<c->pb.N, 256, 0, c->stream>>>(d_sigma_re, d_sigma_im, d_Z, c->d_xij, n, w0, dw, d_A, d_A_fl);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? QPFRG_OK : cuda_fail(c, e, "spectral_kernel");
}
