// View-space forms shared by the forward and adjoint tile kernels: a Gaussian
// in the frame of a detector view, the footprint coefficients, the rays of the
// general path and the parameter chains from view-space moments (the closed
// form they rewrite is derived at the head of project.cu).
#pragma once
#include "pair.cuh"

namespace rgrt {
namespace {

constexpr float M_PER_ARG = -1.38629436111989061f;        // m = arg * (-2 ln 2)
constexpr float CUT_ARG = -6.49212768400033233f;          // arg at m = 9
constexpr int NG = 10;            // general path: dmu[3], G_P[6], drho

// a Gaussian in the view of the current tile (shared memory)
// The Q coefficients carry the factor -log2(e)/2 (and, for parallel rays, 1/A)
// so that arg = Q/A * (-log2(e)/2) feeds ex2 directly; m = -2 ln2 arg.
struct VRec {
    float4 c0;  // u0, v0, k M_uu, 2 k M_uv               (k = -log2(e)/2, x 1/A for parallel rays)
    float4 c1;  // k M_vv, A0 (cone) | 1/A (parallel), 2 a_u (cone) | 1/sqrt(A) (parallel), 2 a_v
    float4 c2;  // P'_uu, 2 P'_uv, P'_vv, alpha = rho sqrt(2 pi) (cone) | alpha/sqrt(A) (parallel)
    float4 bb;  // u_lo, u_hi, v_lo, v_hi of the detector box (skip test)
    float4 g0;  // mu, rho                      (general path)
    float4 g1;  // P00 P01 P02 P11              (general path)
    float4 g2;  // P12 P22, gid bits, 1 = view-space path / 0 = general path
    float4 t4;  // parallel rays: the closest approach along the ray, t* = x + y du + z dv, and 1/A (w)
};

__device__ __forceinline__ bool cone_interval(float K2, float dsd, float ae, float aw, float see,
                                              float sew, float sww, float &lo, float &hi)
{
    float alpha = aw * aw - K2 * sww;
    if (!(alpha > 0.0f)) return false;
    float beta = dsd * (ae * aw - K2 * sew);
    float disc = aw * aw * see - 2.0f * ae * aw * sew + ae * ae * sww - K2 * (see * sww - sew * sew);
    disc = fmaxf(disc, 0.0f);
    float r = dsd * sqrtf(K2 * disc);
    lo = (beta - r) / alpha;
    hi = (beta + r) / alpha;
    return true;
}

// Every detector geometry's view frame is a rotation about z (geom_tables):
// e_v = (0, 0, 1), e_u = (a, b, 0), e_w = (p, q, 0).  The transforms below
// use that shape: a symmetric X in the frame costs 18 operations instead of
// six general quadratic forms, and a frame matrix back to world as many.
struct AxFrame {
    float a, b, p, q;
};
__device__ __forceinline__ AxFrame ax_frame(const float *F)
{
    AxFrame f;
    f.a = F[0]; f.b = F[1]; f.p = F[6]; f.q = F[7];
    return f;
}

// X (symmetric, packed 00 01 02 11 12 22) in the frame: (uu, uv, uw, vv, vw, ww)
__device__ __forceinline__ void to_frame_ax(const float *X, const AxFrame &f, float *o)
{
    const float xa = X[0] * f.a + X[1] * f.b, xb = X[1] * f.a + X[3] * f.b;   // X e_u (x, y)
    const float xp = X[0] * f.p + X[1] * f.q, xq = X[1] * f.p + X[3] * f.q;   // X e_w (x, y)
    o[0] = f.a * xa + f.b * xb;
    o[1] = X[2] * f.a + X[4] * f.b;
    o[2] = f.a * xp + f.b * xq;
    o[3] = X[5];
    o[4] = X[2] * f.p + X[4] * f.q;
    o[5] = f.p * xp + f.q * xq;
}

// symmetric G' (packed uu uv uw vv vw ww) back to world, G = E G' E^T with
// E = [e_u e_v e_w]: world x = a u + p w, y = b u + q w, z = v
__device__ __forceinline__ void from_frame_ax(const float *Gf, const AxFrame &f, float *G)
{
    const float hu0 = Gf[0] * f.a + Gf[2] * f.p, hw0 = Gf[2] * f.a + Gf[5] * f.p;
    const float hu1 = Gf[0] * f.b + Gf[2] * f.q, hw1 = Gf[2] * f.b + Gf[5] * f.q;
    G[0] = f.a * hu0 + f.p * hw0;
    G[1] = f.a * hu1 + f.p * hw1;
    G[2] = f.a * Gf[1] + f.p * Gf[4];
    G[3] = f.b * hu1 + f.q * hw1;
    G[4] = f.b * Gf[1] + f.q * Gf[4];
    G[5] = Gf[3];
}

// The footprint of a cone-beam record on the detector: rays at offset
// (du, dv) from (u0, v0) with m <= K^2 satisfy Q - K^2 A <= 0, Q and A
// quadratics in (du, dv):
//   G(du, dv) = a du^2 + 2 b du dv + c dv^2 + 2 d du + 2 e dv + f <= 0.
// When the quadratic part is positive definite (an ellipse: the K-sigma
// ellipsoid lies in front of the source) G is convex, and G(x) >= G(x0) +
// grad G(x0).(x - x0) bounds it from below over a rectangle around x0.
struct Conic {
    float a, b, c, d, e, f;
    bool ok;
};

// the footprint conic of a cone-beam view-space record (offsets from u0, v0)
template <int KER>
__device__ __forceinline__ Conic cone_conic(const VRec &r)
{
    const float4 c0 = r.c0, c1 = r.c1, c2 = r.c2;
    const float K2 = Kern<KER>::SKIP, ik = 1.0f / Kern<KER>::QSCALE;
    Conic cn;
    cn.a = c0.z * ik - K2 * c2.x;
    cn.b = 0.5f * (c0.w * ik - K2 * c2.y);
    cn.c = c1.x * ik - K2 * c2.z;
    cn.d = -0.5f * K2 * c1.z;
    cn.e = -0.5f * K2 * c1.w;
    cn.f = -K2 * c1.y;
    cn.ok = cn.a > 0.0f && cn.a * cn.c - cn.b * cn.b > 1e-3f * cn.a * cn.c;
    return cn;
}

// gather one record and turn it into its view-space form for frame F
// (3-D PET: kap0, kap1 are the extreme LOR slopes of the tile's columns)
template <int GM, int KER>
__device__ __forceinline__ void prep_record(const DevGeom &g, const float *F, uint32_t gid,
                                            const float4 *__restrict__ rec,
                                            const float4 *__restrict__ crec, VRec &out,
                                            float kap0 = 0.0f, float kap1 = 0.0f)
{
    constexpr bool CONE = GM == GM_CONE;
    const float4 *r = rec + REC_F4 * (size_t)gid;
    float4 r0 = __ldg(r), r1 = __ldg(r + 1), r2 = __ldg(r + 2), r3 = __ldg(r + 3), r4 = __ldg(r + 4);
    out.t4 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    float4 k1 = __ldg(crec + CREC_F4 * (size_t)gid + 1), k2 = __ldg(crec + CREC_F4 * (size_t)gid + 2);
    const float Sg[6] = { k1.x, k1.y, k1.z, k1.w, k2.x, k2.y };
    const float P[6] = { r1.x, r1.y, r1.z, r1.w, r2.x, r2.y };
    const float Sh[6] = { r2.z, r2.w, r3.x, r3.y, r3.z, r3.w };
    const float m[3] = { r0.x, r0.y, r0.z };
    const float rho = r0.w, smax = r4.x;
    const AxFrame fr = ax_frame(F);
    const float mu_u = m[0] * fr.a + m[1] * fr.b;
    const float mu_v = m[2];
    const float mu_w = m[0] * fr.p + m[1] * fr.q;
    float Pf[6], Sf[6], Gf[6];   // P, Sigma / det Sigma and Sigma in the frame
    to_frame_ax(P, fr, Pf);
    to_frame_ax(Sh, fr, Sf);
    to_frame_ax(Sg, fr, Gf);
    float ulo = -INFINITY, uhi = INFINITY, vlo = -INFINITY, vhi = INFINITY;
    bool sat;
    if (CONE) {
        const float D = mu_w + g.dso;           // depth of mu from the source
        float suu = Gf[0], svv = Gf[3], sww = Gf[5];
        float suw = Gf[2], svw = Gf[4];
        float lo, hi;
        if (cone_interval(Kern<KER>::SKIP, g.dsd, mu_u, D, suu, suw, sww, lo, hi)) { ulo = lo; uhi = hi; }
        if (cone_interval(Kern<KER>::SKIP, g.dsd, mu_v, D, svv, svw, sww, lo, hi)) { vlo = lo; vhi = hi; }
        const float iD = 1.0f / D;
        const float u0 = g.dsd * mu_u * iD, v0 = g.dsd * mu_v * iD;
        // A(du, dv) = d~^T P' d~, d~ = (u0 + du, v0 + dv, dsd)
        const float au = Pf[0] * u0 + Pf[1] * v0 + Pf[2] * g.dsd;
        const float av = Pf[1] * u0 + Pf[3] * v0 + Pf[4] * g.dsd;
        const float aw = Pf[2] * u0 + Pf[4] * v0 + Pf[5] * g.dsd;
        const float A0 = au * u0 + av * v0 + aw * g.dsd;
        // g_u = e_u x delta = (0, D, -mu_v), g_v = e_v x delta = (-D, 0, mu_u)
        const float guv = D, guw = -mu_v, gvu = -D, gvw = mu_u;
        const float cu1 = Sf[3] * guv + Sf[4] * guw, cu2 = Sf[4] * guv + Sf[5] * guw;  // (S' g_u)_{v,w}
        const float cv0 = Sf[0] * gvu + Sf[2] * gvw, cv1 = Sf[1] * gvu + Sf[4] * gvw,
                    cv2 = Sf[2] * gvu + Sf[5] * gvw;                                  // S' g_v
        const float Muu = guv * cu1 + guw * cu2;
        const float Muv = guv * cv1 + guw * cv2;
        const float Mvv = gvu * cv0 + gvw * cv2;
        const float k = Kern<KER>::QSCALE;
        out.c0 = make_float4(u0, v0, k * Muu, 2.0f * k * Muv);
        out.c1 = make_float4(k * Mvv, A0, 2.0f * au, 2.0f * av);
        out.c2 = make_float4(Pf[0], 2.0f * Pf[1], Pf[3], rho * Kern<KER>::FAC);

        // both segment ends (source, detector plane) beyond the 8.66-sigma ball
        sat = D >= Kern<KER>::BALL * smax && (g.dsd - D) >= Kern<KER>::BALL * smax;
    } else if (GM == GM_PET3D) {
        // LOR through (u, z) at w = 0 with direction d~ = e_w + kappa e_v:
        // with du = u - mu_u and v~ = z - mu_v + kappa mu_w (the LOR's height
        // at depth mu_w, relative to mu), c = d~ x delta = (-v~, du, -kappa du),
        //   Q = du^2 (S'_vv - 2 kappa S'_vw + kappa^2 S'_ww)
        //     + 2 du v~ (kappa S'_uw - S'_uv) + v~^2 S'_uu,
        //   A = d~^T P' d~ = P'_ww (1 + kappa (2 P'_vw + kappa P'_vv) / P'_ww),
        // and the integral along the unit ray is |d~| rho sqrt(2 pi / A)
        // exp(-Q / 2A); the coefficients carry the 1/P'_ww.
        float hu = sqrtf(Kern<KER>::SKIP * Gf[0]);
        ulo = mu_u - hu; uhi = mu_u + hu;
        // heights z whose LORs can meet the box ellipsoid (the bounds at the
        // two extreme slopes span those of every slope between them)
        const float svv = Gf[3], svw = Gf[4], sww = Gf[5];
        vlo = INFINITY; vhi = -INFINITY;
#pragma unroll
        for (int e = 0; e < 2; e++) {
            const float kap = e ? kap1 : kap0;
            const float zc = mu_v - kap * mu_w;
            const float half = sqrtf(fmaxf(Kern<KER>::SKIP * (svv - 2.0f * kap * svw + kap * kap * sww), 0.0f));
            vlo = fminf(vlo, zc - half);
            vhi = fmaxf(vhi, zc + half);
        }
        const float iP = 1.0f / Pf[5];
        const float k = Kern<KER>::QSCALE * iP;
        out.c0 = make_float4(mu_u, mu_v, mu_w, k * Sf[0]);
        out.c1 = make_float4(k * Sf[3], -2.0f * k * Sf[4], k * Sf[5], -2.0f * k * Sf[1]);
        out.c2 = make_float4(2.0f * k * Sf[2], 2.0f * Pf[4] * iP, Pf[3] * iP, rho * Kern<KER>::FAC * sqrtf(iP));
        // the LOR ends on the ring: beyond the ball if the ball is inside it
        const float rxy = sqrtf(m[0] * m[0] + m[1] * m[1]);
        sat = rxy + Kern<KER>::BALL * smax <= sqrtf(g.radius2);
    } else {
        float hu = sqrtf(Kern<KER>::SKIP * Gf[0]);
        float hv = sqrtf(Kern<KER>::SKIP * Gf[3]);
        ulo = mu_u - hu; uhi = mu_u + hu; vlo = mu_v - hv; vhi = mu_v + hv;
        const float iA = 1.0f / Pf[5];
        const float rA = sqrtf(iA);
        // c = du e_v - dv e_u: M_uu = S'_vv, M_uv = -S'_uv, M_vv = S'_uu
        const float k = Kern<KER>::QSCALE * iA;
        out.c0 = make_float4(mu_u, mu_v, k * Sf[3], -2.0f * k * Sf[1]);
        out.c1 = make_float4(k * Sf[0], iA, rA, 0.0f);
        out.c2 = make_float4(0.0f, 0.0f, 0.0f, rho * Kern<KER>::FAC * rA);
        // along the ray (direction e_w) the exponent is smallest at
        // t* = mu_w - (P'_uw du + P'_vw dv) / P'_ww
        out.t4 = make_float4(mu_w, -Pf[2] * iA, -Pf[4] * iA, iA);

        if (g.pet) {
            float rxy = sqrtf(m[0] * m[0] + m[1] * m[1]);
            sat = rxy + Kern<KER>::BALL * smax <= sqrtf(g.radius2);
        } else {
            sat = mu_w - Kern<KER>::BALL * smax >= g.t_a && mu_w + Kern<KER>::BALL * smax <= g.t_b;
        }
    }
    out.bb = make_float4(ulo, uhi, vlo, vhi);
    out.g0 = r0;
    out.g1 = r1;
    out.g2 = make_float4(r2.x, r2.y, __uint_as_float(gid), sat ? 1.0f : 0.0f);
}

// ray of detector pixel (u, v) in view frame F (FP32), for the general path
// (3-D PET: v is the LOR's mid-height, kap its slope dz/dw)
template <int GM>
__device__ __forceinline__ Ray make_ray(const DevGeom &g, const float *F, float u, float v, float kap = 0.0f)
{
    float op0, op1, op2, dp0, dp1, dp2, ta, tb;
    if (GM == GM_PET3D) {
        // o' = (u, v, 0), d' = (0, kappa, 1)/L, L = sqrt(1 + kappa^2); the LOR
        // runs over w in [-h, h], h = sqrt(R^2 - u^2), i.e. t = w L
        const float L = sqrtf(1.0f + kap * kap), iL = 1.0f / L;
        const float h = sqrtf(fmaxf(g.radius2 - u * u, 0.0f));
        op0 = u; op1 = v; op2 = 0.0f;
        dp0 = 0.0f; dp1 = kap * iL; dp2 = iL;
        ta = -h * L; tb = h * L;
    } else if (GM == GM_CONE) {
        // d' = (u, v, dsd)/L;  o' = closest point to the origin on the ray,
        // o' = dso/L^2 (dsd u, dsd v, -(u^2+v^2)) (no cancellation);
        // segment from the source (t_a) to the pixel (t_b), measured from o'
        float uv2 = u * u + v * v;
        float L2 = uv2 + g.dsd * g.dsd;
        float iL = rsqrtf(L2);
        float c = g.dso / L2;
        dp0 = u * iL; dp1 = v * iL; dp2 = g.dsd * iL;
        op0 = c * g.dsd * u; op1 = c * g.dsd * v; op2 = -c * uv2;
        ta = -g.dso * g.dsd * iL;
        tb = (uv2 + g.dsd * (g.dsd - g.dso)) * iL;
    } else {
        op0 = u; op1 = v; op2 = 0.0f;
        dp0 = 0.0f; dp1 = 0.0f; dp2 = 1.0f;
        if (g.pet) {
            float h = sqrtf(fmaxf(g.radius2 - u * u, 0.0f));
            ta = -h; tb = h;
        } else {
            ta = g.t_a; tb = g.t_b;
        }
    }
    Ray r;
    r.ox = op0 * F[0] + op1 * F[3] + op2 * F[6];
    r.oy = op0 * F[1] + op1 * F[4] + op2 * F[7];
    r.oz = op0 * F[2] + op1 * F[5] + op2 * F[8];
    r.dx = dp0 * F[0] + dp1 * F[3] + dp2 * F[6];
    r.dy = dp0 * F[1] + dp1 * F[4] + dp2 * F[7];
    r.dz = dp0 * F[2] + dp1 * F[5] + dp2 * F[8];
    r.ta = ta;
    r.tb = tb;
    return r;
}

// 3-D PET: LOR slope dz/dw at radial position u (dz: axial rise over the chord)
__device__ __forceinline__ float pet3d_slope(const DevGeom &g, float dz, float u)
{
    return 0.5f * dz / sqrtf(fmaxf(g.radius2 - u * u, 1e-30f));
}

// 3-D PET view: (offset of the row heights, axial rise, rows with a ring pair)
__device__ __forceinline__ void pet3d_view(const DevGeom &g, int view, float &zoff, float &dz, int &rows)
{
    const int delta = pet3d_delta(g, view), ad = abs(delta);
    zoff = 0.5f * (float)ad * g.ring_pitch;
    dz = (float)delta * g.ring_pitch;
    rows = g.n_rows - ad;
}

// 3-D PET: LOR slopes at the extreme |u| of columns c0..c1
__device__ __forceinline__ void pet3d_slopes(const DevGeom &g, float dz, int c0, int c1, float &k0, float &k1)
{
    const float ua = __ldg(g.utab + c0), ub = __ldg(g.utab + c1);
    const float amin = (ua <= 0.0f && ub >= 0.0f) ? 0.0f : fminf(fabsf(ua), fabsf(ub));
    const float amax = fmaxf(fabsf(ua), fabsf(ub));
    k0 = pet3d_slope(g, dz, amin);
    k1 = pet3d_slope(g, dz, amax);
}

__device__ __forceinline__ float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float rsqrt_approx(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ void cross_acc(const float *a, const float *b, float s, float *o)
{
    o[0] += s * (a[1] * b[2] - a[2] * b[1]);
    o[1] += s * (a[2] * b[0] - a[0] * b[2]);
    o[2] += s * (a[0] * b[1] - a[1] * b[0]);
}

// Gradient w.r.t. (mu, rho, G_P, G_S) of one Gaussian from its view-space
// moments s[] summed over the tile's rays:
//   cone:  s = [SQ_u, SQ_v, SQ_uu, SQ_uv, SQ_vv, SA, SA_u, SA_v, SA_uu, SA_uv, SA_vv, Sw]
//   par.:  s = [SQ_u, SQ_v, SQ_uu, SQ_uv, SQ_vv, SA, Sw]
// where SQ_x = sum (dL/dQ / alpha) x, SA_x = sum (dL/dA / alpha) x (x a
// monomial in du, dv), Sw = sum dL/dI |d~| A^-1/2 e^{-m/2} and
// alpha = rho sqrt(2 pi).  With c = du g_u + dv g_v and d~ = d~0 + (du, dv, 0):
//   dL/dS'  = sum dL/dQ c c^T
//   dL/dP'  = sum dL/dA d~ d~^T
//   dL/dmu' = -2 sum dL/dQ (S' c) x d~      (Q = c^T S' c, c = d~ x (S - mu'))
//   dL/drho = sqrt(2 pi) Sw
// out16 = (dmu[3], drho, G_P[6], G_S[6]) in world coordinates.
// tof4 (nullable; parallel rays with time of flight): the moments of the
// TOF weight's derivatives (rows_tof in adjoint.cu), added to dL/dmu' and dL/dP'.
template <int GM, int KER>
__device__ __forceinline__ void view_chain(const DevGeom &g, const float *F, const float4 *rec,
                                           uint32_t gid, const float *s, float *out16,
                                           const float *tof4 = nullptr)
{
    constexpr bool CONE = GM == GM_CONE;
    const float4 *r = rec + REC_F4 * (size_t)gid;
    const float4 r0 = __ldg(r), r2 = __ldg(r + 2), r3 = __ldg(r + 3);
    const float Sh[6] = { r2.z, r2.w, r3.x, r3.y, r3.z, r3.w };
    const float m[3] = { r0.x, r0.y, r0.z };
    const float alpha = r0.w * Kern<KER>::FAC;
    const AxFrame fr = ax_frame(F);
    float Sf[6];
    to_frame_ax(Sh, fr, Sf);
    const float mu_u = m[0] * fr.a + m[1] * fr.b;
    const float mu_v = m[2];
    const float mu_w = m[0] * fr.p + m[1] * fr.q;
    const float SQu = alpha * s[0], SQv = alpha * s[1], SQuu = alpha * s[2], SQuv = alpha * s[3],
                SQvv = alpha * s[4];
    float gu[3], gv[3], d0[3], GPf[6], GSf[6];
    float Sw;
    if (CONE) {
        const float D = mu_w + g.dso;
        const float u0 = g.dsd * mu_u / D, v0 = g.dsd * mu_v / D;
        gu[0] = 0.0f; gu[1] = D; gu[2] = -mu_v;
        gv[0] = -D; gv[1] = 0.0f; gv[2] = mu_u;
        d0[0] = u0; d0[1] = v0; d0[2] = g.dsd;
        const float SA = alpha * s[5], SAu = alpha * s[6], SAv = alpha * s[7], SAuu = alpha * s[8],
                    SAuv = alpha * s[9], SAvv = alpha * s[10];
        Sw = s[11];
        // dL/dP' = SA d0 d0^T + (d0 m^T + m d0^T) + N,  m = (SAu, SAv, 0)
        GPf[0] = SA * d0[0] * d0[0] + 2.0f * d0[0] * SAu + SAuu;
        GPf[1] = SA * d0[0] * d0[1] + d0[0] * SAv + SAu * d0[1] + SAuv;
        GPf[2] = SA * d0[0] * d0[2] + SAu * d0[2];
        GPf[3] = SA * d0[1] * d0[1] + 2.0f * d0[1] * SAv + SAvv;
        GPf[4] = SA * d0[1] * d0[2] + SAv * d0[2];
        GPf[5] = SA * d0[2] * d0[2];
    } else {
        // c = du e_v - dv e_u: "g_u" = e_v, "g_v" = -e_u (frame coordinates), d~ = e_w
        gu[0] = 0.0f; gu[1] = 1.0f; gu[2] = 0.0f;
        gv[0] = -1.0f; gv[1] = 0.0f; gv[2] = 0.0f;
        d0[0] = 0.0f; d0[1] = 0.0f; d0[2] = 1.0f;
        Sw = s[6];
        GPf[0] = GPf[1] = GPf[2] = GPf[3] = GPf[4] = 0.0f;
        GPf[5] = alpha * s[5];
    }
    float cu[3], cv[3];   // S' g_u, S' g_v
    cu[0] = Sf[0] * gu[0] + Sf[1] * gu[1] + Sf[2] * gu[2];
    cu[1] = Sf[1] * gu[0] + Sf[3] * gu[1] + Sf[4] * gu[2];
    cu[2] = Sf[2] * gu[0] + Sf[4] * gu[1] + Sf[5] * gu[2];
    cv[0] = Sf[0] * gv[0] + Sf[1] * gv[1] + Sf[2] * gv[2];
    cv[1] = Sf[1] * gv[0] + Sf[3] * gv[1] + Sf[4] * gv[2];
    cv[2] = Sf[2] * gv[0] + Sf[4] * gv[1] + Sf[5] * gv[2];
    {
        const int ia[6] = { 0, 0, 0, 1, 1, 2 }, ib[6] = { 0, 1, 2, 1, 2, 2 };
#pragma unroll
        for (int e = 0; e < 6; e++) {
            const int a = ia[e], b = ib[e];
            GSf[e] = SQuu * gu[a] * gu[b] + SQuv * (gu[a] * gv[b] + gv[a] * gu[b]) + SQvv * gv[a] * gv[b];
        }
    }
    // T = sum dL/dQ (S'c) x d~ = cu x d0 SQu + cv x d0 SQv
    //     + cu x e_u SQuu + (cu x e_v + cv x e_u) SQuv + cv x e_v SQvv
    // (the last three only for the cone: parallel rays keep d~ = e_w)
    float T[3] = { 0.0f, 0.0f, 0.0f };
    cross_acc(cu, d0, SQu, T);
    cross_acc(cv, d0, SQv, T);
    if (CONE) {
        const float eU[3] = { 1.0f, 0.0f, 0.0f }, eV[3] = { 0.0f, 1.0f, 0.0f };
        cross_acc(cu, eU, SQuu, T);
        cross_acc(cu, eV, SQuv, T);
        cross_acc(cv, eU, SQuv, T);
        cross_acc(cv, eV, SQvv, T);
    }
    float dmuf[3] = { -2.0f * T[0], -2.0f * T[1], -2.0f * T[2] };
    if (!CONE && tof4) {
        // the TOF weight W(t*, s^2): t* = mu_w + k_u du + k_v dv with
        // k_u = -P'_uw / P'_ww, k_v = -P'_vw / P'_ww, s^2 = 1/P'_ww + sigma_T^2.
        // tof4 = alpha-free sums of val dW/dt* (1, du, dv) and val dW/ds^2.
        const float4 r1 = __ldg(rec + REC_F4 * (size_t)gid + 1), r2 = __ldg(rec + REC_F4 * (size_t)gid + 2);
        const float P[6] = { r1.x, r1.y, r1.z, r1.w, r2.x, r2.y };
        float Pf[6];
        to_frame_ax(P, fr, Pf);
        const float ipw = 1.0f / Pf[5];
        const float ku = -Pf[2] * ipw, kv = -Pf[4] * ipw;
        const float T0 = alpha * tof4[0], Tu = alpha * tof4[1], Tv = alpha * tof4[2], S0 = alpha * tof4[3];
        dmuf[0] -= ku * T0;        // du = u - mu_u: dt*/dmu_u = -k_u
        dmuf[1] -= kv * T0;
        dmuf[2] += T0;
        // symmetric-entry gradients (the full matrix holds P'_uw twice)
        GPf[2] -= 0.5f * Tu * ipw;
        GPf[4] -= 0.5f * Tv * ipw;
        GPf[5] -= (ku * Tu + kv * Tv) * ipw + S0 * ipw * ipw;
    }
    out16[0] = dmuf[0] * fr.a + dmuf[2] * fr.p;
    out16[1] = dmuf[0] * fr.b + dmuf[2] * fr.q;
    out16[2] = dmuf[1];
    out16[3] = Kern<KER>::FAC * Sw;
    from_frame_ax(GPf, fr, out16 + 4);
    from_frame_ax(GSf, fr, out16 + 10);
}

// Gradient of one Gaussian from its 3-D PET view-space moments, summed over
// the tile's LORs (d~ = e_w + kappa e_v, c = d~ x (o - mu') = (-v~, du,
// -kappa du), see prep_record), in the normalised variables of the record
// (A_n = A / P'_ww, Q_n = Q / P'_ww; h = -dL/dQ_n / alpha', gA = dL/dA_n /
// alpha', w = dL/dI |d~| A_n^-1/2 K(m), alpha' = alpha / sqrt(P'_ww)):
//   s = [h v~^2, h v~ du, h kappa v~ du, h du^2, h kappa du^2, h kappa^2 du^2,
//        h v~, h v~ kappa, h du, h du kappa, h du kappa^2,
//        gA, gA kappa, gA kappa^2, w]
// With dL/dQ = -alpha P'_ww^-3/2 h and dL/dA = alpha P'_ww^-3/2 gA:
//   dL/dS'  = sum dL/dQ c c^T,   dL/dP' = sum dL/dA d~ d~^T,
//   dL/dmu' = -2 sum dL/dQ (S'c) x d~,  dL/drho = FAC P'_ww^-1/2 sum w.
template <int KER>
__device__ __forceinline__ void pet3d_chain(const float *F, const float4 *rec, uint32_t gid,
                                            const float *s, float *out16)
{
    const float4 *r = rec + REC_F4 * (size_t)gid;
    const float4 r0 = __ldg(r), r1 = __ldg(r + 1), r2 = __ldg(r + 2), r3 = __ldg(r + 3);
    const float P[6] = { r1.x, r1.y, r1.z, r1.w, r2.x, r2.y };
    const float Sh[6] = { r2.z, r2.w, r3.x, r3.y, r3.z, r3.w };
    const AxFrame fr = ax_frame(F);
    float Sf[6];
    to_frame_ax(Sh, fr, Sf);
    const float Pww = (P[0] * fr.p + P[1] * fr.q) * fr.p + (P[1] * fr.p + P[3] * fr.q) * fr.q;
    const float ipw = 1.0f / Pww;
    const float aw = sqrtf(ipw);
    const float ah = r0.w * Kern<KER>::FAC * aw * ipw;
    float GSf[6], GPf[6];
    GSf[0] = -ah * s[0];   // uu: c_u c_u = v~^2
    GSf[1] = ah * s[1];    // uv: -v~ du
    GSf[2] = -ah * s[2];   // uw: kappa v~ du
    GSf[3] = -ah * s[3];   // vv: du^2
    GSf[4] = ah * s[4];    // vw: -kappa du^2
    GSf[5] = -ah * s[5];   // ww: kappa^2 du^2
    GPf[0] = GPf[1] = GPf[2] = 0.0f;
    GPf[3] = ah * s[13];   // vv: kappa^2
    GPf[4] = ah * s[12];   // vw: kappa
    GPf[5] = ah * s[11];   // ww: 1
    // columns of S' and (S' c) x d~ =
    //   -v~ (S'e_u x e_w) - v~ kappa (S'e_u x e_v) + du (S'e_v x e_w)
    //   + du kappa (S'e_v x e_v - S'e_w x e_w) - du kappa^2 (S'e_w x e_v)
    // with x x e_u = (0, x_w, -x_v), x x e_v = (-x_w, 0, x_u), x x e_w = (x_v, -x_u, 0)
    const float cu[3] = { Sf[0], Sf[1], Sf[2] }, cv[3] = { Sf[1], Sf[3], Sf[4] }, cw[3] = { Sf[2], Sf[4], Sf[5] };
    const float M0 = s[6], M1 = s[7], M2 = s[8], M3 = s[9], M4 = s[10];
    float T[3];
    T[0] = -M0 * cu[1] - M1 * (-cu[2]) + M2 * cv[1] + M3 * (-cv[2] - cw[1]) - M4 * (-cw[2]);
    T[1] = -M0 * (-cu[0]) + M2 * (-cv[0]) + M3 * cw[0];
    T[2] = -M1 * cu[0] + M3 * cv[0] - M4 * cw[0];
    const float dmuf[3] = { 2.0f * ah * T[0], 2.0f * ah * T[1], 2.0f * ah * T[2] };
    out16[0] = dmuf[0] * fr.a + dmuf[2] * fr.p;
    out16[1] = dmuf[0] * fr.b + dmuf[2] * fr.q;
    out16[2] = dmuf[1];
    out16[3] = Kern<KER>::FAC * aw * s[14];
    from_frame_ax(GPf, fr, out16 + 4);
    from_frame_ax(GSf, fr, out16 + 10);
}

// Work items of the persistent launches over a batch of scans, numbered scan
// by scan (ScanDesc::item_begin) and taken from an atomic counter; the CTA
// finds its scan by binary search.
__device__ __forceinline__ bool next_item(const ScanDesc *d, int nscan, uint32_t total,
                                          uint32_t *queue, uint32_t &item, int &scan)
{
    __shared__ uint32_t s_item;
    __shared__ int s_scan;
    __syncthreads();   // the previous item is finished by every thread
    if (threadIdx.x == 0) {
        const uint32_t it = atomicAdd(queue, 1u);
        int lo = 0, hi = nscan - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (d[mid].item_begin <= it) lo = mid; else hi = mid - 1;
        }
        s_item = it;
        s_scan = lo;
    }
    __syncthreads();
    item = s_item;
    scan = s_scan;
    return item < total;
}

int sm_count()
{
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n < 1 ? 1 : n;
}

// CTAs of a persistent launch: SMs x resident CTAs per SM
template <class K>
int grid_for(K kernel, int threads)
{
    int per = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, 0);
    return sm_count() * (per < 1 ? 1 : per);
}

}  // namespace
}  // namespace rgrt
