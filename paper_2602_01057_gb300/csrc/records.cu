// Record build (a0) and per-view culling (a2, first half).
//
// Everything that decides which tiles a Gaussian lands in is evaluated with
// explicit round-to-nearest binary32 intrinsics (__fmul_rn, __fadd_rn, ...),
// so no multiply-add is contracted and the result is fixed by the written
// operation order: that order is the culling specification, and the tile
// lists are reproducible bit for bit by any IEEE binary32 implementation of
// it.
#include "rgrt_internal.h"

namespace rgrt {
namespace {

__device__ __forceinline__ float M(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float A(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float S(float a, float b) { return __fsub_rn(a, b); }

// e^x: Cody-Waite reduction x = n ln2 + r, |r| <= ln2/2, and the degree-7
// Taylor polynomial of e^r in Horner form (truncation below 6e-9 relative).
__device__ __forceinline__ float exp_spec(float x)
{
    const float LOG2E = 0x1.715476p+0f;
    const float LN2_HI = 0x1.62e4p-1f;     // ln 2 truncated to 15 significant bits
    const float LN2_LO = 0x1.7f7d1cp-20f;  // ln 2 - LN2_HI
    float n = rintf(M(x, LOG2E));
    float r = S(S(x, M(n, LN2_HI)), M(n, LN2_LO));
    float p = 0x1.a01a02p-13f;
    p = A(M(p, r), 0x1.6c16c2p-10f);
    p = A(M(p, r), 0x1.111112p-7f);
    p = A(M(p, r), 0x1.555556p-5f);
    p = A(M(p, r), 0x1.555556p-3f);
    p = A(M(p, r), 0.5f);
    p = A(M(p, r), 1.0f);
    p = A(M(p, r), 1.0f);
    return ldexpf(p, (int)n);
}

__global__ void k_records(const float *__restrict__ mu, const float *__restrict__ ls,
                          const float *__restrict__ q, const float *__restrict__ rho, int64_t n,
                          float4 *__restrict__ rec, float4 *__restrict__ crec, uint32_t *bad)
{
    int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    float qw = q[4 * k], qx = q[4 * k + 1], qy = q[4 * k + 2], qz = q[4 * k + 3];
    // a non-finite parameter (a diverged optimisation, corrupted input) is
    // reported to the host, which refuses the projection
    if (bad && !(isfinite(mu[3 * k]) && isfinite(mu[3 * k + 1]) && isfinite(mu[3 * k + 2]) &&
                 isfinite(ls[3 * k]) && isfinite(ls[3 * k + 1]) && isfinite(ls[3 * k + 2]) &&
                 isfinite(qw) && isfinite(qx) && isfinite(qy) && isfinite(qz) && isfinite(rho[k])))
        atomicOr(bad, 1u);
    float n2 = A(A(A(M(qw, qw), M(qx, qx)), M(qy, qy)), M(qz, qz));
    float w, x, y, z;
    if (!(n2 > 0.0f) || !(n2 < INFINITY)) {
        w = 1.0f; x = y = z = 0.0f;
    } else {
        float nr = __fsqrt_rn(n2);
        w = __fdiv_rn(qw, nr); x = __fdiv_rn(qx, nr); y = __fdiv_rn(qy, nr); z = __fdiv_rn(qz, nr);
    }
    float R[3][3];
    R[0][0] = S(1.0f, M(2.0f, A(M(y, y), M(z, z))));
    R[0][1] = M(2.0f, S(M(x, y), M(w, z)));
    R[0][2] = M(2.0f, A(M(x, z), M(w, y)));
    R[1][0] = M(2.0f, A(M(x, y), M(w, z)));
    R[1][1] = S(1.0f, M(2.0f, A(M(x, x), M(z, z))));
    R[1][2] = M(2.0f, S(M(y, z), M(w, x)));
    R[2][0] = M(2.0f, S(M(x, z), M(w, y)));
    R[2][1] = M(2.0f, A(M(y, z), M(w, x)));
    R[2][2] = S(1.0f, M(2.0f, A(M(x, x), M(y, y))));
    float l0 = ls[3 * k], l1 = ls[3 * k + 1], l2 = ls[3 * k + 2];
    float s2[3] = { exp_spec(M(2.0f, l0)), exp_spec(M(2.0f, l1)), exp_spec(M(2.0f, l2)) };
    const int ia[6] = { 0, 0, 0, 1, 1, 2 }, ib[6] = { 0, 1, 2, 1, 2, 2 };
    float sig[6];
#pragma unroll
    for (int e = 0; e < 6; e++) {
        int a = ia[e], b = ib[e];
        sig[e] = A(A(M(M(R[a][0], R[b][0]), s2[0]), M(M(R[a][1], R[b][1]), s2[1])),
                   M(M(R[a][2], R[b][2]), s2[2]));
    }
    float m0 = mu[3 * k], m1 = mu[3 * k + 1], m2 = mu[3 * k + 2];
    crec[CREC_F4 * k + 0] = make_float4(m0, m1, m2, 0.0f);
    crec[CREC_F4 * k + 1] = make_float4(sig[0], sig[1], sig[2], sig[3]);
    crec[CREC_F4 * k + 2] = make_float4(sig[4], sig[5], 0.0f, 0.0f);

    // integration record: P = R diag(e^-2l) R^T and S = Sigma / det Sigma =
    // R diag(e^-2(l_b + l_c)) R^T ({k, b, c} = {0, 1, 2}); not part of the
    // culling specification, ordinary arithmetic.
    float p2[3] = { expf(-2.0f * l0), expf(-2.0f * l1), expf(-2.0f * l2) };
    float c2[3] = { expf(-2.0f * (l1 + l2)), expf(-2.0f * (l0 + l2)), expf(-2.0f * (l0 + l1)) };
    float P[6], Sh[6];
#pragma unroll
    for (int e = 0; e < 6; e++) {
        int a = ia[e], b = ib[e];
        P[e] = R[a][0] * R[b][0] * p2[0] + R[a][1] * R[b][1] * p2[1] + R[a][2] * R[b][2] * p2[2];
        Sh[e] = R[a][0] * R[b][0] * c2[0] + R[a][1] * R[b][1] * c2[1] + R[a][2] * R[b][2] * c2[2];
    }
    float smax = expf(fmaxf(l0, fmaxf(l1, l2)));
    rec[REC_F4 * k + 0] = make_float4(m0, m1, m2, rho[k]);
    rec[REC_F4 * k + 1] = make_float4(P[0], P[1], P[2], P[3]);
    rec[REC_F4 * k + 2] = make_float4(P[4], P[5], Sh[0], Sh[1]);
    rec[REC_F4 * k + 3] = make_float4(Sh[2], Sh[3], Sh[4], Sh[5]);
    rec[REC_F4 * k + 4] = make_float4(smax, 0.0f, 0.0f, 0.0f);
}

// e_a^T Sigma e_b, Sigma packed (00,01,02,11,12,22)
__device__ __forceinline__ float form_spec(const float *Sg, const float *a, const float *b)
{
    float t0 = A(A(M(Sg[0], b[0]), M(Sg[1], b[1])), M(Sg[2], b[2]));
    float t1 = A(A(M(Sg[1], b[0]), M(Sg[3], b[1])), M(Sg[4], b[2]));
    float t2 = A(A(M(Sg[2], b[0]), M(Sg[4], b[1])), M(Sg[5], b[2]));
    return A(A(M(a[0], t0), M(a[1], t1)), M(a[2], t2));
}

__device__ __forceinline__ float dot_spec(const float *m, const float *e)
{
    return A(A(M(m[0], e[0]), M(m[1], e[1])), M(m[2], e[2]));
}

// detector interval along one axis whose cone-beam rays meet the K-sigma
// ellipsoid: roots of (n.a)^2 = K^2 n^T Sigma n for the planes through the
// source containing the other detector axis; false if unbounded.
__device__ __forceinline__ bool cone_spec(float K2, float dsd, float ae, float aw, float see,
                                          float sew, float sww, float &lo, float &hi)
{
    float alpha = S(M(aw, aw), M(K2, sww));
    if (!(alpha > 0.0f)) return false;
    float beta = M(dsd, S(M(ae, aw), M(K2, sew)));
    float disc = S(A(S(M(M(aw, aw), see), M(M(M(2.0f, ae), aw), sew)), M(M(ae, ae), sww)),
                   M(K2, S(M(see, sww), M(sew, sew))));
    if (!(disc > 0.0f)) disc = 0.0f;
    float r = M(dsd, __fsqrt_rn(M(K2, disc)));
    lo = __fdiv_rn(S(beta, r), alpha);
    hi = __fdiv_rn(A(beta, r), alpha);
    return true;
}

// first index whose table value is >= x (n if none), and the last whose
// value is <= x (-1 if none), by binary search over the increasing table
__device__ __forceinline__ int lower_idx(const float *tab, int n, float x)
{
    int lo = 0, hi = n;
    while (lo < hi) {
        int mid = (lo + hi) >> 1;
        if (__ldg(tab + mid) >= x) hi = mid; else lo = mid + 1;
    }
    return lo;
}
__device__ __forceinline__ int upper_idx(const float *tab, int n, float x)
{
    int lo = 0, hi = n;
    while (lo < hi) {
        int mid = (lo + hi) >> 1;
        if (__ldg(tab + mid) > x) hi = mid; else lo = mid + 1;
    }
    return lo - 1;
}

// The same two searches started from a guess: for a uniformly spaced table
// (t0 + i step in binary32, inv = 1/step) the guess is within a step of the
// answer and a short walk in the table makes it exact -- the answer is
// defined by the table comparisons alone, so it equals the binary search's.
// inv == 0 (an irregular table) falls back to the binary search; NaN gives
// what the binary search gives (n, n - 1).
__device__ __forceinline__ int lower_idx_g(const float *tab, int n, float x, float t0, float inv)
{
    if (inv == 0.0f || !(x == x)) return lower_idx(tab, n, x);
    int i = (int)fminf(fmaxf(ceilf((x - t0) * inv), 0.0f), (float)n);
    while (i > 0 && __ldg(tab + i - 1) >= x) i--;
    while (i < n && __ldg(tab + i) < x) i++;
    return i;
}
__device__ __forceinline__ int upper_idx_g(const float *tab, int n, float x, float t0, float inv)
{
    if (inv == 0.0f || !(x == x)) return upper_idx(tab, n, x);
    // first index whose value is > x, minus one
    int i = (int)fminf(fmaxf(floorf((x - t0) * inv) + 1.0f, 0.0f), (float)n);
    while (i > 0 && __ldg(tab + i - 1) > x) i--;
    while (i < n && __ldg(tab + i) <= x) i++;
    return i - 1;
}

// A Gaussian in a view's frame: the quantities that its detector box follows from
struct CullFrame {
    float mu_u, mu_v, mu_w, suu, svv, sww, suw, svw;
};

// By the specification's general forms.  Every frame here is a rotation about
// z -- e_v = (0, 0, 1), e_u and e_w in the transaxial plane -- and for finite
// values the products with its zeros change no sum, so the short forms below
// give the same numbers; where one of them is not finite (an overflowed
// covariance times a zero is a NaN) the general ones decide.
template <bool CONE, bool P3>
__device__ __forceinline__ CullFrame cull_frame(const float *m, const float *Sg, const float *F)
{
    const float eu[3] = { __ldg(F + 0), __ldg(F + 1), __ldg(F + 2) };
    const float ew[3] = { __ldg(F + 6), __ldg(F + 7), __ldg(F + 8) };
    CullFrame c;
    c.mu_u = A(M(m[0], eu[0]), M(m[1], eu[1]));
    c.mu_v = m[2];
    c.suu = A(M(eu[0], A(M(Sg[0], eu[0]), M(Sg[1], eu[1]))), M(eu[1], A(M(Sg[1], eu[0]), M(Sg[3], eu[1]))));
    c.svv = Sg[5];
    c.mu_w = c.sww = c.suw = c.svw = 0.0f;
    if (CONE || P3) {
        const float t0 = A(M(Sg[0], ew[0]), M(Sg[1], ew[1])), t1 = A(M(Sg[1], ew[0]), M(Sg[3], ew[1]));
        c.mu_w = A(M(m[0], ew[0]), M(m[1], ew[1]));
        c.sww = A(M(ew[0], t0), M(ew[1], t1));
        c.suw = A(M(eu[0], t0), M(eu[1], t1));
        c.svw = A(M(Sg[2], ew[0]), M(Sg[4], ew[1]));
    }
    const float all = c.mu_u + c.mu_v + c.mu_w + c.suu + c.svv + c.sww + c.suw + c.svw + (Sg[2] + Sg[4]);
    if (!isfinite(all)) {
        const float ev[3] = { __ldg(F + 3), __ldg(F + 4), __ldg(F + 5) };
        c.mu_u = dot_spec(m, eu);
        c.mu_v = dot_spec(m, ev);
        c.mu_w = dot_spec(m, ew);
        c.suu = form_spec(Sg, eu, eu);
        c.svv = form_spec(Sg, ev, ev);
        c.sww = form_spec(Sg, ew, ew);
        c.suw = form_spec(Sg, eu, ew);
        c.svw = form_spec(Sg, ev, ew);
    }
    return c;
}

// number of tiles and pixel box of columns i0..i1, rows j0..j1
__device__ __forceinline__ void cull_write(const DevGeom &g, int i0, int i1, int j0, int j1, uint32_t *cnt, uint2 *rect)
{
    if (i0 > i1 || j0 > j1) {
        *cnt = 0;
        *rect = make_uint2(1u, 1u);   // empty: columns and rows 1..0
        return;
    }
    const TileDiv d(g);
    const unsigned tx0 = d.x(i0), tx1 = d.x(i1), ty0 = d.y(j0), ty1 = d.y(j1);
    *cnt = (tx1 - tx0 + 1) * (ty1 - ty0 + 1);
    // pixel box (the tiles follow from it)
    *rect = make_uint2((unsigned)i0 | ((unsigned)i1 << 16), (unsigned)j0 | ((unsigned)j1 << 16));
}

// one thread per (view of the chunk, Gaussian), view-major; 3-D PET: one per
// (angle, Gaussian), which takes the chunk's ring differences of that angle in
// turn (they share the frame and the columns)
template <int GM>
__global__ void k_cull(DevGeom g, int nv, const float4 *__restrict__ crec, int64_t n,
                       uint32_t *__restrict__ cnt, uint2 *__restrict__ rect, uint32_t *large)
{
    constexpr bool CONE = GM == GM_CONE, P3 = GM == GM_PET3D;
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const float4 c0 = crec[CREC_F4 * k], c1 = crec[CREC_F4 * k + 1], c2 = crec[CREC_F4 * k + 2];
    const float m[3] = { c0.x, c0.y, c0.z };
    const float Sg[6] = { c1.x, c1.y, c1.z, c1.w, c2.x, c2.y };
    const float K2 = CULL_K2;
    const int nf = P3 ? min(nv, g.n_ang) : nv;
    for (int vf = blockIdx.y; vf < nf; vf += gridDim.y) {
        const CullFrame c = cull_frame<CONE, P3>(m, Sg, g.frames + 9 * (size_t)(g.v0 + vf));
        float ulo = -INFINITY, uhi = INFINITY, vlo = -INFINITY, vhi = INFINITY;
        if (CONE) {
            const float aw = A(c.mu_w, g.dso);
            float lo, hi;
            if (cone_spec(K2, g.dsd, c.mu_u, aw, c.suu, c.suw, c.sww, lo, hi)) { ulo = lo; uhi = hi; }
            if (cone_spec(K2, g.dsd, c.mu_v, aw, c.svv, c.svw, c.sww, lo, hi)) { vlo = lo; vhi = hi; }
        } else {
            const float hu = __fsqrt_rn(M(K2, c.suu));
            ulo = S(c.mu_u, hu); uhi = A(c.mu_u, hu);
            if (!P3) {
                const float hv = __fsqrt_rn(M(K2, c.svv));
                vlo = S(c.mu_v, hv); vhi = A(c.mu_v, hv);
            }
        }
        const int i0 = lower_idx_g(g.utab, g.n_cols, ulo, g.u0, g.uinv);
        const int i1 = upper_idx_g(g.utab, g.n_cols, uhi, g.u0, g.uinv);
        if (!P3) {
            const int j0 = lower_idx_g(g.vtab, g.n_rows, vlo, g.v0f, g.vinv);
            const int j1 = upper_idx_g(g.vtab, g.n_rows, vhi, g.v0f, g.vinv);
            cull_write(g, i0, i1, j0, j1, cnt + (int64_t)vf * n + k, rect + (int64_t)vf * n + k);
            if (GM == GM_PARALLEL) {
                const unsigned a = i1 - i0, b = j1 - j0;   // (a + 1) (b + 1) pixels
                if (i0 <= i1 && j0 <= j1 && a * b + a + b >= (unsigned)ADJOINT_LARGE_PX && large) *large = 1u;
            }
            continue;
        }
        // 3-D PET: the LOR of radial position s and mid-height z has
        // direction e_w + kappa e_v, kappa = dz / (2 sqrt(R^2 - s^2)), and
        // a . x = z along it for a = e_v - kappa e_w, so it can meet the
        // K-sigma ellipsoid only if z lies in mu.a +- sqrt(K^2 a^T Sigma a).
        // Both bounds are convex / concave in kappa, so over the columns
        // i0..i1 the union of these intervals is spanned by their values at
        // the two extreme slopes.  Rows are ring pairs (mid-heights
        // vtab + zoff); rows past the segment's last pair hold no LOR.
        float h2a = 0.0f, h2b = 0.0f;
        if (i0 <= i1) {
            const float ua = __ldg(g.utab + i0), ub = __ldg(g.utab + i1);
            const float amin = (ua <= 0.0f && ub >= 0.0f) ? 0.0f : fminf(fabsf(ua), fabsf(ub));
            const float amax = fmaxf(fabsf(ua), fabsf(ub));
            h2a = S(g.radius2, M(amin, amin));
            h2b = S(g.radius2, M(amax, amax));
        }
        const float sa = __fsqrt_rn(h2a), sb = __fsqrt_rn(h2b);
        for (int vl = vf; vl < nv; vl += g.n_ang) {
            int j0 = 0, j1 = -1;
            if (i0 <= i1) {
                const int delta = pet3d_delta(g, g.v0 + vl), ad = abs(delta);
                const float dz = M((float)delta, g.ring_pitch), zoff = M(M(0.5f, (float)ad), g.ring_pitch);
                const int last = g.n_rows - 1 - ad;
                if (!(h2b > 0.0f)) {
                    j1 = last;
                } else {
                    float zlo = INFINITY, zhi = -INFINITY;
#pragma unroll
                    for (int e = 0; e < 2; e++) {
                        const float kap = __fdiv_rn(M(0.5f, dz), e ? sb : sa);
                        const float zc = S(c.mu_v, M(kap, c.mu_w));
                        const float t = A(S(c.svv, M(M(2.0f, kap), c.svw)), M(M(kap, kap), c.sww));
                        const float half = __fsqrt_rn(fmaxf(M(K2, t), 0.0f));
                        zlo = fminf(zlo, S(zc, half));
                        zhi = fmaxf(zhi, A(zc, half));
                    }
                    j0 = lower_idx_g(g.vtab, g.n_rows, S(zlo, zoff), g.v0f, g.vinv);
                    j1 = min(upper_idx_g(g.vtab, g.n_rows, S(zhi, zoff), g.v0f, g.vinv), last);
                }
            }
            cull_write(g, i0, i1, j0, j1, cnt + (int64_t)vl * n + k, rect + (int64_t)vl * n + k);
        }
    }
}

}  // namespace

cudaError_t launch_records(const float *mu, const float *ls, const float *q, const float *rho,
                           int64_t n, float4 *rec, float4 *crec, uint32_t *bad, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    int bs = 256;
    k_records<<<(unsigned)((n + bs - 1) / bs), bs, 0, s>>>(mu, ls, q, rho, n, rec, crec, bad);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_cull(const DevGeom &g, int nv, const float4 *crec, int64_t n, uint32_t *cnt,
                        uint2 *rect, cudaStream_t s, uint32_t *large)
{
    if (nv <= 0 || n <= 0) return cudaSuccess;
    const int nf = g.kind == GM_PET3D && nv > g.n_ang ? g.n_ang : nv;
    const dim3 grid((unsigned)((n + 255) / 256), (unsigned)(nf < 65535 ? nf : 65535));
    if (g.kind == GM_CONE) k_cull<GM_CONE><<<grid, 256, 0, s>>>(g, nv, crec, n, cnt, rect, nullptr);
    else if (g.kind == GM_PET3D) k_cull<GM_PET3D><<<grid, 256, 0, s>>>(g, nv, crec, n, cnt, rect, nullptr);
    else k_cull<GM_PARALLEL><<<grid, 256, 0, s>>>(g, nv, crec, n, cnt, rect, large);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace rgrt
