// Adjoint of the parallel-ray geometries (a5): CT parallel beam and the PET
// ring with or without time of flight, dL/dI back to the Gaussians'
// (mu, rho, G_P, G_S).  (Cone beam and 3-D PET: adjoint_tile.cu.)
//
// Gaussian-stationary: a warp takes up to 32 Gaussians that lie close together in
// space (launch_order) and, with the CTA's other warps,
// a range of views.  Per view
//  * lane k turns record k into its view-space form (shared memory) and reads
//    its pixel box (k_cull's rectangle); the CTA stages the rectangle of dL/dI
//    that holds all its boxes, in bands when it is larger than the buffer;
//  * sub-warps of S = 2^LG lanes take the Gaussians in turn, a lane walking
//    every S-th row of the box along the footprint's chord,
//    two pixels at a time in packed binary32, and reduce the view-space
//    moments across the sub-warp;
//  * lane k chains Gaussian k's moments (view_chain) into the world-space
//    gradient that it keeps over the CTA's views.
// No tile lists, no per-tile atomics: one set of 16 sums per Gaussian and view
// range, added to the accumulator at the end.  Footprints far larger than their
// neighbours', and launches of few Gaussians, are walked in place instead
// (k_adjoint_direct).
//
// Bound by instruction issue (the pixels of the chords, their set-up, and the
// lanes that wait for a longer chord of the same round).  Against one Gaussian
// per thread and tile (record gathers, box searches, a chain and 16 atomics
// for each of the 1.9 tiles of a PET footprint), measured on a GB300: PET ring
// of 288 x 329 x 63, 200,000 Gaussians 9.6 -> 6.8 ms; 8 raw angles, 100,000
// 0.73 -> 0.14 ms; 24 angles x 13 time-of-flight bins 4.96 -> 2.83 ms; parallel
// beam, 1,000 Gaussians on 16 x 64^2 0.34 -> 0.07 ms (that one had 256 CTAs of
// serial pixels).  Sorting a warp's Gaussians by box area per view took the
// ring from 8.0 to 6.9 ms: a round's lanes then have chords of like length.
// Only the Gaussians that meet a band are walked in it (a ring with 13
// time-of-flight bins, 288 angles: 35.7 -> 33.9 ms).
#include <type_traits>

#include "packed.cuh"
#include "view.cuh"

namespace rgrt {
namespace {

constexpr int BS = 128;
constexpr int NW = BS / 32;
template <bool TOF> struct Wide { static constexpr int v = TOF ? 256 : 512; };   // widest band (columns)
constexpr int BH = 256;         // highest band (rows)

// shared floats of the staged band
template <bool TOF> struct Cap { static constexpr int v = TOF ? 5120 : 4096; };

// factors of the moments' derivatives: with h = dL/dI times the kernel's
// profile and p = h arg,  -dL/dQ = A^-3/2 FQ h  and  dL/dA = A^-3/2 (FP p -
// h / 2)  per unit alpha
template <int KER> struct Fac;
template <> struct Fac<0> {
    static constexpr float FQ = 0.5f, FP = 0.5f * M_PER_ARG;
};
template <> struct Fac<1> {
    static constexpr float FQ = 1.5f / 7.0f, FP = -2.0f;
};

// the Gaussian's cut acts on x (dL/dI or what is made of it), so that an
// infinite or NaN dL/dI outside the cut adds nothing
__device__ __forceinline__ float cut(float arg, float x)
{
    return arg >= CUT_ARG ? x : 0.0f;
}

// dL/dI times the kernel's profile, of two pixels: g e^{-m/2} (Gaussian), g sqrt(c)
// inside the support (Epanechnikov, c = 1 + arg); 0 outside the cut or support,
// whatever g is
template <int KER>
__device__ __forceinline__ f2 weighted(float a0, float a1, float2 g)
{
    if (KER == 1) {
        const float x = 1.0f + a0, y = 1.0f + a1;
        return mul2(pk(x > 0.0f ? g.x : 0.0f, y > 0.0f ? g.y : 0.0f), pk(sqrt_approx(fabsf(x)), sqrt_approx(fabsf(y))));
    }
    return mul2(pk(cut(a0, g.x), cut(a1, g.y)), pk(ex2_approx(a0), ex2_approx(a1)));
}

struct Box {
    int ilo, ihi, jlo, jhi;
};

// Pixels of a box, its sides taken as 16,384 at most (a detector of 65,536 x 65,536
// has 2^32): exact where it is compared with the limits of the two walks, and
// it only orders the larger ones.
__device__ __forceinline__ int box_px(int w, int h)
{
    return min(w, 16384) * min(h, 16384);
}

// a staged band: columns [cb, cb + w), rows [rb, rb + h), row stride st
struct Band {
    int cb, rb, w, h, st;
};

// where a walk reads: a staged band, coordinates relative to it ...
struct Staged {
    static constexpr int UNROLL = 1, STEP = 2;
    const float *sg, *su, *sv;
    Band bd;
    __device__ __forceinline__ int cb() const { return bd.cb; }
    __device__ __forceinline__ int rb() const { return bd.rb; }
    __device__ __forceinline__ int w() const { return bd.w; }
    __device__ __forceinline__ int h() const { return bd.h; }
    __device__ __forceinline__ int col0() const { return 0; }
    __device__ __forceinline__ int plane() const { return bd.h * bd.st; }
    __device__ __forceinline__ float2 u2(int i) const { return *reinterpret_cast<const float2 *>(su + i); }
    __device__ __forceinline__ float v(int j) const { return sv[j]; }
    __device__ __forceinline__ const float *row(int j) const { return sg + j * bd.st; }
    __device__ __forceinline__ float2 g2(const float *p, int i) const { return *reinterpret_cast<const float2 *>(p + i); }
};

// ... or the view itself, 2^DIRECT_LG lanes side by side in a row
constexpr int DIRECT_LG = 2;
struct Direct {
    static constexpr int UNROLL = 2, STEP = 2 << DIRECT_LG;
    const DevGeom &g;
    const float *I;
    int lc;
    __device__ __forceinline__ int cb() const { return 0; }
    __device__ __forceinline__ int rb() const { return 0; }
    __device__ __forceinline__ int w() const { return g.n_cols; }
    __device__ __forceinline__ int h() const { return g.n_rows; }
    __device__ __forceinline__ int col0() const { return 2 * lc; }
    __device__ __forceinline__ long long plane() const { return g.stride_tof; }
    __device__ __forceinline__ float2 u2(int i) const
    {
        return make_float2(__ldg(g.utab + i), __ldg(g.utab + min(i + 1, g.n_cols - 1)));
    }
    __device__ __forceinline__ float v(int j) const { return __ldg(g.vtab + j); }
    __device__ __forceinline__ const float *row(int j) const { return I + j * g.stride_row; }
    __device__ __forceinline__ float2 g2(const float *p, int i) const
    {
        return make_float2(__ldg(p + i), i + 1 < g.n_cols ? __ldg(p + i + 1) : 0.0f);
    }
};

// cut of the chords: a little outside the pairs' own, so that rounding in the
// roots loses no pixel (the chord is widened by 0.05 columns as well)
template <int KER>
__device__ __forceinline__ float chord_cut()
{
    return KER == 1 ? -1.0f - 2e-4f : CUT_ARG * (1.0f + 2e-4f);
}

// columns [lo, hi] cut down to the chord al du^2 + be du + ga >= 0 (al < 0),
// xc = the column coordinate of du = 0, iv = columns per unit
__device__ __forceinline__ void chord(float al, float be, float ga, float xc, float iv, int &lo, int &hi)
{
    const float D = fmaf(be, be, -4.0f * al * ga);
    const float sq = sqrt_approx(fmaxf(D, 0.0f)), i2a = __fdividef(0.5f * iv, al);
    const float a = fmaf(sq - be, i2a, xc - 0.05f), b = fmaf(-be - sq, i2a, xc + 0.05f);   // a <= b
    lo = max(lo, (int)ceilf(fmaxf(a, -1.0f)));
    hi = D < 0.0f ? -1 : min(hi, (int)floorf(fminf(b, 65536.0f)));
}

// Moments of one Gaussian over the lane's share of its box within the band:
// rows jlo + r0, + dr, ..., in each the chord of the footprint (every pixel is
// still tested), two columns at a time.  With h = dL/dI times the kernel's
// profile and p = h arg,
//   m[0..5] = sum h {1, du, dv, du^2, du dv, dv^2},  m[6] = sum p;
// A is constant along parallel rays, its powers are left to finish().
template <int KER, class Src>
__device__ __forceinline__ void rows(const DevGeom &g, const float4 &c0, const float4 &c1, const Box &bx, int r0,
                                     int dr, const Src &src, float *m)
{
    const float u0 = c0.x, v0 = c0.y, kMuv2 = c0.w, kMvv = c1.x, thr = chord_cut<KER>();
    const int ilo = max(bx.ilo - src.cb(), 0), ihi = min(bx.ihi - src.cb(), src.w() - 1);
    const float xc = (u0 - g.u0) * g.uinv - (float)src.cb();
    int j = bx.jlo - src.rb() + r0;
    if (j < 0) j += (-j + dr - 1) / dr * dr;
    const int je = min(bx.jhi - src.rb(), src.h() - 1);
    const f2 nu0 = pk(-u0, -u0), Muu = pk(c0.z, c0.z);
#pragma unroll
    for (int q = 0; q < 7; q++) m[q] = 0.0f;
    for (; j <= je; j += dr) {
        const float dv = src.v(j) - v0, dv2 = dv * dv;
        const float a1 = kMuv2 * dv, a0 = kMvv * dv2;
        const f2 A1 = pk(a1, a1), A0 = pk(a0, a0);
        int ia = ilo, ie = ihi;
        if (g.uinv != 0.0f && c0.z < 0.0f) chord(c0.z, a1, a0 - thr, xc, g.uinv, ia, ie);
        const float *gr = src.row(j);
        f2 h0 = 0, h1 = 0, h2 = 0, q0 = 0;
#pragma unroll Src::UNROLL
        for (int i = (ia & ~1) + src.col0(); i <= ie; i += Src::STEP) {
            const float2 uu = src.u2(i), gg = src.g2(gr, i);
            const f2 du = add2(pk(uu.x, uu.y), nu0);
            const f2 q = fma2(fma2(Muu, du, A1), du, A0);
            float qx, qy;
            up(q, qx, qy);
            const f2 h = weighted<KER>(qx, qy, gg);
            const f2 hd = mul2(h, du);
            h0 = add2(h0, h);
            h1 = add2(h1, hd);
            h2 = fma2(hd, du, h2);
            q0 = fma2(h, q, q0);
        }
        const float s0 = hadd(h0), s1 = hadd(h1);
        m[0] += s0;
        m[1] += s1;
        m[2] = fmaf(s0, dv, m[2]);
        m[3] += hadd(h2);
        m[4] = fmaf(s1, dv, m[4]);
        m[5] = fmaf(s0, dv2, m[5]);
        m[6] += hadd(q0);
    }
}

// The same with time of flight (parallel rays, one pixel at a time): a pair's
// value times the bin's weight W_k = N(t* - t_k; 0, s^2), s^2 = 1/A +
// sigma_T^2.  h carries G = sum_k g_k W_k in place of dL/dI, and four more
// sums the weights' own gradients: m[7..10] = val dW/dt* (1, du, dv) and
// val dW/ds^2.
template <class Src>
__device__ __forceinline__ void rows_tof(const DevGeom &g, const float4 &c0, const float4 &c1, const float4 &t4,
                                         const Box &bx, int r0, int dr, const Src &src, float *m)
{
    const float u0 = c0.x, v0 = c0.y;
    const int ilo = max(bx.ilo - src.cb(), 0), ihi = min(bx.ihi - src.cb(), src.w() - 1);
    const float xc = (u0 - g.u0) * g.uinv - (float)src.cb();
    int j = bx.jlo - src.rb() + r0;
    if (j < 0) j += (-j + dr - 1) / dr * dr;
    const int je = min(bx.jhi - src.rb(), src.h() - 1);
    const float s2 = t4.w + g.tof_s2, is2 = 1.0f / s2, ns = Kern<0>::QSCALE * is2;
    const float nrm = rsqrtf(2.0f * 3.14159265358979324f / is2);
    const auto plane = src.plane();
#pragma unroll
    for (int q = 0; q < 11; q++) m[q] = 0.0f;
    const f2 NS = pk(ns, ns), TH = pk(g.tof_h, g.tof_h), MINUS1 = pk(-1.0f, -1.0f);
    // one flat loop over the lane's (row, column pair) items: a pair costs a loop
    // over the bins, so a lane goes on to its next row rather than waiting for
    // the longest chord of each, and 5 CTAs per SM, for the spills that 6 cost
    // (24 angles x 13 bins: 3.27 -> 2.87 ms)
    int i = 1, ie = 0;
    float dv = 0.0f, a1 = 0.0f, a0 = 0.0f;
    j -= dr;
    while (true) {
        if (i > ie) {
            j += dr;
            if (j > je) break;
            dv = src.v(j) - v0;
            const float dv2 = dv * dv;
            a1 = c0.w * dv;
            a0 = c1.x * dv2;
            i = ilo;
            ie = ihi;
            if (g.uinv != 0.0f && c0.z < 0.0f) chord(c0.z, a1, a0 - chord_cut<0>(), xc, g.uinv, i, ie);
            i = (i & ~1) + src.col0();
        }
        if (i <= ie) {
            const float2 uu = src.u2(i);
            const int at = i;
            i += Src::STEP;
            const float du0 = uu.x - u0, du1 = uu.y - u0;
            const float q0 = fmaf(fmaf(c0.z, du0, a1), du0, a0), q1 = fmaf(fmaf(c0.z, du1, a1), du1, a0);
            const float e0 = ex2_approx(q0), e1 = ex2_approx(q1);
            const float tb = t4.x + t4.z * dv - g.tof_t0;
            const f2 ts = pk(tb + t4.y * du0, tb + t4.y * du1);
            f2 Ge = 0, D1 = 0, D2 = 0, nb = 0;      // nb: minus the bin
            const float *gp = src.row(j);
#pragma unroll 2
            for (int b = 0; b < g.n_tof; b++, gp += plane) {
                const f2 x = fma2(nb, TH, ts), x2 = mul2(x, x);
                nb = add2(nb, MINUS1);
                float y0, y1;
                up(mul2(NS, x2), y0, y1);
                const float2 gg = src.g2(gp, at);
                const f2 gw = mul2(pk(gg.x, gg.y), pk(ex2_approx(y0), ex2_approx(y1)));
                Ge = add2(Ge, gw);
                D1 = fma2(gw, x, D1);
                D2 = fma2(gw, x2, D2);
            }
#pragma unroll
            for (int k = 0; k < 2; k++) {
                float G0, G1, d10, d11, d20, d21;
                up(Ge, G0, G1);
                up(D1, d10, d11);
                up(D2, d20, d21);
                const float du = k ? du1 : du0, e = k ? e1 : e0, q = k ? q1 : q0;
                const float ge = cut(q, k ? G1 : G0) * nrm;
                const float v1 = e * (cut(q, k ? d11 : d10) * (-nrm * is2));     // val sum g_k dW_k/dt*
                const float v2 = e * (0.5f * is2 * (nrm * is2 * cut(q, k ? d21 : d20) - ge));   // val sum g_k dW_k/ds^2
                const float h = ge * e, hd = h * du;
                m[0] += h;
                m[1] += hd;
                m[2] = fmaf(h, dv, m[2]);
                m[3] = fmaf(hd, du, m[3]);
                m[4] = fmaf(hd, dv, m[4]);
                m[5] = fmaf(h * dv, dv, m[5]);
                m[6] = fmaf(h, q, m[6]);
                m[7] += v1;
                m[8] = fmaf(v1, du, m[8]);
                m[9] = fmaf(v1, dv, m[9]);
                m[10] += v2;
            }
        }
    }
}

// moments of rows() in the layout of view_chain
template <int KER>
__device__ __forceinline__ void finish(const float *m, float iA, float rA, float *s)
{
    constexpr float FQ = Fac<KER>::FQ, FP = Fac<KER>::FP;
    const float f = rA * iA;
    s[0] = -FQ * f * m[1];
    s[1] = -FQ * f * m[2];
    s[2] = -FQ * f * m[3];
    s[3] = -FQ * f * m[4];
    s[4] = -FQ * f * m[5];
    s[5] = f * (FP * m[6] - 0.5f * m[0]);
    s[6] = rA * (KER == 1 ? m[0] + m[6] : m[0]);
}

// Sum the N moments over sub-warps of 2^LG lanes, transposed (each halving of
// the sub-warp also halves the values a lane keeps), and add this lane's sums
// to out[0..N) (on, the same over a sub-warp: not where it has no Gaussian of its
// own, whose out may be another sub-warp's).
template <int N, int LG>
__device__ __forceinline__ void reduce_add(float *v, int sl, float *out, bool on = true)
{
    constexpr int H1 = (N + 1) / 2, H2 = (H1 + 1) / 2, H3 = (H2 + 1) / 2, H4 = (H3 + 1) / 2, H5 = (H4 + 1) / 2;
    constexpr int HN[6] = { N, H1, H2, H3, H4, H5 };
    int p = 0, len = N;
    if (LG >= 1) { tr_stage<N, 1>(v, sl); const int h = H1; if (sl & 1) { p += h; len -= h; } else len = h; }
    if (LG >= 2) { tr_stage<H1, 2>(v, sl); const int h = H2; if (sl & 2) { p += h; len -= h; } else len = min(len, h); }
    if (LG >= 3) { tr_stage<H2, 4>(v, sl); const int h = H3; if (sl & 4) { p += h; len -= h; } else len = min(len, h); }
    if (LG >= 4) { tr_stage<H3, 8>(v, sl); const int h = H4; if (sl & 8) { p += h; len -= h; } else len = min(len, h); }
    if (LG >= 5) { tr_stage<H4, 16>(v, sl); const int h = H5; if (sl & 16) { p += h; len -= h; } else len = min(len, h); }
    constexpr int LAST = HN[LG];
#pragma unroll
    for (int q = 0; q < LAST; q++)
        if (on && q < len) out[p + q] += v[q];
}

// A Gaussian near a segment end, in world coordinates: the warp shares the
// pixels of its box; the owner lane adds the sums to its gradient.  Out of
// line: it is rarely taken.
template <int KER, bool TOF>
__device__ __noinline__ void general_box(const DevGeom &g, int view, const float4 *rec,
                                         uint32_t gid, int ilo, int ihi, int jlo, int jhi, const float *dLdI,
                                         float *val)
{
    const int lane = threadIdx.x & 31;
    float F[9];
    for (int q = 0; q < 9; q++) F[q] = __ldg(g.frames + 9 * (size_t)view + q);
    struct { float4 g0, g1, g2; } r;
    r.g0 = __ldg(rec + REC_F4 * (size_t)gid);
    r.g1 = __ldg(rec + REC_F4 * (size_t)gid + 1);
    r.g2 = __ldg(rec + REC_F4 * (size_t)gid + 2);
    const int w = ihi - ilo + 1, di = 32 % w, dj = 32 / w;     // 32 pixels on, row by row
    for (int q = 0; q < NG; q++) val[q] = 0.0f;
    for (int i = ilo + lane % w, j = jlo + lane / w; j <= jhi; i += di, j += dj, j += i > ihi, i -= i > ihi ? w : 0) {
        const Ray ray = make_ray<GM_PARALLEL>(g, F, __ldg(g.utab + i), __ldg(g.vtab + j));
        PairGeo q;
        pair_geo(ray, r, q);
        if (!(q.m <= PAIR_CUT2)) continue;
        const long long idx = (long long)view * g.stride_view + (long long)j * g.stride_row + i;
        for (int b = 0; b < (TOF ? g.n_tof : 1); b++) {
            const float gw = __ldg(dLdI + idx + (TOF ? b * g.stride_tof : 0));
            if (gw == 0.0f) continue;
            float pv[NG];
            if (TOF) general_grad<KER>(ray, q, r.g0.w, gw, pv, g.tof_t0 + (float)b * g.tof_h, g.tof_tau);
            else general_grad<KER>(ray, q, r.g0.w, gw, pv);
            for (int k = 0; k < NG; k++) val[k] += pv[k];
        }
    }
    for (int q = 0; q < NG; q++)
        for (int o = 16; o > 0; o >>= 1) val[q] += __shfl_xor_sync(0xffffffffu, val[q], o);
}

// The warp's Gaussians that meet a band, of the n first that lane k's turn names:
// their number << 8 | the one of this lane (0 past them).
__device__ __forceinline__ uint32_t band_list(const int2 *box, uint8_t *list, int turn, int n, Band bd)
{
    const int lane = threadIdx.x & 31;
    const int2 b = box[turn];
    const bool on = lane < n && (b.x & 0xffff) < bd.cb + bd.w && (int)((unsigned)b.x >> 16) >= bd.cb &&
                    (b.y & 0xffff) < bd.rb + bd.h && (int)((unsigned)b.y >> 16) >= bd.rb;
    const uint32_t bal = __ballot_sync(0xffffffffu, on);
    if (on) list[__popc(bal & ((1u << lane) - 1u))] = (uint8_t)turn;
    const uint32_t num = (uint32_t)__popc(bal);
    __syncwarp();
    return num << 8 | (lane < (int)num ? list[lane] : 0u);
}

// Without time of flight a view is mostly one band, and the list out of line
// leaves the walk its registers (PET ring 6.99 -> 6.77 ms; but 13 bins, several
// bands a view, 2.83 -> 3.03, and Epanechnikov, 20,000 on 90 x 256^2, 1.39 -> 1.42:
// those keep it in line).
__device__ __noinline__ uint32_t band_list_call(const int2 *box, uint8_t *list, int turn, int n, Band bd)
{
    return band_list(box, list, turn, n, bd);
}

// views staged by the CTA and its warps' records and moments
template <bool TOF> struct Shared {
    static constexpr int BW = Wide<TOF>::v;
    static constexpr int NM = TOF ? 11 : 7;
    float sg[Cap<TOF>::v];
    float su[BW + 2], sv[BH + 2];
    int4 sbox[2][NW];
    float4 c0[BS], c1[BS], t4[TOF ? BS : 1];
    int2 box[BS];                // the Gaussian's rectangle (packed as k_cull's)
    uint8_t list[NW][32];        // a warp's Gaussians that meet the band
    float mom[BS * NM];
    float acc[16][BS];
};

template <int KER, bool TOF, int LG>
__global__ void __launch_bounds__(BS, TOF ? 5 : 6) k_adjoint(DevGeom g, int nv, int64_t n, int gw, int vper, int max_px,
                                                   const uint32_t *__restrict__ order,
                                                   const float4 *__restrict__ rec,
                                                   const float4 *__restrict__ crec,
                                                   const uint2 *__restrict__ rect,
                                                   const float *__restrict__ dLdI, float4 *__restrict__ grad)
{
    using Sh = Shared<TOF>;
    constexpr int NM = Sh::NM, S = 1 << LG, BW = Sh::BW;
    __shared__ __align__(16) Sh sh;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, wb = 32 * w;
    const int sl = lane & (S - 1), sw = lane >> LG;
    const int64_t slot = ((int64_t)blockIdx.x * NW + w) * gw + lane;
    const bool active = lane < gw && slot < n;
    const uint32_t gid = !active ? 0u : order ? __ldg(order + slot) : (uint32_t)slot;
    const int va = blockIdx.y * vper, vb = min(nv, va + vper);
    const int nb = TOF ? g.n_tof : 1;
#pragma unroll
    for (int q = 0; q < 16; q++) sh.acc[q][threadIdx.x] = 0.0f;
    uint2 rc_next = active && va < vb ? __ldg(rect + (int64_t)va * n + gid) : make_uint2(1u, 1u);
    for (int vl = va; vl < vb; vl++) {
        const uint2 rc = rc_next;
        if (vl + 1 < vb && active) rc_next = __ldg(rect + (int64_t)(vl + 1) * n + gid);
        Box me;
        me.ilo = rc.x & 0xffff; me.ihi = rc.x >> 16; me.jlo = rc.y & 0xffff; me.jhi = rc.y >> 16;
        const int area = box_px(me.ihi - me.ilo + 1, me.jhi - me.jlo + 1);
        const bool vis = active && me.ilo <= me.ihi && area <= max_px;   // (the others: k_adjoint_direct)
        // the rectangle that holds the CTA's boxes
        {
            int4 b;
            b.x = __reduce_min_sync(0xffffffffu, vis ? me.ilo : 0x7fffffff);
            b.y = __reduce_max_sync(0xffffffffu, vis ? me.ihi : -1);
            b.z = __reduce_min_sync(0xffffffffu, vis ? me.jlo : 0x7fffffff);
            b.w = __reduce_max_sync(0xffffffffu, vis ? me.jhi : -1);
            if (lane == 0) sh.sbox[vl & 1][w] = b;
        }
        __syncthreads();   // (also: every thread is done with the previous view's band)
        int4 ub = sh.sbox[vl & 1][0];
#pragma unroll
        for (int k = 1; k < NW; k++) {
            const int4 b = sh.sbox[vl & 1][k];
            ub.x = min(ub.x, b.x); ub.y = max(ub.y, b.y); ub.z = min(ub.z, b.z); ub.w = max(ub.w, b.w);
        }
        if (ub.y < 0) continue;   // no Gaussian of the CTA on the detector
        const int view = g.v0 + vl;
        // this lane's record in the view; a footprint far larger than its
        // warp's others is left to the whole warp instead of one sub-warp
        bool gen = false;
        uint32_t bigs;
        int turn;
        {
            const int mean = (int)(__reduce_add_sync(0xffffffffu, vis ? (unsigned)area : 0u) >> 5);
            const bool big = vis && area > 64 * S && area > 4 * mean;
            bool sat = false;
            if (vis) {
                float F[9];
#pragma unroll
                for (int q = 0; q < 9; q++) F[q] = __ldg(g.frames + 9 * (size_t)view + q);
                VRec r;
                prep_record<GM_PARALLEL, KER>(g, F, gid, rec, crec, r);
                sat = r.g2.w != 0.0f;
                sh.c0[threadIdx.x] = r.c0;
                sh.c1[threadIdx.x] = r.c1;
                if (TOF) sh.t4[threadIdx.x] = r.t4;
            }
            gen = vis && !sat;
            bigs = __ballot_sync(0xffffffffu, big && sat);
            // the warp's Gaussians by the size of their boxes, largest first:
            // sub-warps walk side by side, so those of a round should be alike
            uint32_t key = ((vis && sat ? (uint32_t)area : 0u) << 5) | (uint32_t)lane;
#pragma unroll
            for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
                for (int j = k >> 1; j > 0; j >>= 1) {
                    const uint32_t o = __shfl_xor_sync(0xffffffffu, key, j);
                    const bool lower = (lane & j) == 0, desc = (lane & k) == 0;
                    key = lower == desc ? max(key, o) : min(key, o);
                }
            turn = (int)(key & 31u);
            sh.box[threadIdx.x] = vis && sat ? make_int2((int)rc.x, (int)rc.y) : make_int2(1, 1);
#pragma unroll
            for (int q = 0; q < NM; q++) sh.mom[threadIdx.x * NM + q] = 0.0f;
        }
        const int n_vs = __popc(__ballot_sync(0xffffffffu, vis && !gen));
        Band bd;
        const int uw = ub.y - ub.x + 1, uh = ub.w - ub.z + 1;
        const bool many = uw > BW || uh > BH || uh * ((uw + 1) & ~1) * nb > Cap<TOF>::v;
        for (bd.cb = ub.x; bd.cb <= ub.y; bd.cb += BW) {
            bd.w = min(BW, ub.y - bd.cb + 1);
            bd.st = (bd.w + 1) & ~1;
            const int hmax = min(BH, Cap<TOF>::v / (bd.st * nb));
            for (bd.rb = ub.z; bd.rb <= ub.w; bd.rb += hmax) {
                bd.h = min(hmax, ub.w - bd.rb + 1);
                int now = turn, n_now = n_vs;
                if (many) {
                    // several bands: the Gaussians that meet this one, and no
                    // staging where there is none
                    const uint32_t r = TOF || KER == 1 ? band_list(sh.box + wb, sh.list[w], turn, n_vs, bd)
                                                       : band_list_call(sh.box + wb, sh.list[w], turn, n_vs, bd);
                    n_now = (int)(r >> 8);
                    if (!__syncthreads_or(n_now)) continue;     // (also: every warp is done with the band before)
                    now = (int)(r & 255u);
                }
                // stage dL/dI of the band, a warp taking 1, 2 or 4 rows at a time
                for (int i = threadIdx.x; i < bd.st; i += BS)
                    sh.su[i] = __ldg(g.utab + min(bd.cb + i, g.n_cols - 1));
                for (int j = threadIdx.x; j < bd.h; j += BS) sh.sv[j] = __ldg(g.vtab + bd.rb + j);
                const int sh_ = bd.st <= 8 ? 3 : bd.st <= 16 ? 4 : 5;
                const int lc = lane & ((1 << sh_) - 1), lr = (w << (5 - sh_)) + (lane >> sh_), rstep = NW << (5 - sh_);
                // (time of flight: plane by plane), four loads in flight (PET ring
                // 7.1 -> 6.85 ms against one)
                const int nr = TOF ? nb * bd.h : bd.h;
                const float ih = 1.0f / (float)bd.h;
                for (int c = lc; c < bd.st; c += 1 << sh_) {
                    const float *src = dLdI + (long long)view * g.stride_view + (long long)bd.rb * g.stride_row + (bd.cb + c);
                    for (int j0 = lr; j0 < nr; j0 += 4 * rstep) {
                        float x[4];
#pragma unroll
                        for (int u = 0; u < 4; u++) {
                            const int jj = j0 + u * rstep, b = TOF ? (int)(((float)jj + 0.5f) * ih) : 0;
                            x[u] = 0.0f;
                            if (jj < nr && c < bd.w)
                                x[u] = __ldg(src + (long long)(jj - b * bd.h) * g.stride_row + (TOF ? b * g.stride_tof : 0));
                        }
#pragma unroll
                        for (int u = 0; u < 4; u++)
                            if (j0 + u * rstep < nr) sh.sg[(j0 + u * rstep) * bd.st + c] = x[u];
                    }
                }
                __syncthreads();
                // the sub-warps take the warp's Gaussians in turn ...
                auto take = [&](int k, int l, auto lgc, bool on) {
                    constexpr int L = decltype(lgc)::value;
                    const int2 b = sh.box[wb + k];
                    Box bx;
                    bx.ilo = b.x & 0xffff; bx.ihi = (int)((unsigned)b.x >> 16);
                    bx.jlo = b.y & 0xffff; bx.jhi = (int)((unsigned)b.y >> 16);
                    if (!on) { bx.jlo = 1; bx.jhi = 0; bx.ilo = 1; bx.ihi = 0; }
                    const float4 c0 = sh.c0[wb + k], c1 = sh.c1[wb + k];
                    float m[NM];
                    const Staged src = { sh.sg, sh.su, sh.sv, bd };
                    if constexpr (TOF) rows_tof(g, c0, c1, sh.t4[wb + k], bx, l, 1 << L, src, m);
                    else rows<KER>(g, c0, c1, bx, l, 1 << L, src, m);
                    __syncwarp();
                    reduce_add<NM, L>(m, l, sh.mom + (wb + k) * NM, on);
                };
                __syncwarp();
                {
                    for (int t = 0; t < n_now; t += 32 / S) {
                        const int k = __shfl_sync(0xffffffffu, now, t + sw);
                        take(k, sl, std::integral_constant<int, LG>{}, t + sw < n_now && !((bigs >> k) & 1u));
                    }
                    // ... and the whole warp the big ones
                    for (uint32_t bm = bigs; bm; bm &= bm - 1u)
                        take(__ffs(bm) - 1, lane, std::integral_constant<int, 5>{}, true);
                }
            }
        }
        __syncwarp();
        if (vis && !gen) {
            float m[NM], o[16];
            bool any = false;
#pragma unroll
            for (int q = 0; q < NM; q++) {
                m[q] = sh.mom[threadIdx.x * NM + q];
                any |= m[q] != 0.0f;
            }
            if (any) {
                float F[9];
#pragma unroll
                for (int q = 0; q < 9; q++) F[q] = __ldg(g.frames + 9 * (size_t)view + q);
                const float4 c1 = sh.c1[threadIdx.x];
                float s[12], tof4[4];
                finish<KER>(m, c1.y, c1.z, s);
                if (TOF) {
#pragma unroll
                    for (int q = 0; q < 4; q++) tof4[q] = c1.z * m[TOF ? 7 + q : 0];
                }
                view_chain<GM_PARALLEL, KER>(g, F, rec, gid, s, o, TOF ? tof4 : nullptr);
#pragma unroll
                for (int q = 0; q < 16; q++) sh.acc[q][threadIdx.x] += o[q];
            }
        }
        // Gaussians near a segment end
        uint32_t gm = __ballot_sync(0xffffffffu, gen);
        while (gm) {
            const int owner = __ffs(gm) - 1;
            gm &= gm - 1u;
            float val[NG];
            general_box<KER, TOF>(g, view, rec, __shfl_sync(0xffffffffu, gid, owner),
                                      __shfl_sync(0xffffffffu, me.ilo, owner), __shfl_sync(0xffffffffu, me.ihi, owner),
                                      __shfl_sync(0xffffffffu, me.jlo, owner), __shfl_sync(0xffffffffu, me.jhi, owner),
                                      dLdI, val);
            if (lane == owner) {
                const int slot_of[NG] = { 0, 1, 2, 4, 5, 6, 7, 8, 9, 3 };
#pragma unroll
                for (int q = 0; q < NG; q++) sh.acc[slot_of[q]][threadIdx.x] += val[q];
            }
        }
    }
    if (active) {
        float acc[16];
        bool any = false;
#pragma unroll
        for (int q = 0; q < 16; q++) {
            acc[q] = sh.acc[q][threadIdx.x];
            any |= acc[q] != 0.0f;
        }
        if (any) {
            float4 *gp = grad + GRAD_F4 * (size_t)gid;
#pragma unroll
            for (int q = 0; q < 4; q++)
                atomicAdd(gp + q, make_float4(acc[4 * q], acc[4 * q + 1], acc[4 * q + 2], acc[4 * q + 3]));
        }
    }
}

// The Gaussians whose boxes exceed min_px pixels, dL/dI read in place (no band
// to stage, nothing shared with the neighbours).  A CTA takes 128 Gaussians of a
// view and cuts the boxes into strips of whole rows of about strip_px pixels;
// its warps, and those of the gridDim.z CTAs with the same Gaussians, take the
// strips in equal shares, 32 at a time: lane k prepares strip k's record and
// chains its moments, the whole warp walks each, 8 rows by 8 columns at a step (4
// or 16 rows: 20,000 Gaussians of 150 x 150 px on 8 x 512^2 4.5 and 6.1 ms against
// 4.2).  Bound by issue for large footprints and by latency for few.  Against
// the staged walk, and (last) one Gaussian per thread and tile: 64 of 10^5 px on
// one view 8.1, 0.16, 0.18 ms; 8 of 960 px 0.12, 0.015, 0.014; 1,000 of 23,000
// px on 8 views 0.82, 0.23, 0.26.
template <int KER, bool TOF>
__global__ void __launch_bounds__(BS, TOF ? 3 : 6) k_adjoint_direct(DevGeom g, int nv, int64_t n, int min_px, int strip_px,
                                                                    const float4 *__restrict__ rec,
                                                                    const float4 *__restrict__ crec,
                                                                    const uint2 *__restrict__ rect,
                                                                    const float *__restrict__ dLdI,
                                                                    float4 *__restrict__ grad)
{
    constexpr int NM = TOF ? 11 : 7, ROWS = 32 >> DIRECT_LG;
    __shared__ uint32_t ids[BS], first[BS];      // the view's Gaussians, and the first of their strips
    __shared__ uint2 box[BS], wsum[NW];
    __shared__ float4 sc0[BS], sc1[BS], st4[TOF ? BS : 1];
    __shared__ uint2 strip[BS];
    __shared__ float mom[BS * NM];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, wb = 32 * w;
    const int64_t k = (int64_t)blockIdx.x * BS + threadIdx.x;
    // rows of a strip
    auto rows_of = [&](int wd) { return (max(strip_px / wd, 1) + ROWS - 1) / ROWS * ROWS; };
    for (int vl = blockIdx.y; vl < nv; vl += gridDim.y) {
        const uint2 rc = k < n ? __ldg(rect + (int64_t)vl * n + k) : make_uint2(1u, 1u);
        const int bw = (int)(rc.x >> 16) - (int)(rc.x & 0xffff) + 1, bh = (int)(rc.y >> 16) - (int)(rc.y & 0xffff) + 1;
        const bool on = bw > 0 && box_px(bw, bh) > min_px;
        if (!__syncthreads_or(on)) continue;
        const uint32_t mine = on ? (uint32_t)((bh - 1) / rows_of(bw) + 1) : 0u;
        uint32_t inc = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        const uint32_t bal = __ballot_sync(0xffffffffu, on);
        if (lane == 31) wsum[w] = make_uint2(__popc(bal), inc);
        __syncthreads();
        uint32_t at = __popc(bal & ((1u << lane) - 1u)), num = 0, strips = 0;
        inc -= mine;
#pragma unroll
        for (int q = 0; q < NW; q++) {
            if (q < w) {
                at += wsum[q].x;
                inc += wsum[q].y;
            }
            num += wsum[q].x;
            strips += wsum[q].y;
        }
        if (on) {
            ids[at] = (uint32_t)k;
            box[at] = rc;
            first[at] = inc;
        }
        __syncthreads();
        const int view = g.v0 + vl;
        const float *I = dLdI + (long long)view * g.stride_view;
        float F[9];
#pragma unroll
        for (int q = 0; q < 9; q++) F[q] = __ldg(g.frames + 9 * (size_t)view + q);
        const uint32_t share = blockIdx.z * NW + w, shares = gridDim.z * NW;
        const uint32_t sa = (uint32_t)((uint64_t)strips * share / shares), sb = (uint32_t)((uint64_t)strips * (share + 1) / shares);
        for (uint32_t s0 = sa; s0 < sb; s0 += 32) {
            // lane k: strip s0 + k
            const uint32_t st = s0 + lane;
            const bool vis = st < sb;
            uint32_t gid = 0;
            Box bx = { 1, 0, 1, 0 };
            bool gen = false;
            if (vis) {
                uint32_t e = 0;
                for (uint32_t hi = num - 1; e < hi;) {
                    const uint32_t mid = (e + hi + 1) >> 1;
                    if (first[mid] <= st) e = mid; else hi = mid - 1;
                }
                gid = ids[e];
                const uint2 b = box[e];
                bx.ilo = b.x & 0xffff; bx.ihi = b.x >> 16; bx.jlo = b.y & 0xffff; bx.jhi = b.y >> 16;
                const int per = rows_of(bx.ihi - bx.ilo + 1);
                bx.jlo += (int)(st - first[e]) * per;
                bx.jhi = min(bx.jhi, bx.jlo + per - 1);
                VRec r;
                prep_record<GM_PARALLEL, KER>(g, F, gid, rec, crec, r);
                gen = r.g2.w == 0.0f;
                sc0[threadIdx.x] = r.c0;
                sc1[threadIdx.x] = r.c1;
                if (TOF) st4[threadIdx.x] = r.t4;
            }
            strip[threadIdx.x] = make_uint2((uint32_t)bx.ilo | ((uint32_t)bx.ihi << 16),
                                            (uint32_t)bx.jlo | ((uint32_t)bx.jhi << 16));
#pragma unroll
            for (int q = 0; q < NM; q++) mom[threadIdx.x * NM + q] = 0.0f;
            __syncwarp();
            for (uint32_t m32 = __ballot_sync(0xffffffffu, vis && !gen); m32; m32 &= m32 - 1u) {
                const int t = wb + __ffs(m32) - 1;
                const uint2 b = strip[t];
                Box s;
                s.ilo = b.x & 0xffff; s.ihi = b.x >> 16; s.jlo = b.y & 0xffff; s.jhi = b.y >> 16;
                const Direct src = { g, I, lane & ((1 << DIRECT_LG) - 1) };
                float v[NM];
                if constexpr (TOF) rows_tof(g, sc0[t], sc1[t], st4[t], s, lane >> DIRECT_LG, ROWS, src, v);
                else rows<KER>(g, sc0[t], sc1[t], s, lane >> DIRECT_LG, ROWS, src, v);
                __syncwarp();
                reduce_add<NM, 5>(v, lane, mom + t * NM);
            }
            __syncwarp();
            float o[16];
            bool any = false;
#pragma unroll
            for (int q = 0; q < 16; q++) o[q] = 0.0f;
            if (vis && !gen) {
                float m[NM], sm[12], tof4[4];
#pragma unroll
                for (int q = 0; q < NM; q++) {
                    m[q] = mom[threadIdx.x * NM + q];
                    any |= m[q] != 0.0f;
                }
                const float4 c1 = sc1[threadIdx.x];
                if (any) {
                    finish<KER>(m, c1.y, c1.z, sm);
                    if (TOF) {
#pragma unroll
                        for (int q = 0; q < 4; q++) tof4[q] = c1.z * m[TOF ? 7 + q : 0];
                    }
                    view_chain<GM_PARALLEL, KER>(g, F, rec, gid, sm, o, TOF ? tof4 : nullptr);
                }
            }
            // Gaussians near a segment end
            for (uint32_t gm = __ballot_sync(0xffffffffu, vis && gen); gm; gm &= gm - 1u) {
                const int owner = __ffs(gm) - 1;
                const uint2 b = strip[wb + owner];
                float val[NG];
                general_box<KER, TOF>(g, view, rec, __shfl_sync(0xffffffffu, gid, owner), b.x & 0xffff, b.x >> 16,
                                      b.y & 0xffff, b.y >> 16, dLdI, val);
                if (lane == owner) {
                    const int slot_of[NG] = { 0, 1, 2, 4, 5, 6, 7, 8, 9, 3 };
#pragma unroll
                    for (int q = 0; q < NG; q++) {
                        o[slot_of[q]] = val[q];
                        any |= val[q] != 0.0f;
                    }
                }
            }
            if (any) {
                float4 *gp = grad + GRAD_F4 * (size_t)gid;
#pragma unroll
                for (int q = 0; q < 4; q++)
                    atomicAdd(gp + q, make_float4(o[4 * q], o[4 * q + 1], o[4 * q + 2], o[4 * q + 3]));
            }
            __syncwarp();   // the strips' records are done with
        }
        __syncthreads();   // the list is done before another view's
    }
}

// ---- spatial order ---------------------------------------------------------
//
// The Gaussians sorted by a cell code: the bounding box of the centres is
// halved along whichever axis is then longest until a cell of an evenly filled
// box would hold CELL_N Gaussians, so cells are near cubes and consecutive
// codes lie together.  Within a cell any order will do.
constexpr int CELL_N = 4;
constexpr int CODE_BITS = 15, CELLS = 1 << CODE_BITS;
constexpr int SMALL_BS = 1024, SMALL_BITS = 12, SMALL_N = 16384;

// monotone map of binary32 to u32
__device__ __forceinline__ uint32_t ord_enc(float x)
{
    const uint32_t b = __float_as_uint(x);
    return b & 0x80000000u ? ~b : b | 0x80000000u;
}
__device__ __forceinline__ float ord_dec(uint32_t u)
{
    return __uint_as_float(u & 0x80000000u ? u & 0x7fffffffu : ~u);
}

// box: enc(max) of x, y, z, then ~enc(min) (zeroed buffer = empty)
__device__ __forceinline__ uint32_t cell_code(const float4 *__restrict__ crec, int64_t k, const uint32_t *box, int bits)
{
    const float4 c0 = __ldg(crec + CREC_F4 * k);
    const float m[3] = { c0.x, c0.y, c0.z };
    float e[3], f[3];
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const float hi = ord_dec(box[a]), lo = ord_dec(~box[3 + a]);
        e[a] = hi - lo;
        f[a] = e[a] > 0.0f ? (m[a] - lo) / e[a] : 0.0f;
    }
    uint32_t code = 0;
    for (int b = 0; b < bits; b++) {
        const int a = e[0] >= e[1] && e[0] >= e[2] ? 0 : e[1] >= e[2] ? 1 : 2;
        const float x = 2.0f * (a == 0 ? f[0] : a == 1 ? f[1] : f[2]);
        const uint32_t bit = x >= 1.0f;
        code = (code << 1) | bit;
        const float y = x - (float)bit;
        if (a == 0) { f[0] = y; e[0] *= 0.5f; }
        else if (a == 1) { f[1] = y; e[1] *= 0.5f; }
        else { f[2] = y; e[2] *= 0.5f; }
    }
    return code;
}

__device__ __forceinline__ void box_add(const float *m, uint32_t *b)
{
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const uint32_t u = ord_enc(m[a]);
        b[a] = max(b[a], u);
        b[3 + a] = max(b[3 + a], ~u);
    }
}

__global__ void __launch_bounds__(256) k_order_box(const float4 *__restrict__ crec, int64_t n, uint32_t *box)
{
    __shared__ uint32_t sb[6];
    if (threadIdx.x < 6) sb[threadIdx.x] = 0;
    __syncthreads();
    uint32_t b[6] = { 0, 0, 0, 0, 0, 0 };
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        const float4 c = __ldg(crec + CREC_F4 * k);
        const float m[3] = { c.x, c.y, c.z };
        box_add(m, b);
    }
#pragma unroll
    for (int a = 0; a < 6; a++) {
        b[a] = __reduce_max_sync(0xffffffffu, b[a]);
        if ((threadIdx.x & 31) == 0) atomicMax(&sb[a], b[a]);
    }
    __syncthreads();
    if (threadIdx.x < 6) atomicMax(box + threadIdx.x, sb[threadIdx.x]);
}

// code << 32 | rank within the cell, per Gaussian
__global__ void k_order_cells(const float4 *__restrict__ crec, int64_t n, int bits,
                              const uint32_t *__restrict__ box, uint32_t *__restrict__ cells, uint2 *__restrict__ where)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const uint32_t c = cell_code(crec, k, box, bits);
    where[k] = make_uint2(c, atomicAdd(cells + c, 1u));
}

// exclusive scan of cnt[0..4 V SMALL_BS) in place by one CTA of SMALL_BS
// threads, V 16-byte loads each
template <int V>
__device__ __forceinline__ void cta_scan(uint32_t *cnt, uint32_t *wsum)
{
    uint4 *p = reinterpret_cast<uint4 *>(cnt) + V * threadIdx.x;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint4 q[V];
    uint32_t s = 0;
#pragma unroll
    for (int j = 0; j < V; j++) q[j] = p[j];
#pragma unroll
    for (int j = 0; j < V; j++) s += q[j].x + q[j].y + q[j].z + q[j].w;
    uint32_t inc = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[w] = inc;
    __syncthreads();
    if (w == 0) {
        const uint32_t v = wsum[lane];
        uint32_t x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        wsum[lane] = x - v;
    }
    __syncthreads();
    uint32_t run = wsum[w] + inc - s;
#pragma unroll
    for (int j = 0; j < V; j++) {
        uint4 o;
        o.x = run;
        o.y = o.x + q[j].x;
        o.z = o.y + q[j].y;
        o.w = o.z + q[j].z;
        run = o.w + q[j].w;
        p[j] = o;
    }
}

__global__ void __launch_bounds__(SMALL_BS) k_order_scan(uint32_t *cells)
{
    __shared__ uint32_t wsum[32];
    cta_scan<CELLS / (4 * SMALL_BS)>(cells, wsum);
}

__global__ void k_order_scatter(int64_t n, const uint32_t *__restrict__ cells, const uint2 *__restrict__ where,
                                uint32_t *__restrict__ order)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const uint2 p = where[k];
    order[cells[p.x] + p.y] = (uint32_t)k;
}

// the whole order by one CTA: small sets, where the launches would dominate
__global__ void __launch_bounds__(SMALL_BS) k_order_small(const float4 *__restrict__ crec, int n, int bits,
                                                          uint32_t *order)
{
    __shared__ __align__(16) uint32_t cells[1 << SMALL_BITS];
    __shared__ uint32_t wsum[32], box[6];
    for (int k = threadIdx.x; k < (1 << SMALL_BITS); k += SMALL_BS) cells[k] = 0;
    if (threadIdx.x < 6) box[threadIdx.x] = 0;
    __syncthreads();
    uint32_t b[6] = { 0, 0, 0, 0, 0, 0 };
    for (int k = threadIdx.x; k < n; k += SMALL_BS) {
        const float4 c = __ldg(crec + CREC_F4 * k);
        const float m[3] = { c.x, c.y, c.z };
        box_add(m, b);
    }
#pragma unroll
    for (int a = 0; a < 6; a++) {
        b[a] = __reduce_max_sync(0xffffffffu, b[a]);
        if ((threadIdx.x & 31) == 0) atomicMax(&box[a], b[a]);
    }
    __syncthreads();
    constexpr int PER = SMALL_N / SMALL_BS;
    uint32_t code[PER], rank[PER];
#pragma unroll
    for (int q = 0; q < PER; q++) {
        const int k = threadIdx.x + q * SMALL_BS;
        if (k >= n) break;
        code[q] = cell_code(crec, k, box, bits);
        rank[q] = atomicAdd(&cells[code[q]], 1u);
    }
    __syncthreads();
    cta_scan<(1 << SMALL_BITS) / (4 * SMALL_BS)>(cells, wsum);
    __syncthreads();
#pragma unroll
    for (int q = 0; q < PER; q++) {
        const int k = threadIdx.x + q * SMALL_BS;
        if (k < n) order[cells[code[q]] + rank[q]] = (uint32_t)k;
    }
}

}  // namespace

size_t order_tmp_bytes(int64_t n)
{
    return n <= SMALL_N ? 16 : sizeof(uint2) * (size_t)n + sizeof(uint32_t) * (CELLS + 8);
}

cudaError_t launch_order(const float4 *crec, int64_t n, void *tmp, uint32_t *order, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    const int most = n <= SMALL_N ? SMALL_BITS : CODE_BITS;
    int bits = 0;
    while (bits < most && (n >> bits) > CELL_N) bits++;
    if (n <= SMALL_N) {
        k_order_small<<<1, SMALL_BS, 0, s>>>(crec, (int)n, bits, order);
        count_launches(1);
        return cudaGetLastError();
    }
    // the counters first: they are read as 16-byte vectors
    uint32_t *cells = (uint32_t *)tmp, *box = cells + CELLS;
    uint2 *where = (uint2 *)(box + 8);
    cudaError_t e = cudaMemsetAsync(cells, 0, sizeof(uint32_t) * (CELLS + 6), s);
    if (e != cudaSuccess) return e;
    const unsigned nb = (unsigned)((n + 255) / 256);
    const unsigned sms = (unsigned)sm_count();
    k_order_box<<<nb < sms ? nb : sms, 256, 0, s>>>(crec, n, box);
    k_order_cells<<<nb, 256, 0, s>>>(crec, n, bits, box, cells, where);
    k_order_scan<<<1, SMALL_BS, 0, s>>>(cells);
    k_order_scatter<<<nb, 256, 0, s>>>(n, cells, where, order);
    count_launches(4);
    return cudaGetLastError();
}

namespace {

// average footprint of a launch in pixels, from its tile entries per (view,
// Gaussian): a w x w box lands on about (1 + w / tile)^2 tiles
double footprint_px(const DevGeom &g, int nv, int64_t n, int64_t entries)
{
    const double per = (double)entries / ((double)nv * (double)n);
    const double side = per > 1.0 ? sqrt(per) - 1.0 : 0.0;
    return side * side * g.tile_w * g.tile_h;
}

template <int KER, bool TOF>
void adjoint_staged_launch(double px, int max_px, const DevGeom &g, int nv, int64_t n, const uint32_t *order,
                           const float4 *rec, const float4 *crec, const uint2 *rect, const float *dLdI, float4 *grad,
                           cudaStream_t s)
{
    // Gaussians per warp: fewer where 32 would leave the GPU short of CTAs (10 per SM)
    const int64_t sms = sm_count();
    int gw = 32;
    while (gw > 2 && (n / (gw * NW)) * nv < sms * 10) gw >>= 1;
    const int64_t bx = (n + NW * gw - 1) / (NW * gw);
    int64_t chunks = (sms * 5 * 12 + bx - 1) / bx;
    if (chunks > nv) chunks = nv;
    if (chunks > 65535) chunks = 65535;
    const int vper = (int)((nv + chunks - 1) / chunks);
    const dim3 grid((unsigned)bx, (unsigned)((nv + vper - 1) / vper));
    // lanes per Gaussian: measured 2 / 4 / 8 lanes at 36 px (PET ring) 6.9 / 7.2 /
    // 8.4 ms, at 65 px (raw PET) 0.143 / 0.143 / 0.163, at 180 px (20,000 on 90 x
    // 256^2) 4 / 8 lanes 0.706 / 0.744, at 5,900 px 10.9 / 10.65
    const int lg = px > 80.0 ? 2 : 1;
#define RGRT_ADJ(L) k_adjoint<KER, TOF, L><<<grid, BS, 0, s>>>(g, nv, n, gw, vper, max_px, order, rec, crec, rect, dLdI, grad)
    if (lg == 1) RGRT_ADJ(1);
    else RGRT_ADJ(2);
#undef RGRT_ADJ
    count_launches(1);
}

template <int KER, bool TOF>
void adjoint_direct_launch(double px, int min_px, const DevGeom &g, int nv, int64_t n, const float4 *rec,
                           const float4 *crec, const uint2 *rect, const float *dLdI, float4 *grad, cudaStream_t s)
{
    // CTAs for a few waves, each looking through the boxes of several views; where
    // the Gaussians are too few for that, several share a set's strips
    const int64_t sms = sm_count(), bx = (n + BS - 1) / BS;
    int64_t by = (sms * 48 + bx - 1) / bx;
    if (by > nv) by = nv;
    if (by > 65535) by = 65535;
    // strips for about 64 warps per SM
    const double pairs = (double)n * (double)nv, strip = px * pairs / (64.0 * (double)sms);
    const int strip_px = strip < 256.0 ? 256 : strip > 4096.0 ? 4096 : (int)strip;
    const double most = pairs * (1.0 + px / strip_px) / (double)(bx * by * NW * 4);   // four strips a warp
    int64_t z = sms * 40 / (bx * by);
    if (z > (int64_t)most) z = (int64_t)most;
    z = z < 1 ? 1 : z;
    const dim3 grid((unsigned)bx, (unsigned)by, (unsigned)z);
    k_adjoint_direct<KER, TOF><<<grid, BS, 0, s>>>(g, nv, n, min_px, strip_px, rec, crec, rect, dLdI, grad);
    count_launches(1);
}

}  // namespace

// k_adjoint needs enough (view, Gaussian) pairs that neighbours share bands and
// the CTAs that hold far-apart Gaussians are a small part; below that every pair
// goes to k_adjoint_direct, whose cost is its own pixels.  Measured staged /
// direct: 64 Gaussians on one view of 512^2 0.15 / 0.01 ms, 16,000 pairs of 470
// px 0.088 / 0.068, 90,000 of 180 px 0.16 / 0.095, 160,000 of 960 px 0.38 / 0.29;
// 200,000 of 75 px 2.5 / 3.7 (a batch's step), 800,000 of 65 px 0.14 / 0.73.
bool adjoint_staged(const DevGeom &g, int nv, int64_t n, int64_t entries)
{
    const int64_t pairs = n * nv;
    return pairs > 262144 || (pairs > 32768 && footprint_px(g, nv, n, entries) <= 200.0);
}

cudaError_t launch_adjoint(const DevGeom &g, int nv, int64_t n, int64_t entries, bool large, const uint32_t *order,
                           const float4 *rec, const float4 *crec, const uint2 *rect, const float *dLdI,
                           float4 *grad, int ker, cudaStream_t s)
{
    if (nv <= 0 || n <= 0) return cudaSuccess;
    const double px = footprint_px(g, nv, n, entries);
    const bool staged = adjoint_staged(g, nv, n, entries);
    // Footprints beyond max_px are walked in place: staged, each would take band
    // after band of its CTA's union.  2,048 px: 50,000 Gaussians of 50 px and 100
    // of 10^4 px on 90 x 256^2 11.5 -> 4.4 ms, log-sizes with a deviation of 1.0
    // 4.9 -> 3.0 (1,024 px 2.9, 4,096 3.0), a PET ring with 0.7 15.3 -> 14.5;
    // where the average is itself larger, up to four times that, eight times
    // (20,000 of 5,900 px: 12.8 ms at 2,048 px, 10.0 at 8,192, 8.9 at 16,384; of
    // 23,000 px 4.3, 4.3 and 4.7).
    const bool alike = px > ADJOINT_LARGE_PX && px <= 4 * ADJOINT_LARGE_PX;
    const int max_px = !staged ? 0 : alike ? 8 * ADJOINT_LARGE_PX : ADJOINT_LARGE_PX;
#define RGRT_ADJ(K, T)                                                                                          \
    {                                                                                                           \
        if (staged) adjoint_staged_launch<K, T>(px, max_px, g, nv, n, order, rec, crec, rect, dLdI, grad, s);   \
        if (!staged || large) adjoint_direct_launch<K, T>(px, max_px, g, nv, n, rec, crec, rect, dLdI, grad, s); \
    }
    // time of flight: PET ring, Gaussian kernel (checked by the caller)
    if (g.n_tof > 0) RGRT_ADJ(0, true)
    else if (ker == 1) RGRT_ADJ(1, false)
    else RGRT_ADJ(0, false)
#undef RGRT_ADJ
    return cudaGetLastError();
}

}  // namespace rgrt
