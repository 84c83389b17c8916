// Adjoint of the cone-beam and fully 3-D PET geometries, tile by tile (a5).
// (Parallel rays walk Gaussian by Gaussian instead, adjoint.cu.  Measured that
// way too, the cone beam gained little -- its footprints span several tiles,
// so its cost is the pixels -- and 3-D PET nothing.)
//
// Adjoint, one Gaussian per thread.  A CTA takes a tile: it stages the
// tile's dL/dI (times |d~| for cone beam) and pixel coordinates in shared
// memory, then every thread walks the tile's rays for one Gaussian of the
// list at a time (all lanes of a warp read the same ray: broadcasts), keeping
// that Gaussian's view-space moments in registers -- no cross-thread
// reduction -- and finishes with the parameter chain and one set of vector
// atomics per (Gaussian, tile).  On the cone beam the tile list is ordered by
// footprint position, so the 32 Gaussians of a warp sit close together: rows and
// 4-column groups that none of their boxes touches are skipped.  Within a row
// the Q and A quadratics are evaluated in Horner form in du with the dv terms
// hoisted.  For 3-D PET the LOR slope kappa varies from column to column:
// the moments carry its powers (pet3d_chain).
#include "packed.cuh"
#include "view.cuh"

namespace rgrt {
namespace {

constexpr int ADJ_BS = 128;       // threads of a CTA (one Gaussian each)
constexpr int NV_CONE = 12;       // view-space moments, cone beam
// A tile's list is shared by up to 16 CTAs while the launch has fewer CTAs than
// SPLIT_CTAS and a share of an average list stays above SPLIT_LIST entries
// (the sums go to the accumulator by atomics either way).  Measured without
// and with it: 8 cone-beam views of 256^2 (2,048 tiles of 1,270 entries, a few
// of them several times longer) 0.815 -> 0.54 ms, 7 views of 201 x 333 0.50 ->
// 0.39 ms; 180 views (46,080 tiles, one CTA each) 10.2 ms.
constexpr int64_t SPLIT_CTAS = 16384, SPLIT_LIST = 128;

// indices [lo, hi] of the m increasing table values within [a, b]
__device__ __forceinline__ void tile_span(float a, float b, const float *tab, int m, float inv, int &lo, int &hi)
{
    if (inv != 0.0f) {
        const float x = (a - tab[0]) * inv, y = (b - tab[0]) * inv;
        lo = (int)ceilf(fminf(fmaxf(x - 0.02f, 0.0f), (float)m));
        hi = (int)floorf(fmaxf(fminf(y + 0.02f, (float)(m - 1)), -1.0f));
        return;
    }
    for (int j = 0; j < m; j++) {
        const bool in = tab[j] >= a && tab[j] <= b;
        lo = in && j < lo ? j : lo;
        hi = in ? j : hi;
    }
}

template <int GM, int TW, int KER>
__device__ __forceinline__ void adjoint_tile(const DevGeom &g, uint32_t tile, uint32_t part, uint32_t parts,
                                             const float4 *__restrict__ rec,
                                             const float4 *__restrict__ crec,
                                             const uint32_t *__restrict__ gids,
                                             const uint2 *__restrict__ ranges,
                                             const float *__restrict__ dLdI,
                                             float4 *__restrict__ grad)
{
    constexpr bool CONE = GM == GM_CONE, P3 = GM == GM_PET3D;
    // dL/dI |d~| of the tile's rays, row-major (0 outside the detector)
    __shared__ float sgl[P3 ? 256 + 32 : 256];   // (3-D PET: and a row of zeros below)
    __shared__ float su[32], svr[P3 ? 33 : 32];
    __shared__ float skap[P3 ? 32 : 1];   // 3-D PET: LOR slope of every column
    __shared__ float Fs[9];
    const int T = g.tiles_x * g.tiles_y;
    const int vl = (int)(tile / (uint32_t)T);
    const int tin = (int)tile - vl * T;
    const int ty = tin / g.tiles_x, tx = tin - ty * g.tiles_x;
    const int view = g.v0 + vl;
    const int TH = g.tile_h;
    const int c0 = tx * TW, r0 = ty * TH;
    float zoff = 0.0f, dz = 0.0f, kap0 = 0.0f, kap1 = 0.0f;
    int rows = g.n_rows;
    if (P3) {
        pet3d_view(g, view, zoff, dz, rows);
        pet3d_slopes(g, dz, c0, min(c0 + TW - 1, g.n_cols - 1), kap0, kap1);
    }
    if (threadIdx.x < 9) Fs[threadIdx.x] = __ldg(g.frames + 9 * (size_t)view + threadIdx.x);
    if (threadIdx.x < TW) {
        su[threadIdx.x] = __ldg(g.utab + min(c0 + (int)threadIdx.x, g.n_cols - 1));
        if (P3) skap[threadIdx.x] = pet3d_slope(g, dz, su[threadIdx.x]);
    }
    if (P3) {
        if (threadIdx.x == 0) svr[TH] = 0.0f;
        if (threadIdx.x < TW) sgl[TW * TH + threadIdx.x] = 0.0f;
    }
    if (threadIdx.x < TH) svr[threadIdx.x] = __ldg(g.vtab + min(r0 + (int)threadIdx.x, g.n_rows - 1)) + zoff;
    for (int r = threadIdx.x; r < TW * TH; r += blockDim.x) {
        const int col = c0 + r % TW, row = r0 + r / TW;
        float gl = 0.0f;
        if (col < g.n_cols && row < rows) {
            const long long idx = (long long)view * g.stride_view + (long long)row * g.stride_row + col;
            gl = __ldg(dLdI + idx);
            if (CONE) {
                const float u = __ldg(g.utab + col), v = __ldg(g.vtab + row);
                gl *= sqrtf(u * u + v * v + g.dsd * g.dsd);
            }
            if (P3) {
                const float kap = pet3d_slope(g, dz, __ldg(g.utab + col));
                gl *= sqrtf(1.0f + kap * kap);
            }
        }
        sgl[r] = gl;
    }
    __syncthreads();
    float F[9];
#pragma unroll
    for (int i = 0; i < 9; i++) F[i] = Fs[i];
    const uint2 rg = ranges[tile];
    // every lane of a warp runs the same number of rounds (inactive lanes idle)
    const uint32_t n = rg.y - rg.x;
    const uint32_t all = (n + blockDim.x - 1) / blockDim.x;
    const uint32_t rounds = (uint32_t)((uint64_t)all * (part + 1) / parts);
    for (uint32_t rd = (uint32_t)((uint64_t)all * part / parts); rd < rounds; rd++) {
        const uint32_t k = rg.x + rd * blockDim.x + threadIdx.x;
        const bool active = k < rg.y;
        VRec r;
        uint32_t gid = 0;
        if (active) {
            gid = __ldg(gids + k);
            prep_record<GM, KER>(g, F, gid, rec, crec, r, kap0, kap1);
        } else {
            r.bb = make_float4(INFINITY, -INFINITY, INFINITY, -INFINITY);
            r.g2 = make_float4(0.0f, 0.0f, 0.0f, 1.0f);
        }
        const float4 bb = r.bb;
        const bool vs = r.g2.w != 0.0f;
        // the Gaussian's box in tile pixels (rows jlo..jhi, columns ilo..ihi)
        int jlo = TH, jhi = -1, ilo = TW, ihi = -1;
        if (P3) {
            tile_span(bb.z, bb.w, svr, TH, g.vinv, jlo, jhi);
            tile_span(bb.x, bb.y, su, TW, g.uinv, ilo, ihi);
        }
        for (int j = 0; j < (P3 ? 0 : TH); j++) {
            const bool in = svr[j] >= bb.z && svr[j] <= bb.w;
            jlo = in && j < jlo ? j : jlo;
            jhi = in ? j : jhi;
        }
#pragma unroll
        for (int i = 0; i < (P3 ? 0 : TW); i++) {
            const bool in = su[i] >= bb.x && su[i] <= bb.y;
            ilo = in && i < ilo ? i : ilo;
            ihi = in ? i : ihi;
        }
        // 4-column groups of the tile the box touches (cone beam)
        uint32_t groups4 = 0;
        if (ilo <= ihi) groups4 = (2u << (ihi >> 2)) - (1u << (ilo >> 2));
        float o[16];
        bool any = false;
        if (!P3 && __any_sync(0xffffffffu, active && vs)) {
            // view-space moments (see view_chain for their meaning)
            const float u0 = r.c0.x, v0 = r.c0.y, kMuu = r.c0.z, kMuv2 = r.c0.w, kMvv = r.c1.x;
            float s[NV_CONE];
#pragma unroll
            for (int q = 0; q < NV_CONE; q++) s[q] = 0.0f;
            for (int j = 0; j < TH; j++) {
                const float vj = svr[j];
                const bool rowin = active && vs && j >= jlo && j <= jhi;
                // rows and 4-column groups that no Gaussian of the warp touches
                // are skipped (the lists are ordered by footprint position, so
                // a warp's Gaussians sit close together in the tile)
                const uint32_t need = __reduce_or_sync(0xffffffffu, rowin ? groups4 : 0u);
                if (need == 0u || !rowin) continue;
                const float dv = vj - v0, dv2 = dv * dv;
                const float a1 = kMuv2 * dv, a0 = kMvv * dv2;
                const float b2 = r.c2.x;
                const float b1 = r.c1.z + r.c2.y * dv;
                const float b0 = r.c1.y + r.c1.w * dv + r.c2.z * dv2;
                float H0 = 0.0f, H1 = 0.0f, H2 = 0.0f, G0 = 0.0f, G1 = 0.0f, G2 = 0.0f, Sw = 0.0f;
                const float *gl_row = sgl + j * TW;
                auto pixel = [&](int i) {
                    const float du = su[i] - u0;
                    const float qv = (kMuu * du + a1) * du + a0;
                    const float A = (b2 * du + b1) * du + b0;
                    const float rA = rsqrt_approx(A);
                    const float iA = rA * rA;
                    const float arg = qv * iA;
                    float wv, h, gA;
                    if (KER == 1) {
                        // f = alpha A^-1/2 c^3/2, c = 1 - Q/(kappa^2 A): -dL/dQ / alpha =
                        // 1.5 w rA iA sqrt(c) / kappa^2, dL/dA / alpha = w rA iA sqrt(c) (1.5 - 2c)
                        const float c = 1.0f + arg;
                        const float sc = c > 0.0f ? sqrt_approx(c) : 0.0f;
                        const float t = (c > 0.0f ? gl_row[i] : 0.0f) * rA * sc;
                        wv = t * c;
                        h = (1.5f / Kern<1>::KAPPA2) * t * iA;
                        gA = t * iA * (1.5f - 2.0f * c);
                    } else {
                        wv = arg >= CUT_ARG ? gl_row[i] * rA * ex2_approx(arg) : 0.0f;
                        h = 0.5f * wv * iA;
                        gA = h * (arg * M_PER_ARG - 1.0f);
                    }
                    const float hd = h * du, gd = gA * du;
                    H0 += h; H1 += hd; H2 += hd * du;
                    G0 += gA; G1 += gd; G2 += gd * du;
                    Sw += wv;
                };
                // 4-column groups that some Gaussian of the warp needs
#pragma unroll
                for (int c4 = 0; c4 < TW / 4; c4++) {
                    if (!((need >> c4) & 1u)) continue;
#pragma unroll
                    for (int i = 4 * c4; i < 4 * c4 + 4; i++) pixel(i);
                }
                // dL/dQ = -h:  SQ_x = -sum h x ;  SA_x = sum gA x
                s[0] -= H1;
                s[1] -= H0 * dv;
                s[2] -= H2;
                s[3] -= H1 * dv;
                s[4] -= H0 * dv2;
                s[5] += G0;
                s[6] += G1;
                s[7] += G0 * dv;
                s[8] += G2;
                s[9] += G1 * dv;
                s[10] += G0 * dv2;
                s[11] += Sw;
            }
            if (active && vs) {
#pragma unroll
                for (int q = 0; q < NV_CONE; q++) any |= s[q] != 0.0f;
                if (any) view_chain<GM, KER>(g, F, rec, gid, s, o);
            }
        }
        if (P3 && __any_sync(0xffffffffu, active && vs)) {
            // every lane its own box, columns outer: the LOR slope kappa is
            // fixed along a column, so the column's kappa terms are taken once
            // and its rows, two at a time in packed binary32, need only five
            // kappa-free sums (h, h v~, h v~^2, p = h arg), folded into the 15
            // moments with the column's du and kappa powers afterwards.  (The
            // list's order by box size keeps the loops of a warp alike: 54.9 ms
            // on 3-D PET of 200,000 Gaussians and 33 million bins, 59.4 ordered
            // by position; walking the union of a warp's boxes in step, row by
            // row, took 76.7.)
            const float4 c0 = r.c0, c1 = r.c1, c2 = r.c2;
            float s[15];
#pragma unroll
            for (int q = 0; q < 15; q++) s[q] = 0.0f;
            const f2 Cvv = pk(c0.w, c0.w);
            const int ie = active && vs && jlo <= jhi ? ihi : -1;
#pragma unroll 1
            for (int i = ilo; i <= ie; i++) {
                const float du = su[i] - c0.x, kap = skap[i];
                const float muu = fmaf(fmaf(c1.z, kap, c1.y), kap, c1.x);
                const float muv2 = fmaf(c2.x, kap, c1.w);
                const float rA = rsqrt_approx(fmaf(fmaf(c2.z, kap, c2.y), kap, 1.0f));
                const float iA = rA * rA;
                const float Kq = muu * du * du, Lq = muv2 * du;
                const float vt0 = fmaf(kap, c0.z, -c0.y);     // v~ = v + vt0
                const f2 VT0 = pk(vt0, vt0), LQ = pk(Lq, Lq), KQ = pk(Kq, Kq), IA = pk(iA, iA);
                f2 h0 = 0, hv = 0, hvv = 0, p0 = 0;
                const float *gc = sgl + i;
                // the rows' values past a box's last row are the tile's own or
                // zero (sgl has a row of padding): pixels outside the footprint
                // add nothing
#pragma unroll 1
                for (int j = jlo; j <= jhi; j += 2) {
                    const f2 vt = add2(pk(svr[j], svr[j + 1]), VT0);
                    float g0 = gc[j * TW], g1 = gc[(j + 1) * TW];
                    // du (muu du + muv2 v~) + S_uu v~^2
                    const f2 q = mul2(fma2(fma2(Cvv, vt, LQ), vt, KQ), IA);
                    float q0, q1, e0, e1;
                    up(q, q0, q1);
                    // the cut acts on g: an infinite or NaN g outside it adds nothing
                    if (KER == 1) {
                        const float x0 = 1.0f + q0, x1 = 1.0f + q1;
                        g0 = x0 > 0.0f ? g0 : 0.0f;
                        g1 = x1 > 0.0f ? g1 : 0.0f;
                        e0 = x0 > 0.0f ? sqrt_approx(x0) : 0.0f;
                        e1 = x1 > 0.0f ? sqrt_approx(x1) : 0.0f;
                    } else {
                        g0 = q0 >= CUT_ARG ? g0 : 0.0f;
                        g1 = q1 >= CUT_ARG ? g1 : 0.0f;
                        e0 = ex2_approx(q0);
                        e1 = ex2_approx(q1);
                    }
                    const f2 h = mul2(pk(g0, g1), pk(e0, e1));
                    const f2 hd = mul2(h, vt);
                    h0 = add2(h0, h);
                    hv = add2(hv, hd);
                    hvv = fma2(hd, vt, hvv);
                    p0 = fma2(h, q, p0);
                }
                // per unit alpha: base = rA h, -dL/dQ = FQ iA base, dL/dA =
                // iA base (FP arg - 1/2)
                constexpr float FQ = KER == 1 ? 1.5f / Kern<1>::KAPPA2 : 0.5f, FP = KER == 1 ? -2.0f : 0.5f * M_PER_ARG;
                const float b0 = hadd(h0), bp = hadd(p0), ra = rA * iA, fq = FQ * ra;
                const float H0 = fq * b0, Hv = fq * hadd(hv), Hvv = fq * hadd(hvv), G0 = ra * (FP * bp - 0.5f * b0);
                const float hd = H0 * du, hvd = Hv * du, kk = kap * kap;
                s[0] += Hvv;
                s[1] += hvd;
                s[2] = fmaf(kap, hvd, s[2]);
                s[3] = fmaf(hd, du, s[3]);
                s[4] = fmaf(kap * hd, du, s[4]);
                s[5] = fmaf(kk * hd, du, s[5]);
                s[6] += Hv;
                s[7] = fmaf(kap, Hv, s[7]);
                s[8] += hd;
                s[9] = fmaf(kap, hd, s[9]);
                s[10] = fmaf(kk, hd, s[10]);
                s[11] += G0;
                s[12] = fmaf(kap, G0, s[12]);
                s[13] = fmaf(kk, G0, s[13]);
                s[14] += rA * (KER == 1 ? b0 + bp : b0);
            }
            __syncwarp();
            if (active && vs) {
#pragma unroll
                for (int q = 0; q < 15; q++) any |= s[q] != 0.0f;
                if (any) pet3d_chain<KER>(F, rec, gid, s, o);
            }
        }
        if (__any_sync(0xffffffffu, active && !vs)) {
            float val[NG];
#pragma unroll
            for (int q = 0; q < NG; q++) val[q] = 0.0f;
            if (active && !vs) {
                for (int j = jlo; j <= jhi; j++) {
                    const float vj = svr[j];
                    for (int i = ilo; i <= ihi; i++) {
                        const float gw0 = sgl[j * TW + i];
                        if (gw0 == 0.0f) continue;
                        const float u = su[i];
                        const Ray ray = make_ray<GM>(g, F, u, vj, P3 ? skap[i] : 0.0f);
                        PairGeo q;
                        pair_geo(ray, r, q);
                        if (!(q.m <= PAIR_CUT2)) continue;
                        // sgl holds dL/dI |d~|; the general form wants dL/dI
                        const float gw = CONE ? gw0 * rsqrtf(u * u + vj * vj + g.dsd * g.dsd)
                                       : P3 ? gw0 * rsqrtf(1.0f + skap[i] * skap[i]) : gw0;
                        float pv[NG];
                        general_grad<KER>(ray, q, r.g0.w, gw, pv);
#pragma unroll
                        for (int qq = 0; qq < NG; qq++) val[qq] += pv[qq];
                    }
                }
#pragma unroll
                for (int q = 0; q < NG; q++) any |= val[q] != 0.0f;
                o[0] = val[0]; o[1] = val[1]; o[2] = val[2]; o[3] = val[9];
                o[4] = val[3]; o[5] = val[4]; o[6] = val[5]; o[7] = val[6];
                o[8] = val[7]; o[9] = val[8];
#pragma unroll
                for (int q = 10; q < 16; q++) o[q] = 0.0f;
            }
        }
        if (active && any) {
            float4 *gp = grad + GRAD_F4 * (size_t)gid;
            atomicAdd(gp, make_float4(o[0], o[1], o[2], o[3]));
            atomicAdd(gp + 1, make_float4(o[4], o[5], o[6], o[7]));
            atomicAdd(gp + 2, make_float4(o[8], o[9], o[10], o[11]));
            if (vs) atomicAdd(gp + 3, make_float4(o[12], o[13], o[14], o[15]));
        }
    }
}

// 3-D PET: 5 CTAs per SM (4: 64.3 ms, 6 with spills: 70.2); the cone-beam kernel's
// registers are the compiler's own choice
template <int TW, int KER>
__global__ void __launch_bounds__(ADJ_BS) k_adjoint(DevGeom g, uint32_t parts, const float4 *__restrict__ rec,
                                                 const float4 *__restrict__ crec,
                                                 const uint32_t *__restrict__ gids,
                                                 const uint2 *__restrict__ ranges,
                                                 const float *__restrict__ dLdI,
                                                 float4 *__restrict__ grad)
{
    adjoint_tile<GM_CONE, TW, KER>(g, blockIdx.x / parts, blockIdx.x % parts, parts, rec, crec, gids, ranges, dLdI, grad);
}

template <int TW, int KER>
__global__ void __launch_bounds__(ADJ_BS, 5) k_adjoint_pet3d(DevGeom g, uint32_t parts, const float4 *__restrict__ rec,
                                                 const float4 *__restrict__ crec,
                                                 const uint32_t *__restrict__ gids,
                                                 const uint2 *__restrict__ ranges,
                                                 const float *__restrict__ dLdI,
                                                 float4 *__restrict__ grad)
{
    adjoint_tile<GM_PET3D, TW, KER>(g, blockIdx.x / parts, blockIdx.x % parts, parts, rec, crec, gids, ranges, dLdI, grad);
}

// Persistent form over a batch of cone-beam scans: every CTA takes (scan,
// tile) work items from an atomic counter until all are done (next_item).
template <int TW>
__global__ void __launch_bounds__(ADJ_BS) k_adjoint_persistent(const ScanDesc *__restrict__ d, int nscan,
                                                              uint32_t total, uint32_t *queue)
{
    uint32_t item;
    int scan;
    while (next_item(d, nscan, total, queue, item, scan)) {
        const ScanDesc &sd = d[scan];
        adjoint_tile<GM_CONE, TW, 0>(sd.g, item - sd.item_begin, 0, 1, sd.rec, sd.crec, sd.gids, sd.ranges,
                               sd.dLdI, sd.grad);
    }
}

}  // namespace

cudaError_t launch_adjoint_persistent(int tile_w, const ScanDesc *d, int nscan, uint32_t total, uint32_t *queue,
                                      cudaStream_t s)
{
    if (total == 0) return cudaSuccess;
#define RGRT_ADJP(TW) k_adjoint_persistent<TW><<<grid_for(k_adjoint_persistent<TW>, ADJ_BS), ADJ_BS, 0, s>>>(d, nscan, total, queue)
    if (tile_w == 8) RGRT_ADJP(8);
    else if (tile_w == 16) RGRT_ADJP(16);
    else RGRT_ADJP(32);
#undef RGRT_ADJP
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_adjoint_tiles(const DevGeom &g, int nv, int64_t entries, const float4 *rec, const float4 *crec,
                                 const uint32_t *gids, const uint2 *ranges, const float *dLdI, float4 *grad,
                                 int ker, cudaStream_t s)
{
    const int64_t nt = (int64_t)nv * g.tiles_x * g.tiles_y;
    if (nt <= 0) return cudaSuccess;
    uint32_t parts = 1;
    while (parts < 16 && nt * parts < SPLIT_CTAS && entries / (nt * parts) >= SPLIT_LIST) parts *= 2;
#define RGRT_ADJ(M, TW, K) M<TW, K><<<(unsigned)(nt * parts), ADJ_BS, 0, s>>>(g, parts, rec, crec, gids, ranges, dLdI, grad)
#define RGRT_ADJ_W(M, K)                                      \
    {                                                         \
        if (g.tile_w == 8) RGRT_ADJ(M, 8, K);                 \
        else if (g.tile_w == 16) RGRT_ADJ(M, 16, K);          \
        else RGRT_ADJ(M, 32, K);                              \
    }
#define RGRT_ADJ_K(K) if (g.kind == GM_CONE) RGRT_ADJ_W(k_adjoint, K) else RGRT_ADJ_W(k_adjoint_pet3d, K)
    if (ker == 1) { RGRT_ADJ_K(1) } else { RGRT_ADJ_K(0) }
#undef RGRT_ADJ_K
#undef RGRT_ADJ_W
#undef RGRT_ADJ
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace rgrt
