// Per-tile ray integration (a3).
//
// One CTA per detector tile of tile_w x tile_h rays, one ray per thread,
// warps laid out as 8 x 4 ray blocks.  The tile's Gaussian list (ordered by
// footprint position, then id) is walked in chunks: the CTA gathers each
// chunk's records, turning every Gaussian into its view-space form for this
// view (see below) together with its detector bounding box, into one of two
// shared-memory buffers.  A warp skips a Gaussian whose box misses its 8 x 4
// block, or (cone beam) whose footprint ellipse misses it (a warp-uniform
// branch); otherwise every lane evaluates its pair and the pair counts when
// m <= 9 (3-sigma cut).  FP32 throughout, FP32 accumulation per ray.
// 3-D PET LORs (direction e_w + kappa e_v, kappa per detector column) have a
// view-space form of their own (prep_record, pet3d_chain).
//
// The closed form (Eqs. 7-11) for a ray and one Gaussian is
//   rho sqrt(2 pi / A) exp(-m/2),  A = d^T P d,  m = C - B^2/A,
// with unit d.  Two exact rewritings make the per-pair work small:
//  * m does not depend on the length of d, and
//      A C - B^2 = (d x delta)^T cof(P) (d x delta),  cof(P) = Sigma / det Sigma,
//    so m = Q / A with Q = c^T S c, c = d x delta, S = Sigma / det Sigma.
//  * In the frame (e_u, e_v, e_w) of a view every ray is fixed by its
//    detector coordinates (u, v).  For parallel rays (CT parallel beam, PET)
//    d = e_w: A = P'_ww is a per-(Gaussian, view) constant and
//    c = du e_v - dv e_u with (du, dv) = (u - mu_u, v - mu_v), so Q is a 2x2
//    quadratic form.  For cone-beam rays from the source S, d~ = (u, v, dsd)
//    and delta = S - mu is the same for every ray of the view; writing
//    d~ = d~0 + (du, dv, 0) with d~0 the ray through mu, c = du g_u + dv g_v
//    (g_u = e_u x delta, g_v = e_v x delta) and A(du, dv) = d~^T P' d~ are
//    both quadratic in (du, dv), and the integral along the physical ray is
//    |d~| rho sqrt(2 pi / A) exp(-Q/(2A)).
// Both forms avoid the cancellation of C - B^2/A entirely.  Segment ends
// (erf terms) only matter for a Gaussian whose 3-sigma ball lies within
// 5.66 sigma of a segment end (then |w| < 4 is possible); such Gaussians take
// the general path below, in world coordinates, with the ray re-based at the
// foot of the perpendicular from mu.
#include "view.cuh"

namespace rgrt {
namespace {

constexpr int CH = 256;             // records per chunk (one per thread in the prep)
// chunk buffers of the forward: with two, a chunk's records are prepared into
// one buffer while slower warps still read the other, and a single barrier
// per chunk suffices.  The staged records (52 B each) leave the general-path
// fields in global memory so that two buffers still fit 4 CTAs per SM.
constexpr int NBUF = 2;

// the forward's copy of a VRec: the view-space coefficients and the gid
// (general-path records read mu, rho and P from the global records by gid)
struct SRec {
    float4 c0, c1, c2;
    uint32_t gid;
};

// a chunk of staged records in shared memory, one array per field: the
// preparing threads write consecutive 16-byte (4-byte) words, free of bank
// conflicts, and a warp reads one record at a time (broadcast)
struct SChunk {
    float4 c0[CH], c1[CH], c2[CH];
    uint32_t gid[CH];
    __device__ __forceinline__ SRec operator[](int j) const
    {
        SRec r;
        r.c0 = c0[j];
        r.c1 = c1[j];
        r.c2 = c2[j];
        r.gid = gid[j];
        return r;
    }
};

// the general-path fields of record gid (mu, rho | P00 P01 P02 P11 | P12 P22)
struct GRec {
    float4 g0, g1, g2;
};
__device__ __forceinline__ GRec load_grec(const float4 *__restrict__ rec, uint32_t gid)
{
    const float4 *r = rec + REC_F4 * (size_t)gid;
    GRec o;
    o.g0 = __ldg(r);
    o.g1 = __ldg(r + 1);
    o.g2 = __ldg(r + 2);
    return o;
}

struct TileCtx {
    int vl, tx, ty, view, col, row;
    bool valid;                        // the thread's pixel is on the detector
    bool live;                         // ... and has a ray (3-D PET: a ring pair)
    float wu_lo, wu_hi, wv_lo, wv_hi;  // detector box of this warp's (half-warp's) rays
    float zoff, dz;                    // 3-D PET: mid-height offset of the rows, axial LOR rise
    float kap0, kap1;                  // 3-D PET: LOR slopes at the tile's extreme columns
    long long out_idx;
};

// Half-warp blocks (4 x 4 rays per half-warp) for the parallel-ray and 3-D
// PET geometries, whose footprints span a few bins; cone-beam footprints are
// large enough that whole-warp 8 x 4 blocks waste little and build their
// lists for less.
template <int GM>
struct HalfBlocks {
    static constexpr bool value = GM != GM_CONE;
};

template <int GM>
__device__ __forceinline__ TileCtx tile_ctx(const DevGeom &g, uint32_t tile)
{
    constexpr bool HALF = HalfBlocks<GM>::value;
    TileCtx c;
    int T = g.tiles_x * g.tiles_y;
    c.vl = (int)(tile / (uint32_t)T);
    int tin = (int)tile - c.vl * T;
    c.ty = tin / g.tiles_x;
    c.tx = tin - c.ty * g.tiles_x;
    c.view = g.v0 + c.vl;
    // a warp takes an 8 x 4 block of rays (HALF: each half-warp a 4 x 4 half of it)
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int wpr = g.tile_w >> 3;  // warps per tile row
    int wx = w % wpr, wy = w / wpr;
    int c0 = c.tx * g.tile_w + wx * 8 + (HALF ? 4 * (lane >> 4) : 0), r0 = c.ty * g.tile_h + wy * 4;
    c.col = c0 + (HALF ? (lane & 3) : (lane & 7));
    c.row = r0 + (HALF ? ((lane >> 2) & 3) : (lane >> 3));
    c.valid = c.col < g.n_cols && c.row < g.n_rows;
    int rows = g.n_rows;
    c.zoff = c.dz = c.kap0 = c.kap1 = 0.0f;
    if (GM == GM_PET3D) {
        pet3d_view(g, c.view, c.zoff, c.dz, rows);
        const int tc0 = c.tx * g.tile_w;
        pet3d_slopes(g, c.dz, tc0, min(tc0 + g.tile_w - 1, g.n_cols - 1), c.kap0, c.kap1);
    }
    c.live = c.valid && c.row < rows;
    if (c0 < g.n_cols && r0 < rows) {
        int c1 = min(c0 + (HALF ? 3 : 7), g.n_cols - 1), r1 = min(r0 + 3, rows - 1);
        c.wu_lo = __ldg(g.utab + c0); c.wu_hi = __ldg(g.utab + c1);
        c.wv_lo = __ldg(g.vtab + r0) + c.zoff; c.wv_hi = __ldg(g.vtab + r1) + c.zoff;
    } else {
        c.wu_lo = INFINITY; c.wu_hi = -INFINITY; c.wv_lo = INFINITY; c.wv_hi = -INFINITY;
    }
    c.out_idx = (long long)c.view * g.stride_view + (long long)c.row * g.stride_row + c.col;
    return c;
}

// Per chunk: every thread turns one record into its view-space form and tests
// its detector box against the ray block of every warp of the tile (bit w of
// msk), or with half-warp blocks of every half-warp (bit 2w + h, h the half of
// warp w); then each warp compacts, in record order, the records that touch
// its block (each of its halves' blocks) into a list of view-space records and
// a list of general ones.  The two halves of a warp walk their own lists side
// by side: smaller blocks leave fewer lanes evaluating pairs outside the
// footprint.
constexpr uint32_t MSK_VS = 1u << 16;   // msk: the record takes the view-space path
struct ChunkLists {
    uint8_t vs[16][CH];
    uint8_t gen[16][CH];
};

template <int GM, int KER, bool TOF>
__device__ __forceinline__ void prep_chunk(const DevGeom &g, const float *F, const uint32_t *gids,
                                           uint32_t base, uint32_t stride, int cnt,
                                           const float4 *rec, const float4 *crec, SChunk *sv,
                                           const float4 *wbox, int nw, uint32_t *msk,
                                           float kap0, float kap1)
{
    for (int i = threadIdx.x; i < cnt; i += blockDim.x) {
        const uint32_t gid = __ldg(gids + base + (uint32_t)i * stride);
        VRec vr;
        prep_record<GM, KER>(g, F, gid, rec, crec, vr, kap0, kap1);
        if (TOF) {
            // time of flight (parallel rays): the pair's value times the
            // kernel of width s^2 = 1/A + sigma_T^2 at t* - t_k (the
            // convolution of the Gaussian's profile along the ray with the
            // TOF kernel): c1.y = -log2(e) / (2 s^2), c1.z = 1/sqrt(2 pi s^2),
            // c2.xyz = the coefficients of t*
            const float s2 = vr.t4.w + g.tof_s2;
            vr.c1.y = Kern<0>::QSCALE / s2;
            vr.c1.z = rsqrtf(2.0f * 3.14159265358979324f * s2);
            vr.c2.x = vr.t4.x;
            vr.c2.y = vr.t4.y;
            vr.c2.z = vr.t4.z;
        }
        sv->c0[i] = vr.c0;
        sv->c1[i] = vr.c1;
        sv->c2[i] = vr.c2;
        sv->gid[i] = gid;
        const float4 bb = vr.bb;
        // a block inside the footprint's box may still miss the footprint
        // ellipse: skip it when the tangent plane of G at the block centre
        // stays above tol over the block (a pair with m <= 9 + 9e-4 has
        // G <= -0.19 A < 0 at K^2 = 9.2, so none is lost).  Cone beam only:
        // the small footprints of the parallel-ray workloads fill their boxes'
        // blocks, and the test there cost more than it saved.
        Conic cn;
        cn.ok = false;
        float u0 = 0.0f, v0 = 0.0f;
        if (GM == GM_CONE) {
            cn = cone_conic<KER>(vr);
            u0 = vr.c0.x;
            v0 = vr.c0.y;
        }
        const float tol = 1e-3f * fabsf(cn.f);
        uint32_t m = 0;
        for (int w = 0; w < (HalfBlocks<GM>::value ? 2 * nw : nw); w++) {
            const float4 wb = wbox[w];
            bool hit = !(bb.y < wb.x || bb.x > wb.y || bb.w < wb.z || bb.z > wb.w);
            if (GM == GM_CONE && hit && cn.ok) {
                const float cu = 0.5f * (wb.x + wb.y) - u0, cv = 0.5f * (wb.z + wb.w) - v0;
                const float hu = 0.5f * (wb.y - wb.x), hv = 0.5f * (wb.w - wb.z);
                const float gu = cn.a * cu + cn.b * cv + cn.d, gv = cn.b * cu + cn.c * cv + cn.e;
                const float G = cu * (gu + cn.d) + cv * (gv + cn.e) + cn.f;
                hit = G - 2.0f * (fabsf(gu) * hu + fabsf(gv) * hv) <= tol;
            }
            m |= (uint32_t)hit << w;
        }
        if (vr.g2.w != 0.0f) m |= MSK_VS;
        msk[i] = m;
    }
}

// warp-private compaction; returns the list lengths in nvs, ngen
// nvs, ngen: the lengths of this lane's lists
template <bool HALF>
__device__ __forceinline__ void build_lists(int cnt, const uint32_t *msk, ChunkLists &L, int w,
                                            int lane, int &nvs, int &ngen)
{
    const uint32_t lt = (1u << lane) - 1u;
    if (!HALF) {
        nvs = 0;
        ngen = 0;
        for (int b = 0; b < cnt; b += 32) {
            const int i = b + lane;
            const uint32_t m = i < cnt ? msk[i] : 0u;
            const bool in = (m >> w) & 1u;
            const bool vs = (m & MSK_VS) != 0u;
            const uint32_t bv = __ballot_sync(0xffffffffu, in && vs);
            const uint32_t bg = __ballot_sync(0xffffffffu, in && !vs);
            if (in && vs) L.vs[w][nvs + __popc(bv & lt)] = (uint8_t)i;
            if (in && !vs) L.gen[w][ngen + __popc(bg & lt)] = (uint8_t)i;
            nvs += __popc(bv);
            ngen += __popc(bg);
        }
        __syncwarp();
        return;
    }
    int v0 = 0, v1 = 0, g0 = 0, g1 = 0;
    for (int b = 0; b < cnt; b += 32) {
        const int i = b + lane;
        const uint32_t m = i < cnt ? msk[i] : 0u;
        const bool in0 = (m >> (2 * w)) & 1u, in1 = (m >> (2 * w + 1)) & 1u;
        const bool vs = (m & MSK_VS) != 0u;
        const uint32_t bv0 = __ballot_sync(0xffffffffu, in0 && vs);
        const uint32_t bv1 = __ballot_sync(0xffffffffu, in1 && vs);
        const uint32_t bg0 = __ballot_sync(0xffffffffu, in0 && !vs);
        const uint32_t bg1 = __ballot_sync(0xffffffffu, in1 && !vs);
        if (in0 && vs) L.vs[2 * w][v0 + __popc(bv0 & lt)] = (uint8_t)i;
        if (in1 && vs) L.vs[2 * w + 1][v1 + __popc(bv1 & lt)] = (uint8_t)i;
        if (in0 && !vs) L.gen[2 * w][g0 + __popc(bg0 & lt)] = (uint8_t)i;
        if (in1 && !vs) L.gen[2 * w + 1][g1 + __popc(bg1 & lt)] = (uint8_t)i;
        v0 += __popc(bv0);
        v1 += __popc(bv1);
        g0 += __popc(bg0);
        g1 += __popc(bg1);
    }
    __syncwarp();
    const bool h = lane >= 16;
    nvs = h ? v1 : v0;
    ngen = h ? g1 : g0;
}

// the warps' detector boxes, wbox[w] (HALF: the half-warps', wbox[2w + h])
template <bool HALF>
__device__ __forceinline__ void warp_box(const TileCtx &c, float4 *wbox)
{
    if ((threadIdx.x & (HALF ? 15 : 31)) == 0)
        wbox[threadIdx.x >> (HALF ? 4 : 5)] = make_float4(c.wu_lo, c.wu_hi, c.wv_lo, c.wv_hi);
}

// view-space value of one pair (without the |d~| factor of cone beam and
// 3-D PET); returns arg = QSCALE m (Gaussian: -m log2(e)/2; Epanechnikov:
// -m/kappa^2).  kap: the ray's slope (3-D PET).
template <int GM, int KER, class R>
__device__ __forceinline__ float vs_value(const R &r, float u, float v, float kap, float &arg)
{
    const float4 c0 = r.c0, c1 = r.c1, c2 = r.c2;
    float rA = 1.0f;
    if (GM == GM_PET3D) {
        const float du = u - c0.x, vt = fmaf(kap, c0.z, v - c0.y);
        const float muu = fmaf(fmaf(c1.z, kap, c1.y), kap, c1.x);
        const float muv2 = fmaf(c2.x, kap, c1.w);
        const float q = du * (muu * du + muv2 * vt) + c0.w * vt * vt;
        const float An = fmaf(fmaf(c2.z, kap, c2.y), kap, 1.0f);
        rA = rsqrt_approx(An);
        arg = q * (rA * rA);
        if (KER == 1) {
            const float c = 1.0f + arg;
            const float pc = c > 0.0f ? c * sqrt_approx(c) : 0.0f;
            return c2.w * rA * pc;
        }
        return c2.w * rA * ex2_approx(arg);
    }
    const float du = u - c0.x, dv = v - c0.y;
    const float q = du * (c0.z * du + c0.w * dv) + c1.x * dv * dv;
    if (GM == GM_CONE) {
        const float A = c1.y + du * (c1.z + c2.x * du + c2.y * dv) + dv * (c1.w + c2.z * dv);
        rA = rsqrt_approx(A);
        arg = q * (rA * rA);
    } else {
        arg = q;
    }
    if (KER == 1) {
        const float c = 1.0f + arg;                      // 1 - m / kappa^2
        const float pc = c > 0.0f ? c * sqrt_approx(c) : 0.0f;
        return c2.w * rA * pc;
    }
    return c2.w * rA * ex2_approx(arg);
}

// the pair counts (Gaussian: m <= 9; Epanechnikov: inside the support)
template <int KER>
__device__ __forceinline__ bool vs_keep(float arg)
{
    return KER == 1 ? arg > -1.0f : arg >= CUT_ARG;
}

// forward integration of tile `tile` of geometry g (one ray per thread)
template <int GM, bool STATS, int KER, bool TOF = false>
__device__ __forceinline__ void forward_tile(const DevGeom &g, uint32_t tile,
                                             const float4 *__restrict__ rec,
                                             const float4 *__restrict__ crec,
                                             const uint32_t *__restrict__ gids,
                                             const uint2 *__restrict__ ranges,
                                             float *__restrict__ out, Stats *stats)
{
    __shared__ SChunk sv_buf[NBUF];
    __shared__ ChunkLists lists;
    __shared__ uint32_t msk_buf[NBUF][CH];
    __shared__ float4 wbox[16];
    __shared__ float Fs[9];
    constexpr bool CONE = GM == GM_CONE;
    const TileCtx c = tile_ctx<GM>(g, tile);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    constexpr bool HALF = HalfBlocks<GM>::value;
    const int hw = HALF ? threadIdx.x >> 4 : w;   // this lane's lists
    if (threadIdx.x < 9) Fs[threadIdx.x] = __ldg(g.frames + 9 * (size_t)c.view + threadIdx.x);
    warp_box<HALF>(c, wbox);
    __syncthreads();
    float F[9];
#pragma unroll
    for (int i = 0; i < 9; i++) F[i] = Fs[i];
    const float u = __ldg(g.utab + min(c.col, g.n_cols - 1));
    const float v = __ldg(g.vtab + min(c.row, g.n_rows - 1)) + c.zoff;
    const float kap = GM == GM_PET3D ? pet3d_slope(g, c.dz, u) : 0.0f;
    const float L = CONE ? sqrtf(u * u + v * v + g.dsd * g.dsd)
                  : GM == GM_PET3D ? sqrtf(1.0f + kap * kap) : 1.0f;
    const uint2 rg = ranges[tile];
    float acc_vs = 0.0f, acc_gen = 0.0f;
    // time of flight (parallel rays, Gaussian kernel): one sum per bin
    float acc_t[TOF ? TOF_MAX : 1];
#pragma unroll
    for (int q = 0; q < (TOF ? TOF_MAX : 1); q++) acc_t[q] = 0.0f;
    unsigned n_eval = 0, n_kept = 0;
    // chunk c takes list entries c, c + nch, c + 2 nch, ...: the lists are
    // ordered by footprint position, and interleaving spreads every chunk
    // over the whole tile, which keeps the warps' shares of it even
    const uint32_t nlist = rg.y - rg.x;
    const uint32_t nch = (nlist + CH - 1) / CH;
    for (uint32_t ch = 0; ch < nch; ch++) {
        const int cnt = (int)((nlist - ch + nch - 1) / nch);
        const SChunk &sv = sv_buf[ch % NBUF];
        uint32_t *msk = msk_buf[ch % NBUF];
        prep_chunk<GM, KER, TOF>(g, F, gids, rg.x + ch, nch, cnt, rec, crec, &sv_buf[ch % NBUF], wbox, nw, msk,
                                 c.kap0, c.kap1);
        // every thread has prepared this chunk and (with two buffers) left the
        // previous one, whose buffer the next chunk's preparation reuses
        __syncthreads();
        int nvs, ngen;
        build_lists<HALF>(cnt, msk, lists, w, lane, nvs, ngen);
        int k = 0;
        if (TOF) {
            for (; k < nvs; k++) {
                const SRec r = sv[lists.vs[hw][k]];
                float a0;
                const float v0 = vs_value<GM, KER>(r, u, v, kap, a0);
                if (STATS) n_kept += vs_keep<KER>(a0);
                if (!vs_keep<KER>(a0)) continue;
                const float ts = r.c2.x + r.c2.y * (u - r.c0.x) + r.c2.z * (v - r.c0.y) - g.tof_t0;
                const float vn = v0 * r.c1.z;
#pragma unroll
                for (int b = 0; b < TOF_MAX; b++) {
                    if (b >= g.n_tof) break;
                    const float x = ts - (float)b * g.tof_h;
                    acc_t[b] = fmaf(vn, ex2_approx(r.c1.y * x * x), acc_t[b]);
                }
            }
        }
        for (; k + 1 < nvs; k += 2) {
            const int j0 = lists.vs[hw][k], j1 = lists.vs[hw][k + 1];
            float a0, a1;
            const float v0 = vs_value<GM, KER>(sv[j0], u, v, kap, a0);
            const float v1 = vs_value<GM, KER>(sv[j1], u, v, kap, a1);
            acc_vs += vs_keep<KER>(a0) ? v0 : 0.0f;
            acc_vs += vs_keep<KER>(a1) ? v1 : 0.0f;
            if (STATS) n_kept += vs_keep<KER>(a0) + vs_keep<KER>(a1);
        }
        if (k < nvs) {
            float a0;
            const float v0 = vs_value<GM, KER>(sv[lists.vs[hw][k]], u, v, kap, a0);
            acc_vs += vs_keep<KER>(a0) ? v0 : 0.0f;
            if (STATS) n_kept += vs_keep<KER>(a0);
        }
        if (ngen > 0) {
            const Ray ray = make_ray<GM>(g, F, u, v, kap);
            for (int k2 = 0; k2 < ngen; k2++) {
                const GRec r = load_grec(rec, sv.gid[lists.gen[hw][k2]]);
                PairGeo q;
                pair_geo(ray, r, q);
                if (STATS) n_kept += q.m <= PAIR_CUT2;
                if (TOF) {
                    if (q.m <= PAIR_CUT2) {
#pragma unroll
                        for (int b = 0; b < TOF_MAX; b++) {
                            if (b >= g.n_tof) break;
                            acc_t[b] += general_value<KER>(q, r.g0.w, g.tof_t0 + (float)b * g.tof_h, g.tof_tau);
                        }
                    }
                    continue;
                }
                const float val = general_value<KER>(q, r.g0.w);
                acc_gen += q.m <= PAIR_CUT2 ? val : 0.0f;
            }
        }
        if (STATS) n_eval += nvs + ngen;
        if (NBUF == 1) __syncthreads();
    }
    if (TOF) {
        if (c.valid) {
#pragma unroll
            for (int b = 0; b < TOF_MAX; b++) {
                if (b >= g.n_tof) break;
                out[c.out_idx + (long long)b * g.stride_tof] = c.live ? acc_t[b] : 0.0f;
            }
        }
    } else if (c.valid) {
        out[c.out_idx] = c.live ? acc_gen + L * acc_vs : 0.0f;
    }
    if (STATS) {
        unsigned long long e = c.live ? n_eval : 0, kk = c.live ? n_kept : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            e += __shfl_xor_sync(0xffffffffu, e, o);
            kk += __shfl_xor_sync(0xffffffffu, kk, o);
        }
        if (lane == 0) {
            atomicAdd(&stats->pairs_eval, e);
            atomicAdd(&stats->pairs_kept, kk);
        }
    }
}

template <int GM, bool STATS, int KER>
__global__ void __launch_bounds__(256, 4) k_forward(DevGeom g, const float4 *__restrict__ rec,
                                                    const float4 *__restrict__ crec,
                                                    const uint32_t *__restrict__ gids,
                                                    const uint2 *__restrict__ ranges,
                                                    float *__restrict__ out, Stats *stats)
{
    forward_tile<GM, STATS, KER>(g, blockIdx.x, rec, crec, gids, ranges, out, stats);
}

// time-of-flight sinograms (PET ring, Gaussian kernel): one sum per bin per ray
template <bool STATS>
__global__ void __launch_bounds__(256, 2) k_forward_tof(DevGeom g, const float4 *__restrict__ rec,
                                                        const float4 *__restrict__ crec,
                                                        const uint32_t *__restrict__ gids,
                                                        const uint2 *__restrict__ ranges,
                                                        float *__restrict__ out, Stats *stats)
{
    forward_tile<GM_PARALLEL, STATS, 0, true>(g, blockIdx.x, rec, crec, gids, ranges, out, stats);
}

// Persistent form over a batch of scans: every CTA takes (scan, tile) work
// items until all are done (next_item).
template <bool CONE>
__global__ void __launch_bounds__(256, 4) k_forward_persistent(const ScanDesc *__restrict__ d,
                                                               int nscan, uint32_t total,
                                                               uint32_t *queue)
{
    uint32_t item;
    int scan;
    while (next_item(d, nscan, total, queue, item, scan)) {
        const ScanDesc &sd = d[scan];
        forward_tile<CONE ? GM_CONE : GM_PARALLEL, false, 0>(sd.g, item - sd.item_begin, sd.rec, sd.crec, sd.gids, sd.ranges,
                                  sd.out, nullptr);
    }
}

}  // namespace

cudaError_t launch_forward_persistent(bool cone, const ScanDesc *d, int nscan, uint32_t total,
                                      uint32_t *queue, int tile_threads, int grid, cudaStream_t s)
{
    if (total == 0) return cudaSuccess;
    if (cone) k_forward_persistent<true><<<grid, tile_threads, 0, s>>>(d, nscan, total, queue);
    else k_forward_persistent<false><<<grid, tile_threads, 0, s>>>(d, nscan, total, queue);
    count_launches(1);
    return cudaGetLastError();
}

int persistent_grid(bool cone, int tile_threads)
{
    return cone ? grid_for(k_forward_persistent<true>, tile_threads)
                : grid_for(k_forward_persistent<false>, tile_threads);
}

cudaError_t launch_forward(const DevGeom &g, int nv, const float4 *rec, const float4 *crec,
                           const uint32_t *gids, const uint2 *ranges, float *out, Stats *stats,
                           int ker, cudaStream_t s)
{
    unsigned nt = (unsigned)nv * g.tiles_x * g.tiles_y;
    if (nt == 0) return cudaSuccess;
    int bs = g.tile_w * g.tile_h;
#define RGRT_FWD(M, S, K) k_forward<M, S, K><<<nt, bs, 0, s>>>(g, rec, crec, gids, ranges, out, stats)
#define RGRT_FWD_K(M, K) { if (stats) RGRT_FWD(M, true, K); else RGRT_FWD(M, false, K); }
#define RGRT_FWD_M(K)                                  \
    if (g.kind == GM_CONE) RGRT_FWD_K(GM_CONE, K)      \
    else if (g.kind == GM_PET3D) RGRT_FWD_K(GM_PET3D, K) \
    else RGRT_FWD_K(GM_PARALLEL, K)
    if (g.n_tof > 0) {   // PET ring, Gaussian kernel (checked by the caller)
        if (stats) k_forward_tof<true><<<nt, bs, 0, s>>>(g, rec, crec, gids, ranges, out, stats);
        else k_forward_tof<false><<<nt, bs, 0, s>>>(g, rec, crec, gids, ranges, out, stats);
    } else if (ker == 1) { RGRT_FWD_M(1) } else { RGRT_FWD_M(0) }
#undef RGRT_FWD_M
#undef RGRT_FWD_K
#undef RGRT_FWD
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace rgrt
