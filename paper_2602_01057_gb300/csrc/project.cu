// Per-tile ray integration (a3).
//
// One CTA per detector tile of tile_w x tile_h rays (or a cluster of up to 8
// that share the tile's list), two rays per thread, a half- or quarter-warp
// per block of 8 x 4 or 4 x 4 rays.  The tile's Gaussian list (ordered by
// footprint position on the cone beam, by box size on 3-D PET, by id alone on
// parallel rays) is walked in chunks: the CTA gathers each
// chunk's records, turning every Gaussian into its view-space form for this
// view (see below) together with its detector bounding box, into one of two
// shared-memory buffers.  A block skips a Gaussian whose box misses it, or
// (cone beam) whose footprint ellipse misses it; otherwise its lanes evaluate
// their two pairs in packed binary32 and a pair counts when m <= 9 (3-sigma
// cut).  FP32 throughout, FP32 accumulation per ray.
// 3-D PET LORs (direction e_w + kappa e_v, kappa per detector column) have a
// view-space form of their own (prep_record).
//
// Bound by issue: per evaluated record 64 pairs take about 26 arithmetic
// instructions (parallel rays 16), where one ray per thread took the same for
// 32, and the special-function unit two rsqrt and two ex2 per lane.  Measured
// on a GB300 against one ray per thread (8 x 4 warps, 4 x 4 half-warps): cone
// beam 50,000 Gaussians, 180 x 256^2 8.5 -> 6.3 ms; PET ring 200,000, 288 x
// 329 x 63 8.2 -> 5.7 ms; fully 3-D PET (the pair shares its column's slope
// terms) 79 -> 62 ms; time of flight 4.05 -> 3.3 ms before the lists were
// shared (forward_parts).
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
#include <cooperative_groups.h>

#include "packed.cuh"
#include "view.cuh"

namespace cg = cooperative_groups;

namespace rgrt {
namespace {

// records per chunk: at most 256 (8-bit list entries); 192 leave room for two
// more CTAs per SM, which the geometries of small footprints, waiting at the
// chunk barrier, use (3-D PET forward 61.8 -> 58.7 ms; cone beam 6.27 -> 6.32)
template <int GM> struct Chunk {
    static constexpr int N = GM == GM_CONE ? 256 : 192;
};
constexpr int FBS = 128;            // most threads of a CTA (two rays each)
// chunk buffers: with two, a chunk's records are prepared into one buffer
// while slower warps still read the other, and a single barrier per chunk
// suffices.  The staged records leave the general-path fields in global
// memory so that two buffers fit 6 to 8 CTAs per SM.
constexpr int NBUF = 2;
// A tile's list is shared by 2, 4 or 8 CTAs of a cluster while the launch has
// fewer CTAs than FORWARD_SPLIT_CTAS (about 9 waves: tile lists are uneven, and a few
// waves leave most of the SMs waiting for the longest) and a CTA's share of an
// average list stays above FORWARD_SPLIT_LIST records.  Measured without and with it:
// 672 tiles of 2,700 records (8 raw PET angles) 0.46 -> 0.165 ms, 2,016 tiles
// (time of flight, 24 angles) 3.4 -> 2.0, 2,048 of 1,270 (8 cone-beam views)
// 0.55 -> 0.37, 256 of 350 (parallel beam) 0.080 -> 0.036; at 24,000 tiles
// (PET ring) 5.7 either way, so those keep one CTA.

// A lane's two rays: neighbouring columns of one row, or (3-D PET, whose ray
// slope is a column's) neighbouring rows of one column.  The lanes of a group
// share a block of rays and its lists: 8 x 4 rays per half-warp for the cone
// beam, whose footprints are large, 4 x 4 rays per quarter-warp for the others,
// whose footprints span a few bins.
template <int GM>
struct Blocks {
    static constexpr int BWID = GM == GM_CONE ? 8 : 4;
    static constexpr int LANES = GM == GM_CONE ? 16 : 8;
    static constexpr int PER_WARP = 32 / LANES;
    static constexpr int MAX = GM == GM_CONE ? 8 : 16;   // blocks of a tile of 256 rays
};

// a chunk of staged records in shared memory, one array per field: the
// preparing threads write consecutive words, free of bank conflicts, and a
// group of lanes reads one record at a time (broadcast).  Parallel rays need
// c0, M_vv and the amplitude only.
template <bool WIDE, int CH> struct SChunk {
    float4 c0[CH], c1[CH], c2[CH];
    uint32_t gid[CH];
};
template <int CH> struct SChunk<false, CH> {
    float4 c0[CH];
    float2 va[CH];     // k M_vv, alpha / sqrt(A)
    uint32_t gid[CH];
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

// Per chunk: every thread turns records into their view-space form and tests
// their detector boxes against the tile's blocks (bit b of msk: block b);
// then each warp compacts, in record order, the records that touch its groups'
// blocks into one list per group -- of view-space records, and (rarely) of
// general ones.  The groups of a warp walk their own lists side by side.
constexpr uint32_t MSK_VS = 1u << 16;   // msk: the record takes the view-space path
template <int NB, int CH> struct ChunkLists {
    uint8_t vs[NB][CH];
    uint8_t gen[NB][CH];
};

// the intervals of the tile's column and row blocks; wbox: every block's box
// (cone beam, for the ellipse test)
struct TileBoxes {
    float2 cu[8], rv[8];
    float4 wbox[8];
    int ncb, nrb;      // column and row blocks of the tile
};

template <int GM, int KER, bool TOF, class Staged>
__device__ __forceinline__ bool prep_chunk(const DevGeom &g, const float *F, const uint32_t *gids,
                                           uint32_t base, uint32_t stride, int cnt,
                                           const float4 *rec, const float4 *crec, Staged *sv,
                                           const TileBoxes &tb, uint32_t *msk, float kap0, float kap1)
{
    bool gen = false;
    for (int i = threadIdx.x; i < cnt; i += blockDim.x) {
        const uint32_t gid = __ldg(gids + base + (uint32_t)i * stride);
        VRec vr;
        prep_record<GM, KER>(g, F, gid, rec, crec, vr, kap0, kap1);
        if constexpr (TOF) {
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
        if constexpr (GM == GM_PARALLEL && !TOF) {
            sv->va[i] = make_float2(vr.c1.x, vr.c2.w);
        } else {
            sv->c1[i] = vr.c1;
            sv->c2[i] = vr.c2;
        }
        sv->gid[i] = gid;
        const float4 bb = vr.bb;
        uint32_t m = 0;
        if (GM == GM_CONE) {
            // a block inside the footprint's box may still miss the footprint
            // ellipse: skip it when the tangent plane of G at the block centre
            // stays above tol over the block (a pair with m <= 9 + 9e-4 has
            // G <= -0.19 A < 0 at K^2 = 9.2, so none is lost).  Cone beam only:
            // the small footprints of the parallel-ray workloads fill their
            // boxes' blocks, and the test there cost more than it saved.
            const Conic cn = cone_conic<KER>(vr);
            const float u0 = vr.c0.x, v0 = vr.c0.y, tol = 1e-3f * fabsf(cn.f);
            for (int w = 0; w < tb.ncb * tb.nrb; w++) {
                const float4 wb = tb.wbox[w];
                bool hit = !(bb.y < wb.x || bb.x > wb.y || bb.w < wb.z || bb.z > wb.w);
                if (hit && cn.ok) {
                    const float cu = 0.5f * (wb.x + wb.y) - u0, cv = 0.5f * (wb.z + wb.w) - v0;
                    const float hu = 0.5f * (wb.y - wb.x), hv = 0.5f * (wb.w - wb.z);
                    const float gu = cn.a * cu + cn.b * cv + cn.d, gv = cn.b * cu + cn.c * cv + cn.e;
                    const float G = cu * (gu + cn.d) + cv * (gv + cn.e) + cn.f;
                    hit = G - 2.0f * (fabsf(gu) * hu + fabsf(gv) * hv) <= tol;
                }
                m |= (uint32_t)hit << w;
            }
        } else {
            // the blocks are a grid: those hit are columns hit x rows hit
            uint32_t cm = 0;
            for (int c = 0; c < tb.ncb; c++) {
                const float2 x = tb.cu[c];
                cm |= (uint32_t)!(bb.y < x.x || bb.x > x.y) << c;
            }
            for (int r = 0; r < tb.nrb; r++) {
                const float2 x = tb.rv[r];
                m |= bb.w < x.x || bb.z > x.y ? 0u : cm << (r * tb.ncb);
            }
        }
        if (vr.g2.w != 0.0f) m |= MSK_VS;
        else gen = true;
        msk[i] = m;
    }
    return gen;
}

// warp-private compaction into the lists of the warp's groups; returns the
// lengths of this lane's lists
template <int GM, class Lists>
__device__ __forceinline__ void build_lists(int cnt, const uint32_t *msk, bool any_gen, Lists &L, int w,
                                            int lane, int &nvs, int &ngen)
{
    constexpr int PW = Blocks<GM>::PER_WARP;
    const uint32_t lt = (1u << lane) - 1u;
    const int mine = lane / Blocks<GM>::LANES;
    nvs = 0;
    ngen = 0;
    int n[PW], ng[PW];
#pragma unroll
    for (int q = 0; q < PW; q++) n[q] = ng[q] = 0;
    for (int b = 0; b < cnt; b += 32) {
        const int i = b + lane;
        const uint32_t mk = i < cnt ? msk[i] : 0u;
        const uint32_t m = mk >> (w * PW);
        const bool vs = (mk & MSK_VS) != 0u;
#pragma unroll
        for (int q = 0; q < PW; q++) {
            const bool in = ((m >> q) & 1u) && vs;
            const uint32_t bal = __ballot_sync(0xffffffffu, in);
            if (in) L.vs[w * PW + q][n[q] + __popc(bal & lt)] = (uint8_t)i;
            n[q] += __popc(bal);
        }
        if (any_gen) {
#pragma unroll
            for (int q = 0; q < PW; q++) {
                const bool in = ((m >> q) & 1u) && !vs;
                const uint32_t bal = __ballot_sync(0xffffffffu, in);
                if (in) L.gen[w * PW + q][ng[q] + __popc(bal & lt)] = (uint8_t)i;
                ng[q] += __popc(bal);
            }
        }
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < PW; q++)
        if (q == mine) {
            nvs = n[q];
            ngen = ng[q];
        }
}

// the pair counts (Gaussian: m <= 9; Epanechnikov: inside the support)
template <int KER>
__device__ __forceinline__ bool vs_keep(float arg)
{
    return KER == 1 ? arg > -1.0f : arg >= CUT_ARG;
}

// kernel profile of both pairs, arg = QSCALE m (Gaussian: -m log2(e)/2;
// Epanechnikov: -m/kappa^2)
template <int KER>
__device__ __forceinline__ f2 profile2(float a0, float a1)
{
    if (KER == 1) {
        const float x = 1.0f + a0, y = 1.0f + a1;        // 1 - m / kappa^2
        return pk(x > 0.0f ? x * sqrt_approx(x) : 0.0f, y > 0.0f ? y * sqrt_approx(y) : 0.0f);
    }
    return pk(ex2_approx(a0), ex2_approx(a1));
}

// View-space values of a record for the lane's two rays (without the |d~|
// factor of cone beam and 3-D PET).  u, v: the rays' coordinates; kap: their
// slope (3-D PET).
__device__ __forceinline__ f2 quad2(float Muu, float Muv2, float Mvv, f2 du, float dv)
{
    // du (Muu du + 2 Muv dv) + Mvv dv dv
    const f2 t = fma2(pk(Muu, Muu), du, pk(Muv2 * dv, Muv2 * dv));
    const float s = Mvv * dv * dv;
    return fma2(du, t, pk(s, s));
}

template <int KER>
__device__ __forceinline__ f2 value_parallel(const float4 &c0, float Mvv, float alpha, f2 u, float v, float &a0,
                                             float &a1)
{
    const f2 du = add2(u, pk(-c0.x, -c0.x));
    up(quad2(c0.z, c0.w, Mvv, du, v - c0.y), a0, a1);
    return mul2(pk(alpha, alpha), profile2<KER>(a0, a1));
}

template <int KER>
__device__ __forceinline__ f2 value_cone(const float4 &c0, const float4 &c1, const float4 &c2, f2 u, float v,
                                         float &a0, float &a1)
{
    const f2 du = add2(u, pk(-c0.x, -c0.x));
    const float dv = v - c0.y;
    const f2 q = quad2(c0.z, c0.w, c1.x, du, dv);
    // A = c1.y + du (c1.z + c2.x du + c2.y dv) + dv (c1.w + c2.z dv)
    const f2 DV = pk(dv, dv);
    const f2 in = fma2(pk(c2.y, c2.y), DV, fma2(pk(c2.x, c2.x), du, pk(c1.z, c1.z)));
    const float ot = fmaf(c2.z, dv, c1.w);
    float x, y;
    up(fma2(DV, pk(ot, ot), fma2(du, in, pk(c1.y, c1.y))), x, y);
    const f2 rA = pk(rsqrt_approx(x), rsqrt_approx(y));
    up(mul2(q, mul2(rA, rA)), a0, a1);
    return mul2(mul2(pk(c2.w, c2.w), rA), profile2<KER>(a0, a1));
}

template <int KER>
__device__ __forceinline__ f2 value_pet3d(const float4 &c0, const float4 &c1, const float4 &c2, float u, f2 v,
                                          float kap, float &a0, float &a1)
{
    const float du = u - c0.x;
    const float muu = fmaf(fmaf(c1.z, kap, c1.y), kap, c1.x), muv2 = fmaf(c2.x, kap, c1.w);
    const f2 vt = fma2(pk(kap, kap), pk(c0.z, c0.z), add2(v, pk(-c0.y, -c0.y)));
    // du (muu du + muv2 v~) + S_uu v~ v~
    const f2 DU = pk(du, du);
    const f2 t = fma2(pk(muu, muu), DU, mul2(pk(muv2, muv2), vt));
    const f2 q = fma2(mul2(pk(c0.w, c0.w), vt), vt, mul2(DU, t));
    const float rA = rsqrt_approx(fmaf(fmaf(c2.z, kap, c2.y), kap, 1.0f));
    const float iA = rA * rA, al = c2.w * rA;
    up(mul2(q, pk(iA, iA)), a0, a1);
    return mul2(pk(al, al), profile2<KER>(a0, a1));
}

// Forward integration of tile `tile` of geometry g (two rays per thread).  A
// tile's list may be cut into `parts`: part p takes every parts-th chunk, and a
// ray's sum is that of the parts, added in their order.  They belong to the
// CTAs of a cluster, the first adding the others' sums read from their shared
// memory, or (SEQ) to this CTA one after the other, with the same result.
template <int GM, bool STATS, int KER, bool TOF = false, bool SEQ = false>
__device__ __forceinline__ void forward_tile(const DevGeom &g, uint32_t tile, uint32_t part, uint32_t parts,
                                             const float4 *__restrict__ rec,
                                             const float4 *__restrict__ crec,
                                             const uint32_t *__restrict__ gids,
                                             const uint2 *__restrict__ ranges,
                                             float *__restrict__ out, Stats *stats)
{
    using B = Blocks<GM>;
    constexpr bool CONE = GM == GM_CONE, P3 = GM == GM_PET3D, WIDE = GM != GM_PARALLEL || TOF;
    constexpr int CH = Chunk<GM>::N;
    __shared__ SChunk<WIDE, CH> sv_buf[NBUF];
    __shared__ ChunkLists<B::MAX, CH> lists;
    __shared__ uint32_t msk_buf[NBUF][CH];
    __shared__ TileBoxes tb;
    __shared__ float Fs[9];
    __shared__ int s_gen[2];
    const int T = g.tiles_x * g.tiles_y;
    const int vl = (int)(tile / (uint32_t)T);
    const int tin = (int)tile - vl * T;
    const int ty = tin / g.tiles_x, tx = tin - ty * g.tiles_x;
    const int view = g.v0 + vl, tc0 = tx * g.tile_w, tr0 = ty * g.tile_h;
    int rows = g.n_rows;                // rows with a ray
    float zoff = 0.0f, dz = 0.0f, kap0 = 0.0f, kap1 = 0.0f;
    if (P3) {
        pet3d_view(g, view, zoff, dz, rows);
        pet3d_slopes(g, dz, tc0, min(tc0 + g.tile_w - 1, g.n_cols - 1), kap0, kap1);
    }
    const int ncb = g.tile_w / B::BWID, nrb = g.tile_h >> 2;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int blk = w * B::PER_WARP + lane / B::LANES;     // this lane's block (and list)
    // the lane's two rays
    const int l = lane & (B::LANES - 1);
    const int lc = P3 ? l & 3 : 2 * (l & (B::BWID / 2 - 1)), lr = P3 ? 2 * (l >> 2) : l / (B::BWID / 2);
    const int by = blk / ncb, col = tc0 + (blk - by * ncb) * B::BWID + lc, row = tr0 + 4 * by + lr;
    const int col1 = col + (P3 ? 0 : 1), row1 = row + (P3 ? 1 : 0);
    const bool in = blk < ncb * nrb;
    const bool valid0 = in && col < g.n_cols && row < g.n_rows, valid1 = in && col1 < g.n_cols && row1 < g.n_rows;
    const bool live0 = valid0 && row < rows, live1 = valid1 && row1 < rows;
    // the blocks' detector boxes (empty past the detector or the last ring pair)
    if (threadIdx.x < 9) Fs[threadIdx.x] = __ldg(g.frames + 9 * (size_t)view + threadIdx.x);
    if (threadIdx.x < ncb) {
        const int c = tc0 + threadIdx.x * B::BWID;
        tb.cu[threadIdx.x] = c < g.n_cols ? make_float2(__ldg(g.utab + c), __ldg(g.utab + min(c + B::BWID - 1, g.n_cols - 1)))
                                          : make_float2(INFINITY, -INFINITY);
    }
    if (threadIdx.x >= 16 && threadIdx.x < 16 + nrb) {
        const int r = tr0 + 4 * ((int)threadIdx.x - 16);
        tb.rv[threadIdx.x - 16] = r < rows ? make_float2(__ldg(g.vtab + r) + zoff, __ldg(g.vtab + min(r + 3, rows - 1)) + zoff)
                                           : make_float2(INFINITY, -INFINITY);
    }
    if (threadIdx.x == 0) {
        tb.ncb = ncb;
        tb.nrb = nrb;
        s_gen[0] = s_gen[1] = 0;
    }
    __syncthreads();
    if (CONE) {
        if (threadIdx.x < ncb * nrb) {
            const float2 a = tb.cu[threadIdx.x % ncb], b = tb.rv[threadIdx.x / ncb];
            const bool none = a.x > a.y || b.x > b.y;
            tb.wbox[threadIdx.x] = none ? make_float4(INFINITY, -INFINITY, INFINITY, -INFINITY)
                                        : make_float4(a.x, a.y, b.x, b.y);
        }
        __syncthreads();
    }
    float F[9];
#pragma unroll
    for (int i = 0; i < 9; i++) F[i] = Fs[i];
    const float u0 = __ldg(g.utab + min(col, g.n_cols - 1)), u1 = __ldg(g.utab + min(col1, g.n_cols - 1));
    const float v0 = __ldg(g.vtab + min(row, g.n_rows - 1)) + zoff, v1 = __ldg(g.vtab + min(row1, g.n_rows - 1)) + zoff;
    const f2 U = pk(u0, u1), V = pk(v0, v1);
    const float kap = P3 ? pet3d_slope(g, dz, u0) : 0.0f;
    const uint2 rg = ranges[tile];
    f2 acc = 0;
    float gen0 = 0.0f, gen1 = 0.0f;
    // time of flight (parallel rays, Gaussian kernel): one sum per bin
    f2 acc_t[TOF ? TOF_MAX : 1];
#pragma unroll
    for (int q = 0; q < (TOF ? TOF_MAX : 1); q++) acc_t[q] = 0;
    unsigned n_eval = 0, n_kept0 = 0, n_kept1 = 0;
    // chunk c takes list entries c, c + nch, c + 2 nch, ...: a list ordered by
    // footprint position or size is spread over every chunk, which keeps the
    // groups' shares of it even
    const uint32_t nlist = rg.y - rg.x;
    const uint32_t nch = ((nlist + CH - 1) / CH + parts - 1) / parts * parts;
    f2 sum = 0, gsum = 0;      // SEQ: the parts before
    int buf = 0;
next_part:
    for (uint32_t ch = part; ch < nch; ch += parts, buf ^= 1) {
        const int cnt = nlist > ch ? (int)((nlist - ch + nch - 1) / nch) : 0;
        const SChunk<WIDE, CH> &sv = sv_buf[buf];
        uint32_t *msk = msk_buf[buf];
        if (prep_chunk<GM, KER, TOF>(g, F, gids, rg.x + ch, nch, cnt, rec, crec, &sv_buf[buf], tb, msk, kap0, kap1))
            s_gen[buf] = 1;
        // every thread has prepared this chunk and (with two buffers) left the
        // previous one, whose buffer the next chunk's preparation reuses
        __syncthreads();
        const bool any_gen = s_gen[buf] != 0;
        int nvs, ngen;
        build_lists<GM>(cnt, msk, any_gen, lists, w, lane, nvs, ngen);
        const uint8_t *lst = lists.vs[blk & (B::MAX - 1)];
        if constexpr (TOF) {
            for (int k = 0; k < nvs; k++) {
                const int j = lst[k];
                const float4 c0 = sv.c0[j], c1 = sv.c1[j], c2 = sv.c2[j];
                float a0, a1;
                const f2 val = value_parallel<KER>(c0, c1.x, c2.w, U, v0, a0, a1);
                const bool k0 = vs_keep<KER>(a0), k1 = vs_keep<KER>(a1);
                if (STATS) {
                    n_kept0 += k0;
                    n_kept1 += k1;
                }
                if (!k0 && !k1) continue;
                float x0, x1;
                up(mul2(val, pk(c1.z, c1.z)), x0, x1);
                const f2 vn = pk(k0 ? x0 : 0.0f, k1 ? x1 : 0.0f);
                // t* - t_0, then one bin after the other
                const float dv = v0 - c0.y;
                const float t0 = fmaf(c2.z, dv, fmaf(c2.y, u0 - c0.x, c2.x)) - g.tof_t0;
                const float t1 = fmaf(c2.z, dv, fmaf(c2.y, u1 - c0.x, c2.x)) - g.tof_t0;
                const f2 ts = pk(t0, t1), H = pk(g.tof_h, g.tof_h), S = pk(c1.y, c1.y);
#pragma unroll
                for (int b = 0; b < TOF_MAX; b++) {
                    if (b >= g.n_tof) break;
                    const f2 x = fma2(pk(-(float)b, -(float)b), H, ts);
                    float y0, y1;
                    up(mul2(mul2(S, x), x), y0, y1);
                    acc_t[b] = fma2(vn, pk(ex2_approx(y0), ex2_approx(y1)), acc_t[b]);
                }
            }
        } else {
            for (int k = 0; k < nvs; k++) {
                const int j = lst[k];
                float a0, a1;
                f2 val;
                if constexpr (GM == GM_PARALLEL) {
                    const float2 va = sv.va[j];
                    val = value_parallel<KER>(sv.c0[j], va.x, va.y, U, v0, a0, a1);
                } else if constexpr (CONE) {
                    val = value_cone<KER>(sv.c0[j], sv.c1[j], sv.c2[j], U, v0, a0, a1);
                } else {
                    val = value_pet3d<KER>(sv.c0[j], sv.c1[j], sv.c2[j], u0, V, kap, a0, a1);
                }
                float x0, x1;
                up(val, x0, x1);
                acc = add2(acc, pk(vs_keep<KER>(a0) ? x0 : 0.0f, vs_keep<KER>(a1) ? x1 : 0.0f));
                if (STATS) {
                    n_kept0 += vs_keep<KER>(a0);
                    n_kept1 += vs_keep<KER>(a1);
                }
            }
        }
        if (ngen > 0) {
            for (int k2 = 0; k2 < ngen; k2++) {
                const GRec r = load_grec(rec, sv.gid[lists.gen[blk & (B::MAX - 1)][k2]]);
                for (int e = 0; e < 2; e++) {
                    const Ray ray = make_ray<GM>(g, F, e ? u1 : u0, e ? v1 : v0, kap);
                    PairGeo q;
                    pair_geo(ray, r, q);
                    if (STATS) (e ? n_kept1 : n_kept0) += q.m <= PAIR_CUT2;
                    if (!(q.m <= PAIR_CUT2)) continue;
                    if constexpr (TOF) {
#pragma unroll
                        for (int b = 0; b < TOF_MAX; b++) {
                            if (b >= g.n_tof) break;
                            const float x = general_value<KER>(q, r.g0.w, g.tof_t0 + (float)b * g.tof_h, g.tof_tau);
                            acc_t[b] = add2(acc_t[b], pk(e ? 0.0f : x, e ? x : 0.0f));
                        }
                    } else {
                        (e ? gen1 : gen0) += general_value<KER>(q, r.g0.w);
                    }
                }
            }
        }
        if (STATS) n_eval += nvs + ngen;
        // this chunk's flag is read; the next use of it is two chunks on
        if (any_gen) {
            __syncthreads();
            if (threadIdx.x == 0) s_gen[buf] = 0;
        }
    }
    if (SEQ && parts > 1) {
        const f2 gg = pk(gen0, gen1);
        sum = part == 0 ? acc : add2(sum, acc);
        gsum = part == 0 ? gg : add2(gsum, gg);
        if (++part < parts) {
            acc = 0;
            gen0 = gen1 = 0.0f;
            goto next_part;
        }
        acc = sum;
        up(gsum, gen0, gen1);
        part = 0;
    }
    if (!SEQ && parts > 1) {
        // per thread: the sums of its two rays (TOF: bin by bin), in the chunk buffers
        constexpr int NS = TOF ? TOF_MAX : 2;
        f2 *mine = reinterpret_cast<f2 *>(&sv_buf[0]);
        static_assert(sizeof(sv_buf) >= sizeof(f2) * NS * FBS, "a thread's sums fit the chunk buffers");
        __syncthreads();
        if constexpr (TOF) {
#pragma unroll
            for (int b = 0; b < TOF_MAX; b++) mine[b * FBS + threadIdx.x] = acc_t[b];
        } else {
            mine[threadIdx.x] = acc;
            mine[FBS + threadIdx.x] = pk(gen0, gen1);
        }
        cg::cluster_group cluster = cg::this_cluster();
        cluster.sync();
        if (part == 0) {
            for (uint32_t r = 1; r < parts; r++) {
                const f2 *o = cluster.map_shared_rank(mine, r);
                if constexpr (TOF) {
#pragma unroll
                    for (int b = 0; b < TOF_MAX; b++) acc_t[b] = add2(acc_t[b], o[b * FBS + threadIdx.x]);
                } else {
                    float x, y;
                    acc = add2(acc, o[threadIdx.x]);
                    up(o[FBS + threadIdx.x], x, y);
                    gen0 += x;
                    gen1 += y;
                }
            }
        }
        cluster.sync();   // the others' shared memory stays until it has been read
    }
    const bool store0 = valid0 && part == 0, store1 = valid1 && part == 0;
    const long long i0 = (long long)view * g.stride_view + (long long)row * g.stride_row + col;
    const long long i1 = (long long)view * g.stride_view + (long long)row1 * g.stride_row + col1;
    if constexpr (TOF) {
#pragma unroll
        for (int b = 0; b < TOF_MAX; b++) {
            if (b >= g.n_tof) break;
            float x0, x1;
            up(acc_t[b], x0, x1);
            if (store0) out[i0 + (long long)b * g.stride_tof] = x0;
            if (store1) out[i1 + (long long)b * g.stride_tof] = x1;
        }
    } else {
        float x0, x1;
        up(acc, x0, x1);
        const float L0 = CONE ? sqrtf(u0 * u0 + v0 * v0 + g.dsd * g.dsd) : P3 ? sqrtf(1.0f + kap * kap) : 1.0f;
        const float L1 = CONE ? sqrtf(u1 * u1 + v1 * v1 + g.dsd * g.dsd) : L0;
        if (store0) out[i0] = live0 ? gen0 + L0 * x0 : 0.0f;
        if (store1) out[i1] = live1 ? gen1 + L1 * x1 : 0.0f;
    }
    if (STATS) {
        unsigned long long e = (live0 ? n_eval : 0) + (live1 ? n_eval : 0), kk = (live0 ? n_kept0 : 0) + (live1 ? n_kept1 : 0);
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
__global__ void __launch_bounds__(FBS, GM == GM_PARALLEL ? 7 : 6) k_forward(DevGeom g, uint32_t parts, const float4 *__restrict__ rec,
                                                    const float4 *__restrict__ crec,
                                                    const uint32_t *__restrict__ gids,
                                                    const uint2 *__restrict__ ranges,
                                                    float *__restrict__ out, Stats *stats)
{
    forward_tile<GM, STATS, KER>(g, blockIdx.x / parts, blockIdx.x % parts, parts, rec, crec, gids, ranges, out, stats);
}

// time-of-flight sinograms (PET ring, Gaussian kernel): one sum per bin per ray
template <bool STATS>
__global__ void __launch_bounds__(FBS, 5) k_forward_tof(DevGeom g, uint32_t parts, const float4 *__restrict__ rec,
                                                        const float4 *__restrict__ crec,
                                                        const uint32_t *__restrict__ gids,
                                                        const uint2 *__restrict__ ranges,
                                                        float *__restrict__ out, Stats *stats)
{
    forward_tile<GM_PARALLEL, STATS, 0, true>(g, blockIdx.x / parts, blockIdx.x % parts, parts, rec, crec, gids,
                                              ranges, out, stats);
}

// Persistent form over a batch of scans: every CTA takes (scan, tile) work
// items until all are done (next_item).
template <bool CONE>
__global__ void __launch_bounds__(FBS, CONE ? 6 : 7) k_forward_persistent(const ScanDesc *__restrict__ d,
                                                               int nscan, uint32_t total,
                                                               uint32_t *queue)
{
    uint32_t item;
    int scan;
    while (next_item(d, nscan, total, queue, item, scan)) {
        const ScanDesc &sd = d[scan];
        // the parts that a projection of the scan's own would take now
        forward_tile<CONE ? GM_CONE : GM_PARALLEL, false, 0, false, true>(
            sd.g, item - sd.item_begin, 0, forward_parts(sd.n_items, (int64_t)*sd.entries), sd.rec, sd.crec, sd.gids,
            sd.ranges, sd.out, nullptr);
    }
}

}  // namespace

namespace {
// two rays per thread, whole warps
int forward_threads(int tile_rays) { return (tile_rays / 2 + 31) & ~31; }
}  // namespace

cudaError_t launch_forward_persistent(bool cone, const ScanDesc *d, int nscan, uint32_t total,
                                      uint32_t *queue, int tile_rays, int grid, cudaStream_t s)
{
    if (total == 0) return cudaSuccess;
    const int bs = forward_threads(tile_rays);
    if (cone) k_forward_persistent<true><<<grid, bs, 0, s>>>(d, nscan, total, queue);
    else k_forward_persistent<false><<<grid, bs, 0, s>>>(d, nscan, total, queue);
    count_launches(1);
    return cudaGetLastError();
}

int persistent_grid(bool cone, int tile_rays)
{
    const int bs = forward_threads(tile_rays);
    return cone ? grid_for(k_forward_persistent<true>, bs) : grid_for(k_forward_persistent<false>, bs);
}

cudaError_t launch_forward(const DevGeom &g, int nv, int64_t entries, const float4 *rec, const float4 *crec,
                           const uint32_t *gids, const uint2 *ranges, float *out, Stats *stats,
                           int ker, cudaStream_t s)
{
    const int64_t nt = (int64_t)nv * g.tiles_x * g.tiles_y;
    if (nt <= 0) return cudaSuccess;
    const uint32_t parts = forward_parts(nt, entries);
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = parts;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)(nt * parts));
    cfg.blockDim = dim3(forward_threads(g.tile_w * g.tile_h));
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = parts > 1 ? 1 : 0;
    cudaError_t e;
#define RGRT_FWD(M, S, K) e = cudaLaunchKernelEx(&cfg, k_forward<M, S, K>, g, parts, rec, crec, gids, ranges, out, stats)
#define RGRT_FWD_K(M, K) { if (stats) RGRT_FWD(M, true, K); else RGRT_FWD(M, false, K); }
#define RGRT_FWD_M(K)                                  \
    if (g.kind == GM_CONE) RGRT_FWD_K(GM_CONE, K)      \
    else if (g.kind == GM_PET3D) RGRT_FWD_K(GM_PET3D, K) \
    else RGRT_FWD_K(GM_PARALLEL, K)
    if (g.n_tof > 0) {   // PET ring, Gaussian kernel (checked by the caller)
        if (stats) e = cudaLaunchKernelEx(&cfg, k_forward_tof<true>, g, parts, rec, crec, gids, ranges, out, stats);
        else e = cudaLaunchKernelEx(&cfg, k_forward_tof<false>, g, parts, rec, crec, gids, ranges, out, stats);
    } else if (ker == 1) { RGRT_FWD_M(1) } else { RGRT_FWD_M(0) }
#undef RGRT_FWD_M
#undef RGRT_FWD_K
#undef RGRT_FWD
    count_launches(1);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace rgrt
