// dsp_kernels.cu -- the projection-only kernel, the density finalisation and the
// time-segment combination.  Shared device code
// (and the description of the method and of the GB300 design) is in
// dsp_device.cuh.

#include "dsp_device.cuh"

namespace dsp {
namespace {

// Projection of a state already on the device (a launch with no steps).  HBM
// streaming with no CTA-wide barrier: every warp works on its own granules
// (256 points: the density's partial-sum unit) through its own ring of
// shared-memory buffers (ProjShape).  Lane 0 queues both state planes of a
// granule (2 x 4 KB) by 1-D bulk copy (cp.async.bulk) completing on the
// buffer's mbarrier; the copies of the other warps on the SM are in flight
// while one projects (with two buffers a warp also overlaps its own).
// Lane l holds the granule's points l, l + 32, ..., l + 224: the pairwise tree
// of granule_sums (slot j plus slot j + s for s = 128, ..., 1) then takes its
// first three levels inside each lane and the last five across lanes by
// shuffles, the same pairs in the same order, and each point's value comes
// from project_node and store_point as in the evolve kernels, so both give the
// same bits.  Per point: 32 bytes of state read, 4 (FP32_MIXED) or 8 (FP64)
// bytes of map written; FP64-pipe work is one add per point for an FP64 map,
// none for FP32_MIXED.
// Shape per precision: warps per CTA (one CTA per SM) and buffers per warp's
// ring.  Measured on a 4096^2 state (us per launch, FP32_MIXED / FP64): 12
// warps x 2 buffers 109.5 / 258.7, 16 x 1 - / 242.1, 24 x 1 105.7 / 214.0: many
// warps with one buffer each hide both the copies and the latency of the
// double-float arithmetic best.
#ifndef DSP_PROJ32_WARPS
#define DSP_PROJ32_WARPS 24
#endif
#ifndef DSP_PROJ32_BUFS
#define DSP_PROJ32_BUFS 1
#endif
#ifndef DSP_PROJ64_WARPS
#define DSP_PROJ64_WARPS 24
#endif
#ifndef DSP_PROJ64_BUFS
#define DSP_PROJ64_BUFS 1
#endif
template <int PREC>
struct ProjShape {
    static constexpr int warps = PREC == 1 ? DSP_PROJ32_WARPS : DSP_PROJ64_WARPS;
    static constexpr int bufs = PREC == 1 ? DSP_PROJ32_BUFS : DSP_PROJ64_BUFS;
    static constexpr int threads = 32 * warps;
    static constexpr int plane = kGranule * 16;          // bytes of one state plane of a granule
    static constexpr int warp_bytes = bufs * 2 * plane;  // a warp's ring
    static constexpr int smem = warps * (warp_bytes + bufs * 8);
};
constexpr int kProjPer = kGranulePerLane;  // points per lane and granule
static_assert(kTilePoints % kGranule == 0, "tiles hold whole granules");

// The state of a staged granule's point l, as hi/lo pairs.
template <int PREC>
__device__ __forceinline__ SpinorDF granule_spinor(const unsigned char *src, int l)
{
    constexpr int kPlane = ProjShape<PREC>::plane;
    SpinorDF d;
    if constexpr (PREC == 1) {  // hi plane, lo plane
        const float4 u = reinterpret_cast<const float4 *>(src)[l];
        const float4 q = reinterpret_cast<const float4 *>(src + kPlane)[l];
        d = SpinorDF{u.x, q.x, u.y, q.y, u.z, q.z, u.w, q.w};
    } else {  // a plane, b plane
        const double2 u = reinterpret_cast<const double2 *>(src)[l];
        const double2 q = reinterpret_cast<const double2 *>(src + kPlane)[l];
        split_f64(u.x, d.arh, d.arl);
        split_f64(u.y, d.aih, d.ail);
        split_f64(q.x, d.brh, d.brl);
        split_f64(q.y, d.bih, d.bil);
    }
    return d;
}

// A point of the grid that a lane projects, and its nodes.
struct ProjPoint {
    int64_t idx;      // -1: none (past the grid's end)
    int64_t col, row;
    float2 cx, cy;
};

// FP64: the points l and l + 32 of a granule together, in packed FP32x2 (project_df on
// float2: the same operations per point).  Where every lane's values are in the
// ordinary range the conversions take their short forms too; one vote per pair keeps
// the warp together (a branch per lane was slower than the long forms).  Issue-bound
// before: 351 instructions a point, a third of them conversions; 4096^2 state 206 ->
// 153 us, the same bits.
// ALL: both points exist.
template <bool ALL>
__device__ __forceinline__ void project_pair(const ReqDesc &R, const unsigned char *src, int l,
                                             const ProjPoint &p0, const ProjPoint &p1, float2 &v0,
                                             float2 &v1)
{
    const bool in0 = ALL || p0.idx >= 0, in1 = ALL || p1.idx >= 0;
    constexpr unsigned int kAll = 0xffffffffu;
    const double2 *a = reinterpret_cast<const double2 *>(src);
    const double2 *b = reinterpret_cast<const double2 *>(src + ProjShape<0>::plane);
    const double2 one = make_double2(1.0, 1.0);
    const double2 a0 = in0 ? a[l] : one, b0 = in0 ? b[l] : one;
    const double2 a1 = in1 ? a[l + 32] : one, b1 = in1 ? b[l + 32] : one;
    bool ok = in_split_range(a0.x) && in_split_range(a0.y) && in_split_range(b0.x) &&
              in_split_range(b0.y) && in_split_range(a1.x) && in_split_range(a1.y) &&
              in_split_range(b1.x) && in_split_range(b1.y);
    v0 = v1 = make_float2(0.0f, 0.0f);
    if (__all_sync(kAll, ok)) {
        float2 arh, arl, aih, ail, brh, brl, bih, bil, oh, ol;
        split_f64_normal(a0.x, arh.x, arl.x);
        split_f64_normal(a1.x, arh.y, arl.y);
        split_f64_normal(a0.y, aih.x, ail.x);
        split_f64_normal(a1.y, aih.y, ail.y);
        split_f64_normal(b0.x, brh.x, brl.x);
        split_f64_normal(b1.x, brh.y, brl.y);
        split_f64_normal(b0.y, bih.x, bil.x);
        split_f64_normal(b1.y, bih.y, bil.y);
        ok = project_df(make_float2(p0.cx.x, p1.cx.x), make_float2(p0.cx.y, p1.cx.y),
                        make_float2(p0.cy.x, p1.cy.x), make_float2(p0.cy.y, p1.cy.y), arh, arl,
                        aih, ail, brh, brl, bih, bil, oh, ol);
        ok = ok && in_float_range(oh.x) && in_float_range(oh.y) && in_float_range(ol.x) &&
             in_float_range(ol.y);
        const double d0 = __dadd_rn(normal_to_f64(oh.x), normal_to_f64(ol.x));
        const double d1 = __dadd_rn(normal_to_f64(oh.y), normal_to_f64(ol.y));
        ok = ok && in_split_range(d0) && in_split_range(d1);
        if (__all_sync(kAll, ok)) {
            double *map = static_cast<double *>(R.map);
            if (in0) {
                if (map)
                    map[p0.idx] = d0;
                split_f64_normal(d0, v0.x, v0.y);
            }
            if (in1) {
                if (map)
                    map[p1.idx] = d1;
                split_f64_normal(d1, v1.x, v1.y);
            }
            return;
        }
    }
    if (in0)
        v0 = store_point<0>(R.map, p0.idx,
                            project_node_at<0>(R, p0.cx, p0.cy, p0.col, p0.row,
                                               granule_spinor<0>(src, l)));
    if (in1)
        v1 = store_point<0>(R.map, p1.idx,
                            project_node_at<0>(R, p1.cx, p1.cy, p1.col, p1.row,
                                               granule_spinor<0>(src, l + 32)));
}

// GROUPS: the launch has requests that may have gone step by step (ReqDesc::by_groups).
// NEAR: neighbouring granules go to one SM; else they go to the CTAs in turn, so that a small
// grid's spread over the SMs and the last round's over all of them (see launch_project).
template <int PREC, bool GROUPS, bool NEAR>
__global__ void __launch_bounds__(ProjShape<PREC>::threads, 1)
    project_kernel(const __grid_constant__ EvolveArgs args)
{
    using Sh = ProjShape<PREC>;
    constexpr int kProjPlane = Sh::plane;
    constexpr int NB = Sh::bufs;
    extern __shared__ __align__(128) unsigned char proj_dyn[];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    unsigned char *buf = proj_dyn + w * Sh::warp_bytes;  // [buffer][plane][kProjPlane]
    uint64_t *bars = reinterpret_cast<uint64_t *>(proj_dyn + Sh::warps * Sh::warp_bytes) + NB * w;
    constexpr int kGranPerTile = kTilePoints / kGranule;
    const int total = args.total_tiles * kGranPerTile;  // granules of the launch
    const int nw = gridDim.x * Sh::warps;
    const int wid = NEAR ? blockIdx.x * Sh::warps + w : w * gridDim.x + blockIdx.x;
    // A request that went step by step has been projected there: nothing to load or to do.
    // (Looked up once per request: granules of one follow each other.  A warp's first
    // granule is loaded meanwhile, whatever comes of it.)
    int seen = -1;
    bool wanted = true;
    const auto to_project = [&](int r) {
        if (GROUPS && r != seen) {
            seen = r;
            wanted = !args.r[r].by_groups || left_to_groups(args.r[r]);
        }
        return wanted;
    };
    if (lane == 0) {
        for (int b = 0; b < NB; ++b)
            mbar_init(&bars[b], 1);
        fence_mbar_init();
    }
    __syncwarp();
    // lane 0 queues both planes of granule Gi into buffer b (whole 16-byte points);
    // a granule past the end of its grid, or of a request that is not to be projected,
    // completes its phase empty
    const auto issue = [&](int Gi, int b, bool first) {
        const int T = Gi / kGranPerTile;
        const int r = find_request(args, T);
        const ReqDesc &R = args.r[r];
        const int64_t base = static_cast<int64_t>(T - R.tile_begin) * kTilePoints +
                             static_cast<int64_t>(Gi % kGranPerTile) * kGranule;
        const int64_t left = R.n_points - base;
        const uint32_t bytes =
            left <= 0 || !(first || to_project(r))
                ? 0u : 16u * static_cast<uint32_t>(left < kGranule ? left : kGranule);
        mbar_arrive_expect_tx(&bars[b], 2 * bytes);
        if (bytes > 0) {
            const unsigned char *st = static_cast<const unsigned char *>(R.state);
            unsigned char *dst = buf + b * 2 * kProjPlane;
            bulk_load(dst, st + 16 * base, bytes, &bars[b]);
            bulk_load(dst + kProjPlane, st + 16 * (R.n_points + base), bytes, &bars[b]);
        }
    };
    if (lane == 0)
        for (int b = 0; b < NB; ++b)
            if (wid + b * nw < total)
                issue(wid + b * nw, b, true);
    int k = 0;
    for (int Gi = wid; Gi < total; Gi += nw, ++k) {
        const int b = k % NB;
        const int T = Gi / kGranPerTile;
        const int r = find_request(args, T);
        const ReqDesc &R = args.r[r];
        const bool project = to_project(r);
        const bool arrived = mbar_wait_bounded(&bars[b], (k / NB) & 1);
        if (!__all_sync(0xffffffffu, arrived)) {
            if (lane == 0) {  // flag it; give the copies still queued a bounded chance to
                              // land before the warp leaves
                atomicOr(R.err, kErrTimeout);
                for (int j = 1; j < NB; ++j)
                    if (Gi + j * nw < total)
                        (void)mbar_wait_bounded(&bars[(k + j) % NB], ((k + j) / NB) & 1);
            }
            return;
        }
        const int tile = T - R.tile_begin;
        if (project && tile_ok(R, tile, R.err)) {
            const int64_t gbase = static_cast<int64_t>(tile) * kTilePoints +
                                  static_cast<int64_t>(Gi % kGranPerTile) * kGranule;
            // column and row of the granule's first point (one division per granule)
            int64_t col0 = 0, row0 = 0;
            if (lane == 0) {
                col0 = gbase % R.nx;
                row0 = gbase / R.nx;
            }
            col0 = __shfl_sync(0xffffffffu, col0, 0);
            row0 = __shfl_sync(0xffffffffu, row0, 0);
            const unsigned char *src = buf + b * 2 * kProjPlane;
            const auto spinor = [&](int l) { return granule_spinor<PREC>(src, l); };
            float2 v[kProjPer];
            if (gbase + kGranule <= R.n_points && col0 + kGranule <= R.nx) {
                // a whole granule inside one row (every grid whose nx is a multiple of 256):
                // one row node, the column nodes loaded up front, no bounds to check
                const float2 cy = R.nodes_out[R.nx + row0];
                float2 cx[kProjPer];
#pragma unroll
                for (int i = 0; i < kProjPer; ++i)
                    cx[i] = R.nodes_out[col0 + lane + 32 * i];
#pragma unroll
                for (int i = 0; i < kProjPer; i += PREC == 0 ? 2 : 1) {
                    const int l = lane + 32 * i;
                    if constexpr (PREC == 0)
                        project_pair<true>(R, src, l, ProjPoint{gbase + l, col0 + l, row0, cx[i], cy},
                                           ProjPoint{gbase + l + 32, col0 + l + 32, row0,
                                                     cx[i + 1], cy},
                                           v[i], v[i + 1]);
                    else
                        v[i] = store_point<PREC>(
                            R.map, gbase + l,
                            project_node_at<PREC>(R, cx[i], cy, col0 + l, row0, spinor(l)));
                }
            } else {
                int64_t col = col0 + lane, row = row0;
                const auto wrap = [&] {
                    while (col >= R.nx) {
                        col -= R.nx;
                        ++row;
                    }
                };
                wrap();
                // point i of the lane; called in order
                const auto next_point = [&](int i) {
                    const int64_t idx = gbase + lane + 32 * i;
                    ProjPoint p{-1, col, row, make_float2(1.0f, 0.0f), make_float2(1.0f, 0.0f)};
                    if (idx < R.n_points) {
                        p.idx = idx;
                        p.cx = R.nodes_out[col];
                        p.cy = R.nodes_out[R.nx + row];
                    }
                    col += 32;
                    wrap();
                    return p;
                };
#pragma unroll
                for (int i = 0; i < kProjPer; i += PREC == 0 ? 2 : 1) {
                    const int l = lane + 32 * i;
                    const ProjPoint p = next_point(i);
                    if constexpr (PREC == 0) {
                        const ProjPoint q = next_point(i + 1);
                        project_pair<false>(R, src, l, p, q, v[i], v[i + 1]);
                    } else {
                        v[i] = make_float2(0.0f, 0.0f);
                        if (p.idx >= 0)
                            v[i] = store_point<PREC>(R.map, p.idx,
                                                     project_node_at<PREC>(R, p.cx, p.cy, p.col,
                                                                           p.row, spinor(l)));
                    }
                }
            }
            granule_tree(v, lane);
            const int64_t gi = gbase / kGranule;
            if (lane == 0 && gi < (R.n_points + kGranule - 1) / kGranule)
                R.partials[gi] = df_to_f64(v[0].x, v[0].y);
        }
        __syncwarp();  // the warp is done with buffer b
        if (lane == 0 && Gi + NB * nw < total)
            issue(Gi + NB * nw, b, false);
    }
}

// One cluster per density: 1024 fixed-order strided sums of the granule partials (sum t
// takes partials t, t + 1024, ...), then a pairwise tree over them.  The strided sums of
// a large map are a chain of FP64 adds per thread (64 for 4096^2), and one CTA of 1024
// threads puts 32 warps of them on one SM's FP64 pipe: 25 us for 65536 partials.  Spread
// over a cluster of 8 CTAs each scheduler has one warp; the sums meet in rank 0's shared
// memory for the tree.  The order of every addition is the one-CTA kernel's.
constexpr int kFinSums = 1024, kFinCtas = 8, kFinThreads = kFinSums / kFinCtas;
__global__ void __cluster_dims__(kFinCtas, 1, 1) __launch_bounds__(kFinThreads)
    finalize_kernel(const __grid_constant__ FinalizeArgs args)
{
    __shared__ double red[kFinSums];
    const FinDesc &f = args.f[blockIdx.x / kFinCtas];
    const int rank = blockIdx.x % kFinCtas;
    const int slot = rank * kFinThreads + threadIdx.x;
    double acc = 0.0;
#pragma unroll 8
    for (int64_t i = slot; i < f.n_parts; i += kFinSums)
        acc += f.partials[i];
    uint32_t dst;  // rank 0's red[slot]
    asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(dst) : "r"(smem_addr(&red[slot])));
    asm volatile("barrier.cluster.arrive;\n\tbarrier.cluster.wait;" ::: "memory");
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(dst), "d"(acc) : "memory");
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
    if (rank != 0)
        return;
    for (int s = kFinSums / 2; s > 0; s >>= 1) {
        for (int i = threadIdx.x; i < s; i += kFinThreads)
            red[i] += red[i + s];
        __syncthreads();
    }
    if (threadIdx.x == 0)
        *f.out = red[0] * f.scale;
}

// Time-parallel combination, one thread per momentum: psi <- M_s psi for s =
// 0 .. S-1 in time order, starting from v(p + A_in), all in FP64.  Bound by FP64 latency
// on a small grid: 16 FP64 operations per segment, 4 more to bring an FP32_MIXED column
// to double (the conversions themselves are integer operations: a cvt issues on the
// FP64 pipe), the columns of 4 segments loaded ahead.
template <int PREC>
__global__ void __launch_bounds__(128) combine_kernel(const __grid_constant__ CombineArgs a)
{
    const int64_t idx = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (idx >= a.n_points)
        return;
    const double vs = a.valley > 0 ? 1.0 : -1.0;
    const double px = grid_node(a.px_min, a.hx, idx % a.nx);
    const double py = grid_node(a.py_min, a.hy, a.row0 + idx / a.nx);
    double ar, ai, br, bi;
    initial_spinor(px + a.a_in[0], py + a.a_in[1], vs, ar, ai, br, bi);
    const size_t slab = static_cast<size_t>(a.n_points) * 32;
#pragma unroll 4
    for (int s = 0; s < a.n_segments; ++s) {
        const unsigned char *seg = static_cast<const unsigned char *>(a.segs) + s * slab;
        double alr, ali, ber, bei;  // (alpha, beta): first column of M_s
        if constexpr (PREC == 1) {
            const float4 h = reinterpret_cast<const float4 *>(seg)[idx];
            const float4 l = reinterpret_cast<const float4 *>(seg)[a.n_points + idx];
            alr = df_to_f64(h.x, l.x);
            ali = df_to_f64(h.y, l.y);
            ber = df_to_f64(h.z, l.z);
            bei = df_to_f64(h.w, l.w);
        } else {
            const double2 c0 = reinterpret_cast<const double2 *>(seg)[idx];
            const double2 c1 = reinterpret_cast<const double2 *>(seg)[a.n_points + idx];
            alr = c0.x; ali = c0.y; ber = c1.x; bei = c1.y;
        }
        // a' = alpha a - conj(beta) b ; b' = beta a + conj(alpha) b
        const double nar = alr * ar - ali * ai - (ber * br + bei * bi);
        const double nai = alr * ai + ali * ar - (ber * bi - bei * br);
        const double nbr = ber * ar - bei * ai + (alr * br + ali * bi);
        const double nbi = ber * ai + bei * ar + (alr * bi - ali * br);
        ar = nar; ai = nai; br = nbr; bi = nbi;
    }
    if constexpr (PREC == 1) {
        float4 *hi = static_cast<float4 *>(a.state);
        float4 *lo = hi + a.n_points;
        const float h0 = static_cast<float>(ar), h1 = static_cast<float>(ai);
        const float h2 = static_cast<float>(br), h3 = static_cast<float>(bi);
        hi[idx] = make_float4(h0, h1, h2, h3);
        lo[idx] = make_float4(static_cast<float>(ar - h0), static_cast<float>(ai - h1),
                              static_cast<float>(br - h2), static_cast<float>(bi - h3));
    } else {
        double2 *pa = static_cast<double2 *>(a.state);
        pa[idx] = make_double2(ar, ai);
        pa[a.n_points + idx] = make_double2(br, bi);
    }
}

}  // namespace

cudaError_t launch_combine(const CombineArgs &args, int precision, cudaStream_t stream)
{
    if (args.n_points <= 0)
        return cudaSuccess;
    const int64_t blocks = (args.n_points + 127) / 128;
    if (precision == 1)
        combine_kernel<1><<<static_cast<unsigned>(blocks), 128, 0, stream>>>(args);
    else
        combine_kernel<0><<<static_cast<unsigned>(blocks), 128, 0, stream>>>(args);
    return cudaGetLastError();
}

// The FP32_MIXED strip kernels, one object of dsp_strip.cu each.
cudaError_t strip_ctas_per_sm_s0_np2(int *ctas);
cudaError_t strip_ctas_per_sm_s1_np2(int *ctas);
cudaError_t strip_ctas_per_sm_s2_np2(int *ctas);
cudaError_t launch_evolve_strip_s0_np2(const EvolveArgs &args, cudaStream_t stream);
cudaError_t launch_evolve_strip_s0_np1(const EvolveArgs &args, cudaStream_t stream);
cudaError_t launch_evolve_strip_s1_np2(const EvolveArgs &args, cudaStream_t stream);
cudaError_t launch_evolve_strip_s1_np1(const EvolveArgs &args, cudaStream_t stream);
cudaError_t launch_evolve_strip_s2_np2(const EvolveArgs &args, cudaStream_t stream);
cudaError_t launch_evolve_strip_s2_np1(const EvolveArgs &args, cudaStream_t stream);

cudaError_t strip_ctas_per_sm(int scheme, int *ctas)
{
    return scheme == 0   ? strip_ctas_per_sm_s0_np2(ctas)
           : scheme == 1 ? strip_ctas_per_sm_s1_np2(ctas)
                         : strip_ctas_per_sm_s2_np2(ctas);
}

cudaError_t launch_evolve_strip(const EvolveArgs &args, int scheme, int strip_h,
                                cudaStream_t stream)
{
    const bool half = strip_h == 2;
    if (scheme == 0)
        return half ? launch_evolve_strip_s0_np1(args, stream)
                    : launch_evolve_strip_s0_np2(args, stream);
    if (scheme == 1)
        return half ? launch_evolve_strip_s1_np1(args, stream)
                    : launch_evolve_strip_s1_np2(args, stream);
    return half ? launch_evolve_strip_s2_np1(args, stream) : launch_evolve_strip_s2_np2(args, stream);
}

template <int PREC, bool GROUPS, bool NEAR>
static cudaError_t launch_project(const EvolveArgs &args, int grid, cudaStream_t stream)
{
    using Sh = ProjShape<PREC>;
    // the warps' rings are above the 48 KB a kernel gets without asking
    const cudaError_t e = cudaFuncSetAttribute(
        project_kernel<PREC, GROUPS, NEAR>, cudaFuncAttributeMaxDynamicSharedMemorySize, Sh::smem);
    if (e != cudaSuccess)
        return e;
    project_kernel<PREC, GROUPS, NEAR><<<grid, Sh::threads, Sh::smem, stream>>>(args);
    return cudaGetLastError();
}

cudaError_t launch_project(const EvolveArgs &args, int precision, cudaStream_t stream)
{
    if (args.nreq <= 0 || args.total_tiles <= 0)
        return cudaSuccess;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess)
        e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess)
        return e;
    bool groups = false, whole = true;
    for (int i = 0; i < args.nreq; ++i) {
        groups = groups || args.r[i].by_groups;
        whole = whole && args.r[i].nx % kGranule == 0;
    }
    // one CTA per SM, no more CTAs than granules
    const int granules = args.total_tiles * (kTilePoints / kGranule);
    const int grid = granules < sms ? granules : sms;
    if (precision != 1)
        return launch_project<0, false, false>(args, grid, stream);
    // Rows of whole granules, four or more of them a warp: neighbours on one SM (us a launch on
    // buffers not in L2, in turn and neighbours: 2048^2 32.7 and 32.5, 3072 x 2000 44.3 and 43.4,
    // 4096^2 101.9 and 100.2).  Fewer or ragged ones in turn (100 x 75 6.1 and 7.6, 1024^2 8.4
    // and 10.4, 1801 x 2001 31.1 and 31.6); the order as a constant, since one picked in the
    // kernel costs every grid up to 1% (1500^2 22.6 and 22.9).
    if (whole && granules >= 4 * grid * ProjShape<1>::warps)
        return groups ? launch_project<1, true, true>(args, grid, stream)
                      : launch_project<1, false, true>(args, grid, stream);
    return groups ? launch_project<1, true, false>(args, grid, stream)
                  : launch_project<1, false, false>(args, grid, stream);
}

cudaError_t launch_finalize(const FinalizeArgs &args, cudaStream_t stream)
{
    if (args.count <= 0)
        return cudaSuccess;
    finalize_kernel<<<args.count * kFinCtas, kFinThreads, 0, stream>>>(args);
    return cudaGetLastError();
}

}  // namespace dsp
