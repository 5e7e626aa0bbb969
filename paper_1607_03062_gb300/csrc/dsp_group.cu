// dsp_group.cu -- the FP32_MIXED evolve kernel on expanded step groups, and the kernel
// that expands a pulse's groups.  Shared device code is in dsp_device.cuh.

#include "dsp_device.cuh"
#include "dsp_steptable.h"

namespace dsp {
namespace {

// ---------------------------------------------------------------------------
// Expanded step groups
//
// The product of a group's G steps exp(-i sigma.P_n), P_n = dt (p + A_n), is
// exp(-i sigma.w) with w(p) = S + (small), S = G dt p + sum_n dt A_n: what makes w
// differ from S is how A changes inside the group, which does not depend on p, so
// it is expanded once per group and pulse (the Magnus series of the steps,
// prep_groups_kernel) and the evolve kernel evaluates, per momentum and GROUP
// instead of per step,
//   w_z  = C + S x m1 + x (S x n3 + x S x n5)           x = S.S, u x v = u_x v_y - u_y v_x
//   w_xy = S + (S_y, -S_x) (S x u2 + x S x u4) + K S
// (GroupEntry).  A STRANG_XY step is exp(-i sigma.P') with P' = P + cubic(P) in closed
// series, so its groups are those of P': the same w with the cubic and fifth-order terms
// of P' added to w_xy and their part of S x m1 to w_z (group_step).  What the
// expansion drops is summed over the run (GroupSums); the kernels pick G and the level
// from the sums (pick_plan), and where no G passes the step-by-step chains (dsp_strip.cu, dsp_mixed.cu), queued behind, take the run.
//
// S comes as hi + lo (each from an exact sum of the hi/lo halves of G dt p and of
// the group's sum of dt A), so no step's momentum is rounded on the way.  Three levels:
//   lite  drops n5, u2, u4 and K (their sums passed the bound too) and adds the lo
//         part of S to its hi part;
//   full  keeps everything, and takes cos|w| - 1 from the rounded vector part of the
//         operator, so that the operator is unitary to the rounding of its entries;
//   wide  also applies S and the small rest of w apart, because at large group angles
//         the rounding of their sum would show.
//
// What bounds it: FP32 issue.  Per spinor and group 42 (lite), 64 (full) or 76 (wide)
// lane operations plus a column part shared by the warp's rows, against 9 and more per
// spinor and STEP of the chains.  FMA pipe 83% busy (lite; packed instructions hold it
// two cycles), issue 50%, DRAM idle.
//
// Tiles: one warp owns 32 columns x H rows (H = 4, 2: packed FP32x2 row pairs; H =
// 1: scalar), any nx (columns past the row's end idle), and works alone: its own
// double-buffered 1-D bulk copies of 32 group entries (bounded mbarrier waits), its
// own table of the row parts of 32 groups (one lane per group), no CTA-wide
// barrier.  A grid too small to fill the chip with 4-row warps takes lower ones
// (group_rows in dsp_api.cpp); every point's arithmetic is the same for every H.
// The projection is the projection kernel's, on the state this kernel leaves.
//
// Measured (GB300, whole solves, step by step -> expanded): 2048^2 x 1e5 sin^2 pulse
// 209.2 -> 35.2 ms (lite, G = 16); 1024^2 x 3e4 Gaussian pulse 22.6 -> 5.05 ms (wide,
// 16); 1000 x 750 x 2e4 two colours 10.36 -> 2.46 ms (wide, 16; contiguous tiles
// before); 512^2 x 12000 MAGNUS4 3.14 -> 0.575 ms (full); 256^2 x 2e4 paper pulse 1.42
// -> 0.375 ms; 512 x 384 x 12000 STRANG_XY 1.79 -> 0.55 ms (full).  2-norm error of
// |c+|^2 against 64 bits on the last four: 3.7e-7 -> 2.3e-7, 2.0e-7 -> 1.3e-7, 5.0e-7
// -> 2.3e-7, 2.8e-7 -> 1.2e-7.
// ---------------------------------------------------------------------------

constexpr int kGrpChunk = 32;  // group entries per staged chunk: one per lane
constexpr int kGrpStage = kGrpChunk * static_cast<int>(sizeof(GroupEntry));
static_assert(sizeof(GroupEntry) % 16 == 0, "bulk copies of whole entries");

// cos - 1 and sinc - 1 series degrees in |w|^2: at a level's largest angle the
// first omitted terms turn a group by 1e-11 (lite, 0.25), 1e-13 (full, 0.32) and 3e-12
// (wide, 0.72), 1e-7 over 1e4 groups; the cos of full and wide, off by 3e-9 and 4e-11,
// is corrected from the sinc.
constexpr int kLiteDC = 4, kLiteDS = 3, kFullDC = 3, kFullDS = 4, kWideDC = 5, kWideDS = 5;
// Steps outside whole groups, one at a time: theta <= kGroupAngleTan / 2.
constexpr int kSingleDC = 4, kSingleDS = 4;

struct WarpSmem {
    unsigned char stage[2][kGrpStage];  // bulk-copied GroupEntry
    float4 rows[8][kGrpChunk];          // row parts: [pack (or row) and part][group]
    float4 prow[4];                     // per row: G dt p_y as hi + lo
    uint64_t bars[2];
};

template <typename V>
struct GroupPoint {  // spinor(s) as hi + lo
    V ar, ai, br, bi, lar, lai, lbr, lbi;
};

// The column part of a group, one per lane (scalars shared by the lane's rows).
struct GroupCol {
    float Sx, Tx;  // hi of S_x; lite: S_x hi + lo
    float m1y, n3y, n5y, u2y, u4y;
    float kx, Kyx;  // wide: lo of S_x plus Kxx S_x; Kyx
    float C;
};

// The row part of a group (V = float2: the two rows of a pack).
template <typename V>
struct GroupRow {
    V Sy;        // hi of S_y (lite: hi + lo)
    V y2;        // lite: S_y^2
    V r1, r3;    // C - S_y m1x, -S_y n3x
    V r5, e2, e4;  // -S_y n5x, -S_y u2x, -S_y u4x
    V kx, ky;    // Kxy S_y; Kyy S_y plus the lo of S_y
};

__device__ __forceinline__ GroupCol group_col(const float4 *e, float gxh, float gxl, bool wide)
{
    const float4 e0 = e[0];  // sum A_x hi, lo, m1y, n3y
    GroupCol c;
    float lo;
    two_sum(gxh, e0.x, c.Sx, lo);
    lo = __fadd_rn(lo, __fadd_rn(gxl, e0.y));
    c.m1y = e0.z;
    c.n3y = e0.w;
    c.Tx = __fadd_rn(c.Sx, lo);
    if (wide) {
        const float4 e1 = e[1];  // n5y, u2y, u4y, Kxx
        c.n5y = e1.x;
        c.u2y = e1.y;
        c.u4y = e1.z;
        c.kx = __fmaf_rn(c.Sx, e1.w, lo);
        const float4 e2 = e[2];
        c.Kyx = e2.x;
        c.C = e2.w;
    }
    return c;
}

// The row parts of one group entry for a row with G dt p_y = (gyh, gyl), as scalars.
template <bool WIDE>
__device__ __forceinline__ GroupRow<float> group_row(const float4 *e, float gyh, float gyl)
{
    const float4 e2 = e[2], e3 = e[3];  // Kyx, sum A_y hi, lo, C; m1x, n3x, n5x, u2x
    GroupRow<float> r;
    float lo;
    two_sum(gyh, e2.y, r.Sy, lo);
    lo = __fadd_rn(lo, __fadd_rn(gyl, e2.z));
    if constexpr (!WIDE) {
        r.Sy = __fadd_rn(r.Sy, lo);
        r.y2 = __fmul_rn(r.Sy, r.Sy);
    }
    r.r1 = __fmaf_rn(-r.Sy, e3.x, e2.w);
    r.r3 = -__fmul_rn(r.Sy, e3.y);
    if constexpr (WIDE) {
        const float4 e4 = e[4];  // u4x, Kxy, Kyy
        r.r5 = -__fmul_rn(r.Sy, e3.z);
        r.e2 = -__fmul_rn(r.Sy, e3.w);
        r.e4 = -__fmul_rn(r.Sy, e4.x);
        r.kx = __fmul_rn(r.Sy, e4.y);
        r.ky = __fmaf_rn(r.Sy, e4.z, lo);
    }
    return r;
}

// Row parts in shared memory: a pack's are interleaved pairs (lite 2, wide 4
// float4), a single row's packed (lite 1, wide 2).
template <bool WIDE>
__device__ __forceinline__ void put_rows(float4 (*rows)[kGrpChunk], int q, int g,
                                         const GroupRow<float> &a, const GroupRow<float> &b)
{
    float4(*t)[kGrpChunk] = rows + (WIDE ? 4 : 2) * q;
    if constexpr (WIDE) {
        t[0][g] = make_float4(a.Sy, b.Sy, a.r1, b.r1);
        t[1][g] = make_float4(a.r3, b.r3, a.r5, b.r5);
        t[2][g] = make_float4(a.e2, b.e2, a.e4, b.e4);
        t[3][g] = make_float4(a.kx, b.kx, a.ky, b.ky);
    } else {
        t[0][g] = make_float4(a.Sy, b.Sy, a.y2, b.y2);
        t[1][g] = make_float4(a.r1, b.r1, a.r3, b.r3);
    }
}
template <bool WIDE>
__device__ __forceinline__ void put_row(float4 (*rows)[kGrpChunk], int g, const GroupRow<float> &a)
{
    if constexpr (WIDE) {
        rows[0][g] = make_float4(a.Sy, a.r1, a.r3, a.r5);
        rows[1][g] = make_float4(a.e2, a.e4, a.kx, a.ky);
    } else {
        rows[0][g] = make_float4(a.Sy, a.y2, a.r1, a.r3);
    }
}
template <bool WIDE>
__device__ __forceinline__ void get_row(const float4 (*rows)[kGrpChunk], int q, int g,
                                        GroupRow<float2> &r)
{
    const float4(*t)[kGrpChunk] = rows + (WIDE ? 4 : 2) * q;
    const float4 a = t[0][g], b = t[1][g];
    r.Sy = make_float2(a.x, a.y);
    if constexpr (WIDE) {
        const float4 c = t[2][g], d = t[3][g];
        r.r1 = make_float2(a.z, a.w);
        r.r3 = make_float2(b.x, b.y);
        r.r5 = make_float2(b.z, b.w);
        r.e2 = make_float2(c.x, c.y);
        r.e4 = make_float2(c.z, c.w);
        r.kx = make_float2(d.x, d.y);
        r.ky = make_float2(d.z, d.w);
    } else {
        r.y2 = make_float2(a.z, a.w);
        r.r1 = make_float2(b.x, b.y);
        r.r3 = make_float2(b.z, b.w);
    }
}
template <bool WIDE>
__device__ __forceinline__ void get_row(const float4 (*rows)[kGrpChunk], int, int g,
                                        GroupRow<float> &r)
{
    const float4 a = rows[0][g];
    r.Sy = a.x;
    if constexpr (WIDE) {
        const float4 b = rows[1][g];
        r.r1 = a.y;
        r.r3 = a.z;
        r.r5 = a.w;
        r.e2 = b.x;
        r.e4 = b.y;
        r.kx = b.z;
        r.ky = b.w;
    } else {
        r.y2 = a.y;
        r.r1 = a.z;
        r.r3 = a.w;
    }
}

// psi <- exp(-i sigma.w) psi for one group.  The operator's M - I is
// [[m - i q_z, -(q_y + i q_x)], [q_y - i q_x, m + i q_z]], m = cos|w| - 1, q = sinc|w| w.
// STRANG (full and wide): the steps' P' = P + (-P_x P_y^2 (1/3 + (2 P_x^2 + P_y^2)/45),
// P_y P_x^2 (1/6 + 7 P_x^2/360 - 2 P_y^2/45)) at P = S/G, and through its derivative
// S x m1 gains (P_x^2/6 + P_y^2/3)(S_x m1_y + S_y m1_x); g2 = 1/G^2, C the entry's.
template <int LEVEL, bool STRANG, typename V>
__device__ __forceinline__ void group_step(GroupPoint<V> &p, const GroupCol &c,
                                           const GroupRow<V> &r, float g2)
{
    if constexpr (LEVEL == kGroupLite) {
        const V Tx = vbc<V>(c.Tx);
        const V x = vfma(Tx, Tx, r.y2);
        const V A1 = vfma(Tx, vbc<V>(c.m1y), r.r1), A3 = vfma(Tx, vbc<V>(c.n3y), r.r3);
        const V wz = vfma(x, A3, A1);
        const V m = vmul(vhorner<V, kLiteDC, 1, 0>(x), x);
        const V s = vmul(vhorner<V, kLiteDS, 1, 1>(x), x);
        apply_group(p, m, vneg(vfma(s, wz, wz)), vfma(s, r.Sy, r.Sy), vfma(s, Tx, Tx));
    } else {
        const V Sx = vbc<V>(c.Sx), Sy = r.Sy;
        const V v2 = vmul(Sy, Sy);
        const V x0 = vfma(Sx, Sx, v2);
        const V A1 = vfma(Sx, vbc<V>(c.m1y), r.r1), A3 = vfma(Sx, vbc<V>(c.n3y), r.r3);
        const V A5 = vfma(Sx, vbc<V>(c.n5y), r.r5);
        V wz = vfma(x0, vfma(x0, A5, A3), A1);
        const V e = vfma(x0, vfma(Sx, vbc<V>(c.u4y), r.e4), vfma(Sx, vbc<V>(c.u2y), r.e2));
        // w_xy = S + v, v small
        V vx = vfma(Sy, e, vadd(vbc<V>(c.kx), r.kx));
        V vy = vfma(vneg(Sx), e, vfma(Sx, vbc<V>(c.Kyx), r.ky));
        if constexpr (STRANG) {
            // X = P_x^2, Y = P_y^2
            const float Xs = __fmul_rn(g2, __fmul_rn(c.Sx, c.Sx));
            const V X = vbc<V>(Xs), Y = vmul(vbc<V>(g2), v2);
            const V hx = vfma(Y, vbc<V>(1.0f / 45.0f),
                              vbc<V>(__fmaf_rn(Xs, 2.0f / 45.0f, 1.0f / 3.0f)));
            const V hy = vfma(Y, vbc<V>(-2.0f / 45.0f),
                              vbc<V>(__fmaf_rn(Xs, 7.0f / 360.0f, 1.0f / 6.0f)));
            vx = vfma(vmul(vneg(Y), hx), Sx, vx);
            vy = vfma(vmul(X, hy), Sy, vy);
            // S_x m1_y + S_y m1_x = 2 S_x m1_y - (A1 - C)
            const V sym = vfma(vbc<V>(__fadd_rn(c.Sx, c.Sx)), vbc<V>(c.m1y),
                               vadd(vbc<V>(c.C), vneg(A1)));
            wz = vfma(vfma(Y, vbc<V>(1.0f / 3.0f), vbc<V>(__fmul_rn(Xs, 1.0f / 6.0f))), sym, wz);
        }
        // m = cos - 1 with one Newton step on (1 + m)^2 + q.q = 1, y = q.q
        const auto cos1 = [](V m, V y) {
            return vfma(vbc<V>(-0.5f), vfma(vbc<V>(2.0f), m, vfma(m, m, y)), m);
        };
        if constexpr (LEVEL == kGroupFull) {
            const V Tx = vadd(Sx, vx), Ty = vadd(Sy, vy);
            const V x = vfma(Tx, Tx, vfma(Ty, Ty, vmul(wz, wz)));
            const V s = vmul(vhorner<V, kFullDS, 1, 1>(x), x);
            const V qx = vfma(s, Tx, Tx), qy = vfma(s, Ty, Ty), qz = vfma(s, wz, wz);
            const V m = cos1(vmul(vhorner<V, kFullDC, 1, 0>(x), x),
                             vfma(qx, qx, vfma(qy, qy, vmul(qz, qz))));
            apply_group(p, m, vneg(qz), qy, qx);
            return;
        }
        const V Tx = vadd(Sx, vx), Ty = vadd(Sy, vy);
        const V x = vfma(Tx, Tx, vfma(Ty, Ty, vmul(wz, wz)));
        const V s = vmul(vhorner<V, kWideDS, 1, 1>(x), x);
        // q = S + (v + s (S + v)), the outer sum left unrounded for the update; q.q from that
        // sum, rounded (from x (1 + s)^2, one operation less, the error against 64 bits is
        // up to half as large again)
        const V qx = vfma(s, Tx, vx), qy = vfma(s, Ty, vy), qz = vfma(s, wz, wz);
        const V fx = vadd(Sx, qx), fy = vadd(Sy, qy);
        const V m = cos1(vmul(vhorner<V, kWideDC, 1, 0>(x), x),
                         vfma(fx, fx, vfma(fy, fy, vmul(qz, qz))));
        const V nqx = vneg(qx), nqy = vneg(qy), nqz = vneg(qz), nSx = vneg(Sx), nSy = vneg(Sy);
        V dar = vfma(m, p.ar, vfma(qz, p.ai, vfma(nqy, p.br, vfma(qx, p.bi, p.lar))));
        V dai = vfma(m, p.ai, vfma(nqz, p.ar, vfma(nqy, p.bi, vfma(nqx, p.br, p.lai))));
        V dbr = vfma(m, p.br, vfma(nqz, p.bi, vfma(qy, p.ar, vfma(qx, p.ai, p.lbr))));
        V dbi = vfma(m, p.bi, vfma(qz, p.br, vfma(qy, p.ai, vfma(nqx, p.ar, p.lbi))));
        dar = vfma(nSy, p.br, vfma(Sx, p.bi, dar));
        dai = vfma(nSy, p.bi, vfma(nSx, p.br, dai));
        dbr = vfma(Sy, p.ar, vfma(Sx, p.ai, dbr));
        dbi = vfma(Sy, p.ai, vfma(nSx, p.ar, dbi));
        V t;
        t = vadd(p.ar, dar); p.lar = vadd(dar, vneg(vadd(t, vneg(p.ar)))); p.ar = t;
        t = vadd(p.ai, dai); p.lai = vadd(dai, vneg(vadd(t, vneg(p.ai)))); p.ai = t;
        t = vadd(p.br, dbr); p.lbr = vadd(dbr, vneg(vadd(t, vneg(p.br)))); p.br = t;
        t = vadd(p.bi, dbi); p.lbi = vadd(dbi, vneg(vadd(t, vneg(p.bi)))); p.bi = t;
    }
}

// One step alone (outside whole groups): n = (P_x, P_y, n_z), n_z = 0 for EXACT and
// MAGNUS4's commutator part P_x D_y - P_y D_x.
template <typename V>
__device__ __forceinline__ void single_step(GroupPoint<V> &p, V Px, V Py, float dx, float dy)
{
    const V nz = vfma(Px, vbc<V>(dy), vneg(vmul(Py, vbc<V>(dx))));
    const V x = vfma(Px, Px, vfma(Py, Py, vmul(nz, nz)));
    const V m = vmul(vhorner<V, kSingleDC, 1, 0>(x), x);
    const V s = vmul(vhorner<V, kSingleDS, 1, 1>(x), x);
    apply_group(p, m, vneg(vfma(s, nz, nz)), vfma(s, Py, Py), vfma(s, Px, Px));
}

template <typename V>
__device__ __forceinline__ void single_step_strang(GroupPoint<V> &p, V Px, V Py)
{  // coeffs_strang's operations
    const V xx = vmul(Px, Px), xy = vmul(Py, Py);
    const V cx = vmul(vhorner<V, kSingleDC, 1, 0>(xx), xx);
    const V cy = vmul(vhorner<V, kSingleDC, 1, 0>(xy), xy);
    const V sx = vfma(vmul(vhorner<V, kSingleDS, 1, 1>(xx), xx), Px, Px);
    const V sy = vfma(vmul(vhorner<V, kSingleDS, 1, 1>(xy), xy), Py, Py);
    apply_group(p, vfma(cx, cy, vadd(cx, cy)), vbc<V>(0.0f), sy, vfma(cy, sx, sx));
}

// A warp's spinors: H rows of one column per lane, as packs of two rows (H = 4, 2)
// or one row alone (H = 1).
template <int H>
struct Rows {
    using V = typename std::conditional<H == 1, float, float2>::type;
    static constexpr int N = H == 1 ? 1 : H / 2;
    GroupPoint<V> p[N];
};

__device__ __forceinline__ float &lane_of(float &v, int) { return v; }
__device__ __forceinline__ float &lane_of(float2 &v, int k) { return (k & 1) ? v.y : v.x; }
__device__ __forceinline__ float2 pair_of(float a, float b, float2 *) { return make_float2(a, b); }
__device__ __forceinline__ float pair_of(float a, float, float *) { return a; }

template <int H, int LEVEL, bool STRANG>
__device__ void body_group(const ReqDesc &R, int size, int tile, WarpSmem &sm, int *err)
{
    constexpr bool WIDE = LEVEL != kGroupLite;  // the entries' parts that full and wide read
    using RowsT = Rows<H>;
    using V = typename RowsT::V;
    constexpr int N = RowsT::N;
    const int lane = threadIdx.x & 31;
    const int ncb = (R.nx + 31) / 32;
    const int rb = tile / ncb, cb = tile - rb * ncb;
    const int64_t row_first = static_cast<int64_t>(rb) * H;
    const int64_t col = static_cast<int64_t>(cb) * 32 + lane;
    const bool col_ok = col < R.nx;
    const double vs = R.valley > 0 ? 1.0 : -1.0;
    const int G = group_size(0) >> size;
    const double gs = static_cast<double>(G) * vs;  // exact scalings of dt p
    const float inv_g = 1.0f / static_cast<float>(G);
    float4 *hi_plane = static_cast<float4 *>(R.state);
    float4 *lo_plane = hi_plane + R.n_points;

    const double px = grid_node(R.px_min, R.hx, col);
    const double tx = gs * (R.dt * px);
    const float gxh = static_cast<float>(tx);
    const float gxl = static_cast<float>(tx - static_cast<double>(gxh));
    RowsT s;
#pragma unroll
    for (int k = 0; k < H; ++k) {
        const int64_t row = row_first + k;
        const bool valid = col_ok && row < R.ny;
        const int64_t idx = row * R.nx + col;
        const double py = grid_node(R.py_min, R.hy, R.row0 + row);
        if (lane == 0) {
            const double ty = gs * (R.dt * py);
            const float h = static_cast<float>(ty);
            sm.prow[k] = make_float4(h, static_cast<float>(ty - static_cast<double>(h)), 0.0f, 0.0f);
        }
        float4 h, l;
        if (R.fresh || !valid) {
            double ar = 1.0, ai = 0.0, br = 0.0, bi = 0.0;  // identity column
            if (!R.init_identity)
                initial_spinor(px + R.a_in[0], py + R.a_in[1], vs, ar, ai, br, bi);
            h = make_float4(static_cast<float>(ar), static_cast<float>(ai), static_cast<float>(br),
                            static_cast<float>(bi));
            l = make_float4(static_cast<float>(ar - static_cast<double>(h.x)),
                            static_cast<float>(ai - static_cast<double>(h.y)),
                            static_cast<float>(br - static_cast<double>(h.z)),
                            static_cast<float>(bi - static_cast<double>(h.w)));
        } else {
            h = hi_plane[idx];
            l = lo_plane[idx];
        }
        GroupPoint<V> &p = s.p[k / 2];
        lane_of(p.ar, k) = h.x; lane_of(p.ai, k) = h.y; lane_of(p.br, k) = h.z; lane_of(p.bi, k) = h.w;
        lane_of(p.lar, k) = l.x; lane_of(p.lai, k) = l.y; lane_of(p.lbr, k) = l.z; lane_of(p.lbi, k) = l.w;
    }
    __syncwarp();  // prow is written

    // a step of the launch outside whole groups
    const auto single = [&](int64_t n) {
        float4 a;  // dt A_x, dt A_y, D_x, D_y
        if (R.scheme == 2) {
            a = __ldg(static_cast<const float4 *>(R.table) + n);
        } else {
            const float2 b = __ldg(static_cast<const float2 *>(R.table) + n);
            a = make_float4(b.x, b.y, 0.0f, 0.0f);
        }
        const float Px = __fadd_rn(gxh * inv_g, __fadd_rn(a.x, gxl * inv_g));
#pragma unroll
        for (int q = 0; q < N; ++q) {
            const float4 p0 = sm.prow[2 * q], p1 = sm.prow[H == 1 ? 0 : 2 * q + 1];
            const float y0 = __fadd_rn(p0.x * inv_g, __fadd_rn(a.y, p0.y * inv_g));
            const float y1 = __fadd_rn(p1.x * inv_g, __fadd_rn(a.y, p1.y * inv_g));
            const V Py = pair_of(y0, y1, static_cast<V *>(nullptr));
            if constexpr (STRANG)
                single_step_strang(s.p[q], vbc<V>(Px), Py);
            else
                single_step(s.p[q], vbc<V>(Px), Py, a.z, a.w);
        }
    };

    // whole groups [g0, g1) of absolute index, steps alone before and after
    int64_t g0 = (R.step_begin + G - 1) / G, g1 = R.step_end / G;
    if (g1 < g0)
        g0 = g1 = R.step_begin / G + 1;  // inside one group: every step alone
#ifdef DSP_BOUNDS_CHECK
    if (R.step_begin < 0 || R.step_end > R.table_steps ||
        R.step_end > R.groups.n_steps) {
        if (lane == 0)
            atomicOr(err, kErrBounds);
        return;
    }
#endif
    const int64_t head_end = g1 > g0 ? g0 * G : R.step_end;
    const int nchunks = static_cast<int>((g1 - g0 + kGrpChunk - 1) / kGrpChunk);
    const GroupEntry *entries =
        R.groups.entries + group_entries_before(R.groups.n_steps, R.groups.first, size) + g0;
    const auto chunk_len = [&](int c) {
        const int64_t rem = g1 - g0 - static_cast<int64_t>(c) * kGrpChunk;
        return rem < kGrpChunk ? static_cast<int>(rem) : kGrpChunk;
    };
    const auto issue = [&](int c) {  // lane 0
        const uint32_t bytes = static_cast<uint32_t>(chunk_len(c)) * sizeof(GroupEntry);
        mbar_arrive_expect_tx(&sm.bars[c & 1], bytes);
        if (!(c == 0 && R.withhold_first_copy))  // test hook: the wait for chunk 0 runs out
            bulk_load(sm.stage[c & 1], entries + static_cast<int64_t>(c) * kGrpChunk, bytes,
                      &sm.bars[c & 1]);
    };
    if (lane == 0) {
        for (int c = 0; c < 2 && c < nchunks; ++c)
            issue(c);
        if (nchunks == 0 && R.withhold_first_copy)
            mbar_arrive_expect_tx(&sm.bars[0], 16);
    }
    if (nchunks == 0 && R.withhold_first_copy) {
        if (!mbar_wait_bounded(&sm.bars[0], 0) && lane == 0)
            atomicOr(err, kErrTimeout);
        return;
    }
    for (int64_t n = R.step_begin; n < head_end; ++n)
        single(n);
    for (int c = 0; c < nchunks; ++c) {
        const bool arrived = mbar_wait_bounded(&sm.bars[c & 1], (c >> 1) & 1);
        if (!__all_sync(0xffffffffu, arrived)) {
            if (lane == 0) {  // flag it; the copy still queued gets a bounded chance to land
                atomicOr(err, kErrTimeout);
                if (c + 1 < nchunks)
                    (void)mbar_wait_bounded(&sm.bars[(c + 1) & 1], ((c + 1) >> 1) & 1);
            }
            return;
        }
        const float4 *st = reinterpret_cast<const float4 *>(sm.stage[c & 1]);
        constexpr int kE = static_cast<int>(sizeof(GroupEntry) / 16);
        const int len = chunk_len(c);
        if (lane < len) {  // the row parts of group `lane`
            if constexpr (H == 1) {
                const float4 p0 = sm.prow[0];
                put_row<WIDE>(sm.rows, lane, group_row<WIDE>(st + lane * kE, p0.x, p0.y));
            } else {
#pragma unroll
                for (int q = 0; q < N; ++q) {
                    const float4 p0 = sm.prow[2 * q], p1 = sm.prow[2 * q + 1];
                    put_rows<WIDE>(sm.rows, q, lane, group_row<WIDE>(st + lane * kE, p0.x, p0.y),
                                   group_row<WIDE>(st + lane * kE, p1.x, p1.y));
                }
            }
        }
        __syncwarp();
#pragma unroll 2
        for (int j = 0; j < len; ++j) {
            const GroupCol cc = group_col(st + j * kE, gxh, gxl, WIDE);
#pragma unroll
            for (int q = 0; q < N; ++q) {
                GroupRow<V> r;
                get_row<WIDE>(sm.rows, q, j, r);
                group_step<LEVEL, STRANG>(s.p[q], cc, r, inv_g * inv_g);
            }
        }
        __syncwarp();  // the warp is done with the stage and the row parts
        if (lane == 0 && c + 2 < nchunks)
            issue(c + 2);
    }
    if (g1 > g0)
        for (int64_t n = g1 * G; n < R.step_end; ++n)
            single(n);

    if (!R.store_state)
        return;
#pragma unroll
    for (int k = 0; k < H; ++k) {
        const int64_t row = row_first + k;
        if (col_ok && row < R.ny) {
            const int64_t idx = row * R.nx + col;
            GroupPoint<V> &p = s.p[k / 2];
            hi_plane[idx] = make_float4(lane_of(p.ar, k), lane_of(p.ai, k), lane_of(p.br, k),
                                        lane_of(p.bi, k));
            lo_plane[idx] = make_float4(lane_of(p.lar, k), lane_of(p.lai, k), lane_of(p.lbr, k),
                                        lane_of(p.lbi, k));
        }
    }
}

template <int H>
__global__ void __launch_bounds__(32 * kGroupWarps, 4)
    evolve_group_kernel(const __grid_constant__ EvolveArgs args)
{
    extern __shared__ __align__(128) unsigned char group_dyn[];
    const int w = threadIdx.x >> 5;
    const int t = static_cast<int>(blockIdx.x) * static_cast<int>(blockDim.x >> 5) + w;
    if (t >= args.total_tiles)
        return;
    WarpSmem &sm = reinterpret_cast<WarpSmem *>(group_dyn)[w];
    if ((threadIdx.x & 31) == 0) {
        mbar_init(&sm.bars[0], 1);
        mbar_init(&sm.bars[1], 1);
        fence_mbar_init();
    }
    __syncwarp();
    const ReqDesc &R = args.r[find_request(args, t)];
    const int tile = t - R.tile_begin;
    if (!tile_ok(R, tile, R.err))
        return;
    const GroupPick pick = pick_plan(R.groups);
    if (pick.size == kNumGroupSizes)
        return;  // step by step
    if (R.scheme == 1)
        pick.level == kGroupWide ? body_group<H, kGroupWide, true>(R, pick.size, tile, sm, R.err)
                                 : body_group<H, kGroupFull, true>(R, pick.size, tile, sm, R.err);
    else if (pick.level == kGroupWide)
        body_group<H, kGroupWide, false>(R, pick.size, tile, sm, R.err);
    else if (pick.level == kGroupFull)
        body_group<H, kGroupFull, false>(R, pick.size, tile, sm, R.err);
    else
        body_group<H, kGroupLite, false>(R, pick.size, tile, sm, R.err);
}

template <int H>
cudaError_t launch_rows(const EvolveArgs &args, int warps, cudaStream_t stream)
{
    const int grid = (args.total_tiles + warps - 1) / warps;
    evolve_group_kernel<H><<<grid, 32 * warps, warps * sizeof(WarpSmem), stream>>>(args);
    return cudaGetLastError();
}
static_assert(kGroupWarps * sizeof(WarpSmem) <= 48 * 1024, "dynamic shared memory without asking");

// ---------------------------------------------------------------------------
// The expansion of a pulse's groups
//
// A group is G consecutive steps exp(-i sigma.P_n), P_n = p + a_n (p and a_n times
// dt and the valley sign here).  With a_n = abar + d_n, sum d_n = 0, its steps are
// exp(-i sigma.Pbar) disturbed by d_n, and their product is exp(-i sigma.w).  Read
// d as a piecewise constant function d(tau) of the step index tau from the group's
// middle, and let z v = 2 Pbar x v (Pbar = S/G, S = G p + sum a_n).  In the
// interaction picture about Pbar (d turned by -tau about it):
//   first order in d, to all orders in Pbar (the derivative of the exponential):
//     w - S = [(Gz/2)/sinh(Gz/2)] int e^{-tau z} d(tau) dtau
//           = (1 - G^2 z^2/24 + 7 G^4 z^4/5760 - 31 G^6 z^6/967680 ...)
//             (-z M1 + z^2 M2/2 - z^3 M3/6 + ...),   Mk = int tau^k d dtau,
//     where odd powers of z give w_z (z v is along sigma_z, and z^2 there is -4
//     |Pbar|^2) and even ones the plane;
//   second order in d: C = int int_{t1>t2} d1 x d2 along sigma_z, and in the plane
//     K S from L_ij = int int_{t1>t2} (t1 d1_i d2_j - t2 d2_i d1_j).
// (Magnus series; Blanes, Casas, Oteo and Ros, Phys. Rep. 470 (2009) 151.)  MAGNUS4
// steps exp(-i (sigma.P_n + sigma_z P_n x D_n)) add the sigma_z parts of their
// commutators, z D/2, to the disturbance: the same integrals one power of z higher, so
// the odd moments of D enter the plane (u2, u4) and the even ones w_z (n1, n3, n5).
// STRANG_XY's P' adds the second derivative of its cubic terms, sum d d, to K (the rest
// of P' depends on S alone and is the evolve kernel's).
// The next power of x = |S|^2 is folded into the kept ones (its Chebyshev
// economisation on [0, eps^2], eps = G theta_max the largest |S| of the box).
//
// What each level drops is estimated per group at |S| = eps and summed over the
// run.  Against the true sum of the groups' largest errors over the box (FP64, CPU):
// smooth pulses 0.7e-6 (Gaussian pulse, eps 0.63), 9e-8 (two colours, 0.36), 2e-10
// (sin^2, 0.16) for estimates about three times that; tables of noise, steps, spikes
// and kinks, and for MAGNUS4 of noise in D alone: at most 0.7 of the estimate (EXACT
// 1.2 where a group drops less than 1e-9).
//
// One thread per group, and two per 16 steps for the per-step table (dt A rounded
// to FP32 so that its running sum keeps to the exact one, dsp_steptable.h); FP64 only
// where those sums and the group's mean need it.  A 1e5-step table takes microseconds, where the host took 18 ns a step.
// ---------------------------------------------------------------------------

struct F2 {
    float x, y;
};
__device__ __forceinline__ F2 operator+(F2 a, F2 b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ F2 operator-(F2 a, F2 b) { return {a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ F2 operator*(float s, F2 a) { return {s * a.x, s * a.y}; }
__device__ __forceinline__ float cross(F2 a, F2 b) { return a.x * b.y - a.y * b.x; }
__device__ __forceinline__ float size1(F2 a) { return fabsf(a.x) + fabsf(a.y); }

// int_j^{j+1} t^k dt
__host__ __device__ constexpr double moment_weight(int k, int j)
{
    double hi = 1.0, lo = 1.0;
    for (int i = 0; i <= k; ++i) {
        hi *= j + 1;
        lo *= j;
    }
    return (hi - lo) / (k + 1);
}

// Potentials of step n, times s dt: the midpoint sample, or MAGNUS4's mean of the
// Gauss points with D = -(sqrt(3)/6) s dt (A2 - A1).
struct StepA {
    double x, y;
    F2 D;
};
__device__ __forceinline__ float gauss_difference(const PrepArgs &a, double p, double q)
{
    constexpr double kappa = -0.28867513459481288225;  // -sqrt(3)/6
    return static_cast<float>(kappa * (a.sdt * (q - p)));
}
__device__ __forceinline__ StepA step_potential(const PrepArgs &a, int64_t n)
{
    if (a.scheme == 2) {
        const double2 p = reinterpret_cast<const double2 *>(a.raw)[2 * n];
        const double2 q = reinterpret_cast<const double2 *>(a.raw)[2 * n + 1];
        return {a.sdt * (0.5 * (p.x + q.x)), a.sdt * (0.5 * (p.y + q.y)),
                {gauss_difference(a, p.x, q.x), gauss_difference(a, p.y, q.y)}};
    }
    const double2 p = reinterpret_cast<const double2 *>(a.raw)[n];
    return {a.sdt * p.x, a.sdt * p.y, {0.0f, 0.0f}};
}

template <int I>  // of group_size
__device__ __forceinline__ void expand_group(const PrepArgs &args, int64_t g, float &wide, float &lite)
{
    constexpr int G = group_size(I);
    const float eps = args.eps / static_cast<float>(1 << I);
    double sx = 0.0, sy = 0.0;
    for (int n = 0; n < G; ++n) {
        const StepA a = step_potential(args, g * G + n);
        sx += a.x;
        sy += a.y;
    }
    const double mx = sx * (1.0 / G), my = sy * (1.0 / G);
    F2 d[G], D[G];
#pragma unroll
    for (int n = 0; n < G; ++n) {
        const StepA a = step_potential(args, g * G + n);
        d[n] = {static_cast<float>(a.x - mx), static_cast<float>(a.y - my)};
        D[n] = a.D;
    }
    F2 M1{0, 0}, M2{0, 0}, M3{0, 0}, M4{0, 0}, M5{0, 0}, M7{0, 0};
    float s_odd = 0.0f, s_even = 0.0f;
#pragma unroll
    for (int j = 0; j < G / 2; ++j) {
        const F2 o = d[G / 2 + j] - d[G / 2 - 1 - j], v = d[G / 2 + j] + d[G / 2 - 1 - j];
        M1 = M1 + static_cast<float>(moment_weight(1, j)) * o;
        M2 = M2 + static_cast<float>(moment_weight(2, j)) * v;
        M3 = M3 + static_cast<float>(moment_weight(3, j)) * o;
        M4 = M4 + static_cast<float>(moment_weight(4, j)) * v;
        M5 = M5 + static_cast<float>(moment_weight(5, j)) * o;
        M7 = M7 + static_cast<float>(moment_weight(7, j)) * o;
        s_odd += size1(o);
        s_even += size1(v);
    }
    float C = 0.0f, Lxx = 0.0f, Lxy = 0.0f, Lyx = 0.0f, Lyy = 0.0f;
    F2 cum{0, 0}, cumt{0, 0};
#pragma unroll
    for (int n = 0; n < G; ++n) {
        const float tau = static_cast<float>(n + 0.5 - 0.5 * G), sixth = 1.0f / 6.0f;
        const F2 t = tau * d[n];
        C += cross(d[n], cum);
        Lxx += t.x * cum.x - cumt.x * d[n].x + d[n].x * d[n].x * sixth;
        Lxy += t.x * cum.y - cumt.x * d[n].y + d[n].x * d[n].y * sixth;
        Lyx += t.y * cum.x - cumt.y * d[n].x + d[n].y * d[n].x * sixth;
        Lyy += t.y * cum.y - cumt.y * d[n].y + d[n].y * d[n].y * sixth;
        cum = cum + d[n];
        cumt = cumt + t;
    }
    constexpr double k = 2.0 / G, k2 = k * k, k3 = k2 * k, k4 = k2 * k2, k5 = k4 * k, k7 = k5 * k2;
    constexpr double G2 = static_cast<double>(G) * G, G4 = G2 * G2, G6 = G4 * G2;
    F2 n1 = static_cast<float>(-k) * M1;
    F2 n3 = static_cast<float>(k3 / 6.0) * M3 - static_cast<float>(k3 * G2 / 24.0) * M1;
    F2 n5 = static_cast<float>(k5 * G2 / 144.0) * M3 - static_cast<float>(k5 / 120.0) * M5 -
            static_cast<float>(k5 * 7.0 * G4 / 5760.0) * M1;
    const F2 n7 = static_cast<float>(k7 / 5040.0) * M7 - static_cast<float>(k7 * G2 / 2880.0) * M5 +
                  static_cast<float>(k7 * 7.0 * G4 / 34560.0) * M3 -
                  static_cast<float>(k7 * 31.0 * G6 / 967680.0) * M1;
    F2 u2 = static_cast<float>(0.5 * k2) * M2;
    F2 u4 = static_cast<float>(k4 * G2 / 48.0) * M2 - static_cast<float>(k4 / 24.0) * M4;
    const float X = eps * eps, e3 = X * eps, e5 = e3 * X, e7 = e5 * X;
    const float s = s_odd + s_even;
    wide = 0.0f;
    if (args.scheme == 2) {
        F2 D0{0, 0}, D1{0, 0}, D2{0, 0}, D3{0, 0}, D4{0, 0};  // int tau^k D dtau
        float sD = 0.0f;
#pragma unroll
        for (int n = 0; n < G; ++n) {
            const float tau = static_cast<float>(n + 0.5 - 0.5 * G), t2 = tau * tau;
            D0 = D0 + D[n];
            D1 = D1 + tau * D[n];
            D2 = D2 + (t2 + 1.0f / 12.0f) * D[n];
            D3 = D3 + (tau * (t2 + 0.25f)) * D[n];
            D4 = D4 + (t2 * t2 + 0.5f * t2 + 1.0f / 80.0f) * D[n];
            C += cross(d[n], D[n]);
            sD += size1(D[n]);
        }
        constexpr double i = 1.0 / G;
        n1 = n1 + static_cast<float>(i) * D0;
        n3 = n3 + static_cast<float>(i / 6.0) * D0 - static_cast<float>(0.5 * k2 * i) * D2;
        n5 = n5 + static_cast<float>(k4 * i * 7.0 * G4 / 5760.0) * D0 -
             static_cast<float>(k4 * i * G2 / 48.0) * D2 + static_cast<float>(k4 * i / 24.0) * D4;
        u2 = u2 - static_cast<float>(k * i) * D1;
        u4 = u4 + static_cast<float>(k4 / 12.0) * D3 - static_cast<float>(k4 * G2 / 48.0) * D1;
        // the next orders of D: z^7 along sigma_z; z^6 in the plane, whose coefficient is
        // at most 0.0065 whatever the D's signs; and D with D, (sD/G)^2 |S|^3
        const float mD = static_cast<float>(i) * sD;
        wide += mD * (s * eps + 0.03f * e7 + 0.01f * e3 * e3) + 0.25f * mD * mD * e3;
    }
    // (the next power of K S, fitted to smooth pulses, at half the box's x)
    const float kk = static_cast<float>(k) * (1.0f + 0.08f * X);
    float Kxx = kk * Lyy, Kxy = -kk * Lxy, Kyx = -kk * Lyx, Kyy = kk * Lxx;
    const float Kn = static_cast<float>(k) * (fabsf(Lxx) + fabsf(Lxy) + fabsf(Lyx) + fabsf(Lyy));
    if (args.scheme == 1) {
        float dxx = 0.0f, dxy = 0.0f, dyy = 0.0f;
#pragma unroll
        for (int n = 0; n < G; ++n) {
            dxx += d[n].x * d[n].x;
            dxy += d[n].x * d[n].y;
            dyy += d[n].y * d[n].y;
        }
        constexpr float third = static_cast<float>(1.0 / (3.0 * G));
        Kxx -= third * dyy;
        Kxy -= 2.0f * third * dxy;
        Kyx += third * dxy;
        Kyy += 0.5f * third * dxx;
        // the derivative of P' at the other terms, the next orders of P'
        const float t2 = X * static_cast<float>(1.0 / G2);
        wide += 0.1f * size1(n1) * eps * t2 * t2 +
                0.7f * t2 * (size1(n3) * e3 + size1(u2) * X + Kn * eps) +
                0.02f * eps * t2 * t2 * t2;
    }
    // x^3 on [0, X] as 3/2 X x^2 - 9/16 X^2 x + X^3/32, off by X^3/32
    n5 = n5 + (1.5f * X) * n7;
    n3 = n3 - (0.5625f * X * X) * n7;
    n1 = n1 + (X * X * X * 0.03125f) * n7;
    wide += size1(n7) * e7 * (0.05f + 0.1f * X) + 0.1f * size1(u4) * e3 * e3 + 0.07f * Kn * e3 +
            0.25f * X * s_odd * s_even + s * s * s * (1.0f / 24.0f);
    const float wz = fabsf(C) + size1(n1) * eps + size1(n3) * e3;
    lite = wide + size1(n5) * e5 + size1(u2) * X + size1(u4) * X * X + Kn * eps +
           0.5f * wz * wz;
    const float xh = static_cast<float>(sx), yh = static_cast<float>(sy);
    float4 *e = reinterpret_cast<float4 *>(
        args.entries + group_entries_before(args.n_steps, args.first, I) + g);
    e[0] = make_float4(xh, static_cast<float>(sx - static_cast<double>(xh)), n1.y, n3.y);
    e[1] = make_float4(n5.y, u2.y, u4.y, Kxx);
    e[2] = make_float4(Kyx, yh, static_cast<float>(sy - static_cast<double>(yh)), C);
    e[3] = make_float4(n1.x, n3.x, n5.x, u2.x);
    e[4] = make_float4(u4.x, Kxy, Kyy, 0.0f);
}

// Adds the threads' estimates to a sum, in fixed point (clamped above the budget).
__device__ __forceinline__ void add_estimate(unsigned long long *sum, float v)
{
    constexpr float most = static_cast<float>(2.0 * kPlanBudget);
    const float c = v <= most ? v : most;  // NaN too
    unsigned long long f =
        static_cast<unsigned long long>(ceilf(c * static_cast<float>(1.0 / kPlanUnit)));
    for (int o = 16; o > 0; o >>= 1)
        f += __shfl_down_sync(0xffffffffu, f, o);
    if ((threadIdx.x & 31) == 0 && f > 0)
        atomicAdd(sum, f);
}

// blockIdx.y: a group size, or (kNumGroupSizes) the per-step table.
constexpr int kPrepThreads = 64;
__global__ void __launch_bounds__(kPrepThreads) prep_groups_kernel(const __grid_constant__ PrepArgs a)
{
    const int64_t g = static_cast<int64_t>(blockIdx.x) * kPrepThreads + threadIdx.x;
    const int what = blockIdx.y;
    if (what < kNumGroupSizes) {
        float wide = 0.0f, lite = 0.0f;
        if (what >= a.first && g < a.n_steps / group_size(what)) {
            if (what == 0)
                expand_group<0>(a, g, wide, lite);
            else if (what == 1)
                expand_group<1>(a, g, wide, lite);
            else
                expand_group<2>(a, g, wide, lite);
        }
        add_estimate(&a.sums->wide[what], wide);
        add_estimate(&a.sums->lite[what], lite);
        return;
    }
    // dt A per step, rounded to FP32 (table_block): a thread per 16 steps and coordinate, so
    // that the chain of FP64 operations is half as long (prep of 12000 MAGNUS4 steps 24.6
    // us with one thread for both, 18.4 with the residual dropped every 16 steps)
    const int64_t block = g >> 1;
    const int c = static_cast<int>(g & 1);
    if (kTableBlock * block >= a.n_steps)
        return;
    const double half = a.scheme == 2 ? 0.5 * a.sdt : a.sdt;  // times the sum of the samples
    const double s0 = a.prefix[2 * block + c], s1 = a.prefix[2 * block + 2 + c];
    float *out = static_cast<float *>(a.table) + c;
    if (a.scheme == 2) {
        table_block(block, a.n_steps, __dmul_rn(half, s0), __dmul_rn(half, s1),
                    [&](int64_t k) {
                        return a.sdt * (0.5 * (a.raw[4 * k + c] + a.raw[4 * k + 2 + c]));
                    },
                    [&](int64_t k, float f) {
                        out[4 * k] = f;
                        out[4 * k + 2] = gauss_difference(a, a.raw[4 * k + c], a.raw[4 * k + 2 + c]);
                    });
    } else {
        table_block(block, a.n_steps, __dmul_rn(half, s0), __dmul_rn(half, s1),
                    [&](int64_t k) { return a.sdt * a.raw[2 * k + c]; },
                    [&](int64_t k, float f) { out[2 * k] = f; });
    }
}

}  // namespace

cudaError_t launch_prep_groups(const PrepArgs &args, cudaStream_t stream)
{
    if (args.n_steps <= 0)
        return cudaSuccess;
    const int64_t most = (args.n_steps + group_size(kNumGroupSizes - 1) - 1) /
                         group_size(kNumGroupSizes - 1);
    const dim3 grid(static_cast<unsigned>((most + kPrepThreads - 1) / kPrepThreads),
                    kNumGroupSizes + 1);
    prep_groups_kernel<<<grid, kPrepThreads, 0, stream>>>(args);
    return cudaGetLastError();
}

cudaError_t launch_evolve_group(const EvolveArgs &args, int rows, int warps, cudaStream_t stream)
{
    if (args.nreq <= 0 || args.total_tiles <= 0)
        return cudaSuccess;
    return rows == 4   ? launch_rows<4>(args, warps, stream)
           : rows == 2 ? launch_rows<2>(args, warps, stream)
                       : launch_rows<1>(args, warps, stream);
}

}  // namespace dsp
