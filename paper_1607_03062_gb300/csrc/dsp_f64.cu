// dsp_f64.cu -- the FP64 evolve kernels.  Shared device code (and the description
// of the method) is in dsp_device.cuh.

#include "dsp_device.cuh"

namespace dsp {
namespace {

// ---------------------------------------------------------------------------
// FP64 step
// ---------------------------------------------------------------------------

struct F64Point {
    double ar, ai, br, bi;
    double tx, ty;  // dt * p (times the valley sign)
};

// ---------------------------------------------------------------------------
// The FP64 EXACT step with its small parts in double-float.
//
// GB300's FP64 pipe runs at 1/64 of the FP32 rate (a warp's DFMA holds a
// scheduler's FP64 unit for ~64 cycles), so only what must accumulate in FP64 is
// done there: the update psi <- psi + m psi - (q conj ...) and q = dt P + s1 dt P.
// The small parts m = cos(theta) - 1 and s1 = sin(theta)/theta - 1 of theta^2 =
// |dt P|^2 are evaluated in double-float FP32 arithmetic (pairs of floats, ~2^-46
// relative): being small (~theta^2/2, ~theta^2/6), they come out to ~1e-19
// absolute, far below an FP64 ulp of the state, so the step is FP64-accurate.
// FP64 operations per spinor-step: 2 (dt P) + 2 (m, s1 to double) + 2 (q) + 12
// (update) = 18 instead of 18 + dc + ds; the ~100 FP32 operations of the series
// issue beside them.
// ---------------------------------------------------------------------------

// dt P squared as a float pair, from the double (split exactly into hi + lo).
__device__ __forceinline__ float2 square_df(double P)
{
    float h, l;
    split_f64(P, h, l);
    const float p = __fmul_rn(h, h);
    const float e = __fmaf_rn(__fadd_rn(h, h), l, __fmaf_rn(h, h, -p));
    const float sh = __fadd_rn(p, e);
    return make_float2(sh, __fadd_rn(e, -__fadd_rn(sh, -p)));
}

// sum_{k=K..D} c_k x^(k-K) in double-float, c_k = (-1)^k / (2k + ODD)!.
template <int D, int K, int ODD>
__device__ __forceinline__ void horner_df(float xh, float xl, float &th, float &tl)
{
    constexpr DFConst c = df_const(((K & 1) ? -1.0 : 1.0) * inv_factorial<2 * K + ODD>());
    if constexpr (K == D) {
        th = c.h;
        tl = c.l;
    } else {
        float uh, ul;
        horner_df<D, K + 1, ODD>(xh, xl, uh, ul);
        df_mul(xh, xl, uh, ul, th, tl);
        df_add(th, tl, c.h, c.l);
    }
}

// The FP64 EXACT step: dt P = (Px, Py), their squares as float pairs.
template <int DC, int DS>
__device__ __forceinline__ void step_f64_exact(F64Point &s, double Px, double Py, float2 px2,
                                               float2 py2)
{
    float xh = px2.x, xl = px2.y;
    df_add(xh, xl, py2.x, py2.y);  // theta^2
    float th, tl, mh, ml, sh, sl;
    horner_df<DC, 1, 0>(xh, xl, th, tl);  // (cos(theta) - 1) / theta^2
    df_mul(xh, xl, th, tl, mh, ml);
    horner_df<DS, 1, 1>(xh, xl, th, tl);  // (sin(theta)/theta - 1) / theta^2
    df_mul(xh, xl, th, tl, sh, sl);
    const double m = df_to_f64(mh, ml), s1 = df_to_f64(sh, sl);
    const double qr = fma(s1, Py, Py), qi = fma(s1, Px, Px);
    // a' = a + m a - q b ; b' = b + m b + conj(q) a, q = qr + i qi
    const double nar = fma(m, s.ar, fma(-qr, s.br, fma(qi, s.bi, s.ar)));
    const double nai = fma(m, s.ai, fma(-qr, s.bi, fma(-qi, s.br, s.ai)));
    const double nbr = fma(m, s.br, fma(qr, s.ar, fma(qi, s.ai, s.br)));
    const double nbi = fma(m, s.bi, fma(qr, s.ai, fma(-qi, s.ar, s.bi)));
    s.ar = nar; s.ai = nai; s.br = nbr; s.bi = nbi;
}

// sum_{k=K..D} c_k x^(k-K), c_k = (-1)^k / (2k + ODD)!, in FP64.
template <int D, int K, int ODD>
__device__ __forceinline__ double horner_f64(double x)
{
    constexpr double c = ((K & 1) ? -1.0 : 1.0) * inv_factorial<2 * K + ODD>();
    if constexpr (K == D)
        return c;
    else
        return fma(horner_f64<D, K + 1, ODD>(x), x, c);
}

// STRANG_XY and MAGNUS4 form their small parts in double-float up to this cosine
// degree (theta below ~0.2, where their ~2^-46 relative error is below an FP64 ulp of
// the state), in FP64 above.
constexpr int kDfDegree = 5;

// The FP64 MAGNUS4 step in the same way: n = (dt Pbar, n_z), n_z = Pbar x D, |n|^2 and
// the small parts in double-float (kDfDegree), the update and q in FP64.  26 FP64
// operations where the FP64 series took 26 + dc + ds.
template <int DC, int DS>
__device__ __forceinline__ void step_f64_magnus(F64Point &s, double Px, double Py, double2 d)
{
    const double nz = fma(Px, d.y, -(Py * d.x));
    double c, qr, qi, qz;
    if constexpr (DC <= kDfDegree) {
        const float2 px2 = square_df(Px), py2 = square_df(Py), nz2 = square_df(nz);
        float xh = px2.x, xl = px2.y;
        df_add(xh, xl, py2.x, py2.y);
        df_add(xh, xl, nz2.x, nz2.y);  // |n|^2
        float th, tl, uh, ul;
        horner_df<DC, 1, 0>(xh, xl, th, tl);
        df_mul(xh, xl, th, tl, uh, ul);
        c = 1.0 + df_to_f64(uh, ul);
        horner_df<DS, 1, 1>(xh, xl, th, tl);
        df_mul(xh, xl, th, tl, uh, ul);
        const double s1 = df_to_f64(uh, ul);
        qr = fma(s1, Py, Py);
        qi = fma(s1, Px, Px);
        qz = fma(s1, nz, nz);
    } else {
        const double x = fma(Px, Px, fma(Py, Py, nz * nz));
        c = horner_f64<DC, 0, 0>(x);
        const double sn = horner_f64<DS, 0, 1>(x);
        qr = sn * Py;
        qi = sn * Px;
        qz = sn * nz;
    }
    // a' = (c - i qz) a - q b ; b' = conj(q) a + (c + i qz) b, q = qr + i qi: the small
    // terms first, one rounding at the state's size (from psi + m psi each term would
    // round there: 1.2 to 1.6 times the error over 12000 and 50000 steps)
    const double nar = fma(c, s.ar, fma(qz, s.ai, fma(-qr, s.br, qi * s.bi)));
    const double nai = fma(c, s.ai, fma(-qz, s.ar, fma(-qr, s.bi, -(qi * s.br))));
    const double nbr = fma(c, s.br, fma(-qz, s.bi, fma(qr, s.ar, qi * s.ai)));
    const double nbi = fma(c, s.bi, fma(qz, s.br, fma(qr, s.ai, -(qi * s.ar))));
    s.ar = nar; s.ai = nai; s.br = nbr; s.bi = nbi;
}

// psi <- U psi for U = [[c, -q], [conj(q), c]] (STRANG_XY), in FP64.
__device__ __forceinline__ void apply_f64(F64Point &s, double c, double qr, double qi)
{
    const double nar = fma(c, s.ar, fma(-qr, s.br, qi * s.bi));
    const double nai = fma(c, s.ai, fma(-qr, s.bi, -(qi * s.br)));
    const double nbr = fma(c, s.br, fma(qr, s.ar, qi * s.ai));
    const double nbi = fma(c, s.bi, fma(qr, s.ai, -(qi * s.ar)));
    s.ar = nar; s.ai = nai; s.br = nbr; s.bi = nbi;
}

// STRANG_XY's parts of one coordinate: {cos P, sin P} (the small parts by kDfDegree);
// and its step from those of x and y, c = cos y cos x, q = sin y + i cos y sin x.  24
// FP64 operations where the FP64 series took 20 + 2 dc + 2 ds; on row tiles the parts
// of a row and of a column are formed once.
template <int DC, int DS>
__device__ __forceinline__ double2 strang_part(double P)
{
    if constexpr (DC <= kDfDegree) {
        const float2 x = square_df(P);
        float th, tl, uh, ul;
        horner_df<DC, 1, 0>(x.x, x.y, th, tl);
        df_mul(x.x, x.y, th, tl, uh, ul);
        const double c1 = df_to_f64(uh, ul);
        horner_df<DS, 1, 1>(x.x, x.y, th, tl);
        df_mul(x.x, x.y, th, tl, uh, ul);
        return make_double2(1.0 + c1, fma(df_to_f64(uh, ul), P, P));
    } else {
        const double x = P * P;
        return make_double2(horner_f64<DC, 0, 0>(x), P * horner_f64<DS, 0, 1>(x));
    }
}
__device__ __forceinline__ void step_f64_strang(F64Point &s, double2 x, double2 y)
{
    apply_f64(s, y.x * x.x, y.y, y.x * x.y);
}

template <int SCHEME, int DC, int DS>
__device__ __forceinline__ void step_f64(F64Point &s, double2 a, double2 d)
{
    const double Px = s.tx + a.x, Py = s.ty + a.y;  // dt * P (times the valley sign)
    if constexpr (SCHEME == 0) {
        step_f64_exact<DC, DS>(s, Px, Py, square_df(Px), square_df(Py));
    } else if constexpr (SCHEME == 2) {
        step_f64_magnus<DC, DS>(s, Px, Py, d);
    } else {
        step_f64_strang(s, strang_part<DC, DS>(Px), strang_part<DC, DS>(Py));
    }
}

// The row part of a step from dt P_y, as step_f64 forms it:
//   EXACT {P_y, (P_y^2 as a float pair, in the second double's bits)};
//   STRANG_XY strang_part.
template <int SCHEME, int DC, int DS>
__device__ __forceinline__ double2 strip64_row(double Py)
{
    if constexpr (SCHEME == 0) {
        const float2 p2 = square_df(Py);
        const unsigned long long bits =
            (static_cast<unsigned long long>(__float_as_uint(p2.y)) << 32) | __float_as_uint(p2.x);
        return make_double2(Py, __longlong_as_double(static_cast<long long>(bits)));
    } else {
        return strang_part<DC, DS>(Py);
    }
}

// One step of the thread's H spinors (step_f64's operations; SCHEME 0 EXACT, 1
// STRANG_XY).
template <int SCHEME, int DC, int DS, int H>
__device__ __forceinline__ void strip64_step(F64Point (&pt)[H], double tx, double ax,
                                             const double2 *rows)
{
    const double Px = tx + ax;  // dt * P_x (times the valley sign)
    if constexpr (SCHEME == 0) {
        const float2 px2 = square_df(Px);
#pragma unroll
        for (int k = 0; k < H; ++k) {
            const double2 r = rows[k];
            const unsigned long long bits = static_cast<unsigned long long>(__double_as_longlong(r.y));
            const float2 py2 = make_float2(__uint_as_float(static_cast<unsigned int>(bits)),
                                           __uint_as_float(static_cast<unsigned int>(bits >> 32)));
            step_f64_exact<DC, DS>(pt[k], Px, r.x, px2, py2);
        }
        return;
    }
    const double2 x = strang_part<DC, DS>(Px);
#pragma unroll
    for (int k = 0; k < H; ++k)
        step_f64_strang(pt[k], x, rows[k]);
}

// ---------------------------------------------------------------------------
// Tiles
//
// What bounds every FP64 launch is the FP64 pipe: a warp's DFMA holds its
// scheduler's unit for 64 cycles (33 ns measured, whatever the number of active
// lanes), so a launch takes as long as the scheduler with the most FP64 instructions.
// Warps work alone (their own double-buffered bulk copies of the table with bounded
// waits, no CTA-wide barrier), and the host picks the shape that loads the fullest
// scheduler least (f64_shape in dsp_api.cpp).  FP64 instructions of a warp per EXACT
// step and its points:
//   rows   32 columns x 4 rows: the dt P_x part once per lane, the dt P_y part once per
//          row and step in a shared table                                65 for 128
//   flat 1 32 consecutive points                                         18 for 32
//   flat 2 16 consecutive points, a lane pair per point: lane 0 holds a, lane 1 b;
//          each forms one of P_x and P_y, of the two series, and of the two parts of
//          q, and they trade by shuffles                                  9 for 16
//   flat 4 8 points, a lane per real component                            6 for 8
// (STRANG_XY: rows 62, flat 24; MAGNUS4: flat 26.)  Every FP64 operation of a point is the same in every shape (same operands, same
// rounding), so its result is bitwise the same.  STRANG_XY takes rows or flat 1,
// MAGNUS4 flat 1.  The projection is the projection kernel's, on the state these
// leave.
//
// Measured: 64^2 x 2000 steps 9.48 -> 1.08 ms (1024-point CTAs held 4 of 152 SMs;
// flat 4 holds 512 warps), 300 x 257 x 1700 steps 8.10 -> 4.20 ms; 1000 steps of 512^2:
// MAGNUS4 19.8 -> 12.4 ms, STRANG_XY 9.48 -> 8.50 ms.
// ---------------------------------------------------------------------------

constexpr int kF64Stage = 1024;  // bytes per staged table chunk and warp
constexpr int kF64Chunk = kF64Stage / 16;

// The table entries of a launch's steps, streamed through a warp's two stages.
template <typename E>
struct WarpStager {
    unsigned char *stage;  // 2 x kF64Stage
    uint64_t *bars;
    const E *table;  // entry of the first step
    int64_t nsteps;
    int nchunks;
    int withhold;
    static constexpr int kCh = kF64Stage / static_cast<int>(sizeof(E));

    __device__ __forceinline__ WarpStager(const ReqDesc &R, unsigned char *s, uint64_t *b)
        : stage(s), bars(b), table(static_cast<const E *>(R.table) + R.step_begin),
          nsteps(R.step_end > R.step_begin ? R.step_end - R.step_begin : 0),
          nchunks(static_cast<int>((nsteps + kCh - 1) / kCh)), withhold(R.withhold_first_copy)
    {
    }
    __device__ __forceinline__ int chunk_len(int c) const
    {
        const int64_t rem = nsteps - static_cast<int64_t>(c) * kCh;
        return rem < kCh ? static_cast<int>(rem) : kCh;
    }
    __device__ __forceinline__ void issue(int c) const  // one lane
    {
        const uint32_t bytes = static_cast<uint32_t>(chunk_len(c)) * sizeof(E);
        mbar_arrive_expect_tx(&bars[c & 1], bytes);
        if (c == 0 && withhold)
            return;  // test hook: the waits for chunk 0 run out
        bulk_load(stage + (c & 1) * kF64Stage, table + static_cast<int64_t>(c) * kCh, bytes,
                  &bars[c & 1]);
    }
    // Runs f(entries, len) on every chunk in order; false (flagged in err) if a wait
    // timed out.  The whole warp calls it.
    template <typename F>
    __device__ __forceinline__ bool run(int *err, F f) const
    {
        const bool first = (threadIdx.x & 31) == 0;
        if (first)
            for (int c = 0; c < 2 && c < nchunks; ++c)
                issue(c);
        for (int c = 0; c < nchunks; ++c) {
            const bool arrived = mbar_wait_bounded(&bars[c & 1], (c >> 1) & 1);
            if (!__all_sync(0xffffffffu, arrived)) {
                if (first) {  // the copy still queued gets a bounded chance to land
                    atomicOr(err, kErrTimeout);
                    if (c + 1 < nchunks)
                        (void)mbar_wait_bounded(&bars[(c + 1) & 1], ((c + 1) >> 1) & 1);
                }
                return false;
            }
            f(reinterpret_cast<const E *>(stage + (c & 1) * kF64Stage), chunk_len(c));
            __syncwarp();  // the warp is done with the stage
            if (first && c + 2 < nchunks)
                issue(c + 2);
        }
        return true;
    }
};

struct F64Smem {
    unsigned char stage[2][kF64Stage];
    double2 rows[kF64Chunk][4];  // rows: per step and row (strip64_row)
    uint64_t bars[2];
};

// The spinor a point starts a launch with.
__device__ __forceinline__ void load_f64(const ReqDesc &R, int64_t idx, bool valid, double px,
                                         double py, double vs, F64Point &p)
{
    if (R.fresh || !valid) {
        if (R.init_identity) {
            p.ar = 1.0; p.ai = 0.0; p.br = 0.0; p.bi = 0.0;
        } else {
            initial_spinor(px + R.a_in[0], py + R.a_in[1], vs, p.ar, p.ai, p.br, p.bi);
        }
    } else {
        const double2 *a_plane = static_cast<const double2 *>(R.state);
        const double2 a = a_plane[idx], b = a_plane[R.n_points + idx];
        p.ar = a.x; p.ai = a.y; p.br = b.x; p.bi = b.y;
    }
}

__device__ __forceinline__ double shfl_x(double v, int mask)
{
    return __shfl_xor_sync(0xffffffffu, v, mask);
}
__device__ __forceinline__ float shfl_x(float v, int mask)
{
    return __shfl_xor_sync(0xffffffffu, v, mask);
}

// sum_{k=K..D} c_k x^(k-K) in double-float as horner_df, for U steps at once, of the cos
// series (odd = false: c_k = (-1)^k/(2k)!, to DC) or the sinc one (odd: (-1)^k/(2k +
// 1)!, to DS); the shorter one starts from zero coefficients, which changes nothing.
template <int DC, int DS, int K, int U>
__device__ __forceinline__ void horner_either(bool odd, const float (&xh)[U], const float (&xl)[U],
                                              float (&th)[U], float (&tl)[U])
{
    constexpr int D = DC > DS ? DC : DS;
    constexpr double sign = (K & 1) ? -1.0 : 1.0;
    constexpr DFConst c = df_const(K <= DC ? sign * inv_factorial<2 * K>() : 0.0);
    constexpr DFConst s = df_const(K <= DS ? sign * inv_factorial<2 * K + 1>() : 0.0);
    const float ch = odd ? s.h : c.h, cl = odd ? s.l : c.l;
    if constexpr (K < D)
        horner_either<DC, DS, K + 1, U>(odd, xh, xl, th, tl);
#pragma unroll
    for (int u = 0; u < U; ++u) {
        if constexpr (K == D) {
            th[u] = ch;
            tl[u] = cl;
        } else {
            float ph, pl;
            df_mul(xh[u], xl[u], th[u], tl[u], ph, pl);
            df_add(ph, pl, ch, cl);
            th[u] = ph;
            tl[u] = pl;
        }
    }
}

// EXACT steps on L = 2 or 4 lanes per point (step_f64_exact's operations).  Lane k of a
// point: L = 2 holds a (k = 0) or b (k = 1) in v[0], v[1]; L = 4 holds Re a, Im a, Re b,
// Im b.  An operator's entries as the lane applies them:
template <int L, int U>
struct LaneOps {
    double m[U], sr[U], si[U];  // cos - 1; -+ Re q; +- Im q (L = 2: Im q)
};

// The operators of U steps, stage by stage for all of them (a step's own chain of
// conversions, shuffles and double-float series takes ~900 cycles).  P: the lane's P_x
// (k even) or P_y (k odd).
template <int DC, int DS, int L, int U>
__device__ __forceinline__ void lane_ops(LaneOps<L, U> &o, const double (&P)[U], int k)
{
    const bool odd = k & 1;
    float2 own[U];
    float xh[U], xl[U], th[U], tl[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
        own[u] = square_df(P[u]);
#pragma unroll
    for (int u = 0; u < U; ++u) {
        th[u] = shfl_x(own[u].x, 1);
        tl[u] = shfl_x(own[u].y, 1);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {  // P_x^2 + P_y^2
        xh[u] = odd ? th[u] : own[u].x;
        xl[u] = odd ? tl[u] : own[u].y;
        df_add(xh[u], xl[u], odd ? own[u].x : th[u], odd ? own[u].y : tl[u]);
    }
    horner_either<DC, DS, 1, U>(odd, xh, xl, th, tl);
    double mine[U], q[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        float ph, pl;
        df_mul(xh[u], xl[u], th[u], tl[u], ph, pl);
        mine[u] = df_to_f64(ph, pl);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const double other = shfl_x(mine[u], 1);
        o.m[u] = odd ? other : mine[u];
        q[u] = fma(odd ? mine[u] : other, P[u], P[u]);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const double p = shfl_x(q[u], 1);
        const double qr = odd ? q[u] : p, qi = odd ? p : q[u];
        if constexpr (L == 2) {
            o.sr[u] = odd ? qr : -qr;
            o.si[u] = qi;
        } else {
            o.sr[u] = (k & 2) ? qr : -qr;
            o.si[u] = odd ? -qi : qi;
        }
    }
}

template <int L, int U>
__device__ __forceinline__ void lane_apply(double (&v)[4 / L], const LaneOps<L, U> &o)
{
#pragma unroll
    for (int u = 0; u < U; ++u) {
        if constexpr (L == 2) {
            const double tr = shfl_x(v[0], 1), ti = shfl_x(v[1], 1);
            const double nr = fma(o.m[u], v[0], fma(o.sr[u], tr, fma(o.si[u], ti, v[0])));
            const double ni = fma(o.m[u], v[1], fma(o.sr[u], ti, fma(-o.si[u], tr, v[1])));
            v[0] = nr;
            v[1] = ni;
        } else {
            const double t1 = shfl_x(v[0], 2), t2 = shfl_x(v[0], 3);
            v[0] = fma(o.m[u], v[0], fma(o.sr[u], t1, fma(o.si[u], t2, v[0])));
        }
    }
}

// A chunk's steps: the operators of the next kLaneSteps steps are formed beside the
// current ones' updates.  A warp waits out the issue of its own FP64 instructions, so
// this hides shuffles and FP32 latency only, and only 4 lanes per point, which run
// where a scheduler has one warp or two, take it (64^2 x 2000: 1.29 -> 1.08 ms); on 2
// lanes the registers push out warps that hide more (4 steps on 256^2: 4.84 -> 5.31
// ms).  a: the lane's component of the chunk's entries (every second double).
template <int L>
constexpr int kLaneSteps = L == 4 ? 4 : 1;
template <int DC, int DS, int L>
__device__ __forceinline__ void lane_steps(double (&v)[4 / L], const double *a, double t, int len,
                                           int k)
{
    constexpr int U = kLaneSteps<L>;
    const auto block = [&](LaneOps<L, U> &o, int j) {
        double P[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            P[u] = t + a[2 * (j + u)];
        lane_ops<DC, DS, L, U>(o, P, k);
    };
    int j = 0;
    if (len >= U) {
        LaneOps<L, U> cur;
        block(cur, 0);
        for (j = U; j + U <= len; j += U) {
            LaneOps<L, U> next;
            block(next, j);
            lane_apply<L, U>(v, cur);
            cur = next;
        }
        lane_apply<L, U>(v, cur);
    }
    for (; j < len; ++j) {
        LaneOps<L, 1> o;
        const double P[1] = {t + a[2 * j]};
        lane_ops<DC, DS, L, 1>(o, P, k);
        lane_apply<L, 1>(v, o);
    }
}

// A flat tile of 32 / L consecutive points.
template <int SCHEME, int DC, int DS, int L>
__device__ void body_flat(const ReqDesc &R, int tile, F64Smem &sm, int *err)
{
    constexpr int PTS = 32 / L;
    const int lane = threadIdx.x & 31;
    const int k = lane % L;
    const int64_t idx = static_cast<int64_t>(tile) * PTS + lane / L;
    const bool valid = idx < R.n_points;
    const double vs = R.valley > 0 ? 1.0 : -1.0;
    double px = 0.0, py = 0.0;
    if (valid) {
        px = grid_node(R.px_min, R.hx, idx % R.nx);
        py = grid_node(R.py_min, R.hy, R.row0 + idx / R.nx);
    }
    F64Point pt;
    pt.tx = vs * (R.dt * px);  // valley K- is stepped as K+ on -P
    pt.ty = vs * (R.dt * py);
    load_f64(R, idx, valid, px, py, vs, pt);
    double2 *a_plane = static_cast<double2 *>(R.state);
    if constexpr (L == 1) {
        using E = typename std::conditional<SCHEME == 2, F64G2, double2>::type;
        const WarpStager<E> st(R, &sm.stage[0][0], sm.bars);
        if (!st.run(err, [&](const E *e, int len) {
#pragma unroll 2
                for (int j = 0; j < len; ++j) {
                    if constexpr (SCHEME == 2)
                        step_f64<SCHEME, DC, DS>(pt, e[j].a, e[j].d);
                    else
                        step_f64<SCHEME, DC, DS>(pt, e[j], make_double2(0.0, 0.0));
                }
            }))
            return;
        if (valid) {
            a_plane[idx] = make_double2(pt.ar, pt.ai);
            a_plane[R.n_points + idx] = make_double2(pt.br, pt.bi);
        }
    } else {
        double v[4 / L];
        if constexpr (L == 2) {
            v[0] = k ? pt.br : pt.ar;
            v[1] = k ? pt.bi : pt.ai;
        } else {
            v[0] = k < 2 ? (k == 0 ? pt.ar : pt.ai) : (k == 2 ? pt.br : pt.bi);
        }
        const double t = (k & 1) ? pt.ty : pt.tx;
        const WarpStager<double2> st(R, &sm.stage[0][0], sm.bars);
        if (!st.run(err, [&](const double2 *e, int len) {
                lane_steps<DC, DS, L>(v, reinterpret_cast<const double *>(e) + (k & 1), t, len, k);
            }))
            return;
        if (valid) {
            if constexpr (L == 2)
                a_plane[(k ? R.n_points : 0) + idx] = make_double2(v[0], v[1]);
            else
                reinterpret_cast<double *>(a_plane)[2 * ((k < 2 ? 0 : R.n_points) + idx) + (k & 1)] =
                    v[0];
        }
    }
}

// A tile of 32 columns x 4 rows (EXACT and STRANG_XY).
template <int SCHEME, int DC, int DS>
__device__ void body_rows(const ReqDesc &R, int tile, F64Smem &sm, int *err)
{
    constexpr int H = 4;
    const int lane = threadIdx.x & 31;
    const int ncb = (R.nx + 31) / 32;
    const int rb = tile / ncb, cb = tile - rb * ncb;
    const int64_t row_first = static_cast<int64_t>(rb) * H;
    const int64_t col = static_cast<int64_t>(cb) * 32 + lane;
    const double vs = R.valley > 0 ? 1.0 : -1.0;
    const double px = grid_node(R.px_min, R.hx, col);
    const double tx = vs * (R.dt * px);  // valley K- is stepped as K+ on -P
    F64Point pt[H];
#pragma unroll
    for (int k = 0; k < H; ++k) {
        const int64_t row = row_first + k;
        const double py = grid_node(R.py_min, R.hy, R.row0 + row);
        pt[k].tx = tx;
        pt[k].ty = vs * (R.dt * py);
        load_f64(R, row * R.nx + col, col < R.nx && row < R.ny, px, py, vs, pt[k]);
    }
    const WarpStager<double2> st(R, &sm.stage[0][0], sm.bars);
    if (!st.run(err, [&](const double2 *e, int len) {
            // the row table of this chunk, from dt P_y = s dt p_y + s dt A_y
            for (int j = lane; j < len; j += 32) {
#pragma unroll
                for (int k = 0; k < H; ++k)
                    sm.rows[j][k] = strip64_row<SCHEME, DC, DS>(pt[k].ty + e[j].y);
            }
            __syncwarp();
#pragma unroll 2
            for (int j = 0; j < len; ++j)
                strip64_step<SCHEME, DC, DS, H>(pt, tx, e[j].x, sm.rows[j]);
        }))
        return;
    double2 *a_plane = static_cast<double2 *>(R.state);
#pragma unroll
    for (int k = 0; k < H; ++k) {
        const int64_t row = row_first + k, idx = row * R.nx + col;
        if (col < R.nx && row < R.ny) {
            a_plane[idx] = make_double2(pt[k].ar, pt[k].ai);
            a_plane[R.n_points + idx] = make_double2(pt[k].br, pt[k].bi);
        }
    }
}

// Warp-uniform dispatch on the request's series level (compile-time degrees).  L: 1, 2,
// 4 flat; 0 rows.
template <int SCHEME, int L, int V>
__device__ __forceinline__ void dispatch_f64(const ReqDesc &R, int tile, F64Smem &sm, int *err)
{
    if (R.level == V || V + 1 == kNumLevels) {
        if constexpr (L == 0)
            body_rows<SCHEME, kLevelsF64[V].dc, kLevelsF64[V].ds>(R, tile, sm, err);
        else
            body_flat<SCHEME, kLevelsF64[V].dc, kLevelsF64[V].ds, L>(R, tile, sm, err);
    } else if constexpr (V + 1 < kNumLevels) {
        dispatch_f64<SCHEME, L, V + 1>(R, tile, sm, err);
    }
}

template <int L>
__global__ void __launch_bounds__(32 * kF64Warps, L == 4 ? 2 : L == 0 ? 4 : 5)
    evolve_f64_kernel(const __grid_constant__ EvolveArgs args)
{
    __shared__ __align__(128) F64Smem smem[kF64Warps];
    const int w = threadIdx.x >> 5;
    const int t = static_cast<int>(blockIdx.x) * static_cast<int>(blockDim.x >> 5) + w;
    if (t >= args.total_tiles)
        return;
    F64Smem &sm = smem[w];
    if ((threadIdx.x & 31) == 0) {
        mbar_init(&sm.bars[0], 1);
        mbar_init(&sm.bars[1], 1);
        fence_mbar_init();
    }
    __syncwarp();
    const ReqDesc &R = args.r[find_request(args, t)];
    const int tile = t - R.tile_begin;
    if (!tile_ok(R, tile, R.err) || !table_range_ok(R, R.step_begin, R.err))
        return;
    if (L > 1 || R.scheme == 0)
        dispatch_f64<0, L, 0>(R, tile, sm, R.err);
    else if constexpr (L <= 1) {
        if (R.scheme == 1)
            dispatch_f64<1, L, 0>(R, tile, sm, R.err);
        else if constexpr (L == 1)
            dispatch_f64<2, L, 0>(R, tile, sm, R.err);
    }
}

template <int L>
cudaError_t launch_lanes(const EvolveArgs &args, int warps, cudaStream_t stream)
{
    const int grid = (args.total_tiles + warps - 1) / warps;
    evolve_f64_kernel<L><<<grid, 32 * warps, 0, stream>>>(args);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_evolve_f64(const EvolveArgs &args, int lanes, int warps, cudaStream_t stream)
{
    if (args.nreq <= 0 || args.total_tiles <= 0)
        return cudaSuccess;
    return lanes == 0   ? launch_lanes<0>(args, warps, stream)
           : lanes == 1 ? launch_lanes<1>(args, warps, stream)
           : lanes == 2 ? launch_lanes<2>(args, warps, stream)
                        : launch_lanes<4>(args, warps, stream);
}

}  // namespace dsp
