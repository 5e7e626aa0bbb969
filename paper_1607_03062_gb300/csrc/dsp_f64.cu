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
// absolute at theta 0.005 (below theta^2 2^-47, 7e-17 at 0.1): below an FP64 ulp of the
// state.
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

// The FP64 EXACT step's operator from dt P = (Px, Py) and their squares as float
// pairs: m = cos(theta) - 1 and q = qr + i qi.
template <int DC, int DS>
__device__ __forceinline__ void operator_f64_exact(double Px, double Py, float2 px2, float2 py2,
                                                   double &m, double &qr, double &qi)
{
    float xh = px2.x, xl = px2.y;
    df_add(xh, xl, py2.x, py2.y);  // theta^2
    float th, tl, mh, ml, sh, sl;
    horner_df<DC, 1, 0>(xh, xl, th, tl);  // (cos(theta) - 1) / theta^2
    df_mul(xh, xl, th, tl, mh, ml);
    horner_df<DS, 1, 1>(xh, xl, th, tl);  // (sin(theta)/theta - 1) / theta^2
    df_mul(xh, xl, th, tl, sh, sl);
    m = df_to_f64(mh, ml);
    const double s1 = df_to_f64(sh, sl);
    qr = fma(s1, Py, Py);
    qi = fma(s1, Px, Px);
}

// The FP64 EXACT step.
template <int DC, int DS>
__device__ __forceinline__ void step_f64_exact(F64Point &s, double Px, double Py, float2 px2,
                                               float2 py2)
{
    double m, qr, qi;
    operator_f64_exact<DC, DS>(Px, Py, px2, py2, m, qr, qi);
    // a' = a + m a - q b ; b' = b + m b + conj(q) a
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

// cos and sinc of STRANG_XY and MAGNUS4 from x = theta^2 in FP64.  Up to cosine degree
// kF64TailDegree (theta below ~0.16) the terms from x^2 on are summed in double-float beside the
// FP64 work: at most theta^4/24, they are off by less than 1e-20 at theta 0.1, so cos and
// sinc are rounded as in the FP64 series (measured on the CPU over random theta: cos the
// same, sinc theta 0.8 of its error), for 2 FP64 operations each, whatever the degree.  (All
// of cos - 1 and sinc - 1 as pairs of floats, 1 each, is off by ~2^-50 of theta^2/2 with one
// sign: 1e5 steps at theta 0.06 put 1.6e-13 into the state instead of 1.7e-14.)
// c = cos - 1 + 1 and s1 = sinc - 1 (DC <= kF64TailDegree).
template <int DC, int DS>
__device__ __forceinline__ void cos_sinc_f64(double x, double &c, double &s1)
{
    float xh, xl, x2h, x2l, th, tl, uh, ul;
    split_f64(x, xh, xl);
    df_mul(xh, xl, xh, xl, x2h, x2l);
    horner_df<DC, 2, 0>(xh, xl, th, tl);
    df_mul(x2h, x2l, th, tl, uh, ul);
    c = 1.0 + fma(x, -0.5, df_to_f64(uh, ul));
    horner_df<DS, 2, 1>(xh, xl, th, tl);
    df_mul(x2h, x2l, th, tl, uh, ul);
    s1 = fma(x, -1.0 / 6.0, df_to_f64(uh, ul));
}

// The FP64 MAGNUS4 step's operator: n = (dt Pbar, n_z), n_z = Pbar x D; c = cos|n|, q and
// qz = sinc|n| n: 31 FP64 operations a step with the update, 26 + dc + ds above kF64TailDegree.
template <int DC, int DS>
__device__ __forceinline__ void operator_f64_magnus(double Px, double Py, double2 d, double &c,
                                                    double &qr, double &qi, double &qz)
{
    const double nz = fma(Px, d.y, -(Py * d.x));
    const double x = fma(Px, Px, fma(Py, Py, nz * nz));
    if constexpr (DC <= kF64TailDegree) {
        double s1;
        cos_sinc_f64<DC, DS>(x, c, s1);
        qr = fma(s1, Py, Py);
        qi = fma(s1, Px, Px);
        qz = fma(s1, nz, nz);
    } else {
        c = horner_f64<DC, 0, 0>(x);
        const double sn = horner_f64<DS, 0, 1>(x);
        qr = sn * Py;
        qi = sn * Px;
        qz = sn * nz;
    }
}
template <int DC, int DS>
__device__ __forceinline__ void step_f64_magnus(F64Point &s, double Px, double Py, double2 d)
{
    double c, qr, qi, qz;
    operator_f64_magnus<DC, DS>(Px, Py, d, c, qr, qi, qz);
    // a' = (c - i qz) a - q b ; b' = conj(q) a + (c + i qz) b, q = qr + i qi: the small
    // terms first, one rounding at the state's size
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

// STRANG_XY's parts of one coordinate, {cos P, sin P}; and its step from those of x and y,
// c = cos y cos x, q = sin y + i cos y sin x.  30 FP64 operations a step, 20 + 2 dc + 2 ds
// above kF64TailDegree; on row tiles the parts of a row and of a column are formed once.
template <int DC, int DS>
__device__ __forceinline__ double2 strang_part(double P)
{
    const double x = P * P;
    if constexpr (DC <= kF64TailDegree) {
        double c, s1;
        cos_sinc_f64<DC, DS>(x, c, s1);
        return make_double2(c, fma(s1, P, P));
    } else {
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
// Warps (in one shape, pairs of warps) work alone: their own double-buffered bulk copies
// of the table with bounded waits, no CTA-wide barrier, and the host picks the shape that
// loads the fullest scheduler least (f64_lanes in dsp_api.cpp).  FP64 instructions per
// step of a tile (EXACT; STRANG_XY and MAGNUS4 up to kF64TailDegree) and its points:
//   rows   32 columns x 4 rows: the dt P_x part once per lane, the dt P_y part once per
//          row and step in a shared table                       65, 65, - for 128
//   flat   32 consecutive points, a lane each                   18, 30, 31 for 32
//   pair   8 points, a lane per real component in one warp, the operators of four
//          steps at once in the other                           4.5, 7.5, 7.8 for 8
// Every FP64 operation of a point is the same in every shape (same operands, same
// rounding), so its result is bitwise the same.  The projection is the projection
// kernel's, on the state these leave.
//
// A step's operator is a chain of ~900 cycles before its update, and a warp cannot run
// the one beside the other: its own FP64 instructions hold its issue.  Flat and rows
// therefore need several warps per scheduler, and pairs take the launches that cannot
// give them.  Measured, 2000 EXACT steps: 64^2 9.48 ms with 1024-point CTAs (4 of 152
// SMs), 1.80 flat, 1.08 with 4 lanes a point on one warp, 0.40 on pairs (0.22 of FP64
// work over the whole chip); 128^2 1.83 flat, 1.12 pairs; 256^2 4.83, 4.31; 300 x 257
// 4.84 flat, 4.92 pairs; 512^2 17.1 rows, 16.5 flat and pairs.
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

// A flat tile of 32 consecutive points.
template <int SCHEME, int DC, int DS>
__device__ void body_flat(const ReqDesc &R, int tile, F64Smem &sm, int *err)
{
    const int lane = threadIdx.x & 31;
    const int64_t idx = static_cast<int64_t>(tile) * 32 + lane;
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
    double2 *a_plane = static_cast<double2 *>(R.state);
    if (valid) {
        a_plane[idx] = make_double2(pt.ar, pt.ai);
        a_plane[R.n_points + idx] = make_double2(pt.br, pt.bi);
    }
}

// 4 lanes per point and two warps per 8 points.  A warp waits out the issue of its own
// FP64 instructions, so one warp cannot form a step's operator beside another step's
// update; here one warp of the pair forms operators, the lanes of a point those of four
// steps at once, and hands them through shared memory, kPairSteps at a time and double
// buffered, to the other, whose lanes hold Re a, Im a, Re b, Im b of a point and only
// apply them.  Waits between the two are bounded like those for the table.
constexpr int kPairSteps = 16;
static_assert(kF64Chunk % kPairSteps == 0 && kF64Chunk / 2 % kPairSteps == 0,
              "table chunks are whole slots");
struct PairSmem {
    unsigned char stage[2][kF64Stage];
    double ops[2][kPairSteps][4][8];  // per step: m or c, qr, qi, qz of the 8 points
    uint64_t bars[2];                 // table chunks
    uint64_t full[2], empty[2];       // slots of ops
};

// A step's operator into out: EXACT m, qr, qi; STRANG_XY c, qr, qi; MAGNUS4 c, qr, qi, qz.
template <int SCHEME, int DC, int DS, typename E>
__device__ __forceinline__ void form_operator(const E &e, double tx, double ty,
                                              double (&out)[4][8], int pt)
{
    double c, qr, qi;
    if constexpr (SCHEME == 2) {
        double qz;
        operator_f64_magnus<DC, DS>(tx + e.a.x, ty + e.a.y, e.d, c, qr, qi, qz);
        out[3][pt] = qz;
    } else {
        const double Px = tx + e.x, Py = ty + e.y;
        if constexpr (SCHEME == 0) {
            operator_f64_exact<DC, DS>(Px, Py, square_df(Px), square_df(Py), c, qr, qi);
        } else {
            const double2 x = strang_part<DC, DS>(Px), y = strang_part<DC, DS>(Py);
            c = y.x * x.x;
            qr = y.y;
            qi = y.x * x.y;
        }
    }
    out[0][pt] = c;
    out[1][pt] = qr;
    out[2][pt] = qi;
}

template <int SCHEME, int DC, int DS>
__device__ void pair_operators(const ReqDesc &R, double tx, double ty, PairSmem &sm, int *err)
{
    const int lane = threadIdx.x & 31, s = lane & 3;
    using E = typename std::conditional<SCHEME == 2, F64G2, double2>::type;
    const WarpStager<E> st(R, &sm.stage[0][0], sm.bars);
    int q = 0;
    bool ok = true;
    st.run(err, [&](const E *e, int len) {
        for (int b = 0; b < len; b += kPairSteps, ++q) {
            if (ok && q >= 2)  // the other warp is done with the slot
                ok = __all_sync(0xffffffffu, mbar_wait_bounded(&sm.empty[q & 1], ((q >> 1) - 1) & 1));
            if (!ok)
                continue;
#pragma unroll
            for (int p = 0; p < kPairSteps; p += 4) {
                const int j = b + p + s;  // past the end: the last one's, not applied
                form_operator<SCHEME, DC, DS>(e[j < len ? j : len - 1], tx, ty,
                                              sm.ops[q & 1][p + s], lane >> 2);
            }
            __syncwarp();
            if (lane == 0)
                mbar_arrive(&sm.full[q & 1]);
        }
    });
    if (!ok && lane == 0)
        atomicOr(err, kErrTimeout);
}

// v with its sign bit flipped where mask is 1 << 31: an integer operation (choosing
// between x and -x negates on the FP64 pipe: 64^2 x 2000 took 0.56 ms, not 0.40).
__device__ __forceinline__ double flip_sign(double v, int mask)
{
    return __hiloint2double(__double2hiint(v) ^ mask, __double2loint(v));
}

template <int SCHEME>
__device__ __forceinline__ bool pair_updates(double &v, int64_t nsteps, PairSmem &sm, int *err)
{
    constexpr int kSign = static_cast<int>(0x80000000u);
    const int lane = threadIdx.x & 31, k = lane & 3;
    const int sr_mask = (k & 2) ? 0 : kSign, si_mask = (k & 1) ? kSign : 0;
    const int sz_mask = k == 1 || k == 2 ? kSign : 0;
    for (int q = 0; static_cast<int64_t>(q) * kPairSteps < nsteps; ++q) {
        if (!__all_sync(0xffffffffu, mbar_wait_bounded(&sm.full[q & 1], (q >> 1) & 1))) {
            if (lane == 0)
                atomicOr(err, kErrTimeout);
            return false;
        }
        const int64_t left = nsteps - static_cast<int64_t>(q) * kPairSteps;
        const int len = left < kPairSteps ? static_cast<int>(left) : kPairSteps;
        const double *o = &sm.ops[q & 1][0][0][lane >> 2];
#pragma unroll 4
        for (int u = 0; u < len; ++u, o += 4 * 8) {
            const double c = o[0];
            const double sr = flip_sign(o[8], sr_mask), si = flip_sign(o[16], si_mask);
            const double t1 = shfl_x(v, 2), t2 = shfl_x(v, 3);
            if constexpr (SCHEME == 0) {
                v = fma(c, v, fma(sr, t1, fma(si, t2, v)));
            } else if constexpr (SCHEME == 1) {
                v = fma(c, v, fma(sr, t1, si * t2));
            } else {
                const double t0 = shfl_x(v, 1);
                v = fma(c, v, fma(flip_sign(o[24], sz_mask), t0, fma(sr, t1, si * t2)));
            }
        }
        __syncwarp();
        if (lane == 0)
            mbar_arrive(&sm.empty[q & 1]);
    }
    return true;
}

// A tile of 8 consecutive points; `forms`: this warp forms the operators.
template <int SCHEME, int DC, int DS>
__device__ void body_pair(const ReqDesc &R, int tile, PairSmem &sm, int *err, bool forms)
{
    const int lane = threadIdx.x & 31, k = lane & 3;
    const int64_t idx = static_cast<int64_t>(tile) * 8 + (lane >> 2);
    const bool valid = idx < R.n_points;
    const double vs = R.valley > 0 ? 1.0 : -1.0;
    double px = 0.0, py = 0.0;
    if (valid) {
        px = grid_node(R.px_min, R.hx, idx % R.nx);
        py = grid_node(R.py_min, R.hy, R.row0 + idx / R.nx);
    }
    if (forms) {  // valley K- is stepped as K+ on -P
        pair_operators<SCHEME, DC, DS>(R, vs * (R.dt * px), vs * (R.dt * py), sm, err);
        return;
    }
    F64Point pt;
    load_f64(R, idx, valid, px, py, vs, pt);
    double v = k < 2 ? (k == 0 ? pt.ar : pt.ai) : (k == 2 ? pt.br : pt.bi);
    if (!pair_updates<SCHEME>(v, R.step_end > R.step_begin ? R.step_end - R.step_begin : 0, sm, err))
        return;
    if (valid)
        static_cast<double *>(R.state)[2 * ((k < 2 ? 0 : R.n_points) + idx) + (k & 1)] = v;
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

// Warp-uniform dispatch on the request's scheme and series level (compile-time
// degrees): body(scheme, dc, ds) as integral constants.
template <int SCHEME, int V, typename Body>
__device__ __forceinline__ void dispatch_level(const ReqDesc &R, Body body)
{
    if (R.level == V || V + 1 == kNumLevels)
        body(std::integral_constant<int, SCHEME>{},
             std::integral_constant<int, kLevelsF64[V].dc>{},
             std::integral_constant<int, kLevelsF64[V].ds>{});
    else if constexpr (V + 1 < kNumLevels)
        dispatch_level<SCHEME, V + 1>(R, body);
}
template <bool MAGNUS, typename Body>
__device__ __forceinline__ void dispatch_f64(const ReqDesc &R, Body body)
{
    if (R.scheme == 0)
        dispatch_level<0, 0>(R, body);
    else if (R.scheme == 1)
        dispatch_level<1, 0>(R, body);
    else if constexpr (MAGNUS)
        dispatch_level<2, 0>(R, body);
}

// Tiles on one warp: ROWS 32 columns x 4 rows, otherwise flat.
template <bool ROWS>
__global__ void __launch_bounds__(32 * kF64Warps, ROWS ? 4 : 5)
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
    dispatch_f64<!ROWS>(R, [&](auto scheme, auto dc, auto ds) {
        if constexpr (ROWS)
            body_rows<decltype(scheme)::value, decltype(dc)::value, decltype(ds)::value>(R, tile,
                                                                                         sm, R.err);
        else
            body_flat<decltype(scheme)::value, decltype(dc)::value, decltype(ds)::value>(R, tile,
                                                                                         sm, R.err);
    });
}

// Warp pairs, kF64Warps / 2 of them or one per CTA.  The CTAs are dealt to the SMs in
// turn, so that swapping the warps' roles from one round of SMs to the next puts both
// kinds on every scheduler.  One kernel per scheme.
template <int SCHEME>
__global__ void __launch_bounds__(32 * kF64Warps, 4)
    evolve_f64_pair_kernel(const __grid_constant__ EvolveArgs args, int sms)
{
    __shared__ __align__(128) PairSmem smem[kF64Warps / 2];
    const int w = threadIdx.x >> 5;
    PairSmem &sm = smem[w >> 1];
    if ((threadIdx.x & 63) == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sm.bars[i], 1);
            mbar_init(&sm.full[i], 1);
            mbar_init(&sm.empty[i], 1);
        }
        fence_mbar_init();
    }
    __syncthreads();
    const int t = static_cast<int>(blockIdx.x) * static_cast<int>(blockDim.x >> 6) + (w >> 1);
    if (t >= args.total_tiles)
        return;
    const ReqDesc &R = args.r[find_request(args, t)];
    const int tile = t - R.tile_begin;
    if (!tile_ok(R, tile, R.err) || !table_range_ok(R, R.step_begin, R.err))
        return;
    const bool forms = (w & 1) != ((blockIdx.x / sms) & 1);
    dispatch_level<SCHEME, 0>(R, [&](auto scheme, auto dc, auto ds) {
        body_pair<decltype(scheme)::value, decltype(dc)::value, decltype(ds)::value>(R, tile, sm,
                                                                                     R.err, forms);
    });
}

}  // namespace

cudaError_t launch_evolve_f64(const EvolveArgs &args, int lanes, int warps, cudaStream_t stream)
{
    if (args.nreq <= 0 || args.total_tiles <= 0)
        return cudaSuccess;
    if (lanes == 4) {
        int dev = 0, sms = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess)
            e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess)
            return e;
        const int pairs = warps > 1 ? warps / 2 : 1;
        const int grid = (args.total_tiles + pairs - 1) / pairs;
        const int scheme = args.r[0].scheme;
        if (scheme == 0)
            evolve_f64_pair_kernel<0><<<grid, 64 * pairs, 0, stream>>>(args, sms);
        else if (scheme == 1)
            evolve_f64_pair_kernel<1><<<grid, 64 * pairs, 0, stream>>>(args, sms);
        else
            evolve_f64_pair_kernel<2><<<grid, 64 * pairs, 0, stream>>>(args, sms);
        return cudaGetLastError();
    }
    const int grid = (args.total_tiles + warps - 1) / warps;
    if (lanes == 0)
        evolve_f64_kernel<true><<<grid, 32 * warps, 0, stream>>>(args);
    else
        evolve_f64_kernel<false><<<grid, 32 * warps, 0, stream>>>(args);
    return cudaGetLastError();
}

}  // namespace dsp
