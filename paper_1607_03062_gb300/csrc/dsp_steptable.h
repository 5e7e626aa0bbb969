// dsp_steptable.h -- the FP32 per-step table of a pulse whose groups may be expanded,
// rounded on the device so that its running sum follows the exact one (not installed).
//
// The phase integrates A over time, so what matters is the running sum of the stored
// entries, not each entry.  Rounding one entry after the other with the residual carried
// along (build_table in dsp_api.cpp) is a chain over the whole run; here every step takes
// its entry from the running sum itself: F_n is the exact sum S_n rounded to a multiple of
// q_n, the spacing of floats at the larger of the steps n and n + 1, and the entry is
// F_n - F_(n-1).  Entries are differences of neighbours, so their sum is F_n however
// long the run: within q_n / 2 of S_n, half an ulp of an entry (or 2^-51 of S_n, where the
// steps are smaller than that).  They are floats exactly (a multiple of the smaller q, below
// 2^24 of it) unless neighbouring steps differ by more than 2^23, where the difference is
// rounded.  S_n starts from a sum per 16 steps made on the host,
// so blocks of 16 steps are independent.
#pragma once

#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define DSP_HD __host__ __device__ __forceinline__
#else
#define DSP_HD inline
#endif

namespace dsp {

constexpr int kTableBlock = 16;  // steps per prefix sum

DSP_HD uint64_t double_bits(double v)
{
#ifdef __CUDA_ARCH__
    return static_cast<uint64_t>(__double_as_longlong(v));
#else
    uint64_t u;
    memcpy(&u, &v, sizeof(u));
    return u;
#endif
}
DSP_HD double bits_double(uint64_t u)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double(static_cast<long long>(u));
#else
    double v;
    memcpy(&v, &u, sizeof(v));
    return v;
#endif
}

// a + b with one rounding (never contracted with the product that made a or b, so that
// two threads with the same sum get the same bits).
DSP_HD double add_rn(double a, double b)
{
#ifdef __CUDA_ARCH__
    return __dadd_rn(a, b);
#else
    return a + b;
#endif
}

// The running sum s rounded to a multiple of q, the spacing of floats at the larger of |v|
// and |w| (those within 2^-20 of the next power of two take its spacing, so that an entry a
// little above them still has it) or 2^-50 of |s|'s power of two if that is more.  Adding and
// taking away 1.5 2^52 q does it: the sum in between has the exponent of 2^52 q, its
// spacing is q.
DSP_HD double table_sum(double s, double v, double w)
{
    const uint64_t a = (double_bits(v) >> 32) & 0x7FFFFFFFu, b = (double_bits(w) >> 32) & 0x7FFFFFFFu;
    const uint64_t e = (((a > b ? a : b) + 1) >> 20) + 29;    // exponent fields: of 2^52 q,
    const uint64_t f = ((double_bits(s) >> 52) & 0x7FFu) + 2;  // and at least this
    const double magic = bits_double(((e > f ? e : f) << 52) | 0x8000000000000ull);
    return add_rn(add_rn(s, magic), -magic);
}

// Entries of the steps [16 g, 16 g + 16) of a table of n steps, one coordinate.  step(k) is
// s dt A of step k (also called for the steps just before and after the block), s0 and s1
// the running sums before the block and after it; put(k, f) takes the entry.
template <typename Step, typename Put>
DSP_HD void table_block(int64_t g, int64_t n, double s0, double s1, Step step, Put put)
{
    const int64_t first = kTableBlock * g;
    const int64_t end = first + kTableBlock < n ? first + kTableBlock : n;
    double v = step(first), inside = 0.0;  // inside: the sum in the block
    double f = first > 0 ? table_sum(s0, step(first - 1), v) : 0.0;
    for (int64_t k = first; k < end; ++k) {
        const double w = step(k + 1 < n ? k + 1 : k);  // (past the end: the last step again)
        inside = add_rn(inside, v);
        // (the next block starts from the same sum)
        const double h = table_sum(k + 1 < end ? add_rn(s0, inside) : s1, v, w);
        put(k, static_cast<float>(add_rn(h, -f)));
        f = h;
        v = w;
    }
}

// Copies a table's samples (A_x, A_y), `per` of them a step, to `to` and writes their running
// sums before every 16 steps, and after the last, to out[2 g], out[2 g + 1]: the blocks' sums
// are added with their rounding errors carried along (TwoSum), so that a sum is good to
// ~1e-16 of itself however long the run.  One pass, x and y side by side, four chains of
// additions: 1e5 steps 48 us on the host, the copy alone 45, copy and sums one after the
// other 80.
inline void copy_with_prefix(const double *a, int64_t n_steps, int per, double *to, double *out)
{
    typedef double Pair __attribute__((vector_size(16)));
    const auto load = [](const double *p) {
        Pair v;
        memcpy(&v, p, sizeof(v));
        return v;
    };
    const auto copy = [&load](const double *p, double *q) {
        const Pair v = load(p);
        memcpy(q, &v, sizeof(v));
        return v;
    };
    Pair sum = {0.0, 0.0}, low = {0.0, 0.0};
    const auto put = [&] {
        const Pair v = sum + low;
        memcpy(out, &v, sizeof(v));
        out += 2;
    };
    const auto add = [&](Pair v) {
        const Pair t = sum + v, b = t - sum;
        low += (sum - (t - b)) + (v - b);
        sum = t;
    };
    const int64_t n = n_steps * per;
    for (int64_t k = 0; k < n; k += 16) {
        if (per == 1 || k % 32 == 0)
            put();
        const double *p = a + 2 * k;
        double *q = to + 2 * k;
        if (n - k >= 16) {
            Pair s0 = copy(p, q), s1 = copy(p + 2, q + 2), s2 = copy(p + 4, q + 4),
                 s3 = copy(p + 6, q + 6);
            for (int i = 8; i < 32; i += 8) {
                s0 += copy(p + i, q + i);
                s1 += copy(p + i + 2, q + i + 2);
                s2 += copy(p + i + 4, q + i + 4);
                s3 += copy(p + i + 6, q + i + 6);
            }
            add((s0 + s1) + (s2 + s3));
        } else {
            for (int64_t i = 0; i < n - k; ++i)
                add(copy(p + 2 * i, q + 2 * i));
        }
    }
    put();
}

}  // namespace dsp
