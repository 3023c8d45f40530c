// lbs_log.cuh — log(1 + x) of the equation of state (Eq. 8) near saturation in
// single precision, rounded as the logarithm in double precision is.
//
// Below x = -1/2 (psi / psi_inf > 1/2) the logarithm is that of double
// precision rounded to single.  Its 60-odd instructions run at 1/64 of the
// single precision rate here, so the value is first formed as an unevaluated
// sum r + t of two floats, r the rounded one; only where t and its error leave
// open which float the logarithm rounds to (about one value in 2^13) is the
// double precision one taken.  The results are the same to the bit.
//
// Argument reduction by a table of reciprocals (P.-T. P. Tang, Table-driven
// implementation of the logarithm function in IEEE floating-point arithmetic,
// ACM TOMS 16, 1990):
//   u = 1 + x (exact) = 2^e m, 1 <= m < 2, c_j of 7 bits near 1 / m,
//   z = c_j m - 1 (exact, |z| <= 2^-6),
//   log u = e ln 2 - log c_j + z - z^2/2 + z^3 (1/3 - z/4 + z^2/5 - ...).
// e ln 2 and -log c_j each as a multiple of 2^-16, whose sum is exact, and a
// remainder.  The host and the device execute the same operations.
//
// Force kernel of a 256 x 128 x 128 grid, BF16 populations, half of the cells
// above 1/2: 165 us with the double precision logarithm, 83 with this one.
#pragma once

#include <cmath>
#include <cstring>

#ifdef __CUDACC__
#define LBS_HD __host__ __device__
#else
#define LBS_HD
#endif

namespace lbs {

struct alignas(16) LogRow {
    float c, hi, lo, pad;  // c_j; -log c_j = hi + lo, hi a multiple of 2^-16
};
struct LogTable {
    LogRow row[64];
};
constexpr double kLn2 = 0.693147180559945309417;
// -log c for 1/2 <= c <= 1: 2 artanh((1 - c) / (1 + c)) by its series
constexpr double minus_log(double c) {
    const double s = (1.0 - c) / (1.0 + c), s2 = s * s;
    double sum = 0.0;
    for (int k = 41; k >= 1; k -= 2) sum = sum * s2 + 1.0 / k;
    return 2.0 * s * sum;
}
constexpr LogTable make_log_table() {
    LogTable t{};
    for (int j = 0; j < 64; j++) {
        // 1 / (middle of [1 + j / 64, 1 + (j + 1) / 64)) to 7 bits
        const double c = double(int(128.0 / (1.0 + (j + 0.5) / 64.0) + 0.5)) / 128.0;
        const double l = minus_log(c), hi = double(int(l * 65536.0 + 0.5)) / 65536.0;
        t.row[j] = LogRow{float(c), float(hi), float(l - hi), 0.0f};
    }
    return t;
}
constexpr LogTable kLogTable = make_log_table();
#ifdef __CUDACC__
static __device__ const LogTable d_log_table = make_log_table();
#endif

LBS_HD inline LogRow log_row(int j) {
#ifdef __CUDA_ARCH__
    const float4 v = __ldg((const float4 *)d_log_table.row + j);
    return LogRow{v.x, v.y, v.z, v.w};
#else
    return kLogTable.row[j];
#endif
}
LBS_HD inline float bits_float(int i) {
#ifdef __CUDA_ARCH__
    return __int_as_float(i);
#else
    float f;
    std::memcpy(&f, &i, 4);
    return f;
#endif
}
LBS_HD inline int float_bits(float f) {
#ifdef __CUDA_ARCH__
    return __float_as_int(f);
#else
    int i;
    std::memcpy(&i, &f, 4);
    return i;
#endif
}
// (sums and products that are not to be contracted)
LBS_HD inline float add_rn(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fadd_rn(a, b);
#else
    return a + b;
#endif
}
LBS_HD inline float mul_rn(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fmul_rn(a, b);
#else
    return a * b;
#endif
}

// log(1 + x), -1 < x < -1/2, as r + t (|t| <= half an ulp of r) to within eps;
// true where that decides the rounding: r is the logarithm rounded to nearest
LBS_HD inline bool log1p_pair(float x, float &r) {
    const float u = 1.0f + x;  // (exact: a multiple of 2^-24 below 1/2)
    const int i = float_bits(u), e = (i >> 23) - 127;
    const LogRow w = log_row((i >> 17) & 63);
    const float m = bits_float((i & 0x7FFFFF) | 0x3F800000), ef = float(e);
    const float z = fmaf(m, w.c, -1.0f);
    constexpr float l2hi = float(22713.0 / 32768.0), l2lo = float(kLn2 - 22713.0 / 32768.0);
    // hi parts: exact, and at least 0.6 in magnitude
    const float a = fmaf(ef, l2hi, w.hi);
    const float s1 = add_rn(a, z), e1 = add_rn(z, -add_rn(s1, -a));
    const float q = mul_rn(z, z), qe = fmaf(z, z, -q), h = 0.5f * q;
    const float s2 = add_rn(s1, -h), e2 = add_rn(add_rn(s1, -s2), -h);
    float p = 1.0f / 7.0f;
    p = fmaf(p, z, -1.0f / 6.0f);
    p = fmaf(p, z, 1.0f / 5.0f);
    p = fmaf(p, z, -1.0f / 4.0f);
    p = fmaf(p, z, 1.0f / 3.0f);
    const float c = fmaf(-0.5f, qe, mul_rn(mul_rn(z, q), p));
    const float lo = add_rn(add_rn(add_rn(e1, e2), fmaf(ef, l2lo, w.lo)), c);
    r = add_rn(s2, lo);
    const float t = add_rn(lo, -add_rn(r, -s2));
    const float eps = -r * 0x1p-38f;  // (r < 0)
    return add_rn(r, add_rn(t, eps)) == r && add_rn(r, add_rn(t, -eps)) == r;
}

}  // namespace lbs
