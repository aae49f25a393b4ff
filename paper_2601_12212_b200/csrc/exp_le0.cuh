// The exponential of the acceptance under sampling (sampled.cu), for device code and for a host compiler (its test
// runs this very code).
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

namespace resps {

#ifdef __CUDACC__
#define RESPS_HD __host__ __device__ __forceinline__
#else
#define RESPS_HD inline
#endif

RESPS_HD int low_word(double v) {
#ifdef __CUDA_ARCH__
    return __double2loint(v);
#else
    int64_t bits;
    std::memcpy(&bits, &v, 8);
    return static_cast<int>(static_cast<uint32_t>(bits));
#endif
}
// v with `step` added to its exponent (where the result is a normal number)
RESPS_HD double add_exponent(double v, int step) {
#ifdef __CUDA_ARCH__
    return __hiloint2double(__double2hiint(v) + (step << 20), __double2loint(v));
#else
    int64_t bits;
    std::memcpy(&bits, &v, 8);
    const uint64_t sum = static_cast<uint64_t>(bits) + (static_cast<uint64_t>(static_cast<int64_t>(step)) << 52);
    std::memcpy(&v, &sum, 8);
    return v;
#endif
}

// e^t for t <= 0 (below -700: 0), to about one unit in the last place: table-driven (P. Tang, "Table-driven
// implementation of the exponential function in IEEE floating-point arithmetic", 1989).  t = k ln2/64 + r,
// |r| <= ln2/128, e^t = 2^(k/64) e^r with 2^(i/64) from a table (in shared memory) and five terms of the series
// for e^r - 1 (the next one is below 4e-17): 11 fp64 operations.
constexpr int kExpTable = 64;
RESPS_HD double exp_le0(double t, const double* table) {
    constexpr double kMagic = 6755399441055744.0;  // 1.5 * 2^52: the sum's low word is the rounded integer
    const double biased = fma(t, 92.33248261689366, kMagic);  // 64 / ln 2
    const int k = low_word(biased);
    const double kd = biased - kMagic;
    double r = fma(kd, -0.010830424696249145, t);  // ln 2 / 64, rounded,
    r = fma(kd, -3.623510646634843e-19, r);        // and the rest of it
    double q = fma(r, 1.0 / 120.0, 1.0 / 24.0);
    q = fma(q, r, 1.0 / 6.0);
    q = fma(q, r, 0.5);
    q = fma(q, r, 1.0) * r;
    const double head = table[k & (kExpTable - 1)];
    const double y = fma(head, q, head);  // about 2^(k/64 mod 1) e^r: 2^(k >> 6) goes into its exponent
    const double v = add_exponent(y, k >> 6);
    return t > -700.0 ? v : 0.0;
}

}  // namespace resps
