// cs_action.cuh -- Benincasa-Dowker action arithmetic shared by the
// single-set and batched action kernels and the host path (Section "The
// Benincasa-Dowker Action"), in double-double FP64.
#pragma once

#include <cmath>

#include "cs_internal.cuh"

namespace cs {

constexpr int kMaxEps = 16;  // eps values per call
constexpr int kActThreads = 256;
constexpr int kActBlocks = 128;  // partial sums per eps

// Powers q^(2^b), q = 1 - eps, of one eps: found on the host, so that a power
// on the device is a product of the few that its exponent's bits ask for (the
// repeated squaring took as many dependent double-double products again).
constexpr int kPowBits = 22;  // every exponent of a set (at most 2^22 elements)
struct EpsPowers {
    dd p[kPowBits];
};
inline EpsPowers eps_powers(double eps) {
    EpsPowers t;
    t.p[0] = dd_two_sum(1.0, -eps);
    for (int b = 1; b < kPowBits; ++b) t.p[b] = dd_mul(t.p[b - 1], t.p[b - 1]);
    return t;
}
// Two chains side by side, the five low bits of k (which differ between the
// lanes) and the bits above them (which do not): one product of all the bits
// made the chain twice as long.
__device__ __forceinline__ dd power_of(const EpsPowers& t, int64_t k) {
    const uint32_t m = uint32_t(k) & ((1u << kPowBits) - 1u);
    uint32_t lo = m & 31u, hi = m & ~31u;
    dd r = dd_from(1.0), s = dd_from(1.0);
    if (lo) r = t.p[__ffs(int(lo)) - 1];
    if (hi) s = t.p[__ffs(int(hi)) - 1];
    lo &= lo - 1u;
    hi &= hi - 1u;
    while (lo | hi) {
        r = dd_mul(r, lo ? t.p[__ffs(int(lo)) - 1] : dd_from(1.0));
        s = dd_mul(s, hi ? t.p[__ffs(int(hi)) - 1] : dd_from(1.0));
        lo &= lo - 1u;
        hi &= hi - 1u;
    }
    r = dd_mul(r, s);
    if (k >> kPowBits) r = dd_mul(r, dd_pow(dd_mul(t.p[kPowBits - 1], t.p[kPowBits - 1]), k >> kPowBits));  // a longer histogram
    return r;
}

// f times a whole number, c as exactly as it stands: one double below 2^53 (every
// count of a set), both halves of the int64 from there on (a caller's histogram).
__host__ __device__ __forceinline__ dd dd_times_i64(dd f, int64_t c) {
    if (c < (int64_t(1) << 53) && c > -(int64_t(1) << 53)) return dd_mul_d(f, static_cast<double>(c));
    return dd_mul(dd_from_i64(c), f);
}

// What smear_poly holds without k, and the values f_d(k), k < deg, found on
// the host: products of q and eps were half of a term's FP64 operations.  What
// is left per k are smear_poly's own products, to the last bit.  (With
// coefficients a - b k + c t - d C(k, 3) rounded on the host a term took up to ten operations
// less, but their roundings are the same in every term: the sum's error was
// 8e-31 of its largest term instead of 3e-31.)
struct SmearCoef {
    dd a, q, e2, d, f[3];  // q^deg; q (3+1: q^2) and q; eps^2; 8 eps^3
    dd q1;
    double e;
};
inline SmearCoef smear_coef(int dim, double eps) {
    const dd q = dd_two_sum(1.0, -eps), e = dd_from(eps), q2 = dd_mul(q, q);
    SmearCoef r;
    r.e = eps;
    r.q1 = q;
    r.q = dim == 4 ? q2 : q;
    r.a = dim == 4 ? dd_mul(q2, q) : q2;
    r.e2 = dd_mul(e, e);
    r.d = dd_mul_d(dd_mul(r.e2, e), 8.0);
    for (int k = 0; k < 3; ++k) r.f[k] = smear_poly(dim, k, q, eps);
    return r;
}
__host__ __device__ __forceinline__ dd smear_poly_at(int dim, const SmearCoef& m, int64_t k) {
    const int64_t t = k * (k - 1) / 2;
    const double x = static_cast<double>(k);
    const dd b = dd_mul(dd_two_prod(m.e, (dim == 2 ? 2.0 : dim == 3 ? 3.375 : 9.0) * x), m.q);
    if (dim == 2) return dd_add(dd_sub(m.a, b), dd_times_i64(m.e2, t));
    if (dim == 3) return dd_add(dd_sub(m.a, b), dd_mul_d(m.e2, 2.25 * static_cast<double>(t)));
    const int64_t w = k - 2;
    const dd c3 = w % 3 == 0 ? dd_two_prod(static_cast<double>(t), static_cast<double>(w / 3))
                             : dd_two_prod(static_cast<double>(t / 3), static_cast<double>(w));  // C(k, 3), exactly
    const dd c = dd_mul(dd_times_i64(m.e2, 16 * t), m.q1);
    return dd_sub(dd_add(dd_sub(m.a, b), c), dd_mul(m.d, c3));
}
// f_d(k).
__device__ __forceinline__ dd smear_term(int dim, const SmearCoef& m, const EpsPowers& t, int64_t k) {
    const int64_t deg = smear_deg(dim);
    if (k < deg) return m.f[k];
    return dd_mul(power_of(t, k - deg), smear_poly_at(dim, m, k));
}

struct EpsArgs {
    double v[kMaxEps];
    int64_t kend[kMaxEps];  // smeared-sum cutoffs (single-set kernels; set on the host)
    dd factor[kMaxEps];     // action_factor (single-set kernels; the batch has one set per dimension)
    int n;
};

__host__ __device__ inline dd dd_div(dd a, dd b) {
    const double q1 = a.hi / b.hi;
    dd r = dd_sub(a, dd_mul_d(b, q1));
    const double q2 = r.hi / b.hi;
    r = dd_sub(r, dd_mul_d(b, q2));
    const double q3 = r.hi / b.hi;
    return dd_add(dd_quick_two_sum(q1, q2), dd_from(q3));
}

// One Newton step on the correctly rounded double root: x + (a - x^2) / (2x).
__host__ __device__ inline dd dd_sqrt(dd a) {
    if (a.hi <= 0.0) return dd_from(0.0);
    const double x = sqrt(a.hi);
    const dd r = dd_sub(a, dd_two_prod(x, x));
    return dd_quick_two_sum(x, r.hi / (2.0 * x));
}

// The integer in parentheses of the local action; in 2+1 eight times it
// (8N - 8n1 + 27n2 - 18n3) so that it stays an integer.
__host__ __device__ inline int64_t bracket_of(int dim, int64_t n, const int64_t* h4) {
    if (dim == 2) return n - 2 * h4[0] + 4 * h4[1] - 2 * h4[2];
    if (dim == 3) return 8 * n - 8 * h4[0] + 27 * h4[1] - 18 * h4[2];
    return n - h4[0] + 9 * h4[1] - 16 * h4[2] + 8 * h4[3];
}

// The 2+1 constant (pi/(3 sqrt 2))^(2/3) / Gamma(5/3) of Eqs. s3d_local and
// b3d_local, 0.90665872967043620699..., in double (a constant factor, 7e-17
// from the exact one; the C libraries' cube root and gamma function gave
// values up to two units in the last place off, and not the same ones).
inline double c3_const() { return 0.9066587296704361; }

__host__ __device__ inline bool is_local(double eps) { return eps <= 0.0 || eps == 1.0; }

// Factors of the actions that depend on eps (and the dimension) alone, found
// on the host: on the device the 2+1 and 3+1 ones are a cube root and two
// double-double divisions, FP64 work in one thread.
//   local:   2 * bracket (1+1), c3 * bracket / 8 (2+1), 4/sqrt(6) * bracket (3+1)
//   smeared, from sum = sum_k N_k f(k, eps):
//     1+1: 2 eps [N - 2 eps sum];  2+1: c3 eps^(2/3) [N - eps sum];
//     3+1: 4 sqrt(eps/6) [N - eps sum].
inline dd local_factor(int dim) {
    if (dim == 2) return dd_from(2.0);
    if (dim == 3) return dd_from(c3_const() * 0.125);
    return dd_div(dd_from(4.0), dd_sqrt(dd_from(6.0)));
}

inline dd smeared_factor(int dim, double eps) {
    if (dim == 2) return dd_mul_d(dd_from(eps), 2.0);
    if (dim == 3) return dd_two_prod(c3_const(), pow(eps, 2.0 / 3.0));  // the power within a unit in the last place
    return dd_mul_d(dd_sqrt(dd_div(dd_from(eps), dd_from(6.0))), 4.0);
}

// The factor of one eps value, local or smeared.
inline dd action_factor(int dim, double eps) { return is_local(eps) ? local_factor(dim) : smeared_factor(dim, eps); }

__host__ __device__ inline dd local_action(dd factor, int64_t bracket) { return dd_mul(factor, dd_from_i64(bracket)); }

__host__ __device__ inline dd smeared_action(int dim, int64_t n, double eps, dd factor, dd sum) {
    const dd e = dim == 2 ? dd_mul_d(dd_from(eps), 2.0) : dd_from(eps);
    return dd_mul(factor, dd_sub(dd_from_i64(n), dd_mul(e, sum)));
}

// Sum of one double-double per lane, in every lane.
__device__ __forceinline__ dd warp_sum_dd(dd v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const dd y{__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
        v = dd_add(v, y);
    }
    return v;
}

// Terms k >= K of the smeared sum that can be dropped.  For k >= deg,
// f_d(k) = q^(k-deg) poly_d(k) with q = 1 - eps and
//   |poly_2| <= (1 + k eps)^2, |poly_3| <= 3.375 (1 + k eps)^2,
//   |poly_4| <= 9 (1 + k eps)^3,
// so |f_d(k)| <= B(k) = C (1 + k eps)^m q^(k-deg), which decreases for
// k >= m / eps.  With R >= the sum of the abundances (n(n-1)/2 bounds it for
// any histogram of n elements) the dropped tail is at most R B(K), and the
// sum enters S multiplied by at most 4 (4 eps^2, c3 eps^(5/3) or
// 4 sqrt(eps/6) eps).  K is the first k >= max(deg, m/eps) with
// 4 R B(K) <= 1e-15: the truncation moves S by less than 1e-15.
__host__ __device__ inline int64_t smear_cutoff(int dim, double eps, double R, int64_t len) {
    const double lq = log1p(-eps);  // ln q < 0
    if (!(lq < 0.0)) return len;
    const double C = dim == 2 ? 1.0 : (dim == 3 ? 3.375 : 9.0);
    const double m = dim == 4 ? 3.0 : 2.0;
    const double deg = dim == 4 ? 3.0 : 2.0;
    const double lhs0 = log(4.0 * fmax(R, 1.0) * C) + 34.6;  // ln(4 R C) - ln(1e-15)
    double k = fmax(deg, ceil(m / eps));
    // Fixed point of k = deg + (lhs0 + m ln(1 + k eps)) / (-ln q), approached
    // from below; the map's slope there is about m / (1 + k eps) < 0.1.  The
    // iterates never decrease, and once one repeats every later one does, so
    // stopping there gives the same k as all 24 steps.
    for (int it = 0; it < 24; ++it) {
        const double kn = fmax(k, deg + (lhs0 + m * log1p(k * eps)) / -lq);
        if (kn == k) break;
        k = kn;
    }
    k = ceil(k) + 8.0;
    return k < double(len) ? int64_t(k) : len;
}


}  // namespace cs
