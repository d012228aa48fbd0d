// Scaled products for the * rules of Sec. 5.1.1 (reduce and reduce_by_index).
//
// The forward sweep of the * rule is re-executed as a map-reduce of
// (number of zeros, lowest zero index, product of the nonzero elements).
// The product of the nonzeros leaves every floating-point range on
// realistic sizes (a product of 65536 values from U[0.5,1.5) is about
// 1e-1287), so it is carried as a mantissa and a 64-bit exponent: 64-bit integer
// mantissas in the reductions (ProdAcc, ProdStateQ; no FP64 instruction per
// element), FP64 ones in [0.5, 1) in finished states (ProdState) and in
// reduce_by_index over FP64 values.
#pragma once

#include <stdint.h>

namespace adpar {

// x != 0 finite:  x = m * 2^e, 0.5 <= |m| < 1 (subnormals included).
__device__ __forceinline__ void split_pow2(double x, double& m, int64_t& e) {
    long long bits = __double_as_longlong(x);
    int ex = (int)((bits >> 52) & 0x7ff);
    int adj = 0;
    if (ex == 0) {  // subnormal: scale into the normal range first
        x *= 18014398509481984.0;  // 2^54
        bits = __double_as_longlong(x);
        ex = (int)((bits >> 52) & 0x7ff);
        adj = -54;
    }
    bits = (bits & ~(0x7ffLL << 52)) | (1022LL << 52);
    m = __longlong_as_double(bits);
    e = (int64_t)(ex - 1022 + adj);
}

// FP32 x != 0 finite:  x = m * 2^e, 0.5 <= |m| < 1
__device__ __forceinline__ void split_pow2_f32m(float x, float& m, int& e) {
    int bits = __float_as_int(x);
    int ex = (bits >> 23) & 0xff;
    int adj = 0;
    if (ex == 0) {  // subnormal
        x *= 16777216.0f;  // 2^24
        bits = __float_as_int(x);
        ex = (bits >> 23) & 0xff;
        adj = -24;
    }
    m = __int_as_float((bits & ~(0xff << 23)) | (126 << 23));
    e = ex - 126 + adj;
}

// Renormalise m (nonzero, normal) into [0.5, 1), moving its exponent into e.
__device__ __forceinline__ void renorm(double& m, int64_t& e) {
    long long bits = __double_as_longlong(m);
    const int ex = (int)((bits >> 52) & 0x7ff);
    bits = (bits & ~(0x7ffLL << 52)) | (1022LL << 52);
    m = __longlong_as_double(bits);
    e += (int64_t)(ex - 1022);
}

struct ProdState {
    double m;       // mantissa of the product of the nonzeros, [0.5, 1)
    int64_t e;      // its binary exponent
    int64_t nz;     // number of zeros
    int64_t first;  // lowest zero index (INT64_MAX when none)

    __device__ static ProdState id() { return {0.5, 1, 0, INT64_MAX}; }  // 0.5 * 2^1 = 1
};

// (zero count, lowest zero index, product of the nonzeros) of a range, as the
// reductions combine it: the product is M * 2^(E - 63) with M in [2^63, 2^64),
// its sign a parity.  A factor's product keeps its top 64 bits with the last one
// set (below), so a factor adds a relative error below 2^-62 of either sign, and
// 2^26 factors stay within 1e-14 (truncation alone drifts one way: 5e-12).  Two
// states combine by rounding to nearest: a tree of exact products stays exact,
// the neutral states of idle threads among them.
struct ProdStateQ {
    unsigned long long M;
    long long E;
    long long nz;
    long long first;
    unsigned sign;  // bit 31: parity of the negative factors

    __device__ static ProdStateQ id() { return {1ull << 63, 0, 0, INT64_MAX, 0u}; }
    __device__ static ProdStateQ comb(const ProdStateQ& x, const ProdStateQ& y);
    __device__ ProdState to_state() const;
};

// M * m for top-aligned mantissas (both in [2^63, 2^64), standing for [1, 2)):
// returns the product's mantissa and its exponent increment (0 or 1).  The
// last bit is set always: the 64 bits kept are the exact product cut off plus
// a half on average, so a long chain does not drift; a product that is exact
// in 63 bits keeps those bits.
__device__ __forceinline__ unsigned long long top_mul(unsigned long long M, unsigned long long m, int& de) {
    const unsigned long long p = __umul64hi(M, m);  // [2^62, 2^64)
    de = (int)(p >> 63);
    return (de ? p : p << 1) | 1ull;
}
// the same for a 32-bit top-aligned mantissa m in [2^31, 2^32): two 32x32-bit products
__device__ __forceinline__ unsigned long long top_mul32(unsigned long long M, unsigned m, int& de) {
    const unsigned long long p = (unsigned long long)(unsigned)(M >> 32) * m +
                                 (((unsigned long long)(unsigned)M * m) >> 32);
    de = (int)(p >> 63);
    return (de ? p : p << 1) | 1ull;
}

// x with its mantissa top-aligned: |x| = m * 2^(e - 63); x != 0 finite
__device__ __forceinline__ void split_top(double x, unsigned long long& m, int& e) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x) << 1 >> 1;
    const int ex = (int)(b >> 52);
    if (ex == 0) {  // subnormal: b * 2^-1074
        const int lz = __clzll((long long)b);
        m = b << lz;
        e = -1011 - lz;
        return;
    }
    m = (b << 11) | (1ull << 63);
    e = ex - 1023;
}

// One thread's running product.  The common factor (normal and nonzero) costs
// a 64-bit high product, a conditional shift and two adds on the integer
// pipes; zeros and subnormals leave by a branch.  E fits 32 bits: a factor
// adds at most 1075, and no thread of a grid meets 2^20 factors of an array
// that fits the memory.
struct ProdAcc {
    unsigned long long M;
    int E;
    unsigned sign, nz;
    long long first;

    __device__ static ProdAcc id() { return {1ull << 63, 0, 0u, 0u, INT64_MAX}; }
    __device__ __forceinline__ void zero(int64_t i) {
        ++nz;
        if (i < first) first = i;
    }
    __device__ __forceinline__ void push(double a, int64_t i) {
        const unsigned hi = (unsigned)__double2hiint(a);
        const unsigned ex = (hi >> 20) & 0x7ffu;
        unsigned long long m = ((unsigned long long)__double_as_longlong(a) << 11) | (1ull << 63);
        int e = (int)ex - 1023;
        if (ex == 0u) {
            if (a == 0.0) {
                zero(i);
                return;
            }
            split_top(a, m, e);
        }
        int de;
        M = top_mul(M, m, de);
        E += e + de;
        sign ^= hi;
    }
    __device__ __forceinline__ void push(float a, int64_t i) {
        const unsigned b = (unsigned)__float_as_int(a);
        const unsigned ex = (b >> 23) & 0xffu;
        unsigned m = (b << 8) | 0x80000000u;
        int e = (int)ex - 127;
        if (ex == 0u) {
            if (a == 0.0f) {
                zero(i);
                return;
            }
            const unsigned f = b & 0x7fffffu;  // subnormal: f * 2^-149
            const int lz = __clz((int)f);
            m = f << lz;
            e = -118 - lz;
        }
        int de;
        M = top_mul32(M, m, de);
        E += e + de;
        sign ^= b;
    }
    // The first factor met the exact 1 of id(), so its product gained the last
    // bit without having lost any: drop it here (a thread's chain is then even).
    __device__ __forceinline__ ProdStateQ state() const {
        return {M & ~1ull, E, (long long)nz, first, sign & 0x80000000u};
    }
};

__device__ __forceinline__ ProdStateQ ProdStateQ::comb(const ProdStateQ& x, const ProdStateQ& y) {
    ProdStateQ r;
    const unsigned long long hi = __umul64hi(x.M, y.M), lo = x.M * y.M;  // hi in [2^62, 2^64 - 2]
    int de = (int)(hi >> 63);
    r.M = de ? hi + (lo >> 63) : ((hi << 1) | (lo >> 63)) + ((lo >> 62) & 1ull);
    if (r.M == 0ull) {  // rounded up to the next power of two
        r.M = 1ull << 63;
        de = 1;
    }
    r.E = x.E + y.E + de;
    r.nz = x.nz + y.nz;
    r.first = x.first < y.first ? x.first : y.first;
    r.sign = x.sign ^ y.sign;
    return r;
}
// the FP64 form: mantissa in [0.5, 1), rounded to nearest
__device__ __forceinline__ ProdState ProdStateQ::to_state() const {
    const bool up = M >= 0xfffffffffffffc00ull;  // rounds to the next power of two
    const unsigned long long r = up ? 1ull << 52 : (M + 0x400ull) >> 11;  // [2^52, 2^53)
    ProdState s;
    s.m = __longlong_as_double((long long)(((unsigned long long)sign << 32) | (1022ull << 52) |
                                           (r & 0xfffffffffffffull)));
    s.e = E + 1 + (up ? 1 : 0);
    s.nz = nz;
    s.first = first;
    return s;
}

// ldexp with the exponent clamped to a range where the result is already
// 0 or infinite, so that a 64-bit exponent never overflows the int argument.
__device__ __forceinline__ double ldexp_clamped(double x, int64_t e) {
    if (e < -2200) e = -2200;
    if (e > 2200) e = 2200;
    return ldexp(x, (int)e);
}

// x * 2^e for a normal x with |x| in [2^-4, 2^4): the exponent field is
// adjusted directly when the result is normal (exact); a result in the
// subnormal range is formed by one multiply by 2^-1000 (one rounding,
// correct); below that it is a signed zero, above it an infinity.
__device__ __forceinline__ double scale_pow2(double x, int64_t e) {
    const long long b = __double_as_longlong(x);
    const int64_t ex = ((b >> 52) & 0x7ff) + e;
    const long long sign = b & (long long)0x8000000000000000ULL;
    if (ex >= 1 && ex <= 2046) return __longlong_as_double((b & ~(0x7ffLL << 52)) | ((long long)ex << 52));
    if (ex > 2046) return __longlong_as_double(sign | (0x7ffLL << 52));
    if (ex < -60) return __longlong_as_double(sign);
    return __longlong_as_double((b & ~(0x7ffLL << 52)) | ((long long)(ex + 1000) << 52)) * 9.332636185032189e-302;
}
// the same for FP32 results (x a float in [2^-4, 2^4))
__device__ __forceinline__ float scale_pow2f(float x, int64_t e) {
    const int b = __float_as_int(x);
    const int64_t ex = ((b >> 23) & 0xff) + e;
    const int sign = b & (int)0x80000000u;
    if (ex >= 1 && ex <= 254) return __int_as_float((b & ~(0xff << 23)) | ((int)ex << 23));
    if (ex > 254) return __int_as_float(sign | (0xff << 23));
    if (ex < -30) return __int_as_float(sign);
    return __int_as_float((b & ~(0xff << 23)) | ((int)(ex + 100) << 23)) * 7.888609052210118e-31f;  // 2^-100
}

// 1 / m for a mantissa with 0.5 <= |m| < 1 in integer arithmetic, so that
// no FP64 instruction runs (GB300 issues FP64 at 1/64 of the FP32 rate):
// the seed r0 is the FP32 reciprocal of |m| truncated to 24 bits (relative
// error below 2^-22); one Newton step r1 = r0 (2 - |m| r0) in 64-bit fixed
// point (r scaled by 2^62, |m| by 2^53, products by __umul64hi) squares the
// error, below 2^-44 relative; r1 never exceeds 1/|m|, so it fits.  The sign
// of m is put back at the end.
__device__ __forceinline__ double recip_mantissa(double m) {
    const unsigned long long bm = (unsigned long long)__double_as_longlong(m);
    const unsigned long long sign = bm & 0x8000000000000000ULL;
    const unsigned long long M = (bm & 0xFFFFFFFFFFFFFULL) | (1ULL << 52);  // |m| * 2^53
    const float mf = __int_as_float(0x3F000000 | (int)((bm >> 29) & 0x7FFFFF));  // |m| truncated, in [0.5, 1)
    const unsigned br = __float_as_uint(__frcp_rn(mf));                          // in (1, 2]
    const int ex = (int)((br >> 23) & 0xff) - 127;                               // 0, or 1 for r0 = 2
    const unsigned long long R0 = (unsigned long long)((br & 0x7FFFFFu) | 0x800000u) << (39 + ex);  // r0 * 2^62
    // |m| r0 * 2^62 = M R0 / 2^53 (M R0 < 2^116)
    const unsigned long long mr = (__umul64hi(M, R0) << 11) | ((M * R0) >> 53);
    const unsigned long long d = (2ULL << 62) - mr;  // (2 - |m| r0) * 2^62
    const unsigned long long R1 = (__umul64hi(R0, d) << 2) | ((R0 * d) >> 62);  // r1 * 2^62, in [2^62, 2^63]
    const int lz = __clzll((long long)R1);  // 0 only for r1 = 2
    const unsigned long long mant = ((R1 << lz) >> 11) & 0xFFFFFFFFFFFFFULL;
    return __longlong_as_double((long long)(sign | ((unsigned long long)(1024 - lz) << 52) | mant));
}

// The map of the * rule over FP64 values: K * 2^ek / x (sign parity in bit 31
// of sk), K a top-aligned mantissa, with no FP64 instruction (GB300 issues
// those at 1/64 of the FP32 rate).  With m the mantissa of x and R the
// hardware reciprocal of its top 24 bits (32-bit fixed point), eps = 1 - m R
// is below 2^-21, and K / m = K R (1 + eps + eps^2) up to eps^3 and the
// 2^-52 resolution of eps: within 2^-50.1 of K / m with the final rounding
// (2e7 mantissa pairs, edges among them, checked on the host).
// Results outside the normal range leave by scale_pow2.  About 100 instructions a
// value in all, on the integer pipes; with the one FP64 multiply and 64-bit Newton step that were
// here, the map over 2^26 values took 414 us, now 226 us with the loads four
// vectors deep (158 us for its bytes); the reduction 275 us, now 102 us (79).
struct QuotF64 {
    unsigned long long K;
    int ek;
    unsigned sk;
    // the numerator k * 2^e, k != 0
    __device__ static QuotF64 make(double k, int64_t e) {
        QuotF64 q;
        int e0;
        split_top(k, q.K, e0);
        e += e0;
        // beyond +-2^20 every quotient is 0 or infinite: 32 bits hold it
        q.ek = (int)(e > (1 << 20) ? (1 << 20) : (e < -(1 << 20) ? -(1 << 20) : e));
        q.sk = (unsigned)__double2hiint(k) & 0x80000000u;
        return q;
    }
    __device__ __forceinline__ double operator()(double x) const {
        const unsigned hi = (unsigned)__double2hiint(x);
        int ex = (int)((hi >> 20) & 0x7ffu) - 1023;
        unsigned long long m = ((unsigned long long)__double_as_longlong(x) << 11) | (1ull << 63);
        if (ex == -1023) split_top(x, m, ex);  // subnormal (x is not zero here)
        float r;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(0x3f800000u | ((unsigned)(m >> 40) & 0x7fffffu))));
        r = fmaxf(fminf(r, 0.99999994f), 0.5f);                               // R in [2^31, 2^32)
        const unsigned R = ((unsigned)__float_as_int(r) << 8) | 0x80000000u;  // r * 2^32, r in [1/2, 1)
        const unsigned long long t = (unsigned long long)(unsigned)(m >> 32) * R +
                                     (((unsigned long long)(unsigned)m * R) >> 32);  // m r * 2^63
        const int e1 = (int)((long long)((1ull << 63) - t) >> 11);                   // eps * 2^52
        const int c = e1 + (int)(((long long)e1 * e1) >> 52);                        // + eps^2
        unsigned long long q = (unsigned long long)(unsigned)(K >> 32) * R +
                               (((unsigned long long)(unsigned)K * R) >> 32);  // K r, in [2^62, 2^64)
        q += (unsigned long long)(((long long)(int)(q >> 33) * c) >> 19);
        const int s = (int)(q >> 63) ^ 1;
        q <<= s;
        const int eb = ek - ex - s + 1023;  // biased exponent of the quotient
        const unsigned long long sg = (unsigned long long)((hi ^ sk) & 0x80000000u) << 32;
        // 53 bits, rounded to nearest (q + 2^10 could wrap); the top one adds 1 to the exponent field
        const unsigned long long mant = (q >> 11) + ((q >> 10) & 1ull);
        if ((unsigned)(eb - 1) < 2045u)  // rounding up may carry into it, up to 2046
            return __longlong_as_double((long long)(sg | (((unsigned long long)(eb - 1) << 52) + mant)));
        return scale_pow2(__longlong_as_double((long long)(sg | ((1022ull << 52) + mant))), eb - 1023);
    }
};

// the same over FP32 values: k * 2^e / x with k an FP32 mantissa, 0.25 <= |k| <= 1:
// one hardware reciprocal and a residual correction
__device__ __forceinline__ float quot_f32(float k, int64_t e, float x) {
    float m, r;
    int ex;
    split_pow2_f32m(x, m, ex);
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(m));
    const float q = k * r;
    return scale_pow2f(fmaf(fmaf(-q, m, k), r, q), e - ex);
}

}  // namespace adpar
