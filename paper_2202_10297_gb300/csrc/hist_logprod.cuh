// The recompute of reduce_by_index * over FP32 values (Sec. 5.1.1's product
// per bin) as exact integer sums of logarithms.
//
// A bin's product of nonzeros is carried as the fixed-point number
//   S = sum over the bin of log2|v|, in units of 2^-54,
// and the parity of its negative factors.  An addition needs no return value
// and no retry, so a bin in global memory takes two fire-and-forget 64-bit
// adds where a product takes a compare-and-swap loop, and the result does not
// depend on the order.  log2 of a 24-bit mantissa is formed in integer
// arithmetic to 2^-55 (one table entry for the top 11 bits, a quartic for the
// rest); each term is off by at most 2^-54.4 with mean below 2^-60 over all
// 2^23 mantissas, so a bin of 2^27 factors stays within 2^-40 (the 63-bit
// products that were here lost 2^-62 per factor one way, 2^-35).
//
// The two words of a bin: x = sum of the terms' low 32 bits (no wrap below
// 2^32 elements); y = sum of their high 32 bits (signed, below 2^62 in all)
// plus 2^63 for every negative factor, modulo 2^64: bits 63 and 62 of y differ
// when the number of those is odd.
#pragma once

#include <stdint.h>

#include "common.cuh"
#include "prod.cuh"

namespace adpar {

constexpr int kLogTab = 2048;
constexpr unsigned long long kLog2eQ61 = 3326628274461080623ull;  // log2(e) * 2^61
constexpr unsigned long long kLn2Q64 = 12786308645202655660ull;   // ln(2) * 2^64

// Entry i of the table: x_i = 1 + (i + 1/2) / 2048,
//   x = log2(x_i) * 2^58,   y = 2^49 / (x_i ln 2).
// log2 by the series of atanh: with z = (x - 1) / (x + 1) (x halved above
// sqrt 2, so |z| <= 0.172), ln x = 2 z (1 + z^2/3 + z^4/5 + ...).
__host__ __device__ inline unsigned long long logtab_mulhi(unsigned long long a, unsigned long long b) {
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (unsigned long long)(((unsigned __int128)a * b) >> 64);
#endif
}
__host__ __device__ inline void logtab_entry(int i, unsigned long long& t0, unsigned long long& t1) {
    const unsigned long long X = 4097ull + 2ull * (unsigned)i;  // x_i * 4096
    t1 = kLog2eQ61 / X;
    const bool half = X > 5792ull;  // above sqrt 2
    const unsigned long long num = half ? 8192ull - X : X - 4096ull, den = half ? 8192ull + X : X + 4096ull;
    const unsigned long long q = (num << 50) / den, rem = (num << 50) - q * den;
    const unsigned long long z = (q << 14) | ((rem << 14) / den);  // |z| * 2^64
    const unsigned long long z2 = logtab_mulhi(z, z);
    unsigned long long acc = (1ull << 63) / 27ull;
#pragma unroll
    for (int k = 12; k >= 0; --k) acc = (1ull << 63) / (2ull * (unsigned)k + 1ull) + logtab_mulhi(z2, acc);
    // z S in 2^-63, times log2(e) in 2^-62: the product's top word is z S log2(e) * 2^61 = log2(x) * 2^60
    const unsigned long long r = (logtab_mulhi(logtab_mulhi(z, acc), kLog2eQ61 << 1) + 2ull) >> 2;
    t0 = half ? (1ull << 58) - r : r;
}

// log2|v| in units of 2^-54 for the bits b (sign ignored) of a normal or
// subnormal FP32 value v != 0.  With y = (m / x_i - 1) / ln 2, |y| < 2^-11.4,
//   log2 m = log2 x_i + y - y^2 ln2/2 + y^3 ln2^2/3 - y^4 ln2^3/4:
// y to 2^-60, the square to 2^-55, the last two terms in FP32.
__host__ __device__ __forceinline__ long long log2_q54(unsigned b, const ulonglong2* tab) {
    int e = (int)((b >> 23) & 0xffu) - 127;
    unsigned f = b & 0x7fffffu;
    if (e == -127) {  // subnormal: f * 2^-149
#ifdef __CUDA_ARCH__
        const int lz = __clz((int)f) - 8;
#else
        const int lz = __builtin_clz(f) - 8;
#endif
        f = (f << lz) & 0x7fffffu;
        e = -126 - lz;
    }
    const ulonglong2 t = tab[f >> 12];
    const int lo = (int)(f & 4095u) - 2048;
    const long long y72 = (long long)t.y * lo;
    const int yi = (int)(y72 >> 30), yr = (int)((unsigned)y72 & 0x3fffffffu);  // y * 2^42, and 30 more bits
    const long long y84 = (long long)yi * yi + (((long long)yi * yr) >> 29);   // y^2 * 2^84
    const unsigned sq = (unsigned)((y84 + (1ll << 29)) >> 30);
    const long long q58 = (long long)(((unsigned long long)sq * 1488522236u + (1ull << 27)) >> 28);  // * ln2/2 * 2^32
    const float yf = (float)yi * 2.2737367544323206e-13f;                                            // 2^-42
    // (y^3 ln2^2/3 - y^4 ln2^3/4) * 2^58, rounded by the addition of 1.5 * 2^23 (it is below 2^22)
    const float t58 = (yf * yf) * yf * (4.61603843e16f - 2.39969552e16f * yf);
    const float tr = t58 + 12582912.0f;
#ifdef __CUDA_ARCH__
    const int t58i = __float_as_int(tr) - 0x4b400000;
#else
    const int t58i = (int)(tr - 12582912.0f);
#endif
    const long long m58 = (long long)t.x + (y72 >> 14) - q58 + t58i;
    return ((long long)e << 54) + ((m58 + 8) >> 4);
}

// A bin's product of nonzeros from its two words: M top-aligned in [2^63, 2^64),
// |product| = M * 2^(E - 63), sign = 0 or 1.  2^f of the fraction by the
// series of exp in 64-bit fixed point (19 terms, within 2^-58).
__host__ __device__ inline unsigned long long exp2_frac(unsigned long long f64) {
    const unsigned long long x = logtab_mulhi(f64, kLn2Q64);  // f ln 2, below 0.694, in 2^-64
    unsigned long long acc = 0;
    unsigned long long c[19];
    c[0] = 1ull << 62;
#pragma unroll
    for (int k = 1; k < 19; ++k) c[k] = c[k - 1] / (unsigned)k;
#pragma unroll
    for (int k = 18; k >= 0; --k) acc = c[k] + logtab_mulhi(x, acc);  // in 2^-62, below 2
    acc <<= 1;
    return (acc >> 63) ? acc : 1ull << 63;
}
__host__ __device__ inline void logprod_decode(ulonglong2 w, unsigned long long& M, long long& E, unsigned& sign) {
    sign = (unsigned)((w.y >> 63) ^ (w.y >> 62)) & 1u;
    // log2 in units of 2^-22 (with the low words' carries), and the low word below
    const long long h = ((long long)(w.y << 1) >> 1) + (long long)(w.x >> 32);
    E = h >> 22;
    M = exp2_frac((((unsigned long long)h & 0x3fffffull) << 42) | ((w.x & 0xffffffffull) << 10));
}

// ---------------------------------------------------------------- kernels
// Bin tiers of the recompute.  Bins [0, kLogHot) have 32 copies per block, one
// per lane, so the hot bins of rank-ordered skewed data (Zipf) meet no
// contention inside a warp; the next kLogSlots bins one copy per block; the
// rest are words in global memory (L2).  The shared copies hold 32-bit limbs,
// as shared memory adds 32 bits natively and 64 only by a retry loop:
//   w0  the low words' sum modulo 2^32;
//   w1  bits 0-30: the high words' sum (with w0's carries) modulo 2^31, from 2^30;
//       bit 31: the parity of (negative factors + wraps counted in w2);
//   w2  the wraps of that sum, up less down (rarely any);
//   wz  the zero count.
constexpr int kLogHot = 64;
constexpr int kLogSlots = 8192;
constexpr int kLogThreads = 1024;
constexpr int kLogMaxSlots = 32 * kLogHot + kLogSlots;
constexpr size_t kLogSmem = kLogTab * 16 + (size_t)kLogMaxSlots * 16;

struct LogProdArgs {
    int64_t n, m;  // n < 2^32, m < 2^31
    const float* vals;
    const void* inds;
    ulonglong2* acc;       // [m]
    unsigned* pz;          // [m] zero counts
    long long* pf;         // [m] lowest zero index, or NULL when nobody asks
    const ulonglong2* tab; // [kLogTab]
};

__device__ __forceinline__ void red_add_u64(unsigned long long* p, unsigned long long v) {
    asm volatile("red.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// four consecutive indices from element 4 v on (16-byte aligned array)
template <class I>
__device__ __forceinline__ void ld_index4(const I* p, int64_t v, int64_t (&b)[4]) {
    if constexpr (sizeof(I) == 4) {
        const int4 x = __ldcs(reinterpret_cast<const int4*>(p) + v);
        b[0] = x.x; b[1] = x.y; b[2] = x.z; b[3] = x.w;
    } else {
        const longlong2 x = __ldcs(reinterpret_cast<const longlong2*>(p) + 2 * v);
        const longlong2 y = __ldcs(reinterpret_cast<const longlong2*>(p) + 2 * v + 1);
        b[0] = x.x; b[1] = x.y; b[2] = y.x; b[3] = y.y;
    }
}

// One block of 1024 threads per SM; four consecutive elements per thread and
// step, the next step's loaded while this one is added.  Bound by the shared
// and L2 atomics: 174 us for 2^25 elements into 2^16 Zipf bins, where the
// compare-and-swap products took 1396 us (reading the input alone: 39 us).
template <class I>
__global__ void __launch_bounds__(kLogThreads, 1) hist_logprod_kernel(LogProdArgs A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ulonglong2* tab = reinterpret_cast<ulonglong2*>(smem_raw);
    const int hot = (int)(A.m < kLogHot ? A.m : kLogHot);
    const int H = (int)(A.m < kLogHot + kLogSlots ? A.m : kLogHot + kLogSlots);  // bins with shared copies
    const int slots = 31 * hot + H;
    unsigned* w0 = reinterpret_cast<unsigned*>(tab + kLogTab);
    unsigned* w1 = w0 + slots;
    unsigned* w2 = w1 + slots;
    unsigned* wz = w2 + slots;
    for (int q = threadIdx.x; q < kLogTab; q += kLogThreads) tab[q] = A.tab[q];
    for (int q = threadIdx.x; q < slots; q += kLogThreads) {
        w0[q] = 0u;
        w1[q] = 0x40000000u;
        w2[q] = 0u;
        wz[q] = 0u;
    }
    __syncthreads();
    const I* inds = static_cast<const I*>(A.inds);
    const int lane = threadIdx.x & 31;
    const int64_t nvec = (A.n + 3) / 4, full = A.n / 4;
    const int64_t stride = (int64_t)gridDim.x * kLogThreads;

    int64_t b[4];
    float x[4];
    auto load = [&](int64_t v) {
        if (v < full) {
            ld_index4(inds, v, b);
            const float4 f = __ldcs(reinterpret_cast<const float4*>(A.vals) + v);
            x[0] = f.x; x[1] = f.y; x[2] = f.z; x[3] = f.w;
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int64_t i = 4 * v + j;
                b[j] = i < A.n ? (int64_t)inds[i] : -1;
                x[j] = i < A.n ? A.vals[i] : 0.f;
            }
        }
    };
    int64_t v = blockIdx.x * (int64_t)kLogThreads + threadIdx.x;
    load(v);
    // v - lane is the same in all lanes of a warp: the warp leaves together
    for (; v - lane < nvec; v += stride) {
        int cb[4];
        float cx[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            cb[j] = (b[j] >= 0 && b[j] < A.m) ? (int)b[j] : -1;
            cx[j] = x[j];
        }
        load(v + stride);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            int bin = cb[j];
            const unsigned bits = (unsigned)__float_as_int(cx[j]);
            if (bin >= 0 && (bits << 1) == 0u) {  // a zero: counted apart
                if (bin < H) atomicAdd(wz + (bin < hot ? 32 * bin + lane : bin + 31 * hot), 1u);
                else atomicAdd(A.pz + bin, 1u);
                const long long i = 4 * v + j;
                if (A.pf && i < *reinterpret_cast<volatile long long*>(A.pf + bin)) atomicMin(A.pf + bin, i);
                bin = -1;
            }
            const long long L = log2_q54((bits << 1) == 0u ? 0x3f800000u : bits, tab);
            const unsigned lo = (unsigned)L, neg = bits & 0x80000000u;
            const int hi = (int)(L >> 32);
            if (bin >= 0 && bin < H) {
                const int q = bin < hot ? 32 * bin + lane : bin + 31 * hot;
                const unsigned o0 = atomicAdd(w0 + q, lo);
                const int add = hi + (o0 + lo < lo ? 1 : 0);
                const unsigned o1 = atomicAdd(w1 + q, (unsigned)add ^ neg);
                const unsigned wrap = (((o1 & 0x7fffffffu) + ((unsigned)add & 0x7fffffffu)) >> 31) -
                                      ((unsigned)add >> 31);
                if (wrap) atomicAdd(w2 + q, wrap);
                bin = -1;
            }
            if (__any_sync(0xffffffffu, bin >= 0)) {
                // a bin's two words lie side by side: two lanes add them in one
                // request to its sector
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const int src = 16 * k + (lane >> 1);
                    const int sb = __shfl_sync(0xffffffffu, bin, src);
                    const unsigned sl = __shfl_sync(0xffffffffu, lo, src);
                    const int sh = __shfl_sync(0xffffffffu, hi, src);
                    const unsigned sn = __shfl_sync(0xffffffffu, neg, src);
                    if (sb >= 0)
                        red_add_u64(reinterpret_cast<unsigned long long*>(A.acc) + 2 * (int64_t)sb + (lane & 1),
                                    (lane & 1) ? (unsigned long long)(long long)sh + ((unsigned long long)sn << 32)
                                               : (unsigned long long)sl);
                }
            }
        }
    }
    __syncthreads();
    // the block's shared bins join the global words
    for (int q = threadIdx.x; q < H; q += kLogThreads) {
        unsigned long long lo = 0, hi = 0;
        unsigned z = 0;
        auto take = [&](int s) {
            lo += w0[s];
            hi += (unsigned long long)((long long)(int)w2[s] * 0x80000000ll + (long long)(w1[s] & 0x7fffffffu) -
                                       0x40000000ll) +
                  ((unsigned long long)((w1[s] >> 31) ^ (w2[s] & 1u)) << 63);
            z += wz[s];
        };
        if (q < hot) {
            for (int c = 0; c < 32; ++c) take(32 * q + ((c + lane) & 31));
        } else {
            take(q + 31 * hot);
        }
        if (lo) red_add_u64(&A.acc[q].x, lo);
        if (hi) red_add_u64(&A.acc[q].y, hi);
        if (z) atomicAdd(A.pz + q, z);
    }
}

__global__ void hist_logprod_init_kernel(WsHeader* hdr, LogProdArgs A, ulonglong2* tab) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t0 < 64) reinterpret_cast<uint32_t*>(hdr)[t0] = 0u;
    for (int64_t i = t0; i < kLogTab; i += stride) logtab_entry((int)i, tab[i].x, tab[i].y);
    for (int64_t b = t0; b < A.m; b += stride) {
        A.acc[b] = make_ulonglong2(0ull, 0ull);
        A.pz[b] = 0u;
        if (A.pf) A.pf[b] = INT64_MAX;
    }
}

// Per-bin factor of the adjoint: P_nz * hsbar_b = qm * 2^qe, qm an FP32
// mantissa in [0.5, 1] (0: the bin gives nothing).  flag (bit 0 of the packed
// exponent): the bin holds exactly one zero, which alone gets the factor.
struct alignas(8) BinQ {
    float qm;
    int qe2;  // qe * 2 + flag
};

// a top-aligned mantissa rounded to FP32, in [0.5, 1]
__device__ __forceinline__ float top_to_f32(unsigned long long M) {
    const unsigned r = (unsigned)(M >> 40) + (unsigned)((M >> 39) & 1ull);
    return __int_as_float(0x3f000000 + (int)(r - 0x800000u));
}

// per bin: the recomputed product and what the call asked for
__global__ void hist_logprod_bins_kernel(LogProdArgs A, const float* hsbar, BinQ* binq, float* hs_out,
                                         adpar_prod_aux* aux, int keep_pow2) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; b < A.m; b += stride) {
        unsigned long long M;
        long long E;
        unsigned sign;
        logprod_decode(A.acc[b], M, E, sign);
        const unsigned nz = A.pz[b];
        if (hs_out) {
            const float p = scale_pow2f(top_to_f32(M), E + 1);
            hs_out[b] = nz ? 0.f : (sign ? -p : p);
        }
        if (binq) {
            BinQ q{0.f, 0};
            const float yb = hsbar[b];
            if (yb != 0.f && nz <= 1) {
                float ym;
                int ye, de;
                split_pow2_f32m(yb, ym, ye);  // in [0.5, 1)
                const unsigned long long P = top_mul32(M, ((unsigned)__float_as_int(ym) << 8) | 0x80000000u, de);
                q.qm = top_to_f32(P);
                if ((sign != 0u) != (yb < 0.f)) q.qm = -q.qm;
                long long e = E + de + ye;
                e = e > (1 << 29) ? (1 << 29) : (e < -(1 << 29) ? -(1 << 29) : e);
                q.qe2 = (int)e * 2 + (int)nz;
            }
            binq[b] = q;
        }
        if (aux || keep_pow2) {
            const ProdState s = ProdStateQ{M, E, 0, 0, sign << 31}.to_state();
            if (aux) {
                adpar_prod_aux x;
                x.nzero = nz;
                x.first_zero = nz ? A.pf[b] : -1;
                x.exp2 = s.e;
                x.mant = s.m;
                x.log_abs_nz = log(fabs(s.m)) + (double)s.e * 0.69314718055994530942;
                x.sign = sign ? -1 : 1;
                x.reserved = 0;
                aux[b] = x;
            }
            if (keep_pow2)  // the log-domain map reads (mantissa, exponent) instead of the sums
                A.acc[b] = make_ulonglong2((unsigned long long)__double_as_longlong(s.m), (unsigned long long)s.e);
        }
    }
}

// per element: the three cases of Sec. 5.1.1 from the bin's factor (a bin
// without zeros: factor / v; with one: the factor at its zero)
__device__ __forceinline__ float binq_adjoint(const BinQ& q, float v) {
    const int64_t e = q.qe2 >> 1;
    if (q.qm == 0.f) return 0.f;
    if (q.qe2 & 1) return v == 0.f ? scale_pow2f(q.qm, e) : 0.f;
    return quot_f32(q.qm, e, v);
}

// Bound by the gather of the factors and HBM: 81 us for 2^25 elements into 2^16
// bins (59 us for its bytes); 155 us with one element and a 16-byte factor per
// thread and step.
template <class I>
__global__ void __launch_bounds__(256) hist_logprod_vjp_kernel(LogProdArgs A, const BinQ* binq, float* vb,
                                                               int accumulate) {
    const I* inds = static_cast<const I*>(A.inds);
    const int64_t nvec = A.n / 4, stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    for (int64_t v = nvec - 1 - t0; v >= 0; v -= stride) {  // from the end: read last, still in L2
        int64_t b[4];
        ld_index4(inds, v, b);
        const float4 f = __ldcs(reinterpret_cast<const float4*>(A.vals) + v);
        const float x[4] = {f.x, f.y, f.z, f.w};
        BinQ q[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            q[j] = BinQ{0.f, 0};
            if (b[j] >= 0 && b[j] < A.m) {
                const int2 w = __ldg(reinterpret_cast<const int2*>(binq) + b[j]);
                q[j] = BinQ{__int_as_float(w.x), w.y};
            }
        }
        float o[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) o[j] = binq_adjoint(q[j], x[j]);
        if (accumulate) {
            const float4 p = reinterpret_cast<const float4*>(vb)[v];
            const float pp[4] = {p.x, p.y, p.z, p.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) o[j] += pp[j];
        }
        __stcs(reinterpret_cast<float4*>(vb) + v, make_float4(o[0], o[1], o[2], o[3]));
    }
    const int64_t i = nvec * 4 + t0;
    if (i < A.n) {
        const int64_t b = (int64_t)inds[i];
        const float c = (b >= 0 && b < A.m) ? binq_adjoint(binq[b], A.vals[i]) : 0.f;
        vb[i] = accumulate ? vb[i] + c : c;
    }
}

}  // namespace adpar
