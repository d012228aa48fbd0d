// The recompute of reduce_by_index * over FP32 values (Sec. 5.1.1's product
// per bin) as exact integer sums of logarithms.
//
// A bin's product of nonzeros is carried as the fixed-point number
//   S = sum over the bin of log2|v|, in units of 2^-63,
// and the parity of its negative factors.  An addition needs no return value
// and no retry, so a bin in global memory takes two fire-and-forget 64-bit
// adds where a product takes a compare-and-swap loop, and the result does not
// depend on the order.  log2 of a 24-bit mantissa is formed in integer
// arithmetic (one table entry for the top 11 bits, a quintic for the rest).
// Over all 2^23 mantissas a term is off by at most 1.06 units, by none for powers
// of two, and by 2^-71 on average: n factors, equal ones at worst, leave a
// relative error below n 2^-63.4, where the 63-bit products that were here left
// n 2^-62.  (With terms in units of 2^-54, n equal factors left n 2^-54.9.)
//
// The two words of a bin: x = sum of the terms' low 36 bits; y = sum of the rest
// (signed) plus 2^63 for every negative factor, modulo 2^64.  Over kLogChunk
// elements x does not wrap and the sum in y stays below 2^62 in magnitude, so
// bits 63 and 62 of y differ when the number of negative factors is odd.
// Longer arrays are taken in chunks, after each of which the integer part moves
// to a third word.
#pragma once

#include <math_constants.h>
#include <stdint.h>

#include "common.cuh"
#include "prod.cuh"

namespace adpar {

constexpr int kLogTab = 2048;
constexpr int kLogLow = 36;   // fraction bits in x
constexpr int kLogHigh = 27;  // fraction bits in y
constexpr int64_t kLogChunk = int64_t(1) << 27;
constexpr unsigned long long kLn2Q64 = 12786308645202655660ull;  // ln(2) * 2^64

// Entry i of the table: x_i = 1 + (i + 1/2) / 2048,
//   t0 = log2(x_i) * 2^63,   h * 2^31 + l = 2^61 / (x_i ln 2).
struct alignas(16) LogEntry {
    unsigned long long t0;
    int h, l;
};
struct LogTable {
    LogEntry e[kLogTab];
};

typedef unsigned __int128 u128;
constexpr u128 logtab_mul96(u128 a, u128 b) {  // a b 2^-96 for a, b < 2^97
    const u128 m = ((u128)1 << 48) - 1;
    return (a >> 48) * (b >> 48) + (((a >> 48) * (b & m) + (a & m) * (b >> 48)) >> 48);
}
// log2 by the series of atanh: with z = (x - 1) / (x + 1) (x halved above
// sqrt 2, so |z| <= 0.172), ln x = 2 z (1 + z^2/3 + z^4/5 + ...), to 2^-90
constexpr LogEntry logtab_entry(int i) {
    constexpr u128 log2e = ((u128)0x171547652ull << 64) | 0xb82fe1777d0ffda1ull;  // * 2^96
    const unsigned X = 4097u + 2u * (unsigned)i;                                  // x_i * 4096
    const bool half = X > 5792u;                                                  // above sqrt 2
    const u128 num = half ? 8192u - X : X - 4096u, den = half ? 8192u + X : X + 4096u;
    const u128 z = (num << 96) / den, z2 = logtab_mul96(z, z);
    u128 acc = ((u128)1 << 96) / 39u;
    for (int k = 18; k >= 0; --k) acc = ((u128)1 << 96) / (unsigned)(2 * k + 1) + logtab_mul96(z2, acc);
    u128 r = 2 * logtab_mul96(logtab_mul96(z, acc), log2e);
    if (half) r = ((u128)1 << 96) - r;
    const unsigned long long t1 = (unsigned long long)(((log2e >> 23) + X / 2) / X);
    return LogEntry{(unsigned long long)((r + ((u128)1 << 32)) >> 33), (int)(t1 >> 31), (int)(t1 & 0x7fffffffull)};
}
constexpr LogTable make_logtab() {
    LogTable t{};
    for (int i = 0; i < kLogTab; ++i) t.e[i] = logtab_entry(i);
    return t;
}

// log2|v| = e + frac * 2^-63 for the bits b (sign ignored) of a normal or
// subnormal FP32 value v != 0 (0 gives some number).  With y = (m / x_i - 1) / ln 2, |y| < 2^-11.4,
//   log2 m = log2 x_i + y - q (1 - g),  q = y^2 ln2/2,
//   g = 2/3 r - r^2/2 + 2/5 r^3,  r = y ln 2,
// y to 2^-74, q to 2^-72, g to 2^-43 with its last two terms in FP32.
__host__ __device__ __forceinline__ int log2_q63(unsigned b, const LogEntry* tab, unsigned long long& frac) {
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
    const LogEntry t = tab[f >> 12];
    const int lo = (int)(f & 4095u) - 2048;
    const long long y74 = (((long long)t.h * lo) << 21) + (((long long)t.l * lo) >> 10);
    const int yi = (int)(y74 >> 32), yr = (int)((unsigned)y74 >> 1);                                  // y * 2^42, 31 more bits
    const unsigned long long z = (unsigned long long)((long long)yi * yi + (((long long)yi * yr) >> 30));  // y^2 * 2^84
    // q * 2^85 = z ln2: the rounding of ln2 * 2^32 to a 32-bit word is made up for in g
    const unsigned long long q = (z >> 32) * 2977044472u + (((z & 0xffffffffull) * 2977044472u) >> 32);
    // g * 2^43: the FP32 terms are rounded by the addition of 1.5 * 2^23 (they are below 2^19)
    const float yf = (float)yi;
    const float g2 = (yf * yf) * fmaf(1.3773576781e-26f, yf, -1.0924236765e-13f);
    const float gr = g2 + 12582912.0f;
#ifdef __CUDA_ARCH__
    const int g2i = __float_as_int(gr) - (0x4b400000 - (533));
#else
    const int g2i = (int)(gr - 12582912.0f) + (533);
#endif
    const int g = (int)(((long long)yi * 1984696315) >> 31) + g2i;
    const long long c = y74 - (long long)(q >> 11) + (((long long)(int)(q >> 30) * g) >> 24);
    frac = t.t0 + (unsigned long long)((c + 1024) >> 11);
    return e;
}

// A bin's product of nonzeros from its words (E: the integer part that chunks
// left): M top-aligned in [2^63, 2^64), |product| = M * 2^(E - 63), sign = 0 or
// 1.  2^f of the fraction by the series of exp in 64-bit fixed point (19 terms,
// within 2^-60).
__host__ __device__ inline unsigned long long logprod_mulhi(unsigned long long a, unsigned long long b) {
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (unsigned long long)(((u128)a * b) >> 64);
#endif
}
__host__ __device__ inline unsigned long long exp2_frac(unsigned long long f64) {
    const unsigned long long x = logprod_mulhi(f64, kLn2Q64);  // f ln 2, below 0.694, in 2^-64
    unsigned long long acc = 0;
    unsigned long long c[19];
    c[0] = 1ull << 63;
#pragma unroll
    for (int k = 1; k < 19; ++k) c[k] = c[k - 1] / (unsigned)k;
#pragma unroll
    for (int k = 18; k >= 0; --k) acc = c[k] + logprod_mulhi(x, acc);  // in 2^-63, below 2: every step rounds down
    return acc;
}
// log2 of the magnitude in units of 2^-kLogHigh (with the low words' carries)
__host__ __device__ inline long long logprod_high(ulonglong2 w, unsigned& sign) {
    sign = (unsigned)((w.y >> 63) ^ (w.y >> 62)) & 1u;
    return ((long long)(w.y << 1) >> 1) + (long long)(w.x >> kLogLow);
}
__host__ __device__ inline void logprod_decode(ulonglong2 w, long long whole, unsigned long long& M, long long& E,
                                               unsigned& sign) {
    const long long h = logprod_high(w, sign);
    E = whole + (h >> kLogHigh);
    M = exp2_frac(((unsigned long long)h << (kLogLow + 1)) | ((w.x & ((1ull << kLogLow) - 1)) << 1));
}

// ---------------------------------------------------------------- kernels
// Bin tiers of the recompute.  Bins [0, kLogHot) have 32 copies per block, one
// per lane, so the hot bins of rank-ordered skewed data (Zipf) meet no
// contention inside a warp; the next kLogSlots bins one copy per block; the
// rest are words in global memory (L2).  The shared copies hold 32-bit limbs,
// as shared memory adds 32 bits natively and 64 only by a retry loop:
//   w0  the sum of the terms' low 32 fraction bits, modulo 2^32;
//   w1  bits 0-30: that of the high 31 and w0's carries, modulo 2^31;
//       bit 31: the parity of the negative factors and of w2;
//   w2  the sum of the whole parts and w1's carries (below 2^30 in magnitude: a
//       block takes 2^22 elements of a chunk at most); factors near 1 add to it
//       only when w1 wraps, as a whole part of -1 and a carry cancel;
//   wz  the zero count.
constexpr int kLogHot = 64;
constexpr int kLogSlots = 8192;
constexpr int kLogThreads = 1024;
// Lanes of a warp up to which each adds both words of its bin in L2 itself: with
// more, neighbouring lanes share the work, a request per bin.  2^25 elements, the
// call, by neighbours always / so / each lane always: into 2^16 Zipf bins (3 such
// lanes in a warp) 282 / 269 / 265 us; into 30000 uniform ones (23) 293 / 298 / 471.
constexpr int kLogFew = 6;
constexpr int kLogMaxSlots = 32 * kLogHot + kLogSlots;
constexpr size_t kLogSmem = kLogTab * 16 + (size_t)kLogMaxSlots * 16;

struct LogProdArgs {
    int64_t n, m;
    const float* vals;
    const void* inds;
    ulonglong2* acc;       // [m]
    long long* whole;      // [m] what earlier chunks carried out, or NULL (a single chunk)
    unsigned* pz;          // [m] zero counts
    long long* pf;         // [m] lowest zero index, or NULL when nobody asks
};

__device__ const LogTable g_logtab = make_logtab();

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

// One block of 1024 threads per SM over the elements [first, last) (a chunk;
// first is a multiple of 4); four consecutive elements per thread and step, the
// next step's loaded while this one is added.  B: int, or int64_t for 2^31 bins
// and more.  Bound by instruction issue: 2^25 elements into 2^16 Zipf bins take
// 177 us (72% of the issue slots), into 256 bins 146 us (74%); reading the input
// alone takes 39, the compare-and-swap products that were here took 1396 us, and
// terms in units of 2^-54 (less closely held) 174 us.
template <class I, class B>
__global__ void __launch_bounds__(kLogThreads, 1) hist_logprod_kernel(LogProdArgs A, int64_t first, int64_t last) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LogEntry* tab = reinterpret_cast<LogEntry*>(smem_raw);
    const int hot = (int)(A.m < kLogHot ? A.m : kLogHot);
    const int H = (int)(A.m < kLogHot + kLogSlots ? A.m : kLogHot + kLogSlots);  // bins with shared copies
    const int slots = 31 * hot + H;
    unsigned* w0 = reinterpret_cast<unsigned*>(tab + kLogTab);
    unsigned* w1 = w0 + slots;
    unsigned* w2 = w1 + slots;
    unsigned* wz = w2 + slots;
    for (int q = threadIdx.x; q < kLogTab; q += kLogThreads) tab[q] = g_logtab.e[q];
    for (int q = threadIdx.x; q < 4 * slots; q += kLogThreads) w0[q] = 0u;
    __syncthreads();
    const I* inds = static_cast<const I*>(A.inds);
    const int lane = threadIdx.x & 31;
    const int64_t nvec = (last + 3) / 4, full = last / 4;
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
                b[j] = i < last ? (int64_t)inds[i] : -1;
                x[j] = i < last ? A.vals[i] : 0.f;
            }
        }
    };
    int64_t v = first / 4 + blockIdx.x * (int64_t)kLogThreads + threadIdx.x;
    load(v);
    // v - lane is the same in all lanes of a warp: the warp leaves together
    for (; v - lane < nvec; v += stride) {
        B cb[4];
        float cx[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            cb[j] = (b[j] >= 0 && b[j] < A.m) ? (B)b[j] : B(-1);
            cx[j] = x[j];
        }
        load(v + stride);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            B bin = cb[j];
            const unsigned bits = (unsigned)__float_as_int(cx[j]);
            if (bin >= 0 && (bits << 1) == 0u) {  // a zero: counted apart
                if (bin < H) atomicAdd(wz + (bin < hot ? 32 * bin + lane : bin + 31 * hot), 1u);
                else atomicAdd(A.pz + bin, 1u);
                const long long i = 4 * v + j;
                if (A.pf && i < *reinterpret_cast<volatile long long*>(A.pf + bin)) atomicMin(A.pf + bin, i);
                bin = -1;
            }
            unsigned long long frac;
            const int e = log2_q63(bits, tab, frac);
            const unsigned lo = (unsigned)frac, hi = (unsigned)(frac >> 32), neg = bits & 0x80000000u;
            if (bin >= 0 && bin < H) {
                const int q = (int)(bin < hot ? 32 * bin + lane : bin + 31 * hot);
                const unsigned o0 = atomicAdd(w0 + q, lo);
                const unsigned mid = hi + (o0 + lo < lo ? 1u : 0u);  // up to 2^31
                const unsigned o1 = atomicAdd(w1 + q, (mid + ((unsigned)e << 31)) ^ neg);
                const unsigned add = (unsigned)e + (((o1 & 0x7fffffffu) + mid) >> 31);
                if (add) atomicAdd(w2 + q, add);
                bin = -1;
            }
            const unsigned far = __ballot_sync(0xffffffffu, bin >= 0);  // lanes whose bins are words in L2
            if (far) {
                const unsigned long long x = ((unsigned long long)(hi & 15u) << 32) | lo;
                const unsigned long long y = (unsigned long long)(((long long)e << kLogHigh) + (long long)(hi >> 4)) +
                                             ((unsigned long long)neg << 32);
                unsigned long long* acc = reinterpret_cast<unsigned long long*>(A.acc);
                if (__popc(far) <= kLogFew) {
                    if (bin >= 0) {
                        red_add_u64(acc + 2 * (int64_t)bin, x);
                        red_add_u64(acc + 2 * (int64_t)bin + 1, y);
                    }
                } else {
                    // a bin's two words lie side by side: two neighbouring lanes add them
                    // in one request to its sector, the even lane's bin's first
                    const bool odd = lane & 1;
                    const unsigned long long other = __shfl_xor_sync(0xffffffffu, odd ? x : y, 1);
                    const B ob = __shfl_xor_sync(0xffffffffu, bin, 1);
                    const B b0 = odd ? ob : bin, b1 = odd ? bin : ob;
                    if (b0 >= 0) red_add_u64(acc + 2 * (int64_t)b0 + odd, odd ? other : x);
                    if (b1 >= 0) red_add_u64(acc + 2 * (int64_t)b1 + odd, odd ? y : other);
                }
            }
        }
    }
    __syncthreads();
    // the block's shared bins join the global words
    for (int q = threadIdx.x; q < H; q += kLogThreads) {
        unsigned long long lo = 0, mid = 0;  // in units of 2^-63 and 2^-31
        long long e = 0;
        unsigned z = 0, neg = 0;
        auto take = [&](int s) {
            lo += w0[s];
            mid += w1[s] & 0x7fffffffu;
            e += (int)w2[s];
            neg ^= (w1[s] >> 31) ^ (w2[s] & 1u);
            z += wz[s];
        };
        if (q < hot) {
            for (int c = 0; c < 32; ++c) take(32 * q + ((c + lane) & 31));
        } else {
            take(q + 31 * hot);
        }
        mid += lo >> 32;
        const unsigned long long x = ((mid & 15u) << 32) | (lo & 0xffffffffull);
        const unsigned long long y = (unsigned long long)((e << kLogHigh) + (long long)(mid >> 4)) +
                                     ((unsigned long long)neg << 63);
        if (x) red_add_u64(&A.acc[q].x, x);
        if (y) red_add_u64(&A.acc[q].y, y);
        if (z) atomicAdd(A.pz + q, z);
    }
}
static_assert(kLogLow + kLogHigh == 63 && kLogLow == 32 + 4, "the flush's shifts");

__global__ void hist_logprod_init_kernel(WsHeader* hdr, LogProdArgs A) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t0 < 64) reinterpret_cast<uint32_t*>(hdr)[t0] = 0u;
    for (int64_t b = t0; b < A.m; b += stride) {
        A.acc[b] = make_ulonglong2(0ull, 0ull);
        A.pz[b] = 0u;
        if (A.whole) A.whole[b] = 0;
        if (A.pf) A.pf[b] = INT64_MAX;
    }
}

// between two chunks: a bin's integer part leaves its two words
__global__ void hist_logprod_carry_kernel(LogProdArgs A) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; b < A.m; b += stride) {
        const ulonglong2 w = A.acc[b];
        unsigned sign;
        const long long h = logprod_high(w, sign);
        A.whole[b] += h >> kLogHigh;
        A.acc[b] = make_ulonglong2(w.x & ((1ull << kLogLow) - 1),
                                   ((unsigned long long)h & ((1ull << kLogHigh) - 1)) | ((unsigned long long)sign << 63));
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

// M * 2^(E - 63) rounded once to FP32, to nearest even (subnormals and infinity too)
__device__ __forceinline__ float prod_to_f32(unsigned long long M, long long E) {
    if (E > 127) return CUDART_INF_F;
    const bool normal = E >= -126;
    const long long drop = normal ? 40 : 40 - 126 - E;  // bits of M below the last place
    if (drop > 64) return 0.f;
    unsigned r = drop == 64 ? 0u : (unsigned)(M >> drop);
    const unsigned long long rest = M << (64 - drop);
    r += rest > (1ull << 63) || (rest == (1ull << 63) && (r & 1u)) ? 1u : 0u;
    return __uint_as_float((normal ? (unsigned)(E + 126) << 23 : 0u) + r);
}

// per bin: the recomputed product and what the call asked for
__global__ void hist_logprod_bins_kernel(LogProdArgs A, const float* hsbar, BinQ* binq, float* hs_out,
                                         adpar_prod_aux* aux, int keep_pow2) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; b < A.m; b += stride) {
        unsigned long long M;
        long long E;
        unsigned sign;
        logprod_decode(A.acc[b], A.whole ? A.whole[b] : 0, M, E, sign);
        const unsigned nz = A.pz[b];
        if (hs_out) {
            const float p = prod_to_f32(M, E);
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
