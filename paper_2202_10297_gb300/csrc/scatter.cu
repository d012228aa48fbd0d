// VJP of scatter (Sec. 5.3) and of map with a free array (Sec. 5.4).
//
// scatter:  ys = scatter xs is vs  (is free of duplicates).  The return
//   sweep gathers vsbar[j] += ysbar[is_j], then zeroes ysbar[is_j], which
//   turns ysbar into xsbar in place, and optionally restores
//   ys[is_j] = xs_saved[j].  Work is O(m), not O(n): the same thread reads
//   and then zeroes ysbar[is_j], and no other thread touches that element.
//
// map_acc:  xs[j] = g(as[is_j, :], ws[j, :]).  Every read of the free array
//   as becomes an accumulation into asbar at the same index (the
//   accumulators of Sec. 5.4, atomic adds on the GPU as in Sec. 6); ws is
//   an ordinary mapped input.  When asbar fits in shared memory each block
//   accumulates privately and flushes once with vector atomics (the
//   reduction form that Sec. 6.1 turns accumulators into).
#include <algorithm>

#include "common.cuh"

namespace adpar {
namespace {

constexpr int kBlk = 256;

template <class I>
__device__ __forceinline__ int64_t ldi(const I* p, int64_t j) {
    return (int64_t)__ldcs(p + j);
}

// Random accesses to an array larger than L2 cost a DRAM fetch and a write-back
// per index (32 bytes and more of each for 4 useful ones).  So a large target is
// taken in regions that L2 holds, last region first (what a preceding copy wrote
// last): every thread goes through its indices once per region and touches only
// those in it, so a line is fetched and written back once for all of its
// indices, at the price of reading the indices once per region.
// Worth it when a 64-byte line holds enough indices on average, how many
// depending on the pass (RegionRule below), and for few regions (16: 6.7 ms
// against 5.2 ms in one, 2^26 indices into 1 GB); not when the indices are local
// already (sorted, say): each block looks at 256 pairs 64 apart, the same pairs in
// all blocks, and takes one region when most lie close.
// Random accesses of 4 bytes on a GB300, in G/s, within 64 MB / over 256 MB:
// loads 286 / 77, stores 209 / 33, exchanges 134 / 36.  Forward and VJP through
// autograd, 2^24 indices into 2^26 FP32 (of it 170 us for the two copies of the
// target): 1557 us with a load and a store per index in one region, 741 us so;
// regions of 32 and 90 MB 1190 and 865 us.
constexpr int64_t kRegionBytes = int64_t(64) << 20;
constexpr int64_t kMaxRegions = 8;
constexpr int64_t kLocalBytes = int64_t(1) << 20;
constexpr int64_t kDenseBytes = 64 * 24;  // 64 indices within this many bytes
constexpr int64_t kDenseMin = int64_t(24) << 20;  // bytes of vs (fewer: exchanges within L2 are as fast)
// blocks per SM, all resident: the grid goes through the regions together
constexpr int kScatBlocks = 6;

// When a pass goes by regions: target bytes, indices per 64-byte line, regions.
// Time by regions over time in one, targets of 128 / 256 MB, FP32:
//   VJP                       1 index per line 1.2 / 0.9, 2 per line 0.9 / 0.8
//   forward                   1 per line 1.4 / 1.1, 2 per line 1.0 / 0.8
//   forward, keeping the old  2 per line 1.0 / 1.0, 4 per line 0.8 / 0.9; of 440 MB
//     values                  1.2 (FP64 4 per line 0.9 / 1.0, 8 per line 0.8 / 1.0)
struct RegionRule {
    int64_t min_bytes;
    int per_line;
    int64_t max_regions;
};
constexpr RegionRule kVjpRule{2 * kRegionBytes, 1, kMaxRegions};
constexpr RegionRule kFwdRule{2 * kRegionBytes, 2, kMaxRegions};
constexpr RegionRule save_rule(size_t esz) { return {kRegionBytes * 3 / 2, esz == 4 ? 4 : 8, 5}; }

// elements per region (below 2^32): all of n where one region will do
inline int64_t region_elems(int64_t n, int64_t m, size_t esz, const RegionRule& rule) {
    const int64_t bytes = n * (int64_t)esz;
    const int64_t regions = (bytes + kRegionBytes - 1) / kRegionBytes;
    if (bytes < rule.min_bytes || regions > rule.max_regions || m < 4096 || m * 64 < bytes * rule.per_line)
        return std::min<int64_t>(std::max<int64_t>(n, 1), int64_t(1) << 31);
    return ((n + regions - 1) / regions + 31) / 32 * 32;
}
// A target that just outgrows L2 (129 MB) and few indices per line: exchanges lose
// to a load and a store per index (FP32, 96 to 224 MB, up to 1.13 times; FP64 1.17)
inline bool beyond_l2(int64_t n, size_t esz) {
    const int64_t bytes = n * (int64_t)esz;
    return bytes >= kRegionBytes * 3 / 2 && bytes < kRegionBytes * 7 / 2;
}

// the region size this launch uses (the same in every block); all threads call
// it.  dense, where asked for: neighbouring indices share lines, as sorted ones
// into a quarter of FP32 do (exchanges then take up to 1.15 times as long as a load
// and a store, and 0.9 where only a 16th is written).
template <class I>
__device__ __forceinline__ int64_t pick_region(const I* is, int64_t n, int64_t m, int64_t region, int esz,
                                               bool* dense = nullptr) {
    const bool one = region >= n || region == int64_t(1) << 31;
    if (dense) *dense = false;
    if (one && !(dense && m * esz >= kDenseMin)) return region;
    const int64_t p = (int64_t)threadIdx.x * ((m - 64) / blockDim.x);
    int64_t d = (int64_t)is[p + 64] - (int64_t)is[p];
    if (d < 0) d = -d;
    if (dense && m * esz >= kDenseMin) *dense = 2 * __syncthreads_count(d <= kDenseBytes / esz) >= (int)blockDim.x;
    if (one) return region;
    const int near = __syncthreads_count(d <= kLocalBytes / esz);
    return 2 * near >= (int)blockDim.x ? (n < (int64_t(1) << 31) ? n : int64_t(1) << 31) : region;
}

// Asks L2 for a region's lines in order, each block for its share, ahead of the
// random accesses (which would fetch them one 32-byte sector at a time).
template <class T>
__device__ __forceinline__ void prefetch_region(const T* p, unsigned size) {
    const char* lo = reinterpret_cast<const char*>(p);
    const int64_t bytes = (int64_t)size * (int64_t)sizeof(T) / 16 * 16;
    const int64_t share = (bytes / gridDim.x / 512 + 1) * 512, first = share * blockIdx.x;
    const int64_t stop = first + share < bytes ? first + share : bytes;
    for (int64_t o = first + threadIdx.x * 512; o < stop; o += kBlk * 512) {
        const unsigned sz = (unsigned)(stop - o < 512 ? stop - o : 512);
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(lo + o), "r"(sz) : "memory");
    }
}

// Puts v at p and returns what was there, in one trip to L2.  A load and then a
// store to a random line is far slower (26 against 36 G/s beyond L2, 62 against
// 134 within): the line's copy on the reading die's side of L2 is made and
// thrown away again.
__device__ __forceinline__ float exchange(float* p, float v) { return atomicExch(p, v); }
__device__ __forceinline__ double exchange(double* p, double v) {
    return __longlong_as_double((long long)atomicExch(reinterpret_cast<unsigned long long*>(p),
                                                      (unsigned long long)__double_as_longlong(v)));
}
template <class T>
__device__ __forceinline__ T take_zero(T* p) {
    return exchange(p, T(0));
}

// Four indices per thread and step, a block apart (neighbouring lanes hold
// neighbouring indices).  Loading the next step's ahead loses (800 against 741 us
// below): the more index lines in flight, the fewer of the region's stay in L2.
constexpr int kScatU = 4;

// fn(r, j) for every index j of this thread whose target lies in [base, base + size),
// r its offset there; out(j) for those outside [0, n).  OUT: call out().
template <bool OUT, class I, class Fn, class Out>
__device__ __forceinline__ void for_region(const I* is, int64_t m, int64_t n, int64_t base, unsigned size, Fn fn,
                                           Out out) {
    constexpr int U = kScatU;
    const int64_t stride = (int64_t)gridDim.x * (kBlk * U);
    for (int64_t j = blockIdx.x * (int64_t)(kBlk * U) + threadIdx.x; j < m; j += stride) {
        I q[U];
        unsigned r[U];
#pragma unroll
        for (int u = 0; u < U; ++u) q[u] = j + u * kBlk < m ? __ldcs(is + j + u * kBlk) : I(-1);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t k = (int64_t)q[u], d = k - base;
            r[u] = (unsigned long long)d < size ? (unsigned)d : 0xffffffffu;
            if (OUT && (k < 0 || k >= n) && j + u * kBlk < m) out(j + u * kBlk);
        }
        fn(r, j);
    }
}

template <class T, class I, bool RESTORE, bool ACC>
__global__ void __launch_bounds__(kBlk, kScatBlocks) scatter_vjp_kernel(int64_t n, int64_t m, const I* is, T* ysbar,
                                                                       T* vsbar, T* ys, const T* xs_saved,
                                                                       int64_t region_arg) {
    constexpr int U = kScatU;
    const int64_t region = pick_region(is, n, m, region_arg, (int)sizeof(T));
    const int64_t last = n > 0 ? (n - 1) / region * region : 0;
    for (int64_t base = last; base >= 0; base -= region) {
        const int64_t left = n - base;
        const unsigned size = (unsigned)(left < region ? left : region);
        if (region < n && region <= kRegionBytes) prefetch_region(ysbar + base, size);
        T* yb = ysbar + base;
        auto fn = [&](const unsigned (&r)[U], int64_t j) {
            T g[U];
#pragma unroll
            for (int u = 0; u < U; ++u) g[u] = r[u] != 0xffffffffu ? take_zero(yb + r[u]) : T(0);
            if (RESTORE) {
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (r[u] != 0xffffffffu) ys[base + r[u]] = __ldcs(xs_saved + j + u * kBlk);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                T* o = vsbar + j + u * kBlk;
                if (r[u] != 0xffffffffu) __stcs(o, ACC ? __ldcs(o) + g[u] : g[u]);
            }
        };
        // an index out of range: vsbar 0 (overwrite), in the first region's pass
        if (!ACC && base == last)
            for_region<true>(is, m, n, base, size, fn, [&](int64_t j) { vsbar[j] = T(0); });
        else
            for_region<false>(is, m, n, base, size, fn, [](int64_t) {});
    }
}

// ------------------------------------------------------------- map_acc
template <class T>
struct MapAccArgs {
    int g;
    int64_t nj, na;
    int width;
    const T* as;
    const void* is;
    const T* ws;
    const T* xsbar;
    T* asbar;
    T* wsbar;
    int acc_w;
    int priv;  // asbar (na * width values) is privatised in shared memory
};

template <class T>
__device__ __forceinline__ void acc_add(T* p, T v) {
    atomicAdd(p, v);
}

template <class T, class I>
__global__ void __launch_bounds__(kBlk) map_acc_kernel(MapAccArgs<T> A) {
    extern __shared__ unsigned char smem_raw[];
    T* sh = reinterpret_cast<T*>(smem_raw);
    const int64_t tot = A.na * A.width;
    if (A.priv) {
        for (int64_t q = threadIdx.x; q < tot; q += blockDim.x) sh[q] = T(0);
        __syncthreads();
    }
    T* dst = A.priv ? sh : A.asbar;
    const I* is = static_cast<const I*>(A.is);
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < A.nj; j += stride) {
        const int64_t i = ldi(is, j);
        const bool in = i >= 0 && i < A.na;
        const T xb = __ldcs(A.xsbar + j);
        if (A.g == ADPAR_G_GATHER) {
            if (in) acc_add(dst + i, xb);
        } else if (A.g == ADPAR_G_SCALE) {
            const T w = __ldcs(A.ws + j);
            T wb = T(0);
            if (in) {
                acc_add(dst + i, w * xb);
                wb = __ldg(A.as + i) * xb;
            }
            if (A.wsbar) {
                if (A.acc_w) A.wsbar[j] += wb;
                else A.wsbar[j] = wb;
            }
        } else {  // SQDIST_ROW, rows of `width`
            for (int k = 0; k < A.width; ++k) {
                const T w = A.ws[j * A.width + k];
                T wb = T(0);
                if (in) {
                    const T diff = w - __ldg(A.as + i * A.width + k);
                    acc_add(dst + i * A.width + k, T(-2) * diff * xb);
                    wb = T(2) * diff * xb;
                }
                if (A.wsbar) {
                    if (A.acc_w) A.wsbar[j * A.width + k] += wb;
                    else A.wsbar[j * A.width + k] = wb;
                }
            }
        }
    }
    if (A.priv) {
        __syncthreads();
        for (int64_t q = threadIdx.x; q < tot; q += blockDim.x)
            if (sh[q] != T(0)) atomicAdd(A.asbar + q, sh[q]);
    }
}

// A load and a store per index, U indices per thread and step.
template <int U, class T, class I>
__device__ __forceinline__ void save_plain(int64_t n, int64_t m, const I* is, const T* vs, T* ys, T* xs_saved) {
    const int64_t stride = (int64_t)gridDim.x * (kBlk * U);
    for (int64_t j = blockIdx.x * (int64_t)(kBlk * U) + threadIdx.x; j < m; j += stride) {
        I k[U];
        T o[U];
#pragma unroll
        for (int u = 0; u < U; ++u) k[u] = j + u * kBlk < m ? __ldcs(is + j + u * kBlk) : I(-1);
#pragma unroll
        for (int u = 0; u < U; ++u) o[u] = k[u] >= 0 && k[u] < n ? ys[k[u]] : T(0);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (j + u * kBlk >= m) break;
            xs_saved[j + u * kBlk] = o[u];
            if (k[u] >= 0 && k[u] < n) ys[k[u]] = __ldcs(vs + j + u * kBlk);
        }
    }
}

// primal of scatter (Sec. 5.3's forward sweep): xs_saved[j] = ys[is_j]
// (optional), then ys[is_j] = vs[j], in place; by regions as above
template <class T, class I, bool SAVE>
__global__ void __launch_bounds__(kBlk, kScatBlocks) scatter_fwd_kernel(int64_t n, int64_t m, const I* is, const T* vs,
                                                                       T* ys, T* xs_saved, int64_t region_arg) {
    constexpr int U = kScatU;
    bool dense = false;
    const int64_t region = pick_region(is, n, m, region_arg, (int)sizeof(T), SAVE ? &dense : nullptr);
    if (SAVE && dense) {
        save_plain<kScatU>(n, m, is, vs, ys, xs_saved);
        return;
    }
    const int64_t last = n > 0 ? (n - 1) / region * region : 0;
    for (int64_t base = last; base >= 0; base -= region) {
        const int64_t left = n - base;
        const unsigned size = (unsigned)(left < region ? left : region);
        if (region < n && region <= kRegionBytes) prefetch_region(ys + base, size);
        T* y = ys + base;
        auto fn = [&](const unsigned (&r)[U], int64_t j) {
            T g[U];
#pragma unroll
            for (int u = 0; u < U; ++u) g[u] = r[u] != 0xffffffffu ? __ldcs(vs + j + u * kBlk) : T(0);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (r[u] == 0xffffffffu) continue;
                if (SAVE) xs_saved[j + u * kBlk] = exchange(y + r[u], g[u]);
                else y[r[u]] = g[u];
            }
        };
        if (SAVE && base == last)
            for_region<true>(is, m, n, base, size, fn, [&](int64_t j) { xs_saved[j] = T(0); });
        else
            for_region<false>(is, m, n, base, size, fn, [](int64_t) {});
    }
}

// the plain loop alone (beyond_l2)
template <class T, class I>
__global__ void __launch_bounds__(kBlk) scatter_save_kernel(int64_t n, int64_t m, const I* is, const T* vs, T* ys,
                                                           T* xs_saved) {
    save_plain<1>(n, m, is, vs, ys, xs_saved);
}

// primal of map: xs[j] = g(as[is_j, :], ws[j, :]) (0 for an index out of range)
template <class T, class I>
__global__ void __launch_bounds__(kBlk) map_fwd_kernel(int g, int64_t nj, int64_t na, int width, const T* as,
                                                      const I* is, const T* ws, T* xs) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < nj; j += stride) {
        const int64_t i = ldi(is, j);
        T x = T(0);
        if (i >= 0 && i < na) {
            if (g == ADPAR_G_GATHER) {
                x = __ldg(as + i);
            } else if (g == ADPAR_G_SCALE) {
                x = __ldg(as + i) * ws[j];
            } else {
                for (int k = 0; k < width; ++k) {
                    const T d = ws[j * width + k] - __ldg(as + i * width + k);
                    x += d * d;
                }
            }
        }
        xs[j] = x;
    }
}

template <class T>
__global__ void zero_kernel(T* p, int64_t n) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += stride) p[i] = T(0);
}

int sm_count() {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms > 0 ? sms : 132;
}

constexpr size_t kPrivBytes = 48 * 1024;

}  // namespace
}  // namespace adpar

extern "C" int adpar_vjp_scatter(int dtype, int64_t n, int64_t m, const void* is, int itype,
                                 void* ysbar_inout, void* vsbar, void* ys_restore, const void* xs_saved,
                                 uint32_t flags, void* stream) {
    using namespace adpar;
    if (n < 0 || m < 0) return ADPAR_ERR_INVALID;
    if (dtype != ADPAR_F32 && dtype != ADPAR_F64) return ADPAR_ERR_INVALID;
    if (itype != ADPAR_I32 && itype != ADPAR_I64) return ADPAR_ERR_INVALID;
    if (flags & ~(uint32_t)(ADPAR_ACCUMULATE | ADPAR_SCATTER_RESTORE)) return ADPAR_ERR_UNSUPPORTED;
    const bool restore = (flags & ADPAR_SCATTER_RESTORE) != 0;
    if (m > 0 && (!is || !vsbar || !ysbar_inout)) return ADPAR_ERR_INVALID;
    if (restore && m > 0 && (!ys_restore || !xs_saved)) return ADPAR_ERR_INVALID;
    const void* ptrs[] = {is, ysbar_inout, vsbar, ys_restore, xs_saved};
    for (const void* p : ptrs)
        if (p && !aligned16(p)) return ADPAR_ERR_ALIGN;
    if (m == 0) return ADPAR_OK;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((m / kScatU + kBlk) / kBlk, (int64_t)sm_count() * kScatBlocks));
    const int64_t region = region_elems(n, m, dtype == ADPAR_F64 ? 8 : 4, kVjpRule);
    const int acc = (flags & ADPAR_ACCUMULATE) ? 1 : 0;
    void* ys = restore ? ys_restore : nullptr;
#define ADPAR_SCATTER_RA(T, I, R, A)                                                                             \
    scatter_vjp_kernel<T, I, R, A><<<grid, kBlk, 0, s>>>(n, m, static_cast<const I*>(is), static_cast<T*>(ysbar_inout), \
                                                         static_cast<T*>(vsbar), static_cast<T*>(ys),            \
                                                         static_cast<const T*>(xs_saved), region)
#define ADPAR_SCATTER(T, I)                                                                                 \
    (ys ? (acc ? ADPAR_SCATTER_RA(T, I, true, true) : ADPAR_SCATTER_RA(T, I, true, false))                  \
        : (acc ? ADPAR_SCATTER_RA(T, I, false, true) : ADPAR_SCATTER_RA(T, I, false, false)))
    if (dtype == ADPAR_F32) {
        if (itype == ADPAR_I32) ADPAR_SCATTER(float, int32_t); else ADPAR_SCATTER(float, int64_t);
    } else {
        if (itype == ADPAR_I32) ADPAR_SCATTER(double, int32_t); else ADPAR_SCATTER(double, int64_t);
    }
#undef ADPAR_SCATTER
#undef ADPAR_SCATTER_RA
    return cudaGetLastError() == cudaSuccess ? ADPAR_OK : ADPAR_ERR_CUDA;
}

extern "C" int adpar_vjp_map_acc(int gfun, int dtype, int64_t nj, int64_t na, int width, const void* as,
                                 const void* is, int itype, const void* ws, const void* xsbar, void* asbar,
                                 void* wsbar, uint32_t flags, void* work, size_t work_bytes, void* stream) {
    using namespace adpar;
    (void)work;
    (void)work_bytes;
    if (nj < 0 || na < 0 || width < 1) return ADPAR_ERR_INVALID;
    if (gfun != ADPAR_G_GATHER && gfun != ADPAR_G_SCALE && gfun != ADPAR_G_SQDIST_ROW) return ADPAR_ERR_INVALID;
    if (gfun != ADPAR_G_SQDIST_ROW && width != 1) return ADPAR_ERR_INVALID;
    if (dtype != ADPAR_F32 && dtype != ADPAR_F64) return ADPAR_ERR_INVALID;
    if (itype != ADPAR_I32 && itype != ADPAR_I64) return ADPAR_ERR_INVALID;
    if (flags & ~(uint32_t)ADPAR_ACCUMULATE) return ADPAR_ERR_UNSUPPORTED;
    if (nj > 0 && (!is || !xsbar || !asbar)) return ADPAR_ERR_INVALID;
    if (gfun != ADPAR_G_GATHER && nj > 0 && (!ws || !as)) return ADPAR_ERR_INVALID;
    const void* ptrs[] = {as, is, ws, xsbar, asbar, wsbar};
    for (const void* p : ptrs)
        if (p && !aligned16(p)) return ADPAR_ERR_ALIGN;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const bool acc = (flags & ADPAR_ACCUMULATE) != 0;
    const size_t esz = dtype == ADPAR_F64 ? 8 : 4;
    const int64_t tot = na * width;
    const int sms = sm_count();
    // asbar is an accumulator: without ADPAR_ACCUMULATE it starts from zero
    if (!acc && tot > 0) {
        const int gz = (int)std::max<int64_t>(1, std::min<int64_t>((tot + 255) / 256, (int64_t)sms * 8));
        if (dtype == ADPAR_F32) zero_kernel<float><<<gz, 256, 0, s>>>(static_cast<float*>(asbar), tot);
        else zero_kernel<double><<<gz, 256, 0, s>>>(static_cast<double*>(asbar), tot);
    }
    if (nj == 0) return cudaGetLastError() == cudaSuccess ? ADPAR_OK : ADPAR_ERR_CUDA;
    const bool priv = (size_t)tot * esz <= kPrivBytes;
    const size_t shm = priv ? (size_t)tot * esz : 0;
    const int64_t blocks = priv ? std::min<int64_t>((nj + kBlk * 16 - 1) / (kBlk * 16), (int64_t)sms * 2)
                                : std::min<int64_t>((nj + kBlk - 1) / kBlk, (int64_t)sms * 8);
    const int grid = (int)std::max<int64_t>(1, blocks);
#define ADPAR_MAPACC(T, I)                                                                   \
    do {                                                                                     \
        MapAccArgs<T> A{gfun, nj, na, width, static_cast<const T*>(as), is,                  \
                        static_cast<const T*>(ws), static_cast<const T*>(xsbar),             \
                        static_cast<T*>(asbar), static_cast<T*>(wsbar), acc ? 1 : 0, priv ? 1 : 0}; \
        map_acc_kernel<T, I><<<grid, kBlk, shm, s>>>(A);                                     \
    } while (0)
    if (dtype == ADPAR_F32) {
        if (itype == ADPAR_I32) ADPAR_MAPACC(float, int32_t); else ADPAR_MAPACC(float, int64_t);
    } else {
        if (itype == ADPAR_I32) ADPAR_MAPACC(double, int32_t); else ADPAR_MAPACC(double, int64_t);
    }
#undef ADPAR_MAPACC
    return cudaGetLastError() == cudaSuccess ? ADPAR_OK : ADPAR_ERR_CUDA;
}

extern "C" int adpar_scatter(int dtype, int64_t n, int64_t m, const void* is, int itype, const void* vs,
                             void* ys_inout, void* xs_saved_out, void* stream) {
    using namespace adpar;
    if (n < 0 || m < 0) return ADPAR_ERR_INVALID;
    if (dtype != ADPAR_F32 && dtype != ADPAR_F64) return ADPAR_ERR_INVALID;
    if (itype != ADPAR_I32 && itype != ADPAR_I64) return ADPAR_ERR_INVALID;
    if (m > 0 && (!is || !vs || !ys_inout)) return ADPAR_ERR_INVALID;
    const void* ptrs[] = {is, vs, ys_inout, xs_saved_out};
    for (const void* p : ptrs)
        if (p && !aligned16(p)) return ADPAR_ERR_ALIGN;
    if (m == 0) return ADPAR_OK;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((m / kScatU + kBlk) / kBlk, (int64_t)sm_count() * kScatBlocks));
    const size_t esz = dtype == ADPAR_F64 ? 8 : 4;
    const int64_t region = region_elems(n, m, esz, xs_saved_out ? save_rule(esz) : kFwdRule);
    const bool plain = xs_saved_out && region >= n && beyond_l2(n, esz);
    const int grid1 = (int)std::max<int64_t>(1, std::min<int64_t>((m + kBlk - 1) / kBlk, (int64_t)sm_count() * 8));
#define ADPAR_SCAT_FWD_S(T, I, S)                                                                                 \
    scatter_fwd_kernel<T, I, S><<<grid, kBlk, 0, s>>>(n, m, static_cast<const I*>(is), static_cast<const T*>(vs), \
                                                      static_cast<T*>(ys_inout), static_cast<T*>(xs_saved_out), region)
#define ADPAR_SCAT_SAVE(T, I)                                                                                     \
    scatter_save_kernel<T, I><<<grid1, kBlk, 0, s>>>(n, m, static_cast<const I*>(is), static_cast<const T*>(vs),  \
                                                     static_cast<T*>(ys_inout), static_cast<T*>(xs_saved_out))
#define ADPAR_SCAT_FWD(T, I)                                                                             \
    (plain ? ADPAR_SCAT_SAVE(T, I)                                                                       \
           : (xs_saved_out ? ADPAR_SCAT_FWD_S(T, I, true) : ADPAR_SCAT_FWD_S(T, I, false)))
    if (dtype == ADPAR_F32) {
        if (itype == ADPAR_I32) ADPAR_SCAT_FWD(float, int32_t); else ADPAR_SCAT_FWD(float, int64_t);
    } else {
        if (itype == ADPAR_I32) ADPAR_SCAT_FWD(double, int32_t); else ADPAR_SCAT_FWD(double, int64_t);
    }
#undef ADPAR_SCAT_FWD
#undef ADPAR_SCAT_FWD_S
#undef ADPAR_SCAT_SAVE
    return cudaGetLastError() == cudaSuccess ? ADPAR_OK : ADPAR_ERR_CUDA;
}

extern "C" int adpar_map_acc(int gfun, int dtype, int64_t nj, int64_t na, int width, const void* as,
                             const void* is, int itype, const void* ws, void* xs_out, void* stream) {
    using namespace adpar;
    if (nj < 0 || na < 0 || width < 1) return ADPAR_ERR_INVALID;
    if (gfun != ADPAR_G_GATHER && gfun != ADPAR_G_SCALE && gfun != ADPAR_G_SQDIST_ROW) return ADPAR_ERR_INVALID;
    if (gfun != ADPAR_G_SQDIST_ROW && width != 1) return ADPAR_ERR_INVALID;
    if (dtype != ADPAR_F32 && dtype != ADPAR_F64) return ADPAR_ERR_INVALID;
    if (itype != ADPAR_I32 && itype != ADPAR_I64) return ADPAR_ERR_INVALID;
    if (nj > 0 && (!is || !xs_out || !as)) return ADPAR_ERR_INVALID;
    if (gfun != ADPAR_G_GATHER && nj > 0 && !ws) return ADPAR_ERR_INVALID;
    const void* ptrs[] = {as, is, ws, xs_out};
    for (const void* p : ptrs)
        if (p && !aligned16(p)) return ADPAR_ERR_ALIGN;
    if (nj == 0) return ADPAR_OK;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((nj + kBlk - 1) / kBlk, (int64_t)sm_count() * 8));
#define ADPAR_MAP_FWD(T, I)                                                                                    \
    map_fwd_kernel<T, I><<<grid, kBlk, 0, s>>>(gfun, nj, na, width, static_cast<const T*>(as),                  \
                                               static_cast<const I*>(is), static_cast<const T*>(ws),            \
                                               static_cast<T*>(xs_out))
    if (dtype == ADPAR_F32) {
        if (itype == ADPAR_I32) ADPAR_MAP_FWD(float, int32_t); else ADPAR_MAP_FWD(float, int64_t);
    } else {
        if (itype == ADPAR_I32) ADPAR_MAP_FWD(double, int32_t); else ADPAR_MAP_FWD(double, int64_t);
    }
#undef ADPAR_MAP_FWD
    return cudaGetLastError() == cudaSuccess ? ADPAR_OK : ADPAR_ERR_CUDA;
}
