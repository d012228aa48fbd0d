// VJP of reduce (Sec. 5.1 and its special cases in Sec. 5.1.1).
//
//   ADD      abar_i = ybar (a broadcast; y itself only if asked for).
//   MIN/MAX  the forward sweep is re-executed as argmin/argmax with the
//            lowest index on ties; abar_{i_y} = ybar and 0 elsewhere.  In
//            overwrite mode the zero fill of abar rides along with the
//            reduction pass, so the whole VJP is one read of a and one
//            write of abar.
//   MUL      the forward sweep is re-executed as a map-reduce of (zero
//            count, lowest zero index, scaled product of the nonzeros);
//            then one map applies the three cases of Sec. 5.1.1.
//
// Pass 1 is a grid-stride map-reduce whose last block to finish (atomic
// ticket) combines the per-block partials, so the reduction needs no second
// launch; the * rule adds one map launch.
#include <algorithm>
#include <type_traits>
#include <math_constants.h>

#include "common.cuh"
#include "prod.cuh"
#include "scan_ops.cuh"

namespace adpar {
namespace {

constexpr int kRedBlock = 256;
constexpr int kRedMaxBlocks = 1024;

template <class T>
struct ArgState {
    T v;
    int64_t i;
};

// max / min with the lowest index on ties
template <class T, bool MAX>
__device__ __forceinline__ ArgState<T> arg_comb(const ArgState<T>& x, const ArgState<T>& y) {
    const bool take_y = MAX ? (y.v > x.v || (y.v == x.v && y.i < x.i))
                            : (y.v < x.v || (y.v == x.v && y.i < x.i));
    return take_y ? y : x;
}

struct ReduceArgs {
    int op;
    int64_t n;
    const void* a;
    const void* ybar;
    void* abar;
    void* y_out;
    int64_t* argidx_out;
    adpar_prod_aux* aux_out;
    int8_t* abar_sign;
    int accumulate;
    int logdomain;
    int primal_only;  // forward operator only: no adjoint is written
    WsHeader* hdr;
    void* partials;  // [gridDim.x] states
    void* final_state;
};

__global__ void header_init_kernel(WsHeader* hdr) {
    reinterpret_cast<uint32_t*>(hdr)[threadIdx.x] = 0u;
}

template <class S, class Comb>
__device__ __forceinline__ S block_reduce(S v, Comb comb, S* s_warp) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        S o = shfl_down_s(v, off);
        v = comb(v, o);
    }
    if (lane == 0) s_warp[warp] = v;
    __syncthreads();
    if (warp == 0) {
        v = lane < (int)(blockDim.x >> 5) ? s_warp[lane] : s_warp[0];
        // lanes past the warp count repeat warp 0: harmless for min/max/argmin;
        // for sums only lanes < nwarps are combined below
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            S o = shfl_down_s(v, off);
            if (lane + off < (int)(blockDim.x >> 5)) v = comb(v, o);
        }
    }
    return v;  // valid in thread 0
}

// Returns true in the block that finished last (all partials are visible).
__device__ __forceinline__ bool last_block(WsHeader* hdr) {
    __shared__ bool s_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const uint32_t t = atomicAdd(&hdr->done[0], 1u);
        s_last = (t == gridDim.x - 1);
    }
    __syncthreads();
    if (s_last) __threadfence();
    return s_last;
}

// ------------------------------------------------------------------ ADD
template <class T>
__global__ void __launch_bounds__(kRedBlock) reduce_add_kernel(ReduceArgs A) {
    __shared__ T s_warp[kRedBlock / 32];
    const T* a = static_cast<const T*>(A.a);
    T* abar = static_cast<T*>(A.abar);
    const T yb = A.primal_only ? T(0) : *static_cast<const T*>(A.ybar);
    constexpr int V = Vec16<T>::N;
    const int64_t nvec = A.n / V;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const bool want_y = A.y_out != nullptr;
    T acc = T(0);
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < nvec; v += stride) {
        if (want_y) {
            Vec16<T> x = ld_vec_stream(a + v * V);
#pragma unroll
            for (int j = 0; j < V; ++j) acc += x.v[j];
        }
        if (A.primal_only) continue;
        Vec16<T> o;
        if (A.accumulate) {
            o = ld_vec(abar + v * V);
#pragma unroll
            for (int j = 0; j < V; ++j) o.v[j] += yb;
        } else {
#pragma unroll
            for (int j = 0; j < V; ++j) o.v[j] = yb;
        }
        st_vec(abar + v * V, o);
    }
    if (blockIdx.x == 0 && threadIdx.x < A.n - nvec * V) {
        const int64_t i = nvec * V + threadIdx.x;
        if (want_y) acc += a[i];
        if (!A.primal_only) abar[i] = A.accumulate ? abar[i] + yb : yb;
    }
    if (!want_y) return;
    auto add = [](T x, T y) { return x + y; };
    T bsum = block_reduce(acc, add, s_warp);
    if (threadIdx.x == 0) static_cast<T*>(A.partials)[blockIdx.x] = bsum;
    if (!last_block(A.hdr)) return;
    T tot = T(0);
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) tot += ld_cg(static_cast<T*>(A.partials) + b);
    __syncthreads();
    tot = block_reduce(tot, add, s_warp);
    if (threadIdx.x == 0) {
        *static_cast<T*>(A.y_out) = tot;
        A.hdr->done[0] = 0u;
    }
}

// -------------------------------------------------------------- MIN/MAX
template <class T, bool MAX>
__global__ void __launch_bounds__(kRedBlock) reduce_arg_kernel(ReduceArgs A) {
    using S = ArgState<T>;
    __shared__ S s_warp[kRedBlock / 32];
    const T* a = static_cast<const T*>(A.a);
    T* abar = static_cast<T*>(A.abar);
    constexpr int V = Vec16<T>::N;
    const int64_t nvec = A.n / V;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const bool fill = !A.accumulate && !A.primal_only;
    S st{MAX ? -pos_inf<T>() : pos_inf<T>(), INT64_MAX};
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < nvec; v += stride) {
        Vec16<T> x = ld_vec_stream(a + v * V);
#pragma unroll
        for (int j = 0; j < V; ++j) st = arg_comb<T, MAX>(st, S{x.v[j], v * V + j});
        if (fill) {
            Vec16<T> z;
#pragma unroll
            for (int j = 0; j < V; ++j) z.v[j] = T(0);
            st_vec(abar + v * V, z);
        }
    }
    if (blockIdx.x == 0 && threadIdx.x < A.n - nvec * V) {
        const int64_t i = nvec * V + threadIdx.x;
        st = arg_comb<T, MAX>(st, S{a[i], i});
        if (fill) abar[i] = T(0);
    }
    auto comb = [](const S& x, const S& y) { return arg_comb<T, MAX>(x, y); };
    S bs = block_reduce(st, comb, s_warp);
    if (threadIdx.x == 0) static_cast<S*>(A.partials)[blockIdx.x] = bs;
    if (!last_block(A.hdr)) return;
    S tot{MAX ? -pos_inf<T>() : pos_inf<T>(), INT64_MAX};
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x)
        tot = arg_comb<T, MAX>(tot, ld_cg(static_cast<S*>(A.partials) + b));
    __syncthreads();
    tot = block_reduce(tot, comb, s_warp);
    if (threadIdx.x == 0) {
        const bool any = A.n > 0;
        if (A.y_out) *static_cast<T*>(A.y_out) = tot.v;
        if (A.argidx_out) *A.argidx_out = any ? tot.i : -1;
        if (any && !A.primal_only) {
            const T yb = *static_cast<const T*>(A.ybar);
            abar[tot.i] = A.accumulate ? abar[tot.i] + yb : yb;
        }
        A.hdr->done[0] = 0u;
    }
}

// ------------------------------------------------------------------ MUL
// y and the product record of a finished product
template <class T>
__device__ __forceinline__ void prod_results(const ReduceArgs& A, const ProdState& tot) {
    if (A.y_out) *static_cast<T*>(A.y_out) = tot.nz > 0 ? T(0) : (T)ldexp_clamped(tot.m, tot.e);
    if (A.aux_out) {
        adpar_prod_aux x;
        x.nzero = tot.nz;
        x.first_zero = tot.nz > 0 ? tot.first : -1;
        x.exp2 = tot.e;
        x.mant = tot.m;
        x.log_abs_nz = log(fabs(tot.m)) + (double)tot.e * 0.69314718055994530942;
        x.sign = tot.m > 0 ? 1 : -1;
        x.reserved = 0;
        *A.aux_out = x;
    }
}

// The recompute multiplies mantissas in fixed point on the integer pipes
// (no FP64 instruction per element for either dtype).
template <class T>
__global__ void __launch_bounds__(kRedBlock, 4) reduce_prod_kernel(ReduceArgs A) {
    using S = ProdStateQ;
    __shared__ S s_warp[kRedBlock / 32];
    const T* a = static_cast<const T*>(A.a);
    constexpr int V = Vec16<T>::N;
    const int64_t nvec = A.n / V;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    ProdAcc st = ProdAcc::id();
    constexpr int U = 4;  // vectors in flight per thread
    int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    for (; v + (U - 1) * stride < nvec; v += U * stride) {
        Vec16<T> x[U];
#pragma unroll
        for (int u = 0; u < U; ++u) x[u] = ld_vec(a + (v + u * stride) * V);
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int j = 0; j < V; ++j) st.push(x[u].v[j], (v + u * stride) * V + j);
    }
    for (; v < nvec; v += stride) {
        Vec16<T> x = ld_vec(a + v * V);
#pragma unroll
        for (int j = 0; j < V; ++j) st.push(x.v[j], v * V + j);
    }
    if (blockIdx.x == 0 && threadIdx.x < A.n - nvec * V) {
        const int64_t i = nvec * V + threadIdx.x;
        st.push(a[i], i);
    }
    auto comb = [](const S& x, const S& y) { return S::comb(x, y); };
    S bs = block_reduce(st.state(), comb, s_warp);
    if (threadIdx.x == 0) static_cast<S*>(A.partials)[blockIdx.x] = bs;
    if (!last_block(A.hdr)) return;
    S totq = S::id();
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x)
        totq = S::comb(totq, ld_cg(static_cast<S*>(A.partials) + b));
    __syncthreads();
    totq = block_reduce(totq, comb, s_warp);
    if (threadIdx.x == 0) {
        const ProdState tot = totq.to_state();
        *static_cast<ProdState*>(A.final_state) = tot;
        prod_results<T>(A, tot);
        A.hdr->done[0] = 0u;
    }
}

// The three cases of Sec. 5.1.1 with z = number of zeros, p = product of
// the nonzeros (scaled):  z = 0: abar_i = p / a_i * ybar;  z = 1: only the
// zero at i0 gets p * ybar;  z >= 2: nothing.  In log mode abar_i holds
// ln|contribution| (-inf for none) and abar_sign its sign.
// The map over elements t0, t0 + stride, ... (t0 = 0 writes the single-
// element cases); st is the recomputed forward state.
template <class T>
__device__ __forceinline__ void prod_adjoint_body(const ReduceArgs& A, const ProdState& st, int64_t t0,
                                                  int64_t stride) {
    const double yb = (double)*static_cast<const T*>(A.ybar);
    T* abar = static_cast<T*>(A.abar);
    const T* a = static_cast<const T*>(A.a);
    // ybar as (mantissa, exponent) so every factor has a bounded mantissa
    double ym = 0.0;
    int64_t ye = 0;
    if (yb != 0.0) split_pow2(yb, ym, ye);
    if (A.logdomain) {
        const double lg_p = log(fabs(st.m)) + (double)st.e * 0.69314718055994530942;
        const double lg_y = yb != 0.0 ? log(fabs(yb)) : -CUDART_INF;
        const int sgn_py = (st.m > 0 ? 1 : -1) * (yb > 0 ? 1 : (yb < 0 ? -1 : 0));
        for (int64_t i = t0; i < A.n; i += stride) {
            double lg = -CUDART_INF;
            int sg = 0;
            if (yb != 0.0) {
                if (st.nz == 0) {
                    const double ai = (double)a[i];
                    lg = lg_p - log(fabs(ai)) + lg_y;
                    sg = sgn_py * (ai > 0 ? 1 : -1);
                } else if (st.nz == 1 && i == st.first) {
                    lg = lg_p + lg_y;
                    sg = sgn_py;
                }
            }
            abar[i] = (T)lg;
            if (A.abar_sign) A.abar_sign[i] = (int8_t)sg;
        }
        return;
    }
    if (A.accumulate && st.nz >= 2) return;  // nothing changes
    if (A.accumulate && st.nz == 1) {
        if (t0 == 0 && yb != 0.0) {
            const double c = ldexp_clamped(st.m * ym, st.e + ye);
            abar[st.first] = (T)((double)abar[st.first] + c);
        }
        return;
    }
    const double kq = st.m * ym;  // the numerator's mantissa, in [0.25, 1)
    if (st.nz == 0 && yb != 0.0) {
        // no zero: abar_i = p / a_i * ybar, from the end (what the recompute
        // read last is still in L2), four 16-byte vectors in flight per thread
        const int64_t eb = st.e + ye;
        const float qf = (float)kq;
        const QuotF64 quot = QuotF64::make(kq, eb);
        auto one = [&](T x) -> T {
            if constexpr (sizeof(T) == 4) return quot_f32(qf, eb, x);
            else return quot(x);
        };
        constexpr int V = Vec16<T>::N, U = 4;
        const int64_t nv = A.n / V;
        int64_t v = nv - 1 - t0;
        for (; v - (U - 1) * stride >= 0; v -= U * stride) {
            Vec16<T> x[U];
#pragma unroll
            for (int u = 0; u < U; ++u) x[u] = ld_vec_stream(a + (v - u * stride) * V);
#pragma unroll
            for (int u = 0; u < U; ++u) {
#pragma unroll
                for (int k = 0; k < V; ++k) x[u].v[k] = one(x[u].v[k]);
                T* o = abar + (v - u * stride) * V;
                if (A.accumulate) {
#pragma unroll
                    for (int k = 0; k < V; ++k) x[u].v[k] += o[k];
                }
                st_vec(o, x[u]);
            }
        }
        for (; v >= 0; v -= stride) {
            Vec16<T> x = ld_vec_stream(a + v * V);
#pragma unroll
            for (int k = 0; k < V; ++k) x.v[k] = A.accumulate ? abar[v * V + k] + one(x.v[k]) : one(x.v[k]);
            st_vec(abar + v * V, x);
        }
        const int64_t i = nv * V + t0;
        if (i < A.n) abar[i] = A.accumulate ? abar[i] + one(a[i]) : one(a[i]);
        return;
    }
    // zeros among the elements (or ybar = 0): 0, and the only zero's own adjoint,
    // which joins the accumulated value before it is rounded to T
    const int64_t at = st.nz == 1 && yb != 0.0 ? st.first : -1;
    auto put = [&](int64_t i) -> T {
        const double c = i == at ? ldexp_clamped(kq, st.e + ye) : 0.0;
        return (T)(A.accumulate ? (double)abar[i] + c : c);
    };
    constexpr int V = Vec16<T>::N;
    const int64_t nv = A.n / V;
    for (int64_t v = t0; v < nv; v += stride) {
        T* p = abar + v * V;
        Vec16<T> o;
        if (at / V == v && at >= 0) {
#pragma unroll
            for (int k = 0; k < V; ++k) o.v[k] = put(v * V + k);
        } else {
#pragma unroll
            for (int k = 0; k < V; ++k) o.v[k] = A.accumulate ? p[k] : T(0);
        }
        st_vec(p, o);
    }
    const int64_t i = nv * V + t0;
    if (i < A.n) abar[i] = put(i);
}

template <class T>
__global__ void __launch_bounds__(kRedBlock, 4) prod_adjoint_kernel(ReduceArgs A) {
    const ProdState st = *static_cast<const ProdState*>(A.final_state);
    prod_adjoint_body<T>(A, st, blockIdx.x * (int64_t)blockDim.x + threadIdx.x, (int64_t)gridDim.x * blockDim.x);
}

// ------------------------------------------------------ one-cluster form
// Short arrays: the whole call in one launch of one cluster of 8 blocks.  Each
// block reduces its share, the blocks read each other's states through
// distributed shared memory (a hardware barrier of the cluster instead of a
// global counter that an earlier launch must clear), and every block maps its
// share with the same total.  65536 FP64 values: 10 us on the device against 17 in
// three launches and their gaps (14 against 18 us per call from Python, on a slow
// host); at 1 MB 18 against 18, at 2 MB 26 against 18.
constexpr int kClusterBlocks = 8;
constexpr int kClusterThreads = 1024;
constexpr int64_t kClusterBytes = int64_t(1) << 20;

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// block `rank`'s copy of the shared variable at p
template <class S>
__device__ __forceinline__ S ld_cluster(const S* p, unsigned rank) {
    static_assert(sizeof(S) % 8 == 0, "8-byte granules");
    constexpr int N = sizeof(S) / 8;
    union {
        S s;
        unsigned long long w[N];
    } u;
    unsigned a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
#pragma unroll
    for (int i = 0; i < N; ++i)
        asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(u.w[i]) : "r"(a + 8u * i));
    return u.s;
}

template <class T>
__global__ void __cluster_dims__(kClusterBlocks, 1, 1) __launch_bounds__(kClusterThreads, 1)
    reduce_prod_cluster_kernel(ReduceArgs A) {
    using S = ProdStateQ;
    __shared__ S s_warp[kClusterThreads / 32];
    __shared__ S s_block;
    __shared__ ProdState s_total;
    const T* a = static_cast<const T*>(A.a);
    constexpr int V = Vec16<T>::N, U = 4;
    const int64_t nvec = A.n / V, stride = kClusterBlocks * kClusterThreads;
    const int64_t t0 = blockIdx.x * (int64_t)kClusterThreads + threadIdx.x;
    if (t0 < 64) reinterpret_cast<uint32_t*>(A.hdr)[t0] = 0u;  // the status word starts at ok
    ProdAcc st = ProdAcc::id();
    for (int64_t v0 = t0; v0 < nvec; v0 += U * stride) {
        Vec16<T> x[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (v0 + u * stride < nvec) x[u] = ld_vec(a + (v0 + u * stride) * V);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (v0 + u * stride >= nvec) break;
#pragma unroll
            for (int j = 0; j < V; ++j) st.push(x[u].v[j], (v0 + u * stride) * V + j);
        }
    }
    if (t0 < A.n - nvec * V) st.push(a[nvec * V + t0], nvec * V + t0);
    auto comb = [](const S& x, const S& y) { return S::comb(x, y); };
    const S bs = block_reduce(st.state(), comb, s_warp);
    if (threadIdx.x == 0) s_block = bs;
    cluster_sync();
    if (threadIdx.x < 32) {
        S q = (int)threadIdx.x < kClusterBlocks ? ld_cluster(&s_block, threadIdx.x) : S::id();
#pragma unroll
        for (int off = kClusterBlocks / 2; off > 0; off >>= 1) q = S::comb(q, shfl_down_s(q, off));
        if (threadIdx.x == 0) s_total = q.to_state();
    }
    __syncthreads();
    if (t0 == 32) prod_results<T>(A, s_total);  // beside the map
    if (!A.primal_only) prod_adjoint_body<T>(A, s_total, t0, stride);
    cluster_sync();  // no block leaves while another may read its state
}

// ------------------------------------------------------------ host side
size_t state_bytes(int op, int dtype) {
    const size_t t = dtype == ADPAR_F64 ? 8 : 4;
    switch (op) {
    case ADPAR_OP_ADD: return t;
    case ADPAR_OP_MIN:
    case ADPAR_OP_MAX: return 16;
    case ADPAR_OP_MUL: return std::max(sizeof(ProdState), sizeof(ProdStateQ));
    }
    return 0;
}

// resident blocks of the * kernels: 4 of 256 threads per SM
int prod_wave() {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return std::min(4 * std::max(sms, 1), kRedMaxBlocks);
}

int grid_for(int64_t n, int dtype) {
    const int64_t per_block = (int64_t)kRedBlock * (dtype == ADPAR_F64 ? 2 : 4) * 8;
    int64_t g = (n + per_block - 1) / per_block;
    return (int)std::max<int64_t>(1, std::min<int64_t>(g, kRedMaxBlocks));
}

template <class T>
int run_reduce(ReduceArgs A, int op, cudaStream_t s) {
    const int grid = grid_for(A.n, sizeof(T) == 8 ? ADPAR_F64 : ADPAR_F32);
    // the "last block" counter must start at zero in a workspace of unknown
    // contents
    // (the log domain's FP64 logarithms would queue on eight SMs: 106 us for 65536
    // values, 30 over the grid)
    const bool cluster = op == ADPAR_OP_MUL && !A.logdomain && A.n * (int64_t)sizeof(T) <= kClusterBytes;
    if (!cluster) header_init_kernel<<<1, 64, 0, s>>>(A.hdr);
    switch (op) {
    case ADPAR_OP_ADD:
        reduce_add_kernel<T><<<grid, kRedBlock, 0, s>>>(A);
        break;
    case ADPAR_OP_MIN:
        reduce_arg_kernel<T, false><<<grid, kRedBlock, 0, s>>>(A);
        break;
    case ADPAR_OP_MAX:
        reduce_arg_kernel<T, true><<<grid, kRedBlock, 0, s>>>(A);
        break;
    case ADPAR_OP_MUL: {
        if (cluster) {
            reduce_prod_cluster_kernel<T><<<kClusterBlocks, kClusterThreads, 0, s>>>(A);
            break;
        }
        // one 16-byte vector per thread, up to a whole wave of resident blocks
        const int64_t per = (int64_t)kRedBlock * (16 / sizeof(T));
        const int wave = prod_wave();
        const int gp = (int)std::max<int64_t>(1, std::min<int64_t>((A.n + per - 1) / per, wave));
        reduce_prod_kernel<T><<<gp, kRedBlock, 0, s>>>(A);
        if (A.primal_only) break;
        // the log domain's threads form two FP64 logarithms of their own: four elements each
        const int ga = A.logdomain ? (int)std::max<int64_t>(1, std::min<int64_t>((A.n + 1023) / 1024, wave)) : gp;
        prod_adjoint_kernel<T><<<ga, kRedBlock, 0, s>>>(A);
        break;
    }
    default:
        return ADPAR_ERR_INVALID;
    }
    return cudaGetLastError() == cudaSuccess ? ADPAR_OK : ADPAR_ERR_CUDA;
}

}  // namespace

size_t reduce_workspace_size(adpar_opdesc d) {
    if (d.dtype != ADPAR_F32 && d.dtype != ADPAR_F64) return (size_t)-1;
    const size_t sb = state_bytes(d.op, d.dtype);
    if (sb == 0) return (size_t)-1;
    return sizeof(WsHeader) + round_up(kRedMaxBlocks * sb, 256) + 256;
}

}  // namespace adpar

extern "C" int adpar_vjp_reduce(adpar_opdesc d, int64_t n, const void* a, const void* ybar, void* abar,
                                void* y_out, int64_t* argidx_out, adpar_prod_aux* aux_out,
                                int8_t* abar_sign, uint32_t flags, void* work, size_t work_bytes,
                                void* stream) {
    using namespace adpar;
    if (n < 0 || d.width != 1) return ADPAR_ERR_INVALID;
    if (d.op != ADPAR_OP_ADD && d.op != ADPAR_OP_MUL && d.op != ADPAR_OP_MIN && d.op != ADPAR_OP_MAX)
        return ADPAR_ERR_INVALID;
    if (d.dtype != ADPAR_F32 && d.dtype != ADPAR_F64) return ADPAR_ERR_INVALID;
    if (flags & ~(uint32_t)(ADPAR_ACCUMULATE | ADPAR_PROD_LOGDOMAIN)) return ADPAR_ERR_UNSUPPORTED;
    const bool logd = (flags & ADPAR_PROD_LOGDOMAIN) != 0;
    if (logd && (d.op != ADPAR_OP_MUL || (flags & ADPAR_ACCUMULATE))) return ADPAR_ERR_UNSUPPORTED;
    if (abar_sign && !logd) return ADPAR_ERR_INVALID;
    if (!ybar || (n > 0 && !abar)) return ADPAR_ERR_INVALID;
    if (n > 0 && !a && !(d.op == ADPAR_OP_ADD && !y_out)) return ADPAR_ERR_INVALID;
    if ((a && !aligned16(a)) || (abar && !aligned16(abar))) return ADPAR_ERR_ALIGN;
    const size_t need = reduce_workspace_size(d);
    if (!work || work_bytes < need || (reinterpret_cast<uintptr_t>(work) & 255u)) return ADPAR_ERR_WORKSPACE;
    ReduceArgs A{};
    A.op = d.op;
    A.n = n;
    A.a = a;
    A.ybar = ybar;
    A.abar = abar;
    A.y_out = y_out;
    A.argidx_out = argidx_out;
    A.aux_out = aux_out;
    A.abar_sign = abar_sign;
    A.accumulate = (flags & ADPAR_ACCUMULATE) ? 1 : 0;
    A.logdomain = logd ? 1 : 0;
    char* w = static_cast<char*>(work);
    A.hdr = reinterpret_cast<WsHeader*>(w);
    A.partials = w + sizeof(WsHeader);
    A.final_state = w + sizeof(WsHeader) + round_up(kRedMaxBlocks * state_bytes(d.op, d.dtype), 256);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (d.dtype == ADPAR_F32) return run_reduce<float>(A, d.op, s);
    return run_reduce<double>(A, d.op, s);
}

extern "C" int adpar_reduce(adpar_opdesc d, int64_t n, const void* a, void* y_out, int64_t* argidx_out,
                            adpar_prod_aux* aux_out, void* work, size_t work_bytes, void* stream) {
    using namespace adpar;
    if (n < 0 || d.width != 1) return ADPAR_ERR_INVALID;
    if (d.op != ADPAR_OP_ADD && d.op != ADPAR_OP_MUL && d.op != ADPAR_OP_MIN && d.op != ADPAR_OP_MAX)
        return ADPAR_ERR_INVALID;
    if (d.dtype != ADPAR_F32 && d.dtype != ADPAR_F64) return ADPAR_ERR_INVALID;
    if (!y_out || (n > 0 && !a)) return ADPAR_ERR_INVALID;
    if (a && !aligned16(a)) return ADPAR_ERR_ALIGN;
    const size_t need = reduce_workspace_size(d);
    if (!work || work_bytes < need || (reinterpret_cast<uintptr_t>(work) & 255u)) return ADPAR_ERR_WORKSPACE;
    ReduceArgs A{};
    A.op = d.op;
    A.n = n;
    A.a = a;
    A.y_out = y_out;
    A.argidx_out = argidx_out;
    A.aux_out = aux_out;
    A.primal_only = 1;
    char* w = static_cast<char*>(work);
    A.hdr = reinterpret_cast<WsHeader*>(w);
    A.partials = w + sizeof(WsHeader);
    A.final_state = w + sizeof(WsHeader) + round_up(kRedMaxBlocks * state_bytes(d.op, d.dtype), 256);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (d.dtype == ADPAR_F32) return run_reduce<float>(A, d.op, s);
    return run_reduce<double>(A, d.op, s);
}
