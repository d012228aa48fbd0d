// VJP of a scan over vectors with an elementwise operator (Sec. 5.2, the
// vectorised case): xs is row-major [n][d] and
//   scan (map (.)) e xs == transpose xs |> map (scan (.) e) |> transpose,
// i.e. d independent scans down the columns.  No transpose is materialised:
// a thread owns one column and one chunk of kVecR rows, so a warp's loads
// cover 32 consecutive columns of a row (coalesced), 8 rows' loads in flight.
// No block waits on another:
//   1. per (chunk, column): the aggregates of the operator's state, then of the
//      return sweep's lin_o state (two launches);
//   2. per column a scan of the chunks' aggregates, left to right and right to
//      left (exclusive carries);
//   3. per (chunk, column): a backward sweep of rs_bar_r = ybar_r +
//      c_{r+1} rs_bar_{r+1} into shared memory, then a forward sweep with
//      the primal prefix writing as_bar = J_right^T rs_bar.
// MIN/MAX, whose J_left needs the primal prefix, take 1 and 2 for the operator
// first and then for the return sweep (re-forming the prefix from the carry).
#include <algorithm>

#include "scan_tiles.cuh"

namespace adpar {
namespace {

constexpr int kVecBlock = 256;
constexpr int kVecOutBlock = 64;  // the output pass keeps 32 rows x width of rs_bar per thread in shared memory
constexpr int kVecR = 32;         // rows per chunk (the J_left bits of a chunk fit one word)

// operators whose return sweep reads the primal (the input a)
template <class Op>
constexpr bool kVecPrimal = Op::kNeedPrimal || Op::kCoefNeedsPrimal || !Op::kCoefOne;

struct VecArgs {
    int64_t n, d, C;  // rows, columns, chunks
    const void* a;
    const void* b;
    const void* ya;
    const void* yb;
    void* abar;
    void* bbar;
    int accumulate;
    void* aggP;  // [C][d] P: chunk aggregates, then exclusive prefixes
    void* aggL;  // [C][d] L: chunk aggregates, then exclusive suffixes
};

// Blocks lie along the columns, a grid row per chunk; with few columns (FLAT)
// consecutive threads take consecutive (chunk, column) pairs, so that narrow
// arrays do not leave most lanes idle: FP64 max over 100000 x 1, 277 -> 220 us;
// 4000 x 300, 76 -> 58 us.  Only where the blocks outnumber the SMs: 2000 x 64
// spread over 63 SMs is faster than over 16.
constexpr int64_t kVecFlat = 1024;
__device__ __forceinline__ int64_t vec_chunk(const VecArgs& V, int64_t i) {
    return (int64_t)((unsigned long long)i / (unsigned)V.d);  // d < kVecFlat
}

// rows whose loads a thread has in flight at once
constexpr int kVecU = 8;  // output pass
template <class Op>
constexpr int kVecUAgg = Op::kWidth == 2 || Op::kCoefOne ? 4 : 8;  // aggregates (LINREC loads two or three arrays)

// p[i], p[i + d], .. for U rows from `row` on (pad past the last row)
template <int U, class T>
__device__ __forceinline__ void vec_rows(const void* p, const VecArgs& V, int64_t row, int64_t col, T pad,
                                         T (&o)[U]) {
    const T* q = static_cast<const T*>(p) + row * V.d + col;
#pragma unroll
    for (int u = 0; u < U; ++u) o[u] = row + u < V.n ? __ldg(q + u * V.d) : pad;
}

// the operator's state over each chunk, top to bottom
template <class Op, class T, bool FLAT>
__global__ void __launch_bounds__(kVecBlock, 6) vec_primal_agg_kernel(VecArgs V) {
    using P = typename Op::P;
    constexpr int W = Op::kWidth, U = kVecUAgg<Op>;
    const int64_t i = blockIdx.x * (int64_t)kVecBlock + threadIdx.x, c = FLAT ? vec_chunk(V, i) : (int64_t)blockIdx.y;
    const int64_t col = FLAT ? i - c * V.d : i;
    if (FLAT ? c >= V.C : col >= V.d) return;
    const int64_t r0 = c * kVecR;
    P acc = Op::pid();
#pragma unroll 1
    for (int q = 0; q < kVecR && r0 + q < V.n; q += U) {
        T a[U], b[U];
        vec_rows<U>(V.a, V, r0 + q, col, Op::pad_a(), a);
        if constexpr (W == 2) vec_rows<U>(V.b, V, r0 + q, col, T(0), b);
#pragma unroll
        for (int u = 0; u < U; ++u) acc = Op::pcomb(acc, Op::pelem(a[u], W == 2 ? b[u] : T(0)));
    }
    static_cast<P*>(V.aggP)[c * V.d + col] = acc;
}

// Turns the chunk aggregates of 32 columns into exclusive prefixes (REV:
// exclusive suffixes, composed right to left).  Thread (x, y) of a 32 x G block
// folds group y of column x's chunks (neighbouring lanes read neighbouring
// columns), the groups' folds are scanned, and each thread runs through its
// chunks again.  8 chunks are loaded at a time; G is a group per 8 chunks, up to
// 32.  The groups' folds: by shuffles, a warp per column, where there are many in
// FP32; few of them, and FP64 ones (a warp's combination takes the FP64 pipe of
// the SM 32 cycles, and 32 columns take five steps each), one after another by a
// thread per column.  FP64 max over 500 x 64, by shuffles and now: the call 57 and
// 39 us; over 500 x 2048, 64 and 49 us (4 or 2 chunks a group: no faster).
constexpr int kVecG = 32;
constexpr int kVecSerialG = 8;
template <bool F64, class S, bool REV, class Comb>
__device__ __forceinline__ void vec_scan_columns(S* agg, int64_t C, int64_t d, S* s_tot, const S& ident, Comb comb) {
    const int x = threadIdx.x & 31, y = threadIdx.x >> 5, G = blockDim.x >> 5;
    const int64_t col = blockIdx.x * (int64_t)32 + x;
    const int64_t per = (C + G - 1) / G;
    const int64_t lo = y * per < C ? y * per : C, hi = lo + per < C ? lo + per : C;
    const bool live = col < d;
    auto at = [&](int64_t q) -> S* { return agg + (REV ? C - 1 - q : q) * d + col; };
    S run = ident;
    if (G > 1) {
        if (live) {
            for (int64_t q = lo; q < hi; q += 8) {
                S v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) v[u] = q + u < hi ? *at(q + u) : ident;
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    if (F64 && q + u >= hi) break;
                    run = comb(run, v[u]);
                }
            }
        }
        s_tot[y * 33 + x] = run;
        __syncthreads();
        const bool serial = F64 || G <= kVecSerialG;
        if (serial && y == 0) {
            S pre = ident;
            for (int w = 0; w < G; ++w) {
                const S t = s_tot[w * 33 + x];
                s_tot[w * 33 + x] = pre;
                pre = comb(pre, t);
            }
        }
        for (int w = serial ? 32 : y; w < 32; w += G) {  // lane x holds group x of column w
            S inc = x < G ? s_tot[x * 33 + w] : ident;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const S o = shfl_up_s(inc, off);
                if (x >= off) inc = comb(o, inc);
            }
            S ex = shfl_up_s(inc, 1);
            if (x == 0) ex = ident;
            __syncwarp();
            if (x < G) s_tot[x * 33 + w] = ex;
        }
        __syncthreads();
        run = s_tot[y * 33 + x];
    }
    if (live) {
        for (int64_t q = lo; q < hi; q += 8) {
            S v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = q + u < hi ? *at(q + u) : ident;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                if (q + u >= hi) break;
                *at(q + u) = run;
                run = comb(run, v[u]);
            }
        }
    }
}

// Scans the aggregates asked for: blockIdx.y 0 the operator's, 1 the return
// sweep's (first: the y of the first grid row)
template <class Op, class T>
__global__ void __launch_bounds__(32 * kVecG) vec_scan_kernel(VecArgs V, int first) {
    using P = typename Op::P;
    using L = Lin<T, Op::kWidth, !Op::kCoefOne>;
    extern __shared__ __align__(16) unsigned char s_dyn[];
    if (blockIdx.y + first == 0) {
        vec_scan_columns<sizeof(T) == 8, P, false>(static_cast<P*>(V.aggP), V.C, V.d, reinterpret_cast<P*>(s_dyn), Op::pid(),
                                   [](const P& l, const P& r) { return Op::pcomb(l, r); });
    } else {
        // scan order is right to left: e holds later rows, l earlier ones
        vec_scan_columns<sizeof(T) == 8, L, true>(static_cast<L*>(V.aggL), V.C, V.d, reinterpret_cast<L*>(s_dyn), L::id(),
                                  [](const L& e, const L& l) { return L::comb(e, l); });
    }
}

// J_left of the chunk's rows as bits (MIN/MAX: needs the primal prefix)
template <class Op, class T>
__device__ __forceinline__ uint32_t vec_coef_bits(const VecArgs& V, int64_t col, int64_t r0,
                                                  const typename Op::P& carry) {
    uint32_t bits = 0u;
    typename Op::P cur = carry;
#pragma unroll 1
    for (int q = 0; q < kVecR && r0 + q < V.n; q += kVecU) {
        T a[kVecU];
        vec_rows(V.a, V, r0 + q, col, Op::pad_a(), a);
#pragma unroll
        for (int u = 0; u < kVecU; ++u) {
            if (Op::coef(cur, a[u]) != T(0)) bits |= 1u << (q + u);
            cur = Op::pcomb(cur, Op::pelem(a[u], T(0)));
        }
    }
    return bits;
}

// J_left of the rows row .. row + U - 1 (q0: the first one's number in the
// chunk); rows past the end have ybar 0 below them, so their value is free
template <class Op, class T, int U>
__device__ __forceinline__ void vec_coefs(const VecArgs& V, int64_t row, int64_t col, uint32_t bits, int q0,
                                          T (&c)[U]) {
    if constexpr (Op::kCoefOne) {
#pragma unroll
        for (int u = 0; u < U; ++u) c[u] = T(1);
    } else if constexpr (Op::kCoefNeedsPrimal) {
#pragma unroll
        for (int u = 0; u < U; ++u) c[u] = ((bits >> (q0 + u)) & 1u) ? T(1) : T(0);
    } else {
        vec_rows<U>(V.a, V, row, col, T(1), c);
#pragma unroll
        for (int u = 0; u < U; ++u) c[u] = Op::coef(Op::pid(), c[u]);
    }
}

// Chunk aggregates of the return sweep: x -> c_r (ybar_r + x) folded bottom to
// top (Horner's order: a contracting recurrence damps the early roundings; the
// growing map of a sweep from the top, fused with the operator's, read each
// array once and took 52 us for 23 + 40, but its FP32 results were further off)
template <class Op, class T, bool FLAT>
__global__ void __launch_bounds__(kVecBlock, Op::kCoefOne && sizeof(T) == 4 ? 8 : 6) vec_adjoint_agg_kernel(VecArgs V) {
    using P = typename Op::P;
    constexpr int W = Op::kWidth, U = kVecUAgg<Op>;
    using L = Lin<T, W, !Op::kCoefOne>;
    const int64_t i = blockIdx.x * (int64_t)kVecBlock + threadIdx.x, c = FLAT ? vec_chunk(V, i) : (int64_t)blockIdx.y;
    const int64_t col = FLAT ? i - c * V.d : i;
    if (FLAT ? c >= V.C : col >= V.d) return;
    const int64_t r0 = c * kVecR;
    uint32_t bits = 0u;
    if constexpr (Op::kCoefNeedsPrimal)
        bits = vec_coef_bits<Op, T>(V, col, r0, static_cast<const P*>(V.aggP)[c * V.d + col]);
    L acc = L::id();
#pragma unroll 1
    for (int q = kVecR - U; q >= 0; q -= U) {
        if (r0 + q >= V.n) continue;
        T cf[U], y1[U], y2[U];
        vec_coefs<Op, T, U>(V, r0 + q, col, bits, q, cf);
        vec_rows<U>(V.ya, V, r0 + q, col, T(0), y1);
        if constexpr (W == 2) vec_rows<U>(V.yb, V, r0 + q, col, T(0), y2);
#pragma unroll
        for (int u = U - 1; u >= 0; --u) {
            if (r0 + q + u >= V.n) continue;
            L el;
            if constexpr (!Op::kCoefOne) {
                el.c = cf[u];
                el.d[0] = cf[u] * y1[u];
                if constexpr (W == 2) el.d[1] = cf[u] * y2[u];
            } else {
                el.d[0] = y1[u];
                if constexpr (W == 2) el.d[1] = y2[u];
            }
            acc = L::comb(acc, el);
        }
    }
    static_cast<L*>(V.aggL)[c * V.d + col] = acc;
}

// Chunks last to first: what the aggregates read last is still in L2.  8 rows'
// loads in flight at 9 blocks an SM (about 110 registers): 72 us for 8192 x 2048
// FP32 LINREC (59 us for its bytes); 64 registers, or one row at a time: 96 and
// 128 us.  The scan of both aggregates takes 11 us (was 13 + 23 with a warp per
// column); the call 245 -> 164 us.
template <class Op, class T, bool FLAT>
__global__ void __launch_bounds__(kVecOutBlock, 9) vec_output_kernel(VecArgs V) {
    using P = typename Op::P;
    constexpr int W = Op::kWidth;
    constexpr bool kP = kVecPrimal<Op>;
    using L = Lin<T, W, !Op::kCoefOne>;
    __shared__ T s_r[kVecR * W * kVecOutBlock];  // rs_bar of the thread's rows, [row][component][thread]
    const int64_t i = blockIdx.x * (int64_t)kVecOutBlock + threadIdx.x, f = FLAT ? vec_chunk(V, i) : (int64_t)blockIdx.y;
    const int64_t col = FLAT ? i - f * V.d : i, c = V.C - 1 - f;
    if (FLAT ? c < 0 : col >= V.d) return;
    const int64_t r0 = c * kVecR;
    const P carry = kP ? static_cast<const P*>(V.aggP)[c * V.d + col] : Op::pid();
    const L suf = static_cast<const L*>(V.aggL)[c * V.d + col];
    uint32_t bits = 0u;
    if constexpr (Op::kCoefNeedsPrimal) bits = vec_coef_bits<Op, T>(V, col, r0, carry);
    // backward: rs_bar of the last row gets the chunks below through suf.d (0 in the
    // last chunk); cn is J_left of the row below.  Rows past the end carry ybar 0 and
    // rs_bar 0 on.
    T ra = suf.d[0], rb = W == 2 ? suf.d[W - 1] : T(0), cn = T(1);
#pragma unroll 1
    for (int q = kVecR - kVecU; q >= 0; q -= kVecU) {
        if (r0 + q >= V.n) continue;
        T cf[kVecU], y1[kVecU], y2[kVecU];
        vec_coefs<Op, T, kVecU>(V, r0 + q, col, bits, q, cf);
        vec_rows(V.ya, V, r0 + q, col, T(0), y1);
        if constexpr (W == 2) vec_rows(V.yb, V, r0 + q, col, T(0), y2);
#pragma unroll
        for (int u = kVecU - 1; u >= 0; --u) {
            ra = fma(cn, ra, y1[u]);
            if constexpr (W == 2) rb = fma(cn, rb, y2[u]);
            cn = cf[u];
            s_r[((q + u) * W) * kVecOutBlock + threadIdx.x] = ra;
            if constexpr (W == 2) s_r[((q + u) * W + 1) * kVecOutBlock + threadIdx.x] = rb;
        }
    }
    // forward: the primal prefix and the adjoints
    T* abar = static_cast<T*>(V.abar) + r0 * V.d + col;
    T* bbar = W == 2 ? static_cast<T*>(V.bbar) + r0 * V.d + col : nullptr;
    P prev = carry;
#pragma unroll 1
    for (int q = 0; q < kVecR && r0 + q < V.n; q += kVecU) {
        T a[kVecU], b[kVecU];
        if constexpr (kP) {
            vec_rows(V.a, V, r0 + q, col, Op::pad_a(), a);
            if constexpr (W == 2) vec_rows(V.b, V, r0 + q, col, T(0), b);
        }
#pragma unroll
        for (int u = 0; u < kVecU; ++u) {
            if (r0 + q + u >= V.n) continue;
            const T av = kP ? a[u] : T(0), bv = kP && W == 2 ? b[u] : T(0);
            const T q1 = s_r[((q + u) * W) * kVecOutBlock + threadIdx.x];
            const T q2 = W == 2 ? s_r[((q + u) * W + 1) * kVecOutBlock + threadIdx.x] : T(0);
            T o1 = T(0), o2 = T(0);
            Op::vjp_right(prev, av, bv, q1, q2, o1, o2);
            if constexpr (kP) prev = Op::pcomb(prev, Op::pelem(av, bv));
            T* oa = abar + (q + u) * V.d;
            if (V.accumulate) {
                *oa += o1;
                if constexpr (W == 2) bbar[(q + u) * V.d] += o2;
            } else {
                *oa = o1;
                if constexpr (W == 2) bbar[(q + u) * V.d] = o2;
            }
        }
    }
}

template <class Op, class T>
size_t vec_workspace(int64_t n, int64_t d) {
    using L = Lin<T, Op::kWidth, !Op::kCoefOne>;
    const int64_t C = (n + kVecR - 1) / kVecR;
    return sizeof(WsHeader) + round_up((size_t)C * d * sizeof(typename Op::P), 256) +
           round_up((size_t)C * d * sizeof(L), 256);
}

template <class Op, class T, bool FLAT>
void launch_vec(const VecArgs& V, cudaStream_t s) {
    using L = Lin<T, Op::kWidth, !Op::kCoefOne>;
    auto grid = [&](int64_t block) {
        if (FLAT) return dim3((unsigned)((V.C * V.d + block - 1) / block));
        return dim3((unsigned)((V.d + block - 1) / block), (unsigned)V.C);
    };
    const unsigned gw = (unsigned)((V.d + 31) / 32);  // 32 columns per block
    const int G = (int)(V.C <= 8 ? 1 : std::min<int64_t>(V.C / 8 + 1, kVecG));
    const size_t sh = std::max(sizeof(typename Op::P), sizeof(L)) * 33 * G;
    constexpr bool kTwo = kVecPrimal<Op> && !Op::kCoefNeedsPrimal;  // both scans from one launch
    if constexpr (kVecPrimal<Op>) vec_primal_agg_kernel<Op, T, FLAT><<<grid(kVecBlock), kVecBlock, 0, s>>>(V);
    if constexpr (Op::kCoefNeedsPrimal) vec_scan_kernel<Op, T><<<dim3(gw, 1), 32 * G, sh, s>>>(V, 0);
    vec_adjoint_agg_kernel<Op, T, FLAT><<<grid(kVecBlock), kVecBlock, 0, s>>>(V);
    vec_scan_kernel<Op, T><<<dim3(gw, kTwo ? 2 : 1), 32 * G, sh, s>>>(V, kTwo ? 0 : 1);
    vec_output_kernel<Op, T, FLAT><<<grid(kVecOutBlock), kVecOutBlock, 0, s>>>(V);
}

template <class Op, class T>
int run_vec(int64_t n, int64_t d, const void* a, const void* b, const void* ya, const void* yb, void* abar,
            void* bbar, uint32_t flags, void* work, size_t work_bytes, cudaStream_t s) {
    using L = Lin<T, Op::kWidth, !Op::kCoefOne>;
    const size_t need = vec_workspace<Op, T>(n, d);
    if (!work || work_bytes < need || (reinterpret_cast<uintptr_t>(work) & 255u)) return ADPAR_ERR_WORKSPACE;
    if (n == 0 || d == 0) return ADPAR_OK;
    VecArgs V{};
    V.n = n; V.d = d; V.C = (n + kVecR - 1) / kVecR;
    V.a = a; V.b = b; V.ya = ya; V.yb = yb; V.abar = abar; V.bbar = bbar;
    V.accumulate = (flags & ADPAR_ACCUMULATE) ? 1 : 0;
    char* w = static_cast<char*>(work);
    cudaMemsetAsync(w, 0, sizeof(WsHeader), s);  // the status word starts at ok
    V.aggP = w + sizeof(WsHeader);
    V.aggL = w + sizeof(WsHeader) + round_up((size_t)V.C * d * sizeof(typename Op::P), 256);
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // (few blocks spread over the SMs as they are)
    if (d < kVecFlat && V.C * ((d + kVecBlock - 1) / kVecBlock) > sms) launch_vec<Op, T, true>(V, s);
    else launch_vec<Op, T, false>(V, s);
    return cudaGetLastError() == cudaSuccess ? ADPAR_OK : ADPAR_ERR_CUDA;
}

template <class T>
int dispatch_vec(int op, int64_t n, int64_t d, const void* a, const void* b, const void* ya, const void* yb,
                 void* abar, void* bbar, uint32_t flags, void* work, size_t work_bytes, cudaStream_t s) {
    switch (op) {
    case ADPAR_OP_ADD: return run_vec<OpAdd<T>, T>(n, d, a, b, ya, yb, abar, bbar, flags, work, work_bytes, s);
    case ADPAR_OP_MUL: return run_vec<OpMul<T>, T>(n, d, a, b, ya, yb, abar, bbar, flags, work, work_bytes, s);
    case ADPAR_OP_MIN: return run_vec<OpMin<T>, T>(n, d, a, b, ya, yb, abar, bbar, flags, work, work_bytes, s);
    case ADPAR_OP_MAX: return run_vec<OpMax<T>, T>(n, d, a, b, ya, yb, abar, bbar, flags, work, work_bytes, s);
    case ADPAR_OP_LINREC:
        return run_vec<OpLinrec<T>, T>(n, d, a, b, ya, yb, abar, bbar, flags, work, work_bytes, s);
    }
    return ADPAR_ERR_INVALID;
}

template <class T>
size_t vec_ws_bytes(int op, int64_t n, int64_t d) {
    switch (op) {
    case ADPAR_OP_ADD: return vec_workspace<OpAdd<T>, T>(n, d);
    case ADPAR_OP_MUL: return vec_workspace<OpMul<T>, T>(n, d);
    case ADPAR_OP_MIN: return vec_workspace<OpMin<T>, T>(n, d);
    case ADPAR_OP_MAX: return vec_workspace<OpMax<T>, T>(n, d);
    case ADPAR_OP_LINREC: return vec_workspace<OpLinrec<T>, T>(n, d);
    }
    return (size_t)-1;
}

}  // namespace

size_t scan_vec_workspace_size(adpar_opdesc desc, int64_t n, int64_t d) {
    if (n < 0 || d < 0) return (size_t)-1;
    if (desc.dtype == ADPAR_F32) return vec_ws_bytes<float>(desc.op, n, d);
    if (desc.dtype == ADPAR_F64) return vec_ws_bytes<double>(desc.op, n, d);
    return (size_t)-1;
}

}  // namespace adpar

extern "C" int adpar_vjp_scan_vec(adpar_opdesc desc, int64_t n, int64_t d, const void* a, const void* b,
                                  const void* ybar_a, const void* ybar_b, void* abar, void* bbar, uint32_t flags,
                                  void* work, size_t work_bytes, void* stream) {
    using namespace adpar;
    if (n < 0 || d < 0) return ADPAR_ERR_INVALID;
    if (desc.op < ADPAR_OP_ADD || desc.op > ADPAR_OP_LINREC) return ADPAR_ERR_INVALID;
    if (desc.dtype != ADPAR_F32 && desc.dtype != ADPAR_F64) return ADPAR_ERR_INVALID;
    const int want_w = desc.op == ADPAR_OP_LINREC ? 2 : 1;
    if (desc.width != want_w) return ADPAR_ERR_INVALID;
    if (flags & ~(uint32_t)ADPAR_ACCUMULATE) return ADPAR_ERR_UNSUPPORTED;
    if (n > 0 && d > 0) {
        if (!ybar_a || !abar) return ADPAR_ERR_INVALID;
        if (desc.op != ADPAR_OP_ADD && !a) return ADPAR_ERR_INVALID;
        if (want_w == 2 && (!b || !ybar_b || !bbar)) return ADPAR_ERR_INVALID;
        const void* ptrs[] = {a, b, ybar_a, ybar_b, abar, bbar};
        for (const void* p : ptrs)
            if (p && !aligned16(p)) return ADPAR_ERR_ALIGN;
    }
    if (n > 0 && d > ((int64_t)1 << 31) / kVecBlock * kVecBlock) return ADPAR_ERR_UNSUPPORTED;  // grid x
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (desc.dtype == ADPAR_F32)
        return dispatch_vec<float>(desc.op, n, d, a, b, ybar_a, ybar_b, abar, bbar, flags, work, work_bytes, s);
    return dispatch_vec<double>(desc.op, n, d, a, b, ybar_a, ybar_b, abar, bbar, flags, work, work_bytes, s);
}
