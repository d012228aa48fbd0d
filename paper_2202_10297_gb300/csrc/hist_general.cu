// reduce_by_index VJP by the GENERAL rule of Sec. 5.1.2, for every operator
// of scan_ops.cuh (LINREC, which has no special rule, included).
//
//   hs[k] = (.) over the elements i with inds_i = k, in increasing i,
//   a_bar_i (+)= d(l_i (.) a_i (.) r_i)/d a_i ^T hs_bar[inds_i],
// where l_i and r_i combine the elements of i's bin before and after i.
// Those are per-bin ("multi-") scans; as Sec. 5.1.2 proposes they come from
// sorting the elements by bin and running a forward and a reverse
// irregular-segmented scan over the sorted sequence.
//
// Sort: least-significant-digit radix passes of up to 8 bits of the bin
// number, each three kernels (digit counts per block, a scan of the counts
// per digit, a stable scatter that ranks each tile by digit, stages it in
// shared memory in digit order and writes every digit's run contiguously).
// The values travel with their keys, so every read of a and b is
// coalesced, and each pass records where every element went.  Elements
// whose index is outside [0, m) leave in the first pass.
// Segmented scans: a segmented scan is a plain scan of (state, flag) pairs,
//   forward  (x1,f1) + (x2,f2) = f2 ? (x2,f2) : (x1 (.) x2, f1)
// with f = "a bin starts here", and its mirror image for the reverse scan
// with f = "a bin ends here".  Both are single-pass look-back scans over
// tiles; the forward one keeps only each tile's carry, the reverse one
// re-forms l inside the tile from that carry, applies the map and writes
// the adjoints in sorted order.
// Return: the recorded destinations of the passes, read backwards, gather
// the adjoints back to the original order (each inverse pass has the
// access pattern of a radix pass, and the last one writes the caller's
// arrays coalesced), instead of one random store per element.
#include <algorithm>

#include "common.cuh"
#include "scan_engine.cuh"
#include "scan_ops.cuh"

namespace adpar {
namespace {

constexpr int kSortBlock = 512;
constexpr int kSortNW = kSortBlock / 32;
// Elements per thread and tile of the scatter, staged in shared memory.  A tile's
// run of one digit is about TILE / 256 elements; a run that ends inside a 32-byte
// sector costs a partial-sector write, so long arrays take large tiles, short
// ones small tiles on more blocks.  10 per thread (5120 elements) is what 64
// registers hold, with two blocks an SM: forward and backward of 2^24 LINREC
// elements in 2^16 Zipf bins 1152 us; 12: 1204, 16: 1325 (spills), 8 with three
// blocks: 1460.
constexpr int kBigItems = 10, kSmallItems = 4;
template <class T, int W>
constexpr int big_items() {
    return sizeof(T) == 8 && W == 2 ? 6 : kBigItems;
}
constexpr int64_t kBigSort = int64_t(1) << 21;  // elements from which tiles are large
constexpr int kRadixBits = 8;
constexpr int kRadix = 1 << kRadixBits;
constexpr int kSortMaxGrid = 2048;
constexpr int kSegBlock = 256;
constexpr int kSegV = 4;  // consecutive elements per thread and chunk
constexpr int kSegK = 2;  // chunks per tile
constexpr int kSegTile = kSegK * kSegBlock * kSegV;
constexpr uint32_t kNoKey = 0xffffffffu;  // above every bin number (m < 2^31)

// One element's values: the pair (a, b) of LINREC side by side, so that a
// scattered element is one store and a gathered one one load.
template <class T, int W>
struct alignas(W * sizeof(T)) Elem {
    T a, b;
};
template <class T>
struct Elem<T, 1> {
    T a;
};
template <class T, int W>
__device__ __forceinline__ Elem<T, W> make_elem(T a, T b) {
    if constexpr (W == 2) return Elem<T, W>{a, b};
    else return Elem<T, W>{a};
}
template <class T, int W>
__device__ __forceinline__ T elem_b(const Elem<T, W>& e) {
    if constexpr (W == 2) return e.b;
    else return T(0);
}

// ------------------------------------------------------------ radix sort
template <class T, int W>
struct SortPass {
    int64_t n, m;          // all elements; bins
    const void* inds;      // first pass: the caller's indices and values
    const T* a;
    const T* b;
    const uint32_t* kin;   // later passes: keys and values
    const Elem<T, W>* ein;
    uint32_t* kout;
    Elem<T, W>* eout;
    uint32_t* dest;        // [input length] where each input element went (kNoKey: left the
                           // sort); NULL when nothing is returned to the input order
    uint32_t* cnt;         // [2^bits][G] digit counts per block, then their exclusive scan
    uint32_t* rowtot;      // [2^bits] elements per digit
    const uint32_t* nsorted;  // in-range elements (set by the first pass)
    int shift, bits, G;
};

// Block c of a pass covers [c * len_c, (c + 1) * len_c) of its input, a
// whole number of tiles.
__host__ __device__ __forceinline__ int64_t block_chunk(int64_t len, int G, int tile) {
    const int64_t c = (len + G - 1) / G;
    return (c + tile - 1) / tile * tile;
}

// Exclusive scan of one value per thread over a block of kSortBlock.
__device__ __forceinline__ uint32_t block_excl_u32(uint32_t x, uint32_t* s_w, uint32_t* total = nullptr) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t inc = x;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t o = __shfl_up_sync(0xffffffffu, inc, off);
        if (lane >= off) inc += o;
    }
    if (lane == 31) s_w[warp] = inc;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t run = 0;
        for (int w = 0; w < kSortNW; ++w) {
            const uint32_t t = s_w[w];
            s_w[w] = run;
            run += t;
        }
        s_w[kSortNW] = run;
    }
    __syncthreads();
    const uint32_t r = s_w[warp] + inc - x;
    if (total) *total = s_w[kSortNW];
    __syncthreads();
    return r;
}

template <class I, class T, int W, bool FIRST>
__device__ __forceinline__ bool sort_key(const SortPass<T, W>& P, int64_t i, uint32_t& key) {
    if constexpr (FIRST) {
        const int64_t ix = (int64_t)static_cast<const I*>(P.inds)[i];
        key = (uint32_t)ix;
        return ix >= 0 && ix < P.m;
    } else {
        key = P.kin[i];
        return true;
    }
}

template <class I, class T, int W, bool FIRST>
__global__ void __launch_bounds__(kSortBlock) hg_count_kernel(SortPass<T, W> P, int tile) {
    __shared__ uint32_t h[kSortNW][kRadix];
    const int warp = threadIdx.x >> 5;
    for (int q = threadIdx.x; q < kSortNW * kRadix; q += kSortBlock) (&h[0][0])[q] = 0u;
    __syncthreads();
    const int64_t len = FIRST ? P.n : (int64_t)*P.nsorted;
    const int64_t bc = block_chunk(len, P.G, tile);
    const int64_t lo = (int64_t)blockIdx.x * bc;
    const int64_t hi = lo + bc < len ? lo + bc : len;
    const uint32_t dmask = (1u << P.bits) - 1u;
    int64_t i = lo + threadIdx.x;
    for (; i + 3 * kSortBlock < hi; i += 4 * kSortBlock) {
        uint32_t key[4];
        bool ok[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) ok[u] = sort_key<I, T, W, FIRST>(P, i + u * kSortBlock, key[u]);
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (ok[u]) atomicAdd(&h[warp][(key[u] >> P.shift) & dmask], 1u);
    }
    for (; i < hi; i += kSortBlock) {
        uint32_t key;
        if (sort_key<I, T, W, FIRST>(P, i, key)) atomicAdd(&h[warp][(key >> P.shift) & dmask], 1u);
    }
    __syncthreads();
    for (int d = threadIdx.x; d < (1 << P.bits); d += kSortBlock) {
        uint32_t t = 0;
#pragma unroll
        for (int w = 0; w < kSortNW; ++w) t += h[w][d];
        P.cnt[(int64_t)d * P.G + blockIdx.x] = t;
    }
}

// Block d turns row d of the counts into its exclusive scan over the
// blocks and records the row total (the first pass also sums the totals
// into the in-range element count).
__global__ void __launch_bounds__(kSortBlock) hg_scan_counts_kernel(uint32_t* cnt, uint32_t* rowtot, int G,
                                                                    uint32_t* nsorted) {
    constexpr int E = 8;
    __shared__ uint32_t s_w[kSortNW + 1];
    uint32_t* row = cnt + (int64_t)blockIdx.x * G;
    uint32_t run = 0;
    for (int base = 0; base < G; base += kSortBlock * E) {
        uint32_t v[E];
        uint32_t s = 0;
#pragma unroll
        for (int j = 0; j < E; ++j) {
            const int q = base + threadIdx.x * E + j;
            v[j] = q < G ? row[q] : 0u;
            s += v[j];
        }
        uint32_t tot;
        uint32_t ex = run + block_excl_u32(s, s_w, &tot);
#pragma unroll
        for (int j = 0; j < E; ++j) {
            const int q = base + threadIdx.x * E + j;
            if (q < G) row[q] = ex;
            ex += v[j];
        }
        run += tot;
    }
    if (threadIdx.x == 0) {
        rowtot[blockIdx.x] = run;
        if (nsorted) atomicAdd(nsorted, run);
    }
}

__device__ __forceinline__ void prefetch_l2(const void* p) {
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

template <class T, int W, int ITEMS>
constexpr size_t sort_smem() {
    return (size_t)kSortBlock * ITEMS * (sizeof(Elem<T, W>) + 4) + kSortNW * kRadix * 2 + 2 * kRadix * 4 +
           (kSortNW + 1) * 4;
}

// Stable scatter of one pass.  A block takes its chunk tile by tile (warp w
// holds the tile's elements [w * 32 ITEMS, (w + 1) * 32 ITEMS), 32 consecutive
// ones per item).  Every element gets its rank among the equal digits before
// it in the tile (the lanes of equal digit from one ballot per digit bit,
// per-warp digit counts, their scan over the warps and the digits), which is
// its place in the tile sorted by digit; the tile is staged in that order in
// shared memory and written out so that each digit's run lands contiguously
// after the block's previous run of that digit.  Blocks and tiles are in input
// order and the counts were scanned over the blocks digit by digit, so equal
// digits keep their input order.
template <class I, class T, int W, bool FIRST, int ITEMS>
__global__ void __launch_bounds__(kSortBlock, 2) hg_scatter_kernel(SortPass<T, W> P) {
    constexpr int kTile = kSortBlock * ITEMS;
    using E = Elem<T, W>;
    extern __shared__ __align__(16) unsigned char s_dyn[];
    E* s_e = reinterpret_cast<E*>(s_dyn);
    uint32_t* s_key = reinterpret_cast<uint32_t*>(s_e + kTile);
    uint32_t* s_off = s_key + kTile;     // [kRadix] the block's next global position per digit
    uint32_t* s_start = s_off + kRadix;  // [kRadix] the digit's first place in the sorted tile
    uint32_t* s_w = s_start + kRadix;    // [kSortNW + 1]
    uint16_t* s_cnt = reinterpret_cast<uint16_t*>(s_w + kSortNW + 1);  // [kSortNW][kRadix]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int R = 1 << P.bits;
    const uint32_t dmask = (uint32_t)R - 1u;
    uint16_t* my_cnt = s_cnt + warp * kRadix;
    {
        const uint32_t rt = threadIdx.x < R ? P.rowtot[threadIdx.x] : 0u;
        const uint32_t ex = block_excl_u32(rt, s_w);
        if (threadIdx.x < R) s_off[threadIdx.x] = ex + P.cnt[(int64_t)threadIdx.x * P.G + blockIdx.x];
    }
    const int64_t len = FIRST ? P.n : (int64_t)*P.nsorted;
    const int64_t bc = block_chunk(len, P.G, kTile);
    const int64_t lo = (int64_t)blockIdx.x * bc;
    const int64_t hi = lo + bc < len ? lo + bc : len;
    const uint32_t lt = (1u << lane) - 1u;
    // the values of the tile at t into L2, while its keys are ranked (asking for
    // the next tile, or for the keys too, measured no better)
    auto prefetch_tile = [&](int64_t t) {
        const int64_t cnt = hi - t < kTile ? hi - t : kTile;
        auto lines = [&](const void* p, int64_t bytes) {
            for (int64_t o = threadIdx.x * 128; o < bytes; o += kSortBlock * 128)
                prefetch_l2(static_cast<const char*>(p) + o);
        };
        if constexpr (FIRST) {
            lines(P.a + t, cnt * (int64_t)sizeof(T));
            if constexpr (W == 2) lines(P.b + t, cnt * (int64_t)sizeof(T));
        } else {
            lines(P.ein + t, cnt * (int64_t)sizeof(E));
        }
    };
    for (int64_t t0 = lo; t0 < hi; t0 += kTile) {
        for (int q = lane; q < kRadix / 2; q += 32) reinterpret_cast<uint32_t*>(my_cnt)[q] = 0u;
        __syncwarp();
        const int64_t i0 = t0 + warp * (32 * ITEMS) + lane;
        uint32_t key[ITEMS], rk[ITEMS / 2];  // ranks, two of 16 bits in a word
        uint32_t okm = 0;
#pragma unroll
        for (int u = 0; u < ITEMS; ++u) {
            key[u] = 0u;
            if (i0 + u * 32 < hi && sort_key<I, T, W, FIRST>(P, i0 + u * 32, key[u])) okm |= 1u << u;
        }
        prefetch_tile(t0);
#pragma unroll
        for (int u = 0; u < ITEMS; ++u) {
            const bool ok = (okm >> u) & 1u;
            const uint32_t d = (key[u] >> P.shift) & dmask;
            // the lanes holding the same digit: one ballot per digit bit
            uint32_t peers = __ballot_sync(0xffffffffu, ok);
#pragma unroll
            for (int b = 0; b < kRadixBits; ++b) {
                const uint32_t mine = (uint32_t)((int)(d << (31 - b)) >> 31);  // all ones or none
                peers &= ~(__ballot_sync(0xffffffffu, mine != 0u) ^ mine);
            }
            const uint32_t base = ok ? my_cnt[d] : 0u;
            __syncwarp();
            if (ok && (peers & lt) == 0u) my_cnt[d] = (uint16_t)(base + __popc(peers));  // the lowest peer
            __syncwarp();
            const uint32_t r = base + __popc(peers & lt);
            rk[u / 2] = (u & 1) ? (rk[u / 2] | (r << 16)) : r;
        }
        __syncthreads();
        // per digit: exclusive over the warps, then over the digits
        uint32_t tot = 0;
        if (threadIdx.x < R) {
#pragma unroll
            for (int w = 0; w < kSortNW; ++w) {
                const uint32_t c = s_cnt[w * kRadix + threadIdx.x];
                s_cnt[w * kRadix + threadIdx.x] = (uint16_t)tot;
                tot += c;
            }
        }
        uint32_t nvalid;
        const uint32_t st = block_excl_u32(tot, s_w, &nvalid);
        if (threadIdx.x < R) s_start[threadIdx.x] = st;
        __syncthreads();
        constexpr int B = ITEMS < 8 ? ITEMS : ITEMS / 2;  // values in flight per thread
        static_assert(ITEMS % B == 0 && ITEMS % 2 == 0, "whole batches, ranks in pairs");
#pragma unroll
        for (int h = 0; h < ITEMS; h += B) {
            E e[B];
#pragma unroll
            for (int u = 0; u < B; ++u) {
                const int64_t i = i0 + (h + u) * 32;
                if (i >= hi) continue;
                if constexpr (FIRST) {
                    e[u] = make_elem<T, W>(__ldcs(P.a + i), W == 2 ? __ldcs(P.b + i) : T(0));
                } else {
                    e[u] = P.ein[i];
                }
            }
#pragma unroll
            for (int u = 0; u < B; ++u) {
                const int64_t i = i0 + (h + u) * 32;
                if (i >= hi) continue;
                const uint32_t k = key[h + u];
                const uint32_t d = (k >> P.shift) & dmask;
                const bool ok = (okm >> (h + u)) & 1u;
                const uint32_t within = my_cnt[d] + ((rk[(h + u) / 2] >> (16 * ((h + u) & 1))) & 0xffffu);
                if (ok) {
                    const uint32_t lpos = s_start[d] + within;
                    s_key[lpos] = k;
                    s_e[lpos] = e[u];
                }
                if (P.dest) __stcs(P.dest + i, ok ? s_off[d] + within : kNoKey);
            }
        }
        __syncthreads();
#pragma unroll 4
        for (int q = threadIdx.x; q < (int)nvalid; q += kSortBlock) {
            const uint32_t k = s_key[q];
            const uint32_t d = (k >> P.shift) & dmask;
            const uint32_t pos = s_off[d] + (uint32_t)q - s_start[d];
            P.kout[pos] = k;
            P.eout[pos] = s_e[q];
        }
        __syncthreads();
        if (threadIdx.x < R) s_off[threadIdx.x] += tot;
    }
}

// Inverse of one pass: out[i] = in[dest[i]] over the pass's input order, a block
// taking kUnsortTile consecutive i at a time (their places lie in at most 256
// runs, whose sectors stay in L1): 49 and 54 us for the two passes of 2^24 pairs,
// 92 and 111 us with the pair in two arrays and a grid-wide stride.  The first pass's inverse writes the caller's
// adjoints (0 or unchanged for an element that left the sort, += with
// accumulation).
constexpr int kUnsortTile = 8 * kSortBlock;
template <class T, int W, bool FIRST>
__global__ void __launch_bounds__(kSortBlock) hg_unsort_kernel(int64_t n, const uint32_t* nsorted,
                                                               const uint32_t* dest, const Elem<T, W>* in, T* oa,
                                                               T* ob, Elem<T, W>* out, int accumulate) {
    using E = Elem<T, W>;
    constexpr int U = 8;
    const int64_t len = FIRST ? n : (int64_t)*nsorted;
    for (int64_t t0 = blockIdx.x * (int64_t)kUnsortTile; t0 < len; t0 += gridDim.x * (int64_t)kUnsortTile) {
        const int64_t i0 = t0 + threadIdx.x;
        uint32_t d[U];
        E v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) d[u] = i0 + u * kSortBlock < len ? __ldcs(dest + i0 + u * kSortBlock) : kNoKey;
#pragma unroll
        for (int u = 0; u < U; ++u) v[u] = d[u] != kNoKey ? in[d[u]] : make_elem<T, W>(T(0), T(0));
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t i = i0 + u * kSortBlock;
            if (i >= len) continue;
            if constexpr (!FIRST) {
                out[i] = v[u];
            } else if (accumulate) {
                if (d[u] != kNoKey) {
                    oa[i] += v[u].a;
                    if constexpr (W == 2) ob[i] += v[u].b;
                }
            } else {
                __stcs(oa + i, v[u].a);
                if constexpr (W == 2) __stcs(ob + i, v[u].b);
            }
        }
    }
}

// ------------------------------------------------------ segmented scans
template <class Op>
struct SegS {
    typename Op::P x;
    uint32_t f;
};

template <class Op>
__device__ __forceinline__ SegS<Op> seg_id() {
    return SegS<Op>{Op::pid(), 0u};
}

// forward: f = a bin starts inside the right operand
template <class Op>
__device__ __forceinline__ SegS<Op> seg_fcomb(const SegS<Op>& l, const SegS<Op>& r) {
    return r.f ? r : SegS<Op>{Op::pcomb(l.x, r.x), l.f};
}

// reverse: e holds later elements, l earlier ones; f = a bin ends inside
template <class Op>
__device__ __forceinline__ SegS<Op> seg_rcomb(const SegS<Op>& e, const SegS<Op>& l) {
    return l.f ? l : SegS<Op>{Op::pcomb(l.x, e.x), e.f};
}

template <class Op, class T>
struct SegArgs {
    const uint32_t* keys;              // sorted bin numbers
    const Elem<T, Op::kWidth>* e;      // sorted values
    const uint32_t* nsorted;
    int64_t tiles;
    SegS<Op>* carry;       // [tiles] forward state before each tile
    unsigned long long* fA;
    unsigned long long* fI;
    unsigned long long* rA;
    unsigned long long* rI;
    WsHeader* hdr;
    const T* hsbar_a;
    const T* hsbar_b;
    Elem<T, Op::kWidth>* o;  // [n] adjoints in sorted order
    T* hs_a;
    T* hs_b;
};

__device__ __forceinline__ void ld_keys(const uint32_t* p, int64_t e, int64_t n, uint32_t (&o)[kSegV]) {
    if (e + kSegV <= n) {
        const uint4 x = __ldcs(reinterpret_cast<const uint4*>(p + e));
        o[0] = x.x; o[1] = x.y; o[2] = x.z; o[3] = x.w;
    } else {
#pragma unroll
        for (int j = 0; j < kSegV; ++j) o[j] = e + j < n ? p[e + j] : kNoKey;
    }
}

// kSegV consecutive elements' values (pads past n), and their store
template <class T, int W>
__device__ __forceinline__ void ld_elems(const Elem<T, W>* p, int64_t e, int64_t n, T pad, T (&a)[kSegV],
                                         T (&b)[kSegV]) {
    constexpr int VV = Vec16<T>::N;
    if (e + kSegV <= n) {
        const T* q = reinterpret_cast<const T*>(p + e);
        T f[W * kSegV];
#pragma unroll
        for (int c = 0; c < W * kSegV / VV; ++c) {
            const Vec16<T> x = ld_vec_stream(q + c * VV);
#pragma unroll
            for (int j = 0; j < VV; ++j) f[c * VV + j] = x.v[j];
        }
#pragma unroll
        for (int j = 0; j < kSegV; ++j) {
            a[j] = f[W * j];
            b[j] = W == 2 ? f[W * j + (W - 1)] : T(0);
        }
    } else {
#pragma unroll
        for (int j = 0; j < kSegV; ++j) {
            a[j] = e + j < n ? p[e + j].a : pad;
            b[j] = e + j < n ? elem_b(p[e + j]) : T(0);
        }
    }
}

template <class T, int W>
__device__ __forceinline__ void st_elems(Elem<T, W>* p, int64_t e, int64_t n, const T (&a)[kSegV],
                                         const T (&b)[kSegV]) {
    constexpr int VV = Vec16<T>::N;
    if (e + kSegV <= n) {
        T* q = reinterpret_cast<T*>(p + e);
        T f[W * kSegV];
#pragma unroll
        for (int j = 0; j < kSegV; ++j) {
            f[W * j] = a[j];
            if (W == 2) f[W * j + (W - 1)] = b[j];
        }
#pragma unroll
        for (int c = 0; c < W * kSegV / VV; ++c) {
            Vec16<T> x;
#pragma unroll
            for (int j = 0; j < VV; ++j) x.v[j] = f[c * VV + j];
            st_vec(q + c * VV, x);
        }
    } else {
#pragma unroll
        for (int j = 0; j < kSegV; ++j)
            if (e + j < n) p[e + j] = make_elem<T, W>(a[j], b[j]);
    }
}

// Forward pass: each tile's forward segmented state before its first
// element (the carry), by look-back.  HS (the forward operator alone): the
// states at the bins' last elements instead, into hs.
template <class Op, class T, bool HS>
__global__ void __launch_bounds__(kSegBlock) hg_seg_fwd_kernel(SegArgs<Op, T> A) {
    using S = SegS<Op>;
    constexpr int NW = kSegBlock / 32, K = kSegK, V = kSegV, W = Op::kWidth;
    __shared__ uint32_t s_tile;
    __shared__ S s_tot[K * NW];
    __shared__ S s_carry;
    if (threadIdx.x == 0) s_tile = atomicAdd(&A.hdr->ticket[0], 1u);
    __syncthreads();
    const int64_t t = s_tile;
    const int64_t ns = (int64_t)*A.nsorted;
    const int64_t base = t * kSegTile;
    uint32_t kk[K][V], kprev[K];
    T av[K][V], bv[K][V];
    S agg[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int64_t e = base + (int64_t)k * kSegBlock * V + threadIdx.x * V;
        ld_keys(A.keys, e, ns, kk[k]);
        ld_elems<T, W>(A.e, e, ns, Op::pad_a(), av[k], bv[k]);
        kprev[k] = (e > 0 && e - 1 < ns) ? A.keys[e - 1] : kNoKey;
        uint32_t prev = kprev[k];
        S acc = seg_id<Op>();
#pragma unroll
        for (int j = 0; j < V; ++j) {
            if (e + j < ns) acc = seg_fcomb<Op>(acc, S{Op::pelem(av[k][j], bv[k][j]), kk[k][j] != prev ? 1u : 0u});
            prev = kk[k][j];
        }
        agg[k] = acc;
    }
    auto fc = [](const S& l, const S& r) { return seg_fcomb<Op>(l, r); };
    S wex[K];
    const S total = block_scan_part1<S, false, K, NW>(agg, wex, s_tot, seg_id<Op>(), fc);
    if ((threadIdx.x >> 5) == 0) {
        LookbackState<S> st{A.fA, A.fI};
        const S pre = lookback(t, st, total, seg_id<Op>(), fc, A.hdr);
        if ((threadIdx.x & 31) == 0) {
            if (HS) s_carry = pre;
            else A.carry[t] = pre;
        }
    }
    if constexpr (HS) {
        __syncthreads();
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int64_t e = base + (int64_t)k * kSegBlock * V + threadIdx.x * V;
            if (e >= ns) continue;
            S lf = block_scan_excl<S, false, K, NW>(k, wex, s_tot, s_carry, fc);
            const uint32_t knext = e + V < ns ? A.keys[e + V] : kNoKey;
            uint32_t prev = kprev[k];
#pragma unroll
            for (int j = 0; j < V; ++j) {
                const uint32_t key = kk[k][j];
                lf = seg_fcomb<Op>(lf, S{Op::pelem(av[k][j], bv[k][j]), key != prev ? 1u : 0u});
                prev = key;
                const bool tail = e + j + 1 >= ns || (j + 1 < V ? kk[k][j + 1 < V ? j + 1 : j] : knext) != key;
                if (e + j < ns && tail) {
                    A.hs_a[key] = Op::out_a(lf.x);
                    if constexpr (W == 2) A.hs_b[key] = Op::out_b(lf.x);
                }
            }
        }
    }
}

// Reverse pass: tiles right to left.  l comes from the tile's carry and a
// forward block scan, r from a reverse block scan and a look-back over the
// tiles to the right; then the map of Sec. 5.1.2 and, at the first element
// of every bin, hs[bin] = a_first (.) r_first.
template <class Op, class T>
__global__ void __launch_bounds__(kSegBlock) hg_seg_bwd_kernel(SegArgs<Op, T> A) {
    using S = SegS<Op>;
    using P = typename Op::P;
    constexpr int NW = kSegBlock / 32, K = kSegK, V = kSegV, W = Op::kWidth;
    __shared__ uint32_t s_tile;
    __shared__ S s_totF[K * NW];
    __shared__ S s_totR[K * NW];
    __shared__ S s_carry;
    __shared__ S s_suf;
    if (threadIdx.x == 0) s_tile = atomicAdd(&A.hdr->ticket[1], 1u);
    __syncthreads();
    const int64_t t_log = s_tile;
    const int64_t tile = A.tiles - 1 - t_log;
    const int64_t ns = (int64_t)*A.nsorted;
    const int64_t base = tile * kSegTile;
    if (threadIdx.x == 0) s_carry = A.carry[tile];

    uint32_t kk[K][V], kprev[K], knext[K];
    T av[K][V], bv[K][V];
    S aggF[K], aggR[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int64_t e = base + (int64_t)k * kSegBlock * V + threadIdx.x * V;
        ld_keys(A.keys, e, ns, kk[k]);
        ld_elems<T, W>(A.e, e, ns, Op::pad_a(), av[k], bv[k]);
        kprev[k] = (e > 0 && e - 1 < ns) ? A.keys[e - 1] : kNoKey;
        knext[k] = (e + V < ns) ? A.keys[e + V] : kNoKey;
        S f = seg_id<Op>();
        uint32_t prev = kprev[k];
#pragma unroll
        for (int j = 0; j < V; ++j) {
            if (e + j < ns) f = seg_fcomb<Op>(f, S{Op::pelem(av[k][j], bv[k][j]), kk[k][j] != prev ? 1u : 0u});
            prev = kk[k][j];
        }
        aggF[k] = f;
        S r = seg_id<Op>();
        uint32_t next = knext[k];
#pragma unroll
        for (int j = V - 1; j >= 0; --j) {
            if (e + j < ns) r = seg_rcomb<Op>(r, S{Op::pelem(av[k][j], bv[k][j]), kk[k][j] != next ? 1u : 0u});
            next = kk[k][j];
        }
        aggR[k] = r;
    }
    auto fc = [](const S& l, const S& r) { return seg_fcomb<Op>(l, r); };
    auto rc = [](const S& e, const S& l) { return seg_rcomb<Op>(e, l); };
    S wexF[K], wexR[K];
    (void)block_scan_part1<S, false, K, NW>(aggF, wexF, s_totF, seg_id<Op>(), fc);
    const S totR = block_scan_part1<S, true, K, NW>(aggR, wexR, s_totR, seg_id<Op>(), rc);
    if ((threadIdx.x >> 5) == 0) {
        LookbackState<S> st{A.rA, A.rI};
        const S suf = lookback(t_log, st, totR, seg_id<Op>(), rc, A.hdr);
        if ((threadIdx.x & 31) == 0) s_suf = suf;
    }
    __syncthreads();

#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int64_t e = base + (int64_t)k * kSegBlock * V + threadIdx.x * V;
        if (e >= ns) continue;
        S lf = block_scan_excl<S, false, K, NW>(k, wexF, s_totF, s_carry, fc);
        P lx[V];
        uint32_t prev = kprev[k];
#pragma unroll
        for (int j = 0; j < V; ++j) {
            const bool head = kk[k][j] != prev;
            lx[j] = head ? Op::pid() : lf.x;
            lf = seg_fcomb<Op>(lf, S{Op::pelem(av[k][j], bv[k][j]), head ? 1u : 0u});
            prev = kk[k][j];
        }
        S rr = block_scan_excl<S, true, K, NW>(k, wexR, s_totR, s_suf, rc);
        uint32_t next = knext[k];
        T oa[V], ob[V];
#pragma unroll
        for (int j = V - 1; j >= 0; --j) {
            const uint32_t key = kk[k][j];
            const bool tail = key != next;
            next = key;
            oa[j] = T(0);
            ob[j] = T(0);
            if (e + j >= ns) continue;
            const P rx = tail ? Op::pid() : rr.x;
            const T ya = A.hsbar_a[key];
            const T yb = W == 2 ? A.hsbar_b[key] : T(0);
            Op::mid_vjp(lx[j], av[k][j], bv[k][j], rx, ya, yb, oa[j], ob[j]);
            const bool head = j > 0 ? kk[k][j - 1] != key : kprev[k] != key;
            if (head && A.hs_a) {
                const P y = Op::pcomb(Op::pelem(av[k][j], bv[k][j]), rx);
                A.hs_a[key] = Op::out_a(y);
                if constexpr (W == 2) A.hs_b[key] = Op::out_b(y);
            }
            rr = seg_rcomb<Op>(rr, S{Op::pelem(av[k][j], bv[k][j]), tail ? 1u : 0u});
        }
        st_elems<T, W>(A.o, e, ns, oa, ob);
    }
}

// hs of a bin without elements is the neutral element
template <class Op, class T>
__global__ void hg_fill_kernel(int64_t m, T* hs_a, T* hs_b) {
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < m; k += (int64_t)gridDim.x * blockDim.x) {
        hs_a[k] = Op::out_a(Op::pid());
        if constexpr (Op::kWidth == 2) hs_b[k] = Op::out_b(Op::pid());
    }
}

// ------------------------------------------------------------ host side
constexpr int kMaxPasses = 4;  // 31 key bits in passes of at most 8

struct HgLayout {
    size_t off_cnt, off_rowtot, off_k[2], off_e[2], off_dest[kMaxPasses], off_carry, off_slots;
    size_t slot_bytes, total;
    int64_t tiles;
};

int key_bits(int64_t m) {
    int bits = 1;
    while (bits < 31 && ((int64_t)1 << bits) < m) ++bits;
    return bits;
}

template <class Op, class T>
HgLayout hg_layout(int64_t n, int64_t m) {
    using S = SegS<Op>;
    HgLayout L{};
    const size_t nn = (size_t)(n > 0 ? n : 1);
    size_t o = sizeof(WsHeader);
    auto take = [&](size_t bytes) {
        const size_t at = o;
        o = round_up(o + bytes, 256);
        return at;
    };
    L.off_cnt = take(sizeof(uint32_t) * kRadix * kSortMaxGrid);
    L.off_rowtot = take(sizeof(uint32_t) * kRadix);
    for (int q = 0; q < 2; ++q) {
        L.off_k[q] = take(sizeof(uint32_t) * nn);
        L.off_e[q] = take(sizeof(Elem<T, Op::kWidth>) * nn);
    }
    const int passes = (key_bits(m) + kRadixBits - 1) / kRadixBits;
    for (int p = 0; p < passes; ++p) L.off_dest[p] = take(sizeof(uint32_t) * nn);
    L.tiles = (n + kSegTile - 1) / kSegTile;
    if (L.tiles < 1) L.tiles = 1;
    L.off_carry = take(sizeof(S) * (size_t)L.tiles);
    L.slot_bytes = 4 * sizeof(unsigned long long) * (size_t)lb_words<S>() * (size_t)L.tiles;
    L.off_slots = take(L.slot_bytes);
    L.total = o;
    return L;
}

int sms_now() {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms > 0 ? sms : 1;
}

// the sort's passes with tiles of ITEMS elements per thread; the sorted data end
// up in buffer (passes & 1)
template <class T, int W, class I, int ITEMS>
int run_sort(SortPass<T, W> SP, char* w, const size_t (&off_k)[2], const size_t (&off_e)[2], const size_t* off_dest,
             bool keep_dest, uint32_t* nsorted, int passes, int bits, cudaStream_t s) {
    constexpr int kTile = kSortBlock * ITEMS;
    constexpr size_t smem = sort_smem<T, W, ITEMS>();
    auto first = hg_scatter_kernel<I, T, W, true, ITEMS>;
    auto later = hg_scatter_kernel<I, T, W, false, ITEMS>;
    if (cudaFuncSetAttribute(first, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        cudaFuncSetAttribute(later, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return ADPAR_ERR_CUDA;
    const int dbits = (bits + passes - 1) / passes;
    // one wave of the scatter kernel (two blocks per SM): every block's chunk is in flight at once
    const int G = (int)std::max<int64_t>(
        1, std::min<int64_t>({(SP.n + kTile - 1) / kTile, (int64_t)kSortMaxGrid, (int64_t)sms_now() * 2}));
    SP.G = G;
    for (int p = 0; p < passes; ++p) {
        const int src = p & 1, dst = (p + 1) & 1;
        SP.shift = p * dbits;
        SP.bits = std::min(dbits, bits - p * dbits);
        SP.kin = reinterpret_cast<const uint32_t*>(w + off_k[src]);
        SP.ein = reinterpret_cast<const Elem<T, W>*>(w + off_e[src]);
        SP.kout = reinterpret_cast<uint32_t*>(w + off_k[dst]);
        SP.eout = reinterpret_cast<Elem<T, W>*>(w + off_e[dst]);
        SP.dest = keep_dest ? reinterpret_cast<uint32_t*>(w + off_dest[p]) : nullptr;
        if (p == 0) {
            hg_count_kernel<I, T, W, true><<<G, kSortBlock, 0, s>>>(SP, kTile);
            hg_scan_counts_kernel<<<1 << SP.bits, kSortBlock, 0, s>>>(SP.cnt, SP.rowtot, G, nsorted);
            first<<<G, kSortBlock, smem, s>>>(SP);
        } else {
            hg_count_kernel<I, T, W, false><<<G, kSortBlock, 0, s>>>(SP, kTile);
            hg_scan_counts_kernel<<<1 << SP.bits, kSortBlock, 0, s>>>(SP.cnt, SP.rowtot, G, nullptr);
            later<<<G, kSortBlock, smem, s>>>(SP);
        }
    }
    return ADPAR_OK;
}

// abar NULL: the forward operator alone (hs_a given)
template <class Op, class T, class I>
int run_hist_general(int64_t n, int64_t m, const void* a, const void* b, const void* inds, const void* hsbar_a,
                     const void* hsbar_b, void* abar, void* bbar, void* hs_a, void* hs_b, uint32_t flags,
                     void* work, size_t work_bytes, cudaStream_t s) {
    using S = SegS<Op>;
    constexpr int W = Op::kWidth;
    using E = Elem<T, W>;
    const HgLayout L = hg_layout<Op, T>(n, m);
    if (work == nullptr || work_bytes < L.total || (reinterpret_cast<uintptr_t>(work) & 255u))
        return ADPAR_ERR_WORKSPACE;
    char* w = static_cast<char*>(work);
    WsHeader* hdr = reinterpret_cast<WsHeader*>(w);
    if (cudaMemsetAsync(hdr, 0, sizeof(WsHeader), s) != cudaSuccess) return ADPAR_ERR_CUDA;
    if (hs_a && m > 0) {
        const int blocks = (int)std::min<int64_t>((m + 255) / 256, 4096);
        hg_fill_kernel<Op, T><<<blocks, 256, 0, s>>>(m, static_cast<T*>(hs_a), static_cast<T*>(hs_b));
    }
    if (n == 0) return cudaGetLastError() == cudaSuccess ? ADPAR_OK : ADPAR_ERR_CUDA;
    if (cudaMemsetAsync(w + L.off_slots, 0, L.slot_bytes, s) != cudaSuccess) return ADPAR_ERR_CUDA;

    // key bits: bin numbers are below m (out-of-range elements leave in pass 0)
    const int bits = key_bits(m);
    const int passes = (bits + kRadixBits - 1) / kRadixBits;
    uint32_t* nsorted = &hdr->done[0];
    SortPass<T, W> SP{};
    SP.n = n;
    SP.m = m;
    SP.inds = inds;
    SP.a = static_cast<const T*>(a);
    SP.b = static_cast<const T*>(b);
    SP.cnt = reinterpret_cast<uint32_t*>(w + L.off_cnt);
    SP.rowtot = reinterpret_cast<uint32_t*>(w + L.off_rowtot);
    SP.nsorted = nsorted;
    const bool vjp = abar != nullptr;
    const int st = n >= kBigSort ? run_sort<T, W, I, big_items<T, W>()>(SP, w, L.off_k, L.off_e, L.off_dest, vjp,
                                                                        nsorted, passes, bits, s)
                                 : run_sort<T, W, I, kSmallItems>(SP, w, L.off_k, L.off_e, L.off_dest, vjp, nsorted,
                                                                  passes, bits, s);
    if (st != ADPAR_OK) return st;
    // the sorted data sit in buffer fin; the other buffer takes the
    // sorted-order adjoints, and the inverse passes alternate between them
    const int fin = passes & 1;
    const size_t wd = (size_t)lb_words<S>() * (size_t)L.tiles;
    unsigned long long* slots = reinterpret_cast<unsigned long long*>(w + L.off_slots);
    SegArgs<Op, T> A{};
    A.keys = reinterpret_cast<const uint32_t*>(w + L.off_k[fin]);
    A.e = reinterpret_cast<const E*>(w + L.off_e[fin]);
    A.nsorted = nsorted;
    A.tiles = L.tiles;
    A.carry = reinterpret_cast<S*>(w + L.off_carry);
    A.fA = slots;
    A.fI = slots + wd;
    A.rA = slots + 2 * wd;
    A.rI = slots + 3 * wd;
    A.hdr = hdr;
    A.hsbar_a = static_cast<const T*>(hsbar_a);
    A.hsbar_b = static_cast<const T*>(hsbar_b);
    A.o = reinterpret_cast<E*>(w + L.off_e[1 - fin]);
    A.hs_a = static_cast<T*>(hs_a);
    A.hs_b = static_cast<T*>(hs_b);
    if (!vjp) {
        hg_seg_fwd_kernel<Op, T, true><<<(unsigned)L.tiles, kSegBlock, 0, s>>>(A);
        return cudaGetLastError() == cudaSuccess ? ADPAR_OK : ADPAR_ERR_CUDA;
    }
    hg_seg_fwd_kernel<Op, T, false><<<(unsigned)L.tiles, kSegBlock, 0, s>>>(A);
    hg_seg_bwd_kernel<Op, T><<<(unsigned)L.tiles, kSegBlock, 0, s>>>(A);
    const int acc = (flags & ADPAR_ACCUMULATE) ? 1 : 0;
    const int ublocks =
        (int)std::max<int64_t>(1, std::min<int64_t>((n + kUnsortTile - 1) / kUnsortTile, (int64_t)sms_now() * 16));
    int cur = 1 - fin;
    for (int p = passes - 1; p >= 0; --p) {
        const uint32_t* dest = reinterpret_cast<const uint32_t*>(w + L.off_dest[p]);
        const E* in = reinterpret_cast<const E*>(w + L.off_e[cur]);
        if (p == 0) {
            hg_unsort_kernel<T, W, true><<<ublocks, kSortBlock, 0, s>>>(n, nsorted, dest, in, static_cast<T*>(abar),
                                                                       static_cast<T*>(bbar), nullptr, acc);
        } else {
            hg_unsort_kernel<T, W, false><<<ublocks, kSortBlock, 0, s>>>(
                n, nsorted, dest, in, nullptr, nullptr, reinterpret_cast<E*>(w + L.off_e[1 - cur]), acc);
            cur = 1 - cur;
        }
    }
    return cudaGetLastError() == cudaSuccess ? ADPAR_OK : ADPAR_ERR_CUDA;
}

template <class T, class I>
int dispatch_hist_general(int op, int64_t n, int64_t m, const void* a, const void* b, const void* inds,
                          const void* ya, const void* yb, void* abar, void* bbar, void* hs_a, void* hs_b,
                          uint32_t flags, void* work, size_t wb, cudaStream_t s) {
    switch (op) {
    case ADPAR_OP_ADD:
        return run_hist_general<OpAdd<T>, T, I>(n, m, a, b, inds, ya, yb, abar, bbar, hs_a, hs_b, flags, work, wb, s);
    case ADPAR_OP_MUL:
        return run_hist_general<OpMul<T>, T, I>(n, m, a, b, inds, ya, yb, abar, bbar, hs_a, hs_b, flags, work, wb, s);
    case ADPAR_OP_MIN:
        return run_hist_general<OpMin<T>, T, I>(n, m, a, b, inds, ya, yb, abar, bbar, hs_a, hs_b, flags, work, wb, s);
    case ADPAR_OP_MAX:
        return run_hist_general<OpMax<T>, T, I>(n, m, a, b, inds, ya, yb, abar, bbar, hs_a, hs_b, flags, work, wb, s);
    case ADPAR_OP_LINREC:
        return run_hist_general<OpLinrec<T>, T, I>(n, m, a, b, inds, ya, yb, abar, bbar, hs_a, hs_b, flags, work, wb,
                                                   s);
    }
    return ADPAR_ERR_INVALID;
}

template <class T>
size_t layout_total(int op, int64_t n, int64_t m) {
    switch (op) {
    case ADPAR_OP_ADD: return hg_layout<OpAdd<T>, T>(n, m).total;
    case ADPAR_OP_MUL: return hg_layout<OpMul<T>, T>(n, m).total;
    case ADPAR_OP_MIN: return hg_layout<OpMin<T>, T>(n, m).total;
    case ADPAR_OP_MAX: return hg_layout<OpMax<T>, T>(n, m).total;
    case ADPAR_OP_LINREC: return hg_layout<OpLinrec<T>, T>(n, m).total;
    }
    return (size_t)-1;
}

}  // namespace

size_t hist_general_workspace_size(adpar_opdesc d, int64_t n, int64_t m) {
    if (n < 0 || m < 0 || d.op < ADPAR_OP_ADD || d.op > ADPAR_OP_LINREC) return (size_t)-1;
    if (d.dtype == ADPAR_F32) return layout_total<float>(d.op, n, m);
    if (d.dtype == ADPAR_F64) return layout_total<double>(d.op, n, m);
    return (size_t)-1;
}

}  // namespace adpar

namespace adpar {
namespace {
int hist_general_impl(adpar_opdesc d, int64_t n, int64_t m, const void* a, const void* b, const void* inds, int itype,
                      const void* hsbar_a, const void* hsbar_b, void* abar, void* bbar, void* hs_a, void* hs_b,
                      uint32_t flags, void* work, size_t work_bytes, void* stream, bool primal_only) {
    if (n < 0 || m < 0) return ADPAR_ERR_INVALID;
    if (d.op < ADPAR_OP_ADD || d.op > ADPAR_OP_LINREC) return ADPAR_ERR_INVALID;
    if (d.dtype != ADPAR_F32 && d.dtype != ADPAR_F64) return ADPAR_ERR_INVALID;
    if (itype != ADPAR_I32 && itype != ADPAR_I64) return ADPAR_ERR_INVALID;
    const int want_w = d.op == ADPAR_OP_LINREC ? 2 : 1;
    if (d.width != want_w) return ADPAR_ERR_INVALID;
    if (flags & ~(uint32_t)ADPAR_ACCUMULATE) return ADPAR_ERR_UNSUPPORTED;
    // positions and bin numbers travel as 32-bit words
    if (n >= (int64_t)0xffffffffu || m > ((int64_t)1 << 31)) return ADPAR_ERR_UNSUPPORTED;
    if (want_w == 2 && hs_a && !hs_b) return ADPAR_ERR_INVALID;
    if (hs_a == nullptr && hs_b != nullptr) return ADPAR_ERR_INVALID;
    if (primal_only) {
        if ((m > 0 && (!hs_a || (want_w == 2 && !hs_b))) || (n > 0 && (!a || !inds || (want_w == 2 && !b))))
            return ADPAR_ERR_INVALID;
    } else if (n > 0) {
        if (!a || !inds || !abar || (m > 0 && !hsbar_a)) return ADPAR_ERR_INVALID;
        if (want_w == 2 && (!b || !bbar || (m > 0 && !hsbar_b))) return ADPAR_ERR_INVALID;
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (d.dtype == ADPAR_F32) {
        if (itype == ADPAR_I32)
            return dispatch_hist_general<float, int32_t>(d.op, n, m, a, b, inds, hsbar_a, hsbar_b, abar, bbar, hs_a,
                                                         hs_b, flags, work, work_bytes, s);
        return dispatch_hist_general<float, int64_t>(d.op, n, m, a, b, inds, hsbar_a, hsbar_b, abar, bbar, hs_a, hs_b,
                                                     flags, work, work_bytes, s);
    }
    if (itype == ADPAR_I32)
        return dispatch_hist_general<double, int32_t>(d.op, n, m, a, b, inds, hsbar_a, hsbar_b, abar, bbar, hs_a,
                                                      hs_b, flags, work, work_bytes, s);
    return dispatch_hist_general<double, int64_t>(d.op, n, m, a, b, inds, hsbar_a, hsbar_b, abar, bbar, hs_a, hs_b,
                                                  flags, work, work_bytes, s);
}
}  // namespace
}  // namespace adpar

extern "C" int adpar_vjp_hist_general(adpar_opdesc d, int64_t n, int64_t m, const void* a, const void* b,
                                      const void* inds, int itype, const void* hsbar_a, const void* hsbar_b,
                                      void* abar, void* bbar, void* hs_a, void* hs_b, uint32_t flags, void* work,
                                      size_t work_bytes, void* stream) {
    return adpar::hist_general_impl(d, n, m, a, b, inds, itype, hsbar_a, hsbar_b, abar, bbar, hs_a, hs_b, flags, work,
                                    work_bytes, stream, false);
}

extern "C" int adpar_hist_general(adpar_opdesc d, int64_t n, int64_t m, const void* a, const void* b, const void* inds,
                                  int itype, void* hs_a, void* hs_b, void* work, size_t work_bytes, void* stream) {
    return adpar::hist_general_impl(d, n, m, a, b, inds, itype, nullptr, nullptr, nullptr, nullptr, hs_a, hs_b, 0u,
                                    work, work_bytes, stream, true);
}
