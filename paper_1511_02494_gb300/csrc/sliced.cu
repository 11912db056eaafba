// SLICED variant (V7): sliced ELL layout, the GPU form of the paper's
// bandwidth (MB) and latency (CML) optimizations on this machine.
//
// Rows are grouped in slices of 32; inside a slice the k-th elements of the
// 32 rows are stored next to each other (column-major), so one lane per row
// reads 32 consecutive values and 32 consecutive column indices per load and
// issues 32 independent gathers of x per instruction.  There is no
// reduction across lanes: each row's sum is one chain of DFMAs in row order,
// so the FP64 pipe spends exactly one instruction slot per element of the
// slice (the CSR kernels with T lanes per row add log2(T) shuffle-adds per
// row, 28 % more FP64 slots on a 27-point stencil).  Lanes whose row is
// shorter than the slice skip the padded slots (the loads and DFMAs are
// predicated), so padding costs issue slots but no memory traffic.
//
// Optionally (sigma > 1) rows are sorted by length, longest first, inside
// windows of sigma rows, so that a slice holds rows of similar length; y is
// then written through the permutation.  Rows longer than a cap are not
// put in slices (their slot has length -1); they are split into segments of
// kSlicedSeg nonzeros computed by one warp each from the CSR arrays, and a
// fix-up adds each such row's segment sums in order.  The layout is that of the oracle's orc_sliced_layout
// and orc_sliced_fill, bit for bit.
#include <cuda_bf16.h>

#include <algorithm>
#include <utility>
#include <vector>

#include "common.cuh"
#include "ptx.cuh"
#include "rowdot.cuh"
#include "sliced.cuh"

namespace spmvlib {
namespace {

using namespace dev;
constexpr int kSB = 256;       // threads per block: 8 slices

// ---- layout (prepare) --------------------------------------------------------
// What the layout kernels find out about the matrix; the scan writes it to
// page-locked host memory, so that a layout costs one wait and no copy.
struct SlStats {
    unsigned long long slots;   // sum of 32 x slice length: padding by unequal rows only
    unsigned long long tot;     // element slots (slices rounded up to `vec` elements a row)
    unsigned n_long, n_seg, n_fix;
    int longest;                // longest slice
    unsigned shortest_c;        // maximum of ~length over the rows
    unsigned reach;             // columns ahead of the diagonal (sampled), then the column-width questions' answers
};
// The slices are cut into at most kTiles tiles of equal length (whole sort
// windows); per tile the element slots and the long rows, their segments and
// those with several segments.  A tile's place is the sum of the tiles before
// it, which every block of the next kernel forms for itself: no block waits
// for another.
constexpr int kTiles = 1024;
struct SlTile {
    unsigned long long len;
    unsigned n_long, n_seg, n_fix, pad;
};
struct SlScratch {
    SlStats stats;
    SlTile tile[kTiles];
};

// a thread's share of a tile
struct TileAcc {
    unsigned long long len = 0, slots = 0;
    unsigned n_long = 0, n_seg = 0, n_fix = 0, shortest_c = 0, reach = 0;
    int longest = 0;

    // one row: its length in the slices, -1 when it is long
    __device__ __forceinline__ int row(int n, int cap) {
        if (n > cap) {
            ++n_long;
            n_seg += (unsigned)(n + kSlicedSeg - 1) / kSlicedSeg;
            n_fix += n > kSlicedSeg;
            n = -1;
        }
        shortest_c = max(shortest_c, ~(unsigned)n);
        return n;
    }
    // one slice (called by one lane)
    __device__ __forceinline__ void slice(int m, int vec) {
        len += 32ull * (unsigned)((m + vec - 1) / vec * vec);
        slots += 32ull * (unsigned)m;
        longest = max(longest, m);
    }
    // adds the block's share to its tile and to the totals
    __device__ __forceinline__ void flush(SlScratch* w, int64_t tile) {
        __shared__ SlTile t;
        __shared__ SlStats g;
        if (threadIdx.x == 0) { t = SlTile{}; g = SlStats{}; }
        __syncthreads();
        const unsigned nl = __reduce_add_sync(FULL, n_long), ns = __reduce_add_sync(FULL, n_seg),
                       nf = __reduce_add_sync(FULL, n_fix), sc = __reduce_max_sync(FULL, shortest_c), re = __reduce_max_sync(FULL, reach);
        const int lo = __reduce_max_sync(FULL, longest);
        unsigned long long l = len, q = slots;
        for (int o = 16; o > 0; o >>= 1) {
            l += __shfl_xor_sync(FULL, l, o);
            q += __shfl_xor_sync(FULL, q, o);
        }
        if ((threadIdx.x & 31) == 0) {
            atomicAdd(&t.len, l);
            atomicAdd(&g.slots, q);
            atomicMax(&g.longest, lo);
            atomicMax(&g.shortest_c, sc);
            if (re) atomicMax(&g.reach, re);
            if (nl) { atomicAdd(&t.n_long, nl); atomicAdd(&t.n_seg, ns); atomicAdd(&t.n_fix, nf); }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            SlTile* T = w->tile + tile;
            SlStats* S = &w->stats;
            atomicAdd(&T->len, t.len);
            atomicAdd(&S->slots, g.slots);
            atomicMax(&S->longest, g.longest);
            atomicMax(&S->shortest_c, g.shortest_c);
            if (g.reach) atomicMax(&S->reach, g.reach);
            if (t.n_long) {
                atomicAdd(&T->n_long, t.n_long); atomicAdd(&T->n_seg, t.n_seg); atomicAdd(&T->n_fix, t.n_fix);
                atomicAdd(&S->n_long, t.n_long); atomicAdd(&S->n_seg, t.n_seg); atomicAdd(&S->n_fix, t.n_fix);
            }
        }
    }
};

// Rows in order: row lengths and slice lengths, a block per tile, a warp per
// slice, four slices' row pointers in flight.
__global__ void __launch_bounds__(kSB)
k_sl_layout(int64_t n_rows, int64_t n_cols, int64_t nnz, int64_t n_slices, const int* __restrict__ rp,
            const int* __restrict__ ci, int cap, int vec, int64_t tile_slices,
            int* __restrict__ rowlen, int* __restrict__ slice_len, SlScratch* __restrict__ w)
{
    constexpr int U = 4;
    const int lane = threadIdx.x & 31;
    const int64_t t0 = blockIdx.x * tile_slices, t1 = min(n_slices, t0 + tile_slices);
    const float ahead = (float)n_cols / (float)n_rows;
    TileAcc acc;
    for (int64_t s0 = t0 + (threadIdx.x >> 5) * U; s0 < t1; s0 += (kSB / 32) * U) {
        int b[U], e[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t row = (s0 + u) * 32 + lane;
            const bool in = s0 + u < t1 && row < n_rows;
            b[u] = in ? rp[row] : 0;
            e[u] = in ? rp[row + 1] : 0;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (s0 + u >= t1) break;  // whole warps
            const int64_t p = (s0 + u) * 32 + lane;
            const int n = p < n_rows ? acc.row(e[u] - b[u], cap) : -1;
            rowlen[p] = n;
            const int m = __reduce_max_sync(FULL, max(n, 0));
            if (lane == 0) {
                slice_len[s0 + u] = m;
                acc.slice(m, vec);
                // how far ahead of the corner-to-corner diagonal the slice's
                // first row reaches (the matrix need not be a valid one yet)
                if (b[u] >= 0 && e[u] > b[u] && e[u] <= nnz) {
                    const int64_t over = (int64_t)__ldg(ci + e[u] - 1) - (int64_t)((float)p * ahead);
                    acc.reach = max(acc.reach, (unsigned)max((int64_t)0, min(over, (int64_t)INT32_MAX)));
                }
            }
        }
    }
    acc.flush(w, blockIdx.x);
}

// Rows sorted by length inside windows of sigma rows (a power of two,
// 32..4096), longest first, ties by row index, long rows as of length 0: a
// block per window, four rows per thread.  A stable radix sort of (longest -
// length, index) in 5-bit digits over only the bits that the window's lengths
// differ in -- one pass for a stencil's rows, two for a cap of 32 -- ranks by
// warp votes (a warp owns 128 consecutive places) and a scan over (digit,
// warp).  A bitonic sort of 64-bit keys, 78 steps with a block barrier each,
// took 70 us for 1M rows in windows of 4096; this takes 17.6.
constexpr int kSortItems = 4;
constexpr int kSortMax = 4096;
__global__ void __launch_bounds__(kSortMax / kSortItems)
k_sl_sort(int64_t n_rows, int64_t n_slices, const int* __restrict__ rp, int sigma, int cap, int vec,
          int64_t tile_slices, int* __restrict__ perm, int* __restrict__ rowlen, int* __restrict__ slice_len,
          SlScratch* __restrict__ w)
{
    __shared__ unsigned buf[kSortMax];
    __shared__ unsigned hist[kSortMax / kSortItems / 32][32];
    __shared__ unsigned warp_sum[32];
    __shared__ unsigned s_max, s_min;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    const int64_t w0 = (int64_t)blockIdx.x * sigma;
    TileAcc acc;
    if (threadIdx.x == 0) { s_max = 0; s_min = 0xffffffffu; }
    __syncthreads();
    // place i of the window: warp * 128 + 32 u + lane
    unsigned klen[kSortItems], lo = 0xffffffffu, hi = 0;
#pragma unroll
    for (int u = 0; u < kSortItems; ++u) {
        const int i = warp * 128 + u * 32 + lane;
        klen[u] = 0xffffffffu;  // no row
        if (i < sigma && w0 + i < n_rows) {
            const int n = acc.row(rp[w0 + i + 1] - rp[w0 + i], cap);
            klen[u] = (unsigned)max(n, 0);
            lo = min(lo, klen[u]);
            hi = max(hi, klen[u]);
        }
    }
    lo = __reduce_min_sync(FULL, lo);
    hi = __reduce_max_sync(FULL, hi);
    if (lane == 0) { atomicMin(&s_min, lo); atomicMax(&s_max, hi); }
    __syncthreads();
    const unsigned longest = s_max, none = longest - min(s_min, longest) + 1;  // places without a row sort last
    const int bits = 32 - __clz((int)none);
    unsigned val[kSortItems];  // key << 12 | index in the window
#pragma unroll
    for (int u = 0; u < kSortItems; ++u) {
        const int i = warp * 128 + u * 32 + lane;
        val[u] = ((klen[u] == 0xffffffffu ? none : longest - klen[u]) << 12) | (unsigned)i;
    }
    for (int shift = 12; shift < 12 + bits; shift += 5) {
        hist[warp][lane] = 0;
        __syncwarp();
        unsigned rank[kSortItems];
#pragma unroll
        for (int u = 0; u < kSortItems; ++u) {
            const bool in = warp * 128 + u * 32 < sigma;  // whole warps
            if (in) {
                const unsigned digit = (val[u] >> shift) & 31u;
                const unsigned peers = __match_any_sync(FULL, digit);
                const unsigned before = hist[warp][digit];
                rank[u] = before + __popc(peers & ((1u << lane) - 1u));
                __syncwarp();
                if ((peers & ((1u << lane) - 1u)) == 0) hist[warp][digit] = before + __popc(peers);
                __syncwarp();
            }
        }
        __syncthreads();
        // exclusive scan over (digit, warp), an entry per thread
        const int e_digit = threadIdx.x / n_warps, e_warp = threadIdx.x % n_warps;
        const unsigned own = hist[e_warp][e_digit];
        unsigned incl = own;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned t = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) warp_sum[warp] = incl;
        __syncthreads();
        unsigned base = 0;
        for (int k = 0; k < warp; ++k) base += warp_sum[k];
        hist[e_warp][e_digit] = base + incl - own;
        __syncthreads();
#pragma unroll
        for (int u = 0; u < kSortItems; ++u)
            if (warp * 128 + u * 32 < sigma) buf[hist[warp][(val[u] >> shift) & 31u] + rank[u]] = val[u];
        __syncthreads();
#pragma unroll
        for (int u = 0; u < kSortItems; ++u)
            if (warp * 128 + u * 32 < sigma) val[u] = buf[warp * 128 + u * 32 + lane];
    }
#pragma unroll
    for (int u = 0; u < kSortItems; ++u) {
        const int i = warp * 128 + u * 32;
        const int64_t p = w0 + i + lane;
        if (i >= sigma || p - lane >= 32 * n_slices) continue;  // whole warps
        int n = -1;
        if (p < n_rows) {
            const int64_t r = w0 + (val[u] & 4095u);
            n = (int)(longest - (val[u] >> 12));
            if (n == 0 && rp[r + 1] - rp[r] > cap) n = -1;
            perm[p] = (int)r;
        }
        rowlen[p] = n;
        const int m = __reduce_max_sync(FULL, max(n, 0));
        if (lane == 0) {
            slice_len[p / 32] = m;
            acc.slice(m, vec);
        }
    }
    acc.flush(w, w0 / 32 / tile_slices);
}

// sums over the tiles before this block's: element slots, long rows,
// segments, rows with several segments (valid in every thread)
__device__ __forceinline__ SlTile tiles_before(const SlScratch* __restrict__ w)
{
    __shared__ SlTile t;
    if (threadIdx.x == 0) t = SlTile{};
    __syncthreads();
    unsigned long long l = 0;
    unsigned nl = 0, ns = 0, nf = 0;
    for (int k = threadIdx.x; k < (int)blockIdx.x; k += kSB) {
        l += w->tile[k].len;
        nl += w->tile[k].n_long;
        ns += w->tile[k].n_seg;
        nf += w->tile[k].n_fix;
    }
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(FULL, l, o);
    nl = __reduce_add_sync(FULL, nl);
    ns = __reduce_add_sync(FULL, ns);
    nf = __reduce_add_sync(FULL, nf);
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&t.len, l);
        atomicAdd(&t.n_long, nl);
        atomicAdd(&t.n_seg, ns);
        atomicAdd(&t.n_fix, nf);
    }
    __syncthreads();
    return t;
}

// block-wide exclusive scan of one value per thread (below 2^31 in total)
__device__ __forceinline__ unsigned block_scan(unsigned v, unsigned* total)
{
    __shared__ unsigned part[kSB / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned incl = v;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned t = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += t;
    }
    __syncthreads();  // part may still be read from the scan before
    if (lane == 31) part[warp] = incl;
    __syncthreads();
    unsigned base = 0, all = 0;
    for (int k = 0; k < kSB / 32; ++k) {
        if (k < warp) base += part[k];
        all += part[k];
    }
    *total = all;
    return base + incl - v;
}

// slice starts from the slice lengths, a block per tile; the last block also
// hands the totals to the host
__global__ void __launch_bounds__(kSB)
k_sl_scan(int64_t n_slices, int64_t tile_slices, int vec, const int* __restrict__ slice_len,
          int64_t* __restrict__ slice_ptr, const SlScratch* __restrict__ w, SlStats* __restrict__ host)
{
    int64_t at = (int64_t)tiles_before(w).len;
    const int64_t t0 = blockIdx.x * tile_slices, t1 = min(n_slices, t0 + tile_slices);
    for (int64_t s0 = t0; s0 < t1; s0 += kSB) {
        const int64_t s = s0 + threadIdx.x;
        const unsigned n = s < t1 ? 32u * (unsigned)((slice_len[s] + vec - 1) / vec * vec) : 0u;
        unsigned all;
        const unsigned before = block_scan(n, &all);
        if (s < t1) slice_ptr[s] = at + before;
        at += all;
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) {
        slice_ptr[n_slices] = at;
        SlStats t = w->stats;
        t.tot = (unsigned long long)at;
        *host = t;
    }
}

// Contents of the slices.  A warp per slice reads its rows' elements with T
// lanes per row (T the power of two that covers the chunk's longest row, at
// most 8), so that a load instruction covers runs of the CSR arrays, straight
// into shared memory (cp.async, no registers held), turned around there (rows
// of 33: no bank conflicts), and writes the chunk column-major, padding
// included: every slot is written, so nothing is zeroed beforehand.  `Out`
// writes the elements of one lane's row in row order, `vec` at a time.
// Bound by HBM: 108 us for a 100^3 27-point stencil (26.5 M nonzeros, 5.9
// TB/s).  A lane per row, as the SpMV walks them, reads 32 places per
// instruction; that and the memsets took 132 + 57 us.  Chunks of 16 or 32
// elements leave fewer blocks resident (125 us either way), 40 registers a
// thread for 48 warps spill (114 us), and warps striding over the slices with
// the next header loaded ahead are slower than many short blocks (138 us).
constexpr int kFillK = 8, kFillWarps = 4;
template <int B>
__device__ __forceinline__ void cp_async(void* dst, const void* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;"
                 :: "r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src), "n"(B) : "memory");
}
template <typename Out>
__global__ void __launch_bounds__(32 * kFillWarps)
k_sl_fill(int64_t n_slices, const int* __restrict__ rp, const int* __restrict__ ci, const double* __restrict__ v,
          const int* __restrict__ perm, const int* __restrict__ rowlen, const int* __restrict__ slice_len,
          const int64_t* __restrict__ slice_ptr, Out out)
{
    __shared__ int s_col[kFillWarps][kFillK * 33];
    __shared__ double s_val[kFillWarps][kFillK * 33];
    const int lane = threadIdx.x & 31;
    int* tc = s_col[threadIdx.x >> 5];
    double* tv = s_val[threadIdx.x >> 5];
    const int64_t s = (int64_t)blockIdx.x * kFillWarps + (threadIdx.x >> 5);
    if (s >= n_slices) return;  // whole warps
    const int64_t p = s * 32 + lane;
    const int len = max(rowlen[p], 0);
    const int r = len > 0 ? (perm ? perm[p] : (int)p) : 0;
    const int b = len > 0 ? rp[r] : 0;
    const int L = slice_len[s], Lp = (L + Out::vec - 1) / Out::vec * Out::vec;
    const int64_t q0 = slice_ptr[s];
    typename Out::Row row;
    out.begin(row, p, r, len > 0 ? ci[b] : 0, len > 0);
    for (int kc = 0; kc < Lp; kc += kFillK) {
        const int width = min(kFillK, L - kc);
        const int lg = width > 1 ? 32 - __clz(width - 1) : 0, T = 1 << lg;
        const int sub = lane >> lg, k = lane & (T - 1);
#pragma unroll 4
        for (int i = 0; i < T; ++i) {
            const int row_of = i * (32 >> lg) + sub;
            const int rb = __shfl_sync(FULL, b, row_of), rl = __shfl_sync(FULL, len, row_of);
            if (kc + k < rl) {
                const int at = k * 33 + row_of;
                cp_async<4>(tc + at, ci + (int64_t)rb + kc + k);
                cp_async<8>(tv + at, v + (int64_t)rb + kc + k);
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();
        for (int k0 = 0; k0 < kFillK && kc + k0 < Lp; k0 += Out::vec) {
            int c[Out::vec];
            double a[Out::vec];
            bool ok[Out::vec];
#pragma unroll
            for (int e = 0; e < Out::vec; ++e) {
                ok[e] = kc + k0 + e < len;
                c[e] = ok[e] ? tc[(k0 + e) * 33 + lane] : 0;
                a[e] = ok[e] ? tv[(k0 + e) * 33 + lane] : 0.0;
            }
            out.put(row, q0 + (int64_t)(kc + k0) * 32 + Out::vec * lane, c, a, ok);
        }
        __syncwarp();
    }
}

// FP64 values; CT int stores the columns, int16_t / int8_t the column minus
// the row index (the range was checked by k_sl_reach)
template <typename CT>
struct OutF64 {
    static constexpr int vec = 1;
    CT* col;
    double* val;
    struct Row { int r; };
    __device__ __forceinline__ void begin(Row& w, int64_t, int r, int, bool) const { w.r = r; }
    __device__ __forceinline__ void put(Row& w, int64_t q, const int* c, const double* a, const bool* ok) const
    {
        col[q] = sizeof(CT) == 4 ? (CT)c[0] : (CT)(ok[0] ? c[0] - w.r : 0);
        val[q] = a[0];
    }
};

// FP64 values with coded columns: MODE 1 deltas and row bases, MODE 2 panel
// offsets and steps
template <int MODE, typename DT>
struct OutCoded {
    static constexpr int vec = 1;
    DT* cs;
    uint8_t* step;
    int* rowbase;
    double* val;
    struct Row { int prev; };
    __device__ __forceinline__ void begin(Row& w, int64_t p, int, int first, bool has) const
    {
        w.prev = MODE == 1 && has ? first : 0;
        if (MODE == 1) rowbase[p] = has ? first : 0;
    }
    __device__ __forceinline__ void put(Row& w, int64_t q, const int* c, const double* a, const bool* ok) const
    {
        const int x = ok[0] ? c[0] : w.prev;
        if (MODE == 1) {
            cs[q] = (DT)(x - w.prev);
        } else {
            cs[q] = ok[0] ? (DT)(x & 0xffff) : (DT)0;
            step[q] = (uint8_t)((x >> 16) - (w.prev >> 16));
        }
        val[q] = a[0];
        w.prev = x;
    }
};

// largest |column - row| over the rows in the slices (the first or the last
// column of a row, its columns being increasing)
__global__ void k_sl_reach(int64_t n_slices, const int* __restrict__ rp, const int* __restrict__ ci,
                           const int* __restrict__ perm, const int* __restrict__ rowlen,
                           unsigned* __restrict__ reach)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= 32 * n_slices) return;
    const int len = rowlen[p];
    if (len <= 0) return;
    const int64_t r = perm ? perm[p] : p;
    const int64_t b = rp[r];
    const int64_t lo = r - ci[b], hi = (int64_t)ci[b + len - 1] - r;
    const int64_t m = lo > hi ? lo : hi;
    atomicMax(reach, (unsigned)(m < 0 ? 0 : (m > 0x7fffffff ? 0x7fffffff : m)));
}

// Coded columns of the FP64 layout: the largest delta between consecutive
// columns of a row (MODE 1) or the largest step between the 65536-column
// panels of consecutive elements, the first from panel 0 (MODE 2), over the
// rows in the slices
template <int MODE>
__global__ void k_sl_code_reach(int64_t n_slices, const int* __restrict__ rp, const int* __restrict__ ci,
                                const int* __restrict__ perm, const int* __restrict__ rowlen,
                                unsigned* __restrict__ reach)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= 32 * n_slices) return;
    const int len = rowlen[p];
    if (len <= 0) return;
    const int64_t b = rp[perm ? perm[p] : p];
    unsigned m = 0;
    int prev = MODE == 1 ? ci[b] : 0;
    for (int k = MODE == 1 ? 1 : 0; k < len; ++k) {
        const int c = ci[b + k];
        const unsigned d = MODE == 1 ? (unsigned)(c - prev) : (unsigned)((c >> 16) - (prev >> 16));
        m = max(m, d);
        prev = c;
    }
    atomicMax(reach, m);
}

// 8 blocks of 256 per SM (32 registers): measured faster than the 40-register
// form on all three regular test matrices (random columns 0.249 against
// 0.258 ms, stencil 0.115 against 0.136 ms, 2-nonzero rows 0.080 against
// 0.093 ms).
// Blocks of two warps (32 per SM), as for k_sliced_long: a block frees its
// slot when its two slices are done (27-point stencil 0.113 against 0.115
// ms with eight-warp blocks, 7-point Laplacian 0.035 against 0.037)
constexpr int kOB = 64;
template <int U, typename CT>
__global__ void __launch_bounds__(kOB, 32)
k_sliced(int64_t n_slices, const int* __restrict__ rowlen, const int* __restrict__ slice_len,
         const int64_t* __restrict__ slice_ptr, const int* __restrict__ perm,
         const CT* __restrict__ col, const double* __restrict__ val,
         const double* __restrict__ x, double* __restrict__ y)
{
    const int64_t s = ((int64_t)blockIdx.x * kOB + threadIdx.x) >> 5;
    if (s >= n_slices) return;  // whole warps only
    slice_rows<U, CT>(s, threadIdx.x & 31, rowlen, slice_len, slice_ptr, perm, col, val, x, y);
}

// The product with x still in the caller's page-locked memory: the first
// blocks pull x over the link into the staging vector, stage by stage in
// ascending order, and the others, a slice per warp as in k_sliced, gather a
// batch of elements once the stage of its largest column is complete.  So the
// upload passes beside the product instead of before it.  A waiting warp
// holds up nothing: the copying blocks come first in the grid and wait for
// nobody.  Every wait is bounded all the same: a warp that gives up sets *late
// in page-locked memory, which the host reads once the kernel has ended (the
// call is then done again with the copy first), and marks every stage's
// counter, so that no other warp waits any longer.  x is read with ordinary
// loads after an acquire: a sector enters L1 only when its stage is complete,
// so none is stale.
// Bound by the link: pulling 16.8 MB takes 87 us (512 warps with 4 x 16
// bytes a lane in flight; 2 x 16 are slower, 8 x 16 or 1024 warps no faster).
// What the waits cost is the looking: 9700 resident warps that look at one
// counter every 0.2 us keep its L2 slice from taking the copies' own counts
// (980 us for the 27-point stencil 128^3), every 1 us 162 us, every 2 us
// 145, every 8 us 138 but longer where the product keeps pace with the link
// (7-point 128^3: 191 us for the call against 167).
constexpr int kXStages = 64;          // at most
constexpr int kXShift = 15;           // columns of a stage, at least (log2)
constexpr unsigned kXWarps = 512;     // copying warps: 64 columns each of a stage's 32768
constexpr int kXStride = 32;          // words from one stage's counter to the next: a line each
constexpr unsigned kXSleepNs = 2048;  // between two looks at a counter
constexpr unsigned kXLate = 0x80000000u;  // in a stage's counter: some wait gave up
struct HostX {
    const double* src;  // device address of the host vector
    double* dst;
    int64_t n;
    int shift;          // log2 of the columns of a stage
    unsigned* count;    // [kXStages kXStride] warps that have finished a stage (each finishes them in order)
    unsigned want;      // of them complete a stage
    uint64_t limit_ns;  // of a wait
    unsigned* late;
};

__device__ __forceinline__ void pull_x(const HostX& h, unsigned w, int lane)
{
    constexpr int U = 4;  // 16 bytes each, in flight per lane
    const int lg = h.shift - kXShift;  // log2 of a warp's items of a stage
    const unsigned n = (unsigned)h.n, per = 1u << lg;
    const unsigned items = (((n - 1) >> h.shift) + 1) << lg;
    const bool wide = ((uintptr_t)h.src & 15) == 0;
    // the lane's first column of item t (item t of a stage: 32768 columns on)
    auto column = [&](unsigned t) { return (t >> lg << h.shift) + ((t & (per - 1)) << kXShift) + w * 64 + 2 * lane; };
    for (unsigned t0 = 0; t0 < items; t0 += U) {
        double2 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const unsigned c = column(t0 + u);
            const bool in = t0 + u < items;
            if (wide && in && c + 1 < n) {
                v[u] = __ldcs(reinterpret_cast<const double2*>(h.src + c));
            } else {
                v[u].x = in && c < n ? __ldcs(h.src + c) : 0.0;
                v[u].y = in && c + 1 < n ? __ldcs(h.src + c + 1) : 0.0;
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const unsigned c = column(t0 + u);
            if (t0 + u < items && c + 1 < n) *reinterpret_cast<double2*>(h.dst + c) = v[u];
            else if (t0 + u < items && c < n) h.dst[c] = v[u].x;
        }
        __threadfence();
        __syncwarp();
        if (lane == 0)
            for (unsigned t = t0; t < t0 + U && t < items; ++t)
                if (((t + 1) & (per - 1)) == 0)
                    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(h.count + kXStride * (t >> lg)) : "memory");
    }
}

// true once all warps have finished the stage, or some wait has given up (for
// the whole warp)
__device__ __forceinline__ bool stage_in(const HostX& h, int stage)
{
    unsigned v = 0;
    if ((threadIdx.x & 31) == 0) {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(h.count + kXStride * stage) : "memory");
    }
    v = __shfl_sync(FULL, v, 0);
    __syncwarp();
    return v >= h.want;
}

// (as a call, with the parameters' addresses taken, the kernel takes 168 us in
// place of 158 for the 27-point stencil 128^3)
__device__ __forceinline__ void give_up(unsigned* count, unsigned* late, int lane)
{
#pragma unroll 1
    for (int i = lane; i < kXStages; i += 32) atomicOr(count + kXStride * i, kXLate);
    if (lane == 0) *late = 1u;
}

template <int U, typename CT>
__global__ void __launch_bounds__(kOB, 32)
k_sliced_host(HostX h, unsigned copy_blocks, int64_t n_slices, const int* __restrict__ rowlen,
              const int* __restrict__ slice_len, const int64_t* __restrict__ slice_ptr,
              const CT* __restrict__ col, const double* __restrict__ val, double* __restrict__ y)
{
    const int lane = threadIdx.x & 31;
    if (blockIdx.x < copy_blocks) {
        pull_x(h, blockIdx.x * (kOB / 32) + (threadIdx.x >> 5), lane);
        return;
    }
    const int64_t s = ((int64_t)(blockIdx.x - copy_blocks) * kOB + threadIdx.x) >> 5;
    if (s >= n_slices) return;  // whole warps only
    const int last = (int)((h.n - 1) >> h.shift);
    const int64_t p = s * 32 + lane;
    const int len = rowlen[p], L = slice_len[s];
    const int64_t q0 = slice_ptr[s] + lane;
    unsigned ready = stage_in(h, last) ? 0xffffffffu : 0u;  // columns below it are in
    const CT* __restrict__ cp = col + q0;
    const double* __restrict__ vp = val + q0;
    double acc = 0.0;
    for (int k = 0; k < L; k += U) {
        int c[U];
        double a[U], xv[U];
        int top = 0;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool ok = k + u < len;
            c[u] = ok ? column_of(__ldcs(cp + (k + u) * 32), (int)p) : 0;
            a[u] = ok ? __ldcs(vp + (k + u) * 32) : 0.0;
            top = max(top, c[u]);
        }
        top = __reduce_max_sync(FULL, top);
        if ((unsigned)top >= ready) {
            const int stage = top >> h.shift;
            uint64_t t0 = 0;
            while (!stage_in(h, stage)) {
                const uint64_t now = __shfl_sync(FULL, ptx::global_ns(), 0);
                if (t0 == 0) t0 = now;
                if (now - t0 > h.limit_ns) {
                    give_up(h.count, h.late, lane);
                    break;
                }
                __nanosleep(kXSleepNs);
            }
            ready = stage == last ? 0xffffffffu : (unsigned)(stage + 1) << h.shift;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) xv[u] = k + u < len ? ldx_of<true>(h.dst + c[u]) : 0.0;
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (k + u < len) acc = fma(a[u], xv[u], acc);
    }
    if (len >= 0) y[p] = acc;
}

// One slice per warp with coded columns (slice_value_coded).
template <int U, int MODE, typename DT>
__global__ void __launch_bounds__(kSB, 8)
k_sliced_coded(int64_t n_slices, const int* __restrict__ rowlen, const int* __restrict__ slice_len,
               const int64_t* __restrict__ slice_ptr, const int* __restrict__ perm,
               const DT* __restrict__ cs, const uint8_t* __restrict__ step,
               const int* __restrict__ rowbase, const double* __restrict__ val,
               const double* __restrict__ x, double* __restrict__ y)
{
    const int64_t s = ((int64_t)blockIdx.x * kSB + threadIdx.x) >> 5;
    if (s >= n_slices) return;  // whole warps only
    int row;
    const double v = slice_value_coded<U, MODE, DT>(s, threadIdx.x & 31, rowlen, slice_len, slice_ptr, perm,
                                                    cs, step, rowbase, val, x, &row);
    if (row >= 0) y[row] = v;
}

// Every row of length L in order, none long (an ELLPACK matrix): R slices
// per warp with no slice header read (uniform_rows); each row is the same
// DFMA chain as in slice_rows / slice_rows_multi.
template <int U, int R, int B, typename CT>
__global__ void __launch_bounds__(kSB, B)
k_sliced_uniform(int64_t n_rows, int64_t n_slices, int L, const CT* __restrict__ col,
                 const double* __restrict__ val, const double* __restrict__ x, double* __restrict__ y)
{
    const int lane = threadIdx.x & 31;
    const int64_t first = (((int64_t)blockIdx.x * kSB + threadIdx.x) >> 5) * R;
    if constexpr (R == 4) {
        // four slices per warp (64 registers, 4 blocks per SM): one resident
        // grid whose warps stride over the slices, instead of many short
        // blocks waiting for an SM slot
        const int64_t step = (int64_t)gridDim.x * (kSB / 32) * R;
        for (int64_t s0 = first; s0 < n_slices; s0 += step)
            uniform_rows<U, R, CT>(s0, n_slices, n_rows, L, lane, col, val, x, y);
    } else {
        if (first >= n_slices) return;  // whole warps only
        uniform_rows<U, R, CT>(first, n_slices, n_rows, L, lane, col, val, x, y);
    }
}

// R consecutive slices per warp (slice_rows_multi), for short slices whose
// few loads per lane leave the warp waiting on latency.
template <int U, int R, int B, typename CT>
__global__ void __launch_bounds__(kSB, B)
k_sliced_multi(int64_t n_slices, const int* __restrict__ rowlen, const int* __restrict__ slice_len,
               const int64_t* __restrict__ slice_ptr, const int* __restrict__ perm,
               const CT* __restrict__ col, const double* __restrict__ val,
               const double* __restrict__ x, double* __restrict__ y)
{
    const int64_t s0 = (((int64_t)blockIdx.x * kSB + threadIdx.x) >> 5) * R;
    if (s0 >= n_slices) return;  // whole warps only
    slice_rows_multi<U, R, CT>(s0, n_slices, threadIdx.x & 31, rowlen, slice_len, slice_ptr, perm, col, val, x,
                               y);
}

// Long rows in ascending order, split into segments of kSlicedSeg nonzeros:
// the list, its segment offsets, each segment's CSR begin and end, its row
// when it is the row's only one (that segment writes y itself; else -1), and
// the rows with several segments with their tickets.  A block per tile.
struct LongTables {
    int* rows; int* seg_off; int64_t* seg_be; int* seg_row; int* seg_fix; int* fix; unsigned* ticket;
};
__global__ void __launch_bounds__(kSB)
k_sl_long_tables(int64_t n_rows, const int* __restrict__ rp, int cap, int64_t tile_slices,
                 const SlScratch* __restrict__ w, int n_long, LongTables o)
{
    if (w->tile[blockIdx.x].n_long == 0) return;
    const SlTile at = tiles_before(w);
    unsigned q0 = at.n_long, j0 = at.n_seg, f0 = at.n_fix;
    const int64_t r0 = blockIdx.x * tile_slices * 32, r1 = min(n_rows, r0 + tile_slices * 32);
    for (int64_t base = r0; base < r1; base += kSB) {
        const int64_t r = base + threadIdx.x;
        const int b = r < r1 ? rp[r] : 0, e = r < r1 ? rp[r + 1] : 0;
        const bool is_long = e - b > cap, several = is_long && e - b > kSlicedSeg;
        if (!__syncthreads_or(is_long)) continue;
        const unsigned segs = is_long ? (unsigned)(e - b + kSlicedSeg - 1) / kSlicedSeg : 0u;
        unsigned nq, nj, nf;
        const unsigned q = q0 + block_scan(is_long, &nq), j = j0 + block_scan(segs, &nj),
                       f = f0 + block_scan(several, &nf);
        if (is_long) {
            o.rows[q] = (int)r;
            o.seg_off[q] = (int)j;
            if ((int)q == n_long - 1) o.seg_off[n_long] = (int)(j + segs);
            if (several) {
                o.fix[f] = (int)q;
                o.ticket[f] = 0u;
            }
            for (unsigned i = 0; i < segs; ++i) {
                const int64_t sb = b + (int64_t)i * kSlicedSeg;
                o.seg_be[2 * (int64_t)(j + i)] = sb;
                o.seg_be[2 * (int64_t)(j + i) + 1] = min((int64_t)e, sb + kSlicedSeg);
                o.seg_row[j + i] = several ? -1 : (int)r;
                o.seg_fix[j + i] = several ? (int)f : -1;
            }
        }
        q0 += nq;
        j0 += nj;
        f0 += nf;
    }
}

__device__ __forceinline__ longlong2 segment_bounds(const int64_t* seg_be, int w)
{
    return __ldg(reinterpret_cast<const longlong2*>(seg_be) + w);
}

// A segment's warp writes its sum to y when it is its row's only segment,
// else to partial; the partials of a row with several segments are summed
// in segment order by the warp finishing the row's last one (finish_segment).
// Lane 0 of segment w's warp, with the segment's sum: y of the row when it
// is the row's only segment; else the partial, and when the atomic ticket
// shows this was the row's last segment to finish, the row's sum of
// partials in segment order, after which the ticket is reset for the next
// call.  Nothing waits.
__device__ __forceinline__ void finish_segment(int w, double sum, const int* __restrict__ seg_row,
                                               const int* __restrict__ seg_fix, const int* __restrict__ fix,
                                               const int* __restrict__ list, const int* __restrict__ seg_off,
                                               unsigned* __restrict__ ticket, double* __restrict__ partial,
                                               double* __restrict__ y)
{
    const int r1 = seg_row[w];
    if (r1 >= 0) {
        y[r1] = sum;
        return;
    }
    partial[w] = sum;
    __threadfence();
    const int t = seg_fix[w];
    const int q = fix[t];
    const int b = seg_off[q], e = seg_off[q + 1];
    if (atomicAdd(ticket + t, 1u) != (unsigned)(e - b - 1)) return;
    __threadfence();
    double s = 0.0;
    for (int i = b; i < e; ++i) s += __ldcg(partial + i);
    y[list[q]] = s;
    ticket[t] = 0u;
}

// Slices and long-row segments in one launch (FP64 values, rows above the
// cap present).  Blocks below seg_blocks take one segment per warp, the
// others the slices (R per warp).  The block scheduler starts blocks
// roughly in index order, so the segments -- long, bound by their gathers of
// x -- start first and the short, latency-bound slices fill in around them
// instead of running as a separate launch after them.  A row with several
// segments has no fix-up launch either: each of its segments stores its
// partial, and the warp that finishes the row's last one (an atomic ticket
// per row) sums the partials in segment order (finish_segment) and resets
// the ticket for the next call.  Nothing waits on another warp.
// Threads per block of k_sliced_long: blocks of two warps, so that a block
// whose warps got segments or slices of unequal length frees its SM slot
// sooner (Zipf rows 0.117 ms against 0.119 with blocks of 128 threads and
// 0.120 with 256; the block order is kept)
constexpr int kLB = 64;
template <int U, int R, int B, typename CT, int MODE = 0, typename DT = uint8_t>
__global__ void __launch_bounds__(kLB, 4 * B)
k_sliced_long(int n_seg, unsigned seg_blocks, int64_t n_slices,
              const int64_t* __restrict__ seg_be, const int* __restrict__ seg_row,
              const int* __restrict__ seg_fix, const int* __restrict__ fix,
              const int* __restrict__ list, const int* __restrict__ seg_off,
              unsigned* __restrict__ ticket, double* __restrict__ partial,
              const int* __restrict__ ci, const double* __restrict__ v,
              const int* __restrict__ rowlen, const int* __restrict__ slice_len,
              const int64_t* __restrict__ slice_ptr, const int* __restrict__ perm,
              const CT* __restrict__ col, const double* __restrict__ val,
              const double* __restrict__ x, double* __restrict__ y,
              const uint8_t* __restrict__ step, const int* __restrict__ rowbase)
{
    const int lane = threadIdx.x & 31;
    if (blockIdx.x < seg_blocks) {
        const int w = (int)(blockIdx.x * (kLB / 32) + (threadIdx.x >> 5));
        if (w >= n_seg) return;  // whole warps only
        const longlong2 be = segment_bounds(seg_be, w);
        const double sum = group_sum(row_partial<32, 4>(be.x, be.y, lane, ColPlain<int>{ci}, v, x), 32);
        if (lane == 0) finish_segment(w, sum, seg_row, seg_fix, fix, list, seg_off, ticket, partial, y);
        return;
    }
    const int64_t s0 = ((int64_t)(blockIdx.x - seg_blocks) * kLB + threadIdx.x) >> 5;
    if constexpr (MODE != 0) {
        if (s0 >= n_slices) return;
        int row;
        const double v = slice_value_coded<U, MODE, DT>(s0, lane, rowlen, slice_len, slice_ptr, perm,
                                                        reinterpret_cast<const DT*>(col), step, rowbase,
                                                        val, x, &row);
        if (row >= 0) y[row] = v;
    } else if constexpr (R == 1) {
        if (s0 >= n_slices) return;
        slice_rows<U, CT>(s0, lane, rowlen, slice_len, slice_ptr, perm, col, val, x, y);
    } else {
        if (s0 * R >= n_slices) return;
        slice_rows_multi<U, R, CT>(s0 * R, n_slices, lane, rowlen, slice_len, slice_ptr, perm, col, val,
                                   x, y);
    }
}

// ---- low-precision values (FP32 or BF16), optionally 16-bit column offsets --
__device__ __forceinline__ float round_to(double v, float*) { return __double2float_rn(v); }
__device__ __forceinline__ __nv_bfloat16 round_to(double v, __nv_bfloat16*) { return __double2bfloat16(v); }
__device__ __forceinline__ float widen32(float a) { return a; }
__device__ __forceinline__ float widen32(__nv_bfloat16 a) { return __bfloat162float(a); }

__global__ void k_sl_span(int64_t n_slices, const int* __restrict__ rp, const int* __restrict__ ci,
                          const int* __restrict__ perm, const int* __restrict__ rowlen,
                          unsigned* __restrict__ span)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= 32 * n_slices) return;
    const int len = rowlen[p];
    if (len <= 0) return;
    const int64_t b = rp[perm ? perm[p] : (int)p];
    atomicMax(span, (unsigned)(ci[b + len - 1] - ci[b]));
}

// low-precision contents, four elements of a row side by side (element k
// at slice_ptr[s] + 128 (k / 4) + 4 l + k % 4); OFF16: offsets from the
// row's first column (rowbase per position), else 32-bit columns
__device__ __forceinline__ void store4(float* p, const float* a) { *reinterpret_cast<float4*>(p) = make_float4(a[0], a[1], a[2], a[3]); }
__device__ __forceinline__ void store4(__nv_bfloat16* p, const __nv_bfloat16* a)
{
    uint2 w;
    w.x = __bfloat16_as_ushort(a[0]) | ((unsigned)__bfloat16_as_ushort(a[1]) << 16);
    w.y = __bfloat16_as_ushort(a[2]) | ((unsigned)__bfloat16_as_ushort(a[3]) << 16);
    *reinterpret_cast<uint2*>(p) = w;
}
template <typename VT, bool OFF16>
struct OutLp {
    static constexpr int vec = 4;
    int* col;
    uint16_t* off;
    int* rowbase;
    VT* val;
    struct Row { int first; };
    __device__ __forceinline__ void begin(Row& w, int64_t p, int, int first, bool has) const
    {
        w.first = has ? first : 0;
        if (OFF16) rowbase[p] = w.first;
    }
    __device__ __forceinline__ void put(Row& w, int64_t q, const int* c, const double* a, const bool* ok) const
    {
        VT x[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) x[e] = round_to(a[e], (VT*)nullptr);
        store4(val + q, x);
        if (OFF16) {
            unsigned o[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) o[e] = ok[e] ? (unsigned)(c[e] - w.first) & 0xffffu : 0u;
            *reinterpret_cast<uint2*>(off + q) = make_uint2(o[0] | (o[1] << 16), o[2] | (o[3] << 16));
        } else {
            *reinterpret_cast<int4*>(col + q) = make_int4(c[0], c[1], c[2], c[3]);
        }
    }
};

__global__ void k_sl_x_to_f32(int64_t n, const double* __restrict__ x, float* __restrict__ x32)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) x32[i] = __double2float_rn(x[i]);
}

// One slice with low-precision values (slice_value_lp).
template <int U, typename VT, bool OFF16, bool ACC32>
__global__ void __launch_bounds__(kSB, 8)
k_sliced_lp(int64_t n_slices, const int* __restrict__ rowlen, const int* __restrict__ slice_len,
            const int64_t* __restrict__ slice_ptr, const int* __restrict__ perm,
            const int* __restrict__ col, const uint16_t* __restrict__ off,
            const int* __restrict__ rowbase, const VT* __restrict__ val,
            const double* __restrict__ x, const float* __restrict__ x32, double* __restrict__ y)
{
    const int64_t s = ((int64_t)blockIdx.x * kSB + threadIdx.x) >> 5;
    if (s >= n_slices) return;
    int row;
    // two groups of four in flight with 16-bit offsets; one with 32-bit
    // columns (gather-bound rows, where registers are worth more as warps)
    const double v = slice_value_lp<OFF16 ? 2 : 1, VT, OFF16, ACC32>(s, threadIdx.x & 31, rowlen, slice_len, slice_ptr,
                                                         perm, col, off, rowbase, val, x, x32, &row);
    if (row >= 0) y[row] = v;
}

// FP32/BF16 values with rows above the cap: slices and long-row segments in
// one launch, as k_sliced_long.  A segment is computed from the CSR arrays
// with each value rounded as the slices' (the same arithmetic per element);
// its lanes are combined by a shuffle tree, in FP32 (ACC32) or FP64.
template <typename VT, bool OFF16, bool ACC32>
__global__ void __launch_bounds__(kSB, 8)
k_sliced_long_lp(int n_seg, unsigned seg_blocks, int64_t n_slices,
                 const int64_t* __restrict__ seg_be, const int* __restrict__ seg_row,
                 const int* __restrict__ seg_fix, const int* __restrict__ fix,
                 const int* __restrict__ list, const int* __restrict__ seg_off,
                 unsigned* __restrict__ ticket, double* __restrict__ partial,
                 const int* __restrict__ ci, const double* __restrict__ v,
                 const int* __restrict__ rowlen, const int* __restrict__ slice_len,
                 const int64_t* __restrict__ slice_ptr, const int* __restrict__ perm,
                 const int* __restrict__ col, const uint16_t* __restrict__ off,
                 const int* __restrict__ rowbase, const VT* __restrict__ val,
                 const double* __restrict__ x, const float* __restrict__ x32, double* __restrict__ y)
{
    const int lane = threadIdx.x & 31;
    if (blockIdx.x < seg_blocks) {
        const int w = (int)(blockIdx.x * (kSB / 32) + (threadIdx.x >> 5));
        if (w >= n_seg) return;  // whole warps only
        const longlong2 be = segment_bounds(seg_be, w);
        double sum;
        if (ACC32) {
            float acc = 0.f;
            for (int64_t j = be.x + lane; j < be.y; j += 32)
                acc = fmaf(widen32(round_to(__ldcs(v + j), (VT*)nullptr)), __ldg(x32 + __ldcs(ci + j)), acc);
            sum = (double)group_sum32(acc, 32);
        } else {
            double acc = 0.0;
            for (int64_t j = be.x + lane; j < be.y; j += 32)
                acc = fma(widen_f32(widen32(round_to(__ldcs(v + j), (VT*)nullptr))), ldx(x + __ldcs(ci + j)), acc);
            sum = group_sum(acc, 32);
        }
        if (lane == 0) finish_segment(w, sum, seg_row, seg_fix, fix, list, seg_off, ticket, partial, y);
        return;
    }
    const int64_t s = ((int64_t)(blockIdx.x - seg_blocks) * kSB + threadIdx.x) >> 5;
    if (s >= n_slices) return;
    int row;
    const double r = slice_value_lp<OFF16 ? 2 : 1, VT, OFF16, ACC32>(s, lane, rowlen, slice_len, slice_ptr,
                                                                    perm, col, off, rowbase, val, x, x32, &row);
    if (row >= 0) y[row] = r;
}

unsigned grid_of(int64_t threads, int64_t cap_blocks)
{
    int64_t g = (threads + kSB - 1) / kSB;
    if (g > cap_blocks) g = cap_blocks;
    return (unsigned)std::max<int64_t>(g, 1);
}

}  // namespace

namespace {

// page-locked memory that kernels write to, one per host thread: the layout's
// totals, and whether a wait of k_sliced_host gave up
struct SlHost {
    SlStats stats;
    unsigned late;
};
thread_local SlHost* t_host = nullptr;
spmv_status host_words()
{
    if (t_host) return SPMV_OK;
    void* p = nullptr;
    if (cudaMallocHost(&p, sizeof(SlHost)) != cudaSuccess) {
        cudaGetLastError();
        return fail(SPMV_ERR_NOMEM, "cudaMallocHost for the SLICED kernels' words failed");
    }
    t_host = static_cast<SlHost*>(p);
    return SPMV_OK;
}

// Places arrays in one allocation, each on a 256-byte boundary, large ones on
// a 2 MB boundary.
struct Arena {
    static constexpr int64_t kPage = 2 << 20, kLarge = 4 << 20;
    int64_t bytes = 0;
    std::vector<std::pair<void**, int64_t>> at;
    template <typename T>
    void add(T** p, int64_t count)
    {
        // large arrays as an allocation of their own would start: FP32 7-point
        // products 2 % faster than with arrays end to end
        const int64_t size = (int64_t)sizeof(T) * std::max<int64_t>(count, 1);
        if (size >= kLarge) bytes = (bytes + kPage - 1) / kPage * kPage;
        at.push_back({reinterpret_cast<void**>(p), bytes});
        bytes += (size + 255) / 256 * 256;
    }
    spmv_status allocate(spmv_prepared* P)
    {
        void* base = nullptr;
        spmv_status st = prepared_alloc(P, &base, bytes);
        if (st != SPMV_OK) return st;
        for (auto& a : at) *a.first = static_cast<char*>(base) + a.second;
        return SPMV_OK;
    }
};

// check: the matrix's validation pass is on the stream; its verdict is read
// at the first wait (what runs before that reads row pointers, each as a
// number, and in k_sl_layout columns of elements that it has found to lie in
// [0, nnz), also as numbers)
spmv_status sliced_build(spmv_prepared* P, SlScratch* w, bool check, cudaStream_t s)
{
    const spmv_csr_t& A = P->A;
    SlicedPlan& d = P->sl;
    SlStats* const host = &t_host->stats;
    int cap = P->c.items_per_warp > 0 ? P->c.items_per_warp : kSlicedCap;
    d.n_slices = (A.n_rows + 31) / 32;
    const int64_t n_pos = 32 * d.n_slices;
    const bool f64 = P->c.value_type == SPMV_VAL_F64;
    // FP64 values: one element per slot row; FP32/BF16: four side by side
    d.vec = f64 ? 1 : 4;
    spmv_status st;
    Arena head;
    head.add(&d.rowlen, n_pos);
    head.add(&d.slice_len, d.n_slices);
    head.add(&d.slice_ptr, d.n_slices + 1);
    if ((st = head.allocate(P)) != SPMV_OK) return st;
    SlStats f = {};
    int64_t tile_slices = 1;
    unsigned n_tiles = 0;
    // one layout pass for window length sigma (1 = rows in order)
    auto layout = [&](int sigma) -> spmv_status {
        if (d.n_slices == 0) {
            SPMV_CUDA_TRY(cudaMemsetAsync(d.slice_ptr, 0, 8, s));
            return SPMV_OK;
        }
        const int64_t unit = sigma > 1 ? sigma / 32 : 32;  // whole windows
        tile_slices = ((d.n_slices + kTiles - 1) / kTiles + unit - 1) / unit * unit;
        n_tiles = (unsigned)((d.n_slices + tile_slices - 1) / tile_slices);
        SPMV_CUDA_TRY(cudaMemsetAsync(w, 0, sizeof(SlStats) + sizeof(SlTile) * n_tiles, s));
        if (sigma == 1) {
            k_sl_layout<<<n_tiles, kSB, 0, s>>>(A.n_rows, A.n_cols, A.nnz, d.n_slices, A.rowptr, A.colind, cap, d.vec,
                                                tile_slices, d.rowlen, d.slice_len, w);
        } else {
            if (!d.perm) {
                st = prepared_alloc(P, reinterpret_cast<void**>(&d.perm), 4 * A.n_rows);
                if (st != SPMV_OK) return st;
            }
            const unsigned n_win = (unsigned)((A.n_rows + sigma - 1) / sigma);
            k_sl_sort<<<n_win, std::max(32, sigma / kSortItems), 0, s>>>(A.n_rows, d.n_slices, A.rowptr, sigma, cap,
                                                                         d.vec, tile_slices, d.perm, d.rowlen,
                                                                         d.slice_len, w);
        }
        SPMV_CUDA_TRY(cudaGetLastError());
        k_sl_scan<<<n_tiles, kSB, 0, s>>>(d.n_slices, tile_slices, d.vec, d.slice_len, d.slice_ptr, w, host);
        SPMV_CUDA_TRY(cudaGetLastError());
        SPMV_CUDA_TRY(cudaStreamSynchronize(s));
        f = *host;
        if (check && (st = feature_pass_verdict(&A)) != SPMV_OK) return st;
        check = false;
        return SPMV_OK;
    };
    int sigma = P->c.block_nnz;
    if (sigma == 0) {
        // rows in order unless that pads the slices by more than a quarter;
        // then rows sorted by length in windows of 4096, and (unless the cap
        // was chosen) every row above 32 nonzeros computed by a warp, so that
        // no lane's chain is longer than one element per lane of a warp
        if ((st = layout(1)) != SPMV_OK) return st;
        if ((int64_t)f.slots > A.nnz + A.nnz / 4) {
            sigma = 4096;
            if (P->c.items_per_warp == 0) cap = 32;
            if ((st = layout(sigma)) != SPMV_OK) return st;
        } else {
            sigma = 1;
        }
    } else if ((st = layout(sigma)) != SPMV_OK) {
        return st;
    }
    P->c.block_nnz = sigma;
    P->c.items_per_warp = cap;
    d.sigma = sigma;
    d.ahead = sigma == 1 ? f.reach : 0;
    // FP64 values: slices per warp, 4 when no slice is longer than four
    // elements (a lane's few loads leave a warp waiting on latency, so one
    // warp takes four slices), else 1 (longer slices keep four elements of
    // one row in flight instead)
    if (!f64) P->c.threads_per_row = 1;
    else if (P->c.threads_per_row == 0) P->c.threads_per_row = f.longest <= 4 ? 4 : 1;
    d.n_long = (int)f.n_long;
    d.n_seg = (int)f.n_seg;
    d.n_fix = (int)f.n_fix;
    d.tot = (int64_t)f.tot;
    // rows all of one length, in order, none long: the slice header is implied
    d.uniform_len = sigma == 1 && d.n_long == 0 && A.n_rows > 0 && (int)~f.shortest_c == f.longest ? f.longest : -1;
    const int64_t tot1 = std::max<int64_t>(d.tot, 1);
    const int* permp = sigma > 1 ? d.perm : nullptr;
    d.value_type = P->c.value_type;
    if (P->c.accumulate == 0) P->c.accumulate = f64 ? 1 : 2;
    d.acc32 = P->c.accumulate == 2;
    // a question about the columns of the rows in the slices (0 without rows)
    auto ask = [&](auto kernel, unsigned* out) -> spmv_status {
        *out = 0;
        if (d.n_slices == 0) return SPMV_OK;
        SPMV_CUDA_TRY(cudaMemsetAsync(&w->stats.reach, 0, 4, s));
        kernel<<<(unsigned)((n_pos + kSB - 1) / kSB), kSB, 0, s>>>(d.n_slices, A.rowptr, A.colind, permp, d.rowlen,
                                                                    &w->stats.reach);
        SPMV_CUDA_TRY(cudaGetLastError());
        SPMV_CUDA_TRY(cudaMemcpyAsync(&host->reach, &w->stats.reach, 4, cudaMemcpyDeviceToHost, s));
        SPMV_CUDA_TRY(cudaStreamSynchronize(s));
        *out = host->reach;
        return SPMV_OK;
    };
    Arena body;
    unsigned r = 0;
    if (f64) {
        // coded columns (Table 2's deltas, or panels) when asked for and
        // every row in the slices fits: deltas in 8 bits, else 16, else (or
        // when panels were asked for) 16-bit panel offsets with 8-bit steps
        d.coding = 0;
        if (P->c.index_coding != 0 && d.n_slices > 0) {
            if (P->c.index_coding == 1) {
                if ((st = ask(k_sl_code_reach<1>, &r)) != SPMV_OK) return st;
                if (r <= 255) { d.coding = 1; d.cbytes = 1; }
                else if (r <= 65535) { d.coding = 1; d.cbytes = 2; }
            }
            if (d.coding == 0) {
                if ((st = ask(k_sl_code_reach<2>, &r)) != SPMV_OK) return st;
                if (r <= 255) { d.coding = 2; d.cbytes = 3; }
            }
        }
        // index_bytes 0: the narrowest form that fits when the rows are all of
        // one length and in order (k_sliced_uniform, where the narrower column
        // stream shortens the launch), else 32-bit columns.  Columns as
        // offsets from the row index in 8 or 16 bits when the caller allows it
        // and every row in the slices stays that close to its diagonal
        const int allowed = d.coding != 0 ? 4
                            : P->c.index_bytes != 0 ? P->c.index_bytes
                            : d.uniform_len >= 0 ? 1 : 4;
        r = 0;
        if (allowed < 4 && (st = ask(k_sl_reach, &r)) != SPMV_OK) return st;
        if (d.coding == 0) d.cbytes = std::max(allowed, r <= 127 ? 1 : (r <= 32767 ? 2 : 4));
        P->c.index_bytes = d.cbytes;
        P->c.index_coding = d.coding;
        if (d.coding != 0) P->c.threads_per_row = 1;  // coded columns: one slice per warp
        const int64_t sbytes = d.coding == 2 ? 2 : d.cbytes;  // panel offsets are 16-bit
        body.add(reinterpret_cast<char**>(&d.scol), sbytes * tot1);
        body.add(&d.val, tot1);
        if (d.coding == 2) body.add(&d.step, tot1);
        if (d.coding == 1) body.add(&d.rowbase, n_pos);
    } else {
        // 16-bit offsets when every row in the slices spans fewer than 65536 columns
        if ((st = ask(k_sl_span, &r)) != SPMV_OK) return st;
        d.off16 = r < 65536;
        body.add(reinterpret_cast<char**>(&d.lowval), (d.value_type == SPMV_VAL_F32 ? 4 : 2) * tot1);
        if (d.off16) {
            body.add(&d.off, tot1);
            body.add(&d.rowbase, n_pos);
        } else {
            body.add(&d.col, tot1);
        }
    }
    if (d.acc32) body.add(&d.x32, A.n_cols);
    LongTables lt = {};
    if (d.n_long > 0) {
        body.add(&d.long_rows, d.n_long);
        body.add(&d.seg_off, (int64_t)d.n_long + 1);
        body.add(&d.partial, d.n_seg);
        body.add(&d.seg_be, 2 * (int64_t)d.n_seg);
        body.add(&d.seg_row, d.n_seg);
        body.add(&d.seg_fix, d.n_seg);
        body.add(&d.fix, d.n_fix);
        body.add(&d.ticket, d.n_fix);
    }
    if ((st = body.allocate(P)) != SPMV_OK) return st;
    if (f64 && d.cbytes == 4) d.col = static_cast<int*>(d.scol);
    if (d.n_slices > 0) {
        const unsigned grid = (unsigned)((d.n_slices + kFillWarps - 1) / kFillWarps);
        auto fill = [&](auto out) {
            k_sl_fill<<<grid, 32 * kFillWarps, 0, s>>>(d.n_slices, A.rowptr, A.colind, A.val, permp, d.rowlen,
                                                       d.slice_len, d.slice_ptr, out);
        };
        if (d.coding == 1 && d.cbytes == 1) fill(OutCoded<1, uint8_t>{static_cast<uint8_t*>(d.scol), nullptr, d.rowbase, d.val});
        else if (d.coding == 1) fill(OutCoded<1, uint16_t>{static_cast<uint16_t*>(d.scol), nullptr, d.rowbase, d.val});
        else if (d.coding == 2) fill(OutCoded<2, uint16_t>{static_cast<uint16_t*>(d.scol), d.step, nullptr, d.val});
        else if (f64 && d.cbytes == 1) fill(OutF64<int8_t>{static_cast<int8_t*>(d.scol), d.val});
        else if (f64 && d.cbytes == 2) fill(OutF64<int16_t>{static_cast<int16_t*>(d.scol), d.val});
        else if (f64) fill(OutF64<int>{d.col, d.val});
        else if (d.value_type == SPMV_VAL_F32 && d.off16) fill(OutLp<float, true>{nullptr, d.off, d.rowbase, static_cast<float*>(d.lowval)});
        else if (d.value_type == SPMV_VAL_F32) fill(OutLp<float, false>{d.col, nullptr, nullptr, static_cast<float*>(d.lowval)});
        else if (d.off16) fill(OutLp<__nv_bfloat16, true>{nullptr, d.off, d.rowbase, static_cast<__nv_bfloat16*>(d.lowval)});
        else fill(OutLp<__nv_bfloat16, false>{d.col, nullptr, nullptr, static_cast<__nv_bfloat16*>(d.lowval)});
        SPMV_CUDA_TRY(cudaGetLastError());
    }
    if (d.n_long > 0) {
        lt = {d.long_rows, d.seg_off, d.seg_be, d.seg_row, d.seg_fix, d.fix, d.ticket};
        k_sl_long_tables<<<n_tiles, kSB, 0, s>>>(A.n_rows, A.rowptr, cap, tile_slices, w, d.n_long, lt);
        SPMV_CUDA_TRY(cudaGetLastError());
    }
    P->n_blocks = d.n_slices;
    return SPMV_OK;
}

}  // namespace

spmv_status sliced_prepare(spmv_prepared* P, bool check, cudaStream_t s)
{
    spmv_status st = host_words();
    if (st != SPMV_OK) return st;
    SlScratch* w = nullptr;
    SPMV_CUDA_TRY(work_alloc(P->device, reinterpret_cast<void**>(&w), sizeof(SlScratch), s));
    st = sliced_build(P, w, check, s);
    cudaFreeAsync(w, s);
    return st;
}

// Where k_sliced_host pays: x of at least half a million columns and rows
// that reach no further than a quarter of them ahead of the diagonal (a
// sample, one row in 32: the speed depends on it, the result does not).  Call
// with the copy first and so, in us: 27-point stencil 96^3 112 and 88, 128^3
// 216 and 158, 160^3 390 and 305; 7-point 128^3 195 and 167; a band of 6 per
// row, 1M rows 104 and 99, 4M 344 and 288; below the limits 27-point 48^3 34
// and 40, 64^3 52 and 53, random columns 1M x 20 136 and 153, 2M x 20 244
// and 276 (nothing passes beside the upload, and the header costs where rows
// are of one length).
bool sliced_host_form(const spmv_prepared* P)
{
    const SlicedPlan& d = P->sl;
    return P->c.variant == SPMV_V7_SLICED && d.value_type == SPMV_VAL_F64 && d.coding == 0 && d.n_long == 0 &&
           d.sigma == 1 && P->A.n_cols >= 1 << 19 && (int64_t)d.ahead * 4 <= P->A.n_cols && P->c.threads_per_row != 2 && P->c.threads_per_row != 4 && P->A.n_rows > 0 && P->A.n_cols > 0;
}

size_t sliced_host_words() { return kXStride * kXStages; }

spmv_status launch_sliced_host(const spmv_prepared* P, const double* x_host, double* y, const PullWait& wait, cudaStream_t s)
{
    const SlicedPlan& d = P->sl;
    spmv_status st = host_words();
    if (st != SPMV_OK) return st;
    t_host->late = 0;
    HostX h{x_host, P->x_stage, P->A.n_cols, kXShift, P->x_count, kXWarps + wait.missing, wait.limit_ns, &t_host->late};
    while (((h.n - 1) >> h.shift) >= kXStages) ++h.shift;
    SPMV_CUDA_TRY(cudaMemsetAsync(P->x_count, 0, sizeof(unsigned) * kXStride * kXStages, s));
    const unsigned copy = kXWarps / (kOB / 32), blocks = copy + (unsigned)((d.n_slices + kOB / 32 - 1) / (kOB / 32));
#define SPMV_SL_HOST(CT)                                                                            \
    k_sliced_host<4, CT><<<blocks, kOB, 0, s>>>(h, copy, d.n_slices, d.rowlen, d.slice_len, d.slice_ptr, \
                                                static_cast<const CT*>(d.scol), d.val, y)
    if (d.cbytes == 1) SPMV_SL_HOST(int8_t);
    else if (d.cbytes == 2) SPMV_SL_HOST(int16_t);
    else SPMV_SL_HOST(int);
#undef SPMV_SL_HOST
    SPMV_CUDA_TRY(cudaGetLastError());
    return SPMV_OK;
}

bool sliced_host_late() { return t_host && *static_cast<volatile unsigned*>(&t_host->late) != 0; }

cudaError_t launch_sliced(const spmv_prepared* P, const double* x, double* y, cudaStream_t s, bool dry)
{
    const spmv_csr_t& A = P->A;
    const SlicedPlan& d = P->sl;
    if (A.n_rows == 0) return cudaSuccess;
    // dry: the same kernels with nothing to do, one block each
    const int64_t n_slices = dry ? 0 : d.n_slices, n_cols = dry ? 0 : A.n_cols;
    const int n_seg = dry ? 0 : d.n_seg;
    const unsigned grid = grid_of(32 * n_slices, INT32_MAX);
    const int* perm = d.sigma > 1 ? d.perm : nullptr;
    cudaError_t e;
    if (d.acc32 && A.n_cols > 0) {
        k_sl_x_to_f32<<<grid_of(n_cols, INT32_MAX), kSB, 0, s>>>(n_cols, x, d.x32);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if (d.value_type == SPMV_VAL_F64 && d.n_long > 0) {
        // slices and long-row segments in one launch, segments first
        const unsigned seg_blocks = (unsigned)((n_seg + kLB / 32 - 1) / (kLB / 32));
        const int R = P->c.threads_per_row == 2 || P->c.threads_per_row == 4 ? P->c.threads_per_row : 1;
        const int64_t slice_warps = (n_slices + R - 1) / R;
        const unsigned blocks = std::max(1u, seg_blocks + (unsigned)((slice_warps + kLB / 32 - 1) / (kLB / 32)));
#define SPMV_SL_LONG(U, RR, B, CT)                                                                  \
    k_sliced_long<U, RR, B, CT><<<blocks, kLB, 0, s>>>(                                           \
        n_seg, seg_blocks, n_slices, d.seg_be, d.seg_row, d.seg_fix, d.fix, d.long_rows,       \
        d.seg_off, d.ticket, d.partial, A.colind, A.val, d.rowlen, d.slice_len, d.slice_ptr, perm,  \
        static_cast<const CT*>(d.scol), d.val, x, y, nullptr, nullptr)
#define SPMV_SL_LONG_CT(CT)                                                                          \
        if (R == 4) SPMV_SL_LONG(1, 4, 4, CT); else if (R == 2) SPMV_SL_LONG(2, 2, 6, CT);           \
        else SPMV_SL_LONG(4, 1, 8, CT);
#define SPMV_SL_LONG_CODED(MODE, DT)                                                                \
    k_sliced_long<4, 1, 8, int, MODE, DT><<<blocks, kLB, 0, s>>>(                                   \
        n_seg, seg_blocks, n_slices, d.seg_be, d.seg_row, d.seg_fix, d.fix, d.long_rows,       \
        d.seg_off, d.ticket, d.partial, A.colind, A.val, d.rowlen, d.slice_len, d.slice_ptr, perm,  \
        static_cast<const int*>(d.scol), d.val, x, y, d.step, d.rowbase)
        if (d.coding == 1 && d.cbytes == 1) { SPMV_SL_LONG_CODED(1, uint8_t); }
        else if (d.coding == 1) { SPMV_SL_LONG_CODED(1, uint16_t); }
        else if (d.coding == 2) { SPMV_SL_LONG_CODED(2, uint16_t); }
        else if (d.cbytes == 1) { SPMV_SL_LONG_CT(int8_t) }
        else if (d.cbytes == 2) { SPMV_SL_LONG_CT(int16_t) }
        else { SPMV_SL_LONG_CT(int) }
#undef SPMV_SL_LONG_CODED
#undef SPMV_SL_LONG_CT
#undef SPMV_SL_LONG
        return cudaGetLastError();
    }
    if (d.value_type == SPMV_VAL_F64 && d.coding != 0) {
#define SPMV_SL_CODED(MODE, DT)                                                                     \
    k_sliced_coded<4, MODE, DT><<<grid, kSB, 0, s>>>(n_slices, d.rowlen, d.slice_len, d.slice_ptr,  \
                                                     perm, static_cast<const DT*>(d.scol), d.step,    \
                                                     d.rowbase, d.val, x, y)
        if (d.coding == 1 && d.cbytes == 1) SPMV_SL_CODED(1, uint8_t);
        else if (d.coding == 1) SPMV_SL_CODED(1, uint16_t);
        else SPMV_SL_CODED(2, uint16_t);
#undef SPMV_SL_CODED
        return cudaGetLastError();
    }
    if (d.value_type == SPMV_VAL_F64 && d.uniform_len >= 0) {
        // rows of one length: no slice header (k_sliced_uniform)
        const int R = P->c.threads_per_row == 2 || P->c.threads_per_row == 4 ? P->c.threads_per_row : 1;
        const unsigned ugrid = grid_of(32 * ((n_slices + R - 1) / R), R == 4 ? (int64_t)P->sm_count * 4 : INT32_MAX);
#define SPMV_SL_U(U, RR, B, CT)                                                                    \
    k_sliced_uniform<U, RR, B, CT><<<ugrid, kSB, 0, s>>>(A.n_rows, n_slices, d.uniform_len,      \
                                                         static_cast<const CT*>(d.scol), d.val, x, y)
#define SPMV_SL_U_CT(CT)                                                                           \
        if (R == 4) SPMV_SL_U(1, 4, 4, CT); else if (R == 2) SPMV_SL_U(2, 2, 6, CT);               \
        else SPMV_SL_U(4, 1, 8, CT);
        if (d.cbytes == 1) { SPMV_SL_U_CT(int8_t) }
        else if (d.cbytes == 2) { SPMV_SL_U_CT(int16_t) }
        else { SPMV_SL_U_CT(int) }
#undef SPMV_SL_U_CT
#undef SPMV_SL_U
        return cudaGetLastError();
    }
    if (d.value_type == SPMV_VAL_F64) {
        // R slices per warp (sliced_prepare chose R, or the caller did);
        // columns stored as CT (sliced_prepare chose the width)
#define SPMV_SL_M(U, RR, B, CT)                                                                    \
    k_sliced_multi<U, RR, B, CT><<<grid_of(32 * ((n_slices + RR - 1) / RR), INT32_MAX), kSB, 0, s>>>( \
        n_slices, d.rowlen, d.slice_len, d.slice_ptr, perm, static_cast<const CT*>(d.scol), d.val, x, y)
#define SPMV_SL_CT(CT)                                                                             \
        switch (P->c.threads_per_row) {                                                            \
            case 2: SPMV_SL_M(2, 2, 6, CT); break;                                                 \
            case 4: SPMV_SL_M(1, 4, 4, CT); break;                                                 \
            default:                                                                               \
                k_sliced<4, CT><<<std::max(1u, (unsigned)((n_slices + kOB / 32 - 1) / (kOB / 32))), kOB, 0, s>>>( \
                    n_slices, d.rowlen, d.slice_len, d.slice_ptr, \
                                                     perm, static_cast<const CT*>(d.scol), d.val, x, y); \
        }
        if (d.cbytes == 1) { SPMV_SL_CT(int8_t) }
        else if (d.cbytes == 2) { SPMV_SL_CT(int16_t) }
        else { SPMV_SL_CT(int) }
#undef SPMV_SL_CT
#undef SPMV_SL_M
    } else if (d.n_long > 0) {
        // FP32/BF16 values with long rows: slices and segments in one launch
        const unsigned seg_blocks = (unsigned)((n_seg + kSB / 32 - 1) / (kSB / 32));
        const unsigned blocks = std::max(1u, seg_blocks + (unsigned)((n_slices + kSB / 32 - 1) / (kSB / 32)));
#define SPMV_SL_LONG_LP(VT, O16, A32)                                                                 \
    k_sliced_long_lp<VT, O16, A32><<<blocks, kSB, 0, s>>>(                                          \
        n_seg, seg_blocks, n_slices, d.seg_be, d.seg_row, d.seg_fix, d.fix, d.long_rows,         \
        d.seg_off, d.ticket, d.partial, A.colind, A.val, d.rowlen, d.slice_len, d.slice_ptr, perm,    \
        d.col, d.off, d.rowbase, static_cast<const VT*>(d.lowval), x, d.x32, y)
#define SPMV_SL_LONG_LP_VT(VT)                                                                         \
    if (d.off16) { if (d.acc32) SPMV_SL_LONG_LP(VT, true, true); else SPMV_SL_LONG_LP(VT, true, false); } \
    else { if (d.acc32) SPMV_SL_LONG_LP(VT, false, true); else SPMV_SL_LONG_LP(VT, false, false); }
        if (d.value_type == SPMV_VAL_F32) { SPMV_SL_LONG_LP_VT(float) } else { SPMV_SL_LONG_LP_VT(__nv_bfloat16) }
#undef SPMV_SL_LONG_LP_VT
#undef SPMV_SL_LONG_LP
    } else {
#define SPMV_SL_LP(VT, O16, A32)                                                                   \
    k_sliced_lp<4, VT, O16, A32><<<grid, kSB, 0, s>>>(n_slices, d.rowlen, d.slice_len,          \
                                                      d.slice_ptr, perm, d.col, d.off, d.rowbase,  \
                                                      static_cast<const VT*>(d.lowval), x, d.x32, y)
#define SPMV_SL_LP_VT(VT)                                                        \
    if (d.off16) { if (d.acc32) SPMV_SL_LP(VT, true, true); else SPMV_SL_LP(VT, true, false); } \
    else { if (d.acc32) SPMV_SL_LP(VT, false, true); else SPMV_SL_LP(VT, false, false); }
        if (d.value_type == SPMV_VAL_F32) { SPMV_SL_LP_VT(float) } else { SPMV_SL_LP_VT(__nv_bfloat16) }
#undef SPMV_SL_LP_VT
#undef SPMV_SL_LP
    }
    return cudaGetLastError();
}

}  // namespace spmvlib
