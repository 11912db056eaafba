// Structural features of Table 1 (Section 3.2.2) and CSR validation, in one
// pass over rowptr and colind.
//
// Per row i (empty rows contribute zeros):
//   nnz_i, bw_i = last - first column (0 when nnz_i <= 1), span_i = bw_i + 1,
//   ngroups_i = maximal runs of consecutive columns,
//   misses_i  = 1 + #{j > first : 8 (c_j - c_{j-1}) > line_bytes},
//   disp q_i  = floor(2^32 nnz_i / span_i), clust q_i = floor(2^32 ngroups_i / nnz_i).
// The aggregates (min, max, sums, sums of squares) are integers; integer
// addition is associative, so global atomics give exact, order-independent
// totals.  128-bit sums are kept as (lo, hi) words with explicit carries.
// The doubles of Table 1 are derived on the host from these integers.
#include <math.h>
#include <string.h>

#include <algorithm>

#include "common.cuh"

namespace spmvlib {
namespace {

typedef unsigned long long u64;
typedef unsigned __int128 u128;

// The pass's result: integer aggregates (min, max, sums; minima are kept as
// the maximum of the bitwise complement so that 0 is the identity), in the
// order of RowAgg's words.  Written by the last block straight into
// page-locked host memory.  The 128-bit sums are carried as three digits of
// 32, 32 and 64 bits, whose sums over blocks need no carries.
constexpr int kFT = 256;        // threads per block of both kernels
constexpr int kFeatBlocks = 3;  // their resident blocks per SM (80 registers)
constexpr int kShortRow = 8;
constexpr int64_t kLongRow = 1024;
constexpr int64_t kPiece = 2048;
constexpr int kFields = 18;
struct FeatAcc {
    u64 nnz_min_c, nnz_max, nnz_sum, nnz_sumsq;
    u64 bw_min_c, bw_max, bw_sum, disp_sum, clust_sum;
    u64 ngroups_sum, misses_sum;
    u64 err;
    u64 bw_sq[3], disp_sq[3];
};
static_assert(sizeof(FeatAcc) == 8 * kFields, "one word per field");

// Device counters and accumulators of one pass, all 0 between calls (the
// last block resets them): long rows listed, their pieces listed, blocks of
// either kernel finished, and kSlots sets of accumulators that the blocks
// add to in turn, so that no address takes an atomic from every block.
constexpr int kSlots = 32;
struct FeatCtl {
    unsigned n_long, n_pieces, done_pass, done_long;
    u64 slot[kSlots][kFields];
};

__device__ __forceinline__ u64 shfl_u64(u64 v, int o) {
    return __shfl_xor_sync(FULL_MASK, v, o);
}

__device__ __forceinline__ u128 warp_sum_u128(u128 v) {
    u64 lo = (u64)v, hi = (u64)(v >> 64);
    for (int o = 16; o > 0; o >>= 1) {
        const u64 lo2 = shfl_u64(lo, o), hi2 = shfl_u64(hi, o);
        const u64 nlo = lo + lo2;
        hi = hi + hi2 + (nlo < lo ? 1ull : 0ull);
        lo = nlo;
    }
    return ((u128)hi << 64) | lo;
}

__device__ __forceinline__ u64 warp_sum_u64(u64 v) {
    for (int o = 16; o > 0; o >>= 1) v += shfl_u64(v, o);
    return v;
}

// floor(a 2^32 / b) for 0 < a < b < 2^31, exactly, without a 64-bit integer
// division and without 64-bit conversions (which run on the FP64 pipe): an
// FP32 estimate of the quotient (a / b < 1, so it fits 32 bits), then the
// integer remainder a 2^32 - q b, converted to FP32 from two 32-bit halves,
// gives a correction, and the remainder is brought into [0, b).  The two
// conversions and the product are off by half an ulp each, the reciprocal by
// at most two ulps: 7 x 2^-24 of a quotient below 2^32 in all, so the first
// estimate is within 1793 < 2^11 of it, |remainder| < 2^42 and the second
// within one, which the last line settles.
// Arguments outside that range come only from rows the pass flags as invalid
// (columns not strictly increasing or out of range), whose results are
// discarded: they give 0.
__device__ __forceinline__ unsigned fixq32(unsigned a, unsigned b)
{
    if (a == 0 || a >= b || b >= (1u << 31)) return 0;
    const float rb = __fdividef(1.0f, __uint2float_rn(b));
    unsigned q = __float2uint_rz(__fmul_rn(__fmul_rn(__uint2float_rn(a), rb), 4294967296.0f));
    int64_t rem = (int64_t)(((u64)a << 32) - (u64)q * b);
    const float rf = __fmaf_rn(__int2float_rn((int)(rem >> 20)), 1048576.0f,
                               __uint2float_rn((unsigned)(rem & 0xFFFFF)));
    const int c = __float2int_rd(__fmul_rn(rf, rb));
    q += (unsigned)c;
    rem -= (int64_t)c * b;
    return rem < 0 ? q - 1 : rem >= (int64_t)b ? q + 1 : q;
}

// A sum of 64-bit terms of which one thread adds fewer than 2^32.
struct Sum96 {
    u64 lo = 0;
    unsigned hi = 0;
    __device__ __forceinline__ void add(u64 v) {
        asm("add.cc.u64 %0, %0, %2;\n\taddc.u32 %1, %1, 0;" : "+l"(lo), "+r"(hi) : "l"(v));
    }
    __device__ __forceinline__ u128 value() const { return ((u128)hi << 64) | lo; }
};

// Per-thread partial aggregates of the rows a thread finalizes.  A ratio of
// exactly 1 (2^32 in fixed point, one bit too wide) is added to the sums'
// upper words, so that every per-row quantity fits 32 bits and its square 64.
struct RowAgg {
    unsigned nnz_min = 0xffffffffu, nnz_max = 0, bw_min = 0xffffffffu, bw_max = 0;
    u64 nnz_sum = 0, nnz_sq = 0, bw_sum = 0, disp_sum = 0, clust_sum = 0, ng_sum = 0, ms_sum = 0;
    Sum96 bw_sq, disp_sq;

    // one row: nz nonzeros, columns first..last, ng / ms counted over its
    // elements after the first (the first element adds one to each)
    __device__ __forceinline__ void add(unsigned nz, int first, int last, unsigned ng, unsigned ms) {
        unsigned bw = 0, dq = 0, cq = 0;
        if (nz > 0) {
            bw = (unsigned)last - (unsigned)first;
            ng += 1;
            ms += 1;
            dq = fixq32(nz, bw + 1);
            cq = fixq32(ng, nz);
            if (nz == bw + 1) { disp_sum += 1ull << 32; ++disp_sq.hi; }
            if (ng == nz) clust_sum += 1ull << 32;
        }
        nnz_min = min(nnz_min, nz);
        nnz_max = max(nnz_max, nz);
        nnz_sum += nz;
        nnz_sq += (u64)nz * nz;
        bw_min = min(bw_min, bw);
        bw_max = max(bw_max, bw);
        bw_sum += bw;
        bw_sq.add((u64)bw * bw);
        disp_sum += dq;
        disp_sq.add((u64)dq * dq);
        clust_sum += cq;
        ng_sum += ng;
        ms_sum += ms;
    }

    // minima as complements; the 128-bit sums apart
    __device__ __forceinline__ void words(u64* t, unsigned err, u128 bw_sq, u128 disp_sq) {
        const u64 m32 = 0xffffffffull;
        t[0] = nnz_min == 0xffffffffu ? 0 : ~(u64)nnz_min;
        t[1] = nnz_max; t[2] = nnz_sum; t[3] = nnz_sq;
        t[4] = bw_min == 0xffffffffu ? 0 : ~(u64)bw_min;
        t[5] = bw_max; t[6] = bw_sum;
        t[7] = disp_sum;
        t[8] = clust_sum;
        t[9] = ng_sum; t[10] = ms_sum; t[11] = err;
        t[12] = (u64)bw_sq & m32; t[13] = (u64)bw_sq >> 32; t[14] = (u64)(bw_sq >> 64);
        t[15] = (u64)disp_sq & m32; t[16] = (u64)disp_sq >> 32; t[17] = (u64)(disp_sq >> 64);
    }
};

// word f of two partials combined: 0, 1, 4 and 5 are maxima, 11 error bits
__device__ __forceinline__ u64 merge_word(int f, u64 a, u64 b)
{
    if (f == 0 || f == 1 || f == 4 || f == 5) return max(a, b);
    return f == 11 ? (a | b) : a + b;
}

// Warp reductions, then the block's words added to one of the kSlots sets.
// Validation alone adds the error bits.  (One set, 15 atomics from every
// block to the same line, took longer than the pass over short matrices.)
template <bool FEATURES>
__device__ void flush_block(RowAgg& r, unsigned err, u64 (*s_red)[kFields], FeatCtl* ctl)
{
    err = __reduce_or_sync(FULL_MASK, err);
    const int w = threadIdx.x >> 5;
    u128 bw_sq = 0, disp_sq = 0;
    if (FEATURES) {
        r.nnz_min = __reduce_min_sync(FULL_MASK, r.nnz_min);
        r.nnz_max = __reduce_max_sync(FULL_MASK, r.nnz_max);
        r.bw_min = __reduce_min_sync(FULL_MASK, r.bw_min);
        r.bw_max = __reduce_max_sync(FULL_MASK, r.bw_max);
        r.nnz_sum = warp_sum_u64(r.nnz_sum);
        r.nnz_sq = warp_sum_u64(r.nnz_sq);
        r.bw_sum = warp_sum_u64(r.bw_sum);
        bw_sq = warp_sum_u128(r.bw_sq.value());
        r.disp_sum = warp_sum_u64(r.disp_sum);
        disp_sq = warp_sum_u128(r.disp_sq.value());
        r.clust_sum = warp_sum_u64(r.clust_sum);
        r.ng_sum = warp_sum_u64(r.ng_sum);
        r.ms_sum = warp_sum_u64(r.ms_sum);
    }
    if ((threadIdx.x & 31) == 0) r.words(s_red[w], err, bw_sq, disp_sq);
    __syncthreads();
    const int f = threadIdx.x;
    if (f < kFields && (FEATURES || f == 11)) {
        u64 t = s_red[0][f];
        for (int k = 1; k < kFT / 32; ++k) t = merge_word(f, t, s_red[k][f]);
        u64* to = &ctl->slot[blockIdx.x % kSlots][f];
        if (t == 0) return;
        if (f == 0 || f == 1 || f == 4 || f == 5) atomicMax(to, t);
        else if (f == 11) atomicOr(to, t);
        else atomicAdd(to, t);
    }
}

// Called by every thread of a block that has flushed: true in the block that
// comes last of n_blocks (nothing waits), which then sees every flush.
__device__ __forceinline__ bool last_to_flush(unsigned* done, unsigned n_blocks)
{
    __shared__ bool s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(done, 1u) == n_blocks - 1;
    __syncthreads();
    if (s_last) __threadfence();
    return s_last;
}

// The last block: the sets' words combined, written to the host's buffer, and
// the counters reset for the next call.
__device__ __forceinline__ void publish(FeatCtl* ctl, FeatAcc* host)
{
    const int f = threadIdx.x;
    if (f < kFields) {
        u64 t = 0;
#pragma unroll 16
        for (int i = 0; i < kSlots; ++i) t = merge_word(f, t, __ldcg(&ctl->slot[i][f]));
        reinterpret_cast<u64*>(host)[f] = t;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kSlots * kFields; i += kFT) (&ctl->slot[0][0])[i] = 0;
    if (threadIdx.x == 0) ctl->n_long = ctl->n_pieces = ctl->done_pass = ctl->done_long = 0;
}

// The warp-wide scan of the columns.  A lane takes eight consecutive elements
// per step (two 16-byte loads), a warp 256, a batch is four steps, whose
// loads are in flight together.  Per element and test one subtraction
// and one funnel shift collect a sign bit:
//   g    1 + prev - c < 0        the column does not follow its predecessor by
//                                one (for increasing columns)
//   m    lb8 + prev - c < 0      it lies more than a line after it: 8 d >
//                                line_bytes, that is d > lb8 =
//                                floor(line_bytes / 8) for an integer d
//   bad  c - prev - 1 < 0        it does not lie after it
// and a running maximum of the columns as unsigned values finds any outside
// [0, n_cols).  Columns in range make every difference exact; with one out of
// range the call returns an error and the counts are not used.  The predecessor
// of a lane's first element is its neighbour lane's last one, below lane 0
// lane 31's of the step before.
// Bound by instruction issue and the waits between a tile's loads
// (ncu: 2.3 instructions a clock, DRAM 34 %).  Measured on a 100^3 27-point
// stencil / 1M Zipf rows: 40 / 39 us; one element per lane with a ballot per
// test (18 instructions where this takes 8) 57 / 66 us; a lane walking its own
// row 56 / 60 us (rows of at most 64; the longer ones then took 93 us).
//
// The bits go to shared memory as bytes, element i of the batch to bit i % 8
// of byte i / 8, so that 32 consecutive elements form a word.
struct ColTest {
    const int* ci;
    int64_t nnz;
    unsigned n_cols;
    int lb8;    // floor(line_bytes / 8)
    int shift;  // elements ci lies past a 16-byte boundary
};
constexpr int kStep = 256, kBatch = 1024;
struct BatchBits {
    unsigned g[kBatch / 32], m[kBatch / 32], bad[kBatch / 32];
};

// eight columns from element j on (ci + j on a 16-byte boundary); elements
// outside [0, nnz) read as 0
__device__ __forceinline__ void load8(const ColTest& t, int64_t j, int (&c)[8])
{
    if (j >= 0 && j + 8 <= t.nnz) {
        const int4 a = __ldg(reinterpret_cast<const int4*>(t.ci + j)), b = __ldg(reinterpret_cast<const int4*>(t.ci + j) + 1);
        c[0] = a.x; c[1] = a.y; c[2] = a.z; c[3] = a.w;
        c[4] = b.x; c[5] = b.y; c[6] = b.z; c[7] = b.w;
    } else {
#pragma unroll
        for (int u = 0; u < 8; ++u) c[u] = j + u >= 0 && j + u < t.nnz ? __ldg(t.ci + j + u) : 0;
    }
}

// the batch that covers element k: its first element (may be negative)
__device__ __forceinline__ int64_t batch_start(const ColTest& t, int64_t k) { return ((k + t.shift) & ~(int64_t)7) - t.shift; }

// one step: the lane's eight columns to its bits of the three tests (of bad
// alone for validation)
template <bool FEATURES>
__device__ __forceinline__ void step_bits(const ColTest& t, const int (&c)[8], int lane, int& carry, unsigned& g, unsigned& m,
                                          unsigned& bad, unsigned& top)
{
    const int turned = __shfl_sync(FULL_MASK, c[7], (lane + 31) & 31);
    const int before = lane == 0 ? carry : turned;
    carry = turned;
    g = m = bad = 0;
#pragma unroll
    for (int u = 7; u >= 0; --u) {
        const unsigned cu = (unsigned)c[u], pu = (unsigned)(u > 0 ? c[u - 1] : before);
        if (FEATURES) {
            g = __funnelshift_l(1u + pu - cu, g, 1);
            m = __funnelshift_l((unsigned)t.lb8 + pu - cu, m, 1);
        }
        bad = __funnelshift_l(cu - pu - 1u, bad, 1);
        top = max(top, cu);
    }
}

// the lane's columns of the batch's four steps, all loads in flight together
__device__ __forceinline__ void load_batch(const ColTest& t, int64_t k0, int len, int lane, int (&c)[4][8], int& carry)
{
    carry = k0 > 0 ? __ldg(t.ci + k0 - 1) : 0;  // the element before, meaningful in lane 0
#pragma unroll
    for (int h = 0; h < kBatch / kStep; ++h) {
        const int i = h * kStep + lane * 8;
        if (i < len) {
            load8(t, k0 + i, c[h]);
        } else {
#pragma unroll
            for (int u = 0; u < 8; ++u) c[h][u] = 0;
        }
    }
}

// scans len <= kBatch elements from k0 = batch_start(...) on (rounded up to a
// step's lanes) and leaves their bits in B
template <bool FEATURES>
__device__ __forceinline__ void scan_batch(const ColTest& t, int64_t k0, int len, int lane, BatchBits& B, unsigned& top)
{
    int c[kBatch / kStep][8], carry;
    load_batch(t, k0, len, lane, c, carry);
    uint8_t* bytes = reinterpret_cast<uint8_t*>(&B) + lane;
#pragma unroll
    for (int h = 0; h < kBatch / kStep; ++h) {
        if (h * kStep >= len) break;  // whole warps
        unsigned g, m, bad;
        step_bits<FEATURES>(t, c[h], lane, carry, g, m, bad, top);
        if (FEATURES) {
            bytes[h * 32] = (uint8_t)g;
            bytes[kBatch / 8 + h * 32] = (uint8_t)m;
        }
        bytes[2 * (kBatch / 8) + h * 32] = (uint8_t)bad;
    }
}

// adds the bits of elements [p, es) of the batch
template <bool FEATURES>
__device__ __forceinline__ void count_bits(const BatchBits& B, int p, int es, unsigned& ng, unsigned& ms, unsigned& any_bad)
{
    while (p < es) {
        const int i = p >> 5, next = (p | 31) + 1;
        unsigned mask = 0xffffffffu << (p & 31);
        if (es < next) mask &= (1u << (es & 31)) - 1u;
        if (FEATURES) {
            ng += __popc(B.g[i] & mask);
            ms += __popc(B.m[i] & mask);
        }
        any_bad |= B.bad[i] & mask;
        p = next;
    }
}

// Rows of at most kLongRow nonzeros: warps take tiles of 32 consecutive
// rows, a lane per row.  A lane walking its own row would read 32 places of
// colind per instruction and run its tile as long as the tile's longest row;
// instead the warp streams the tile's nonzeros, which are contiguous, in
// batches (scan_batch, coalesced), and each lane then counts the bits of its
// row in the batch's words.  The first element of a row has no predecessor:
// its bit is left out.  The per-row arithmetic (two ratios, 128-bit sums)
// runs on all 32 lanes.  Longer rows are listed in pieces of kPiece nonzeros
// for k_feature_long, which their streaming skips: a tile costs at most 32
// kLongRow elements.  One resident grid strides over the tiles.

struct LongScratch {
    FeatCtl* ctl;
    int4* piece;      // [max_pieces] long row's list index, first element, row begin, row end
    int2* row;        // [max_long] ng and ms of a long row's finished pieces
    unsigned* done;   // [max_long] pieces finished
    unsigned max_long, max_pieces;
};

template <bool FEATURES>
__global__ void __launch_bounds__(kFT, kFeatBlocks)
k_feature_pass(int64_t n_rows, int64_t n_cols, int64_t nnz, const int* __restrict__ rp,
               const int* __restrict__ ci, int64_t line_bytes, LongScratch w, FeatAcc* __restrict__ host)
{
    __shared__ u64 s_red[kFT / 32][kFields];
    __shared__ BatchBits s_bits[kFT / 32];
    const int lane = threadIdx.x & 31;
    BatchBits& bits = s_bits[threadIdx.x >> 5];
    RowAgg r;
    unsigned err = 0, top = 0;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (rp[0] != 0) err |= 1;
        if ((int64_t)rp[n_rows] != nnz) err |= 2;
    }
    const int64_t n_tiles = (n_rows + 31) / 32;
    const int64_t n_warps = (int64_t)gridDim.x * (kFT / 32);
    const ColTest t{ci, nnz, (unsigned)n_cols, (int)(line_bytes >> 3), (int)((uintptr_t)ci >> 2 & 3)};
    int64_t tile = ((int64_t)blockIdx.x * kFT + threadIdx.x) / 32;
    // the row pointers of the next tile are loaded one tile ahead
    int nb = 0, ne = 0;
    auto fetch = [&](int64_t tl) {
        const int64_t row = tl * 32 + lane;
        if (row < n_rows) { nb = rp[row]; ne = rp[row + 1]; }
    };
    fetch(tile);
    for (; tile < n_tiles; tile += n_warps) {
        const int64_t row = tile * 32 + lane;
        // [b, e): the row when it is valid and not long, else empty
        int b = nb, e = ne;
        if (tile + n_warps < n_tiles) fetch(tile + n_warps);
        bool row_ok = false, is_long = false;
        if (row < n_rows) {
            if (b < 0 || e < b || e > nnz) err |= 4;
            else if (e - b > kLongRow) is_long = true;
            else row_ok = true;
        }
        // long rows: a list entry each and one per piece (pieces start on the
        // scan's boundaries), with one pair of atomics for the tile's rows
        // (with a pair for each, one after another, 200 rows of 1100 take 48
        // us in place of 33, 20,000 rows of 1030 94 in place of 68);
        // overlapping rows (a rowptr that is not monotone) can list more than
        // the buffers hold, and the error flag is set for them
        if (const unsigned longs = __ballot_sync(FULL_MASK, is_long)) {
            unsigned q = 0, p0 = 0;
            if (lane == 0) q = atomicAdd(&w.ctl->n_long, (unsigned)__popc(longs));
            q = __shfl_sync(FULL_MASK, q, 0) + __popc(longs & ((1u << lane) - 1u));
            const int l0 = (int)batch_start(t, b);
            unsigned np = 0;
            if (is_long && q < w.max_long) {
                np = (unsigned)((e - (int64_t)l0 + kPiece - 1) / kPiece);
                w.row[q] = make_int2(0, 0);
                w.done[q] = 0;
            } else if (is_long) {
                err |= 4;
            }
            unsigned upto = np;  // pieces of the tile's rows up to this one
            if (longs & (longs - 1)) {
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned v = __shfl_up_sync(FULL_MASK, upto, o);
                    if (lane >= o) upto += v;
                }
            }
            const int last_long = 31 - __clz((int)longs);
            if (lane == last_long) p0 = atomicAdd(&w.ctl->n_pieces, upto);
            p0 = __shfl_sync(FULL_MASK, p0, last_long) + upto - np;
            // every entry below n_pieces that the buffer holds is written
            const unsigned room = p0 < w.max_pieces ? w.max_pieces - p0 : 0u;
            if (np > room) err |= 4;
            const unsigned mine = min(np, room);
            for (unsigned todo = longs; todo; todo &= todo - 1) {
                const int src = __ffs(todo) - 1;
                const int rq = __shfl_sync(FULL_MASK, (int)q, src), rl = __shfl_sync(FULL_MASK, l0, src),
                          rb = __shfl_sync(FULL_MASK, b, src), re = __shfl_sync(FULL_MASK, e, src);
                const unsigned rp0 = __shfl_sync(FULL_MASK, p0, src), n = __shfl_sync(FULL_MASK, mine, src);
                for (unsigned p = lane; p < n; p += 32)
                    w.piece[rp0 + p] = make_int4(rq, rl + (int)(p * kPiece), rb, re);
            }
        }
        if (!row_ok) b = e = 0;
        unsigned ng = 0, ms = 0;
        int first = 0, last = 0;
        // A tile of rows of at most kShortRow: a lane's few loads, in flight
        // together, cover what the streaming would, without its batches and
        // shared memory (bound by issue: 8M rows of 2, the call 188 us
        // streamed and 125 so; 7-point stencil 128^3 70 and 56; of at most 4:
        // 118 and 71; more than 8 gains nothing).
        const int nz = e - b;
        if (__reduce_max_sync(FULL_MASK, (unsigned)nz) <= kShortRow) {
            // counted within the row: b + u can pass 2^31 - 1 in the last rows
            int c[kShortRow];
#pragma unroll
            for (int u = 0; u < kShortRow; ++u) c[u] = u < nz ? __ldg(ci + b + u) : 0;
            first = last = c[0];
#pragma unroll
            for (int u = 0; u < kShortRow; ++u) {
                top = max(top, (unsigned)c[u]);
                if (u > 0 && u < nz) {
                    const int d = (int)((unsigned)c[u] - (unsigned)last);
                    if (d <= 0) err |= 16;
                    ng += d > 1;
                    ms += d > t.lb8;
                    last = c[u];
                }
            }
            if (FEATURES && row_ok) r.add((unsigned)nz, first, last, ng, ms);
            continue;
        }
        if (FEATURES && e > b) {
            first = ci[b];
            last = ci[e - 1];
        }
        const int hi = __reduce_max_sync(FULL_MASK, e);
        for (int cur = 0;;) {
            // the next element any row still needs (skips the long rows' parts)
            const unsigned k = __reduce_min_sync(FULL_MASK, e > cur && e > b ? (unsigned)max(b, cur) : 0xffffffffu);
            if (k == 0xffffffffu) break;
            const int64_t k0 = batch_start(t, k);
            const int len = (int)min((int64_t)kBatch, hi - k0);
            scan_batch<FEATURES>(t, k0, len, lane, bits, top);
            __syncwarp();
            // this row's elements in the batch, without the row's first
            const int64_t k1 = k0 + len;
            unsigned any_bad = 0;
            if (e > b && (int64_t)b + 1 < k1) count_bits<FEATURES>(bits, (int)(max((int64_t)max(b + 1, cur), k0) - k0), (int)(min((int64_t)e, k1) - k0), ng, ms, any_bad);
            if (any_bad) err |= 16;
            __syncwarp();
            cur = (int)k1;
        }
        if (FEATURES && row_ok) r.add((unsigned)(e - b), first, last, ng, ms);
    }
    if (top > 0 && top >= t.n_cols) err |= 8;
    flush_block<FEATURES>(r, err, s_red, w.ctl);
    // without long rows the result is complete here
    if (last_to_flush(&w.ctl->done_pass, gridDim.x) && __ldcg(&w.ctl->n_pieces) == 0) publish(w.ctl, host);
}

// The long rows' pieces, a warp each.  A piece's counts, taken from the
// lanes' bits without a detour through shared memory, are added to its row's;
// the warp that completes a row's last piece (a ticket per row) adds the row
// to its aggregates.  Integer sums: the result does not depend on the order.
// The block that finishes last publishes the totals.
template <bool FEATURES>
__global__ void __launch_bounds__(kFT, kFeatBlocks)
k_feature_long(int64_t n_cols, int64_t nnz, const int* __restrict__ ci, int64_t line_bytes, LongScratch w,
               FeatAcc* __restrict__ host)
{
    __shared__ u64 s_red[kFT / 32][kFields];
    const unsigned total = min(__ldcg(&w.ctl->n_pieces), w.max_pieces);
    if (total == 0) return;  // published by the pass
    const int lane = threadIdx.x & 31;
    RowAgg r;
    unsigned err = 0, top = 0;
    const ColTest t{ci, nnz, (unsigned)n_cols, (int)(line_bytes >> 3), (int)((uintptr_t)ci >> 2 & 3)};
    const unsigned n_warps = gridDim.x * (kFT / 32);
    unsigned it = (blockIdx.x * kFT + threadIdx.x) / 32;
    int4 next = it < total ? w.piece[it] : make_int4(0, 0, 0, 0);
    for (; it < total; it += n_warps) {
        const int4 pc = next;
        if (it + n_warps < total) next = w.piece[it + n_warps];
        const int b = pc.z, e = pc.w;
        const int64_t p0 = pc.y;  // may be negative
        const int plen = (int)min((int64_t)e - p0, kPiece);
        unsigned ng = 0, ms = 0, any_bad = 0;
        for (int at = 0; at < plen; at += kBatch) {
            const int64_t k0 = p0 + at;
            const int len = min(kBatch, plen - at);
            int c[kBatch / kStep][8], carry;
            load_batch(t, k0, len, lane, c, carry);
            // elements of the batch that count: after the row's first, before its end
            const int from = (int)max((int64_t)0, (int64_t)b + 1 - k0);
#pragma unroll
            for (int h = 0; h < kBatch / kStep; ++h) {
                unsigned g, m, bad;
                step_bits<FEATURES>(t, c[h], lane, carry, g, m, bad, top);
                const int i = h * kStep + lane * 8;  // the lane's first element of the step
                const unsigned keep = (0xffu << min(max(from - i, 0), 8)) & ((1u << min(max(len - i, 0), 8)) - 1u);
                ng += __popc(g & keep);
                ms += __popc(m & keep);
                any_bad |= bad & keep;
            }
        }
        if (any_bad) err |= 16;
        if (FEATURES) {
            ng = __reduce_add_sync(FULL_MASK, ng);
            ms = __reduce_add_sync(FULL_MASK, ms);
            if (lane == 0) {
                int2* tot = w.row + pc.x;
                atomicAdd(&tot->x, (int)ng);
                atomicAdd(&tot->y, (int)ms);
                __threadfence();
                const unsigned np = (unsigned)((e - batch_start(t, b) + kPiece - 1) / kPiece);
                if (atomicAdd(&w.done[pc.x], 1u) == np - 1) {
                    __threadfence();
                    const int2 all = __ldcg(tot);
                    r.add((unsigned)(e - b), ci[b], ci[e - 1], (unsigned)all.x, (unsigned)all.y);
                }
            }
        }
    }
    if (top > 0 && top >= t.n_cols) err |= 8;
    flush_block<FEATURES>(r, err, s_red, w.ctl);
    if (last_to_flush(&w.ctl->done_long, gridDim.x)) publish(w.ctl, host);
}

double sd_from_sums(u64 n, u64 s1, u128 s2)
{
    const u128 num = (u128)n * s2 - (u128)s1 * (u128)s1;
    return sqrt((double)num) / (double)n;
}

// the 128-bit sum of digits of 32, 32 and 64 bits
u128 digits(const u64 (&d)[3]) { return ((u128)d[2] << 64) + ((u128)d[1] << 32) + d[0]; }

float lg1p(double v) { return (float)log2(1.0 + v); }

// page-locked result buffer the last block writes, one per host thread
thread_local FeatAcc* t_host_acc = nullptr;
// device scratch of the pass (counters first), per host thread; grows, never
// shrinks.  The counters are 0 between calls; after a failed call the scratch
// is cleared again.
thread_local void* t_scratch = nullptr;
thread_local size_t t_scratch_bytes = 0;
thread_local int t_scratch_device = -1;
thread_local bool t_scratch_clean = false;

}  // namespace

int auto_threads_per_row(double mean_nnz)
{
    int T = 1;
    while (T < 32 && T < mean_nnz) T *= 2;
    return T;
}

spmv_status feature_pass_enqueue(const spmv_csr_t* A, int32_t line_bytes, bool features, cudaStream_t s)
{
    spmv_status st = check_csr_args(A);
    if (st != SPMV_OK) return st;
    DeviceInfo dev;
    st = current_device(&dev);
    if (st != SPMV_OK) return st;

    if (!t_host_acc) {
        void* p = nullptr;
        if (cudaMallocHost(&p, sizeof(FeatAcc)) != cudaSuccess)
            return fail(SPMV_ERR_NOMEM, "cudaMallocHost for the feature readback failed");
        t_host_acc = static_cast<FeatAcc*>(p);
    }
    cudaError_t e = cudaSuccess;
    if (A->n_rows > 0) {
        const int64_t n_tiles = (A->n_rows + 31) / 32;
        const int64_t resident = (int64_t)dev.sm_count * kFeatBlocks;
        const unsigned blocks = (unsigned)std::min<int64_t>((n_tiles + kFT / 32 - 1) / (kFT / 32), resident);
        // long rows and pieces a valid matrix can hold
        const int64_t max_long = std::min<int64_t>(A->n_rows, A->nnz / (kLongRow + 1) + 1);
        const int64_t max_pieces = A->nnz / kPiece + 2 * max_long;
        const unsigned lblocks = (unsigned)std::min<int64_t>((max_pieces + kFT / 32 - 1) / (kFT / 32), resident);
        LongScratch w;
        size_t at = 0;
        auto place = [&](size_t bytes) { const size_t p = at; at += (bytes + 15) / 16 * 16; return p; };
        const size_t o_ctl = place(sizeof(FeatCtl)), o_piece = place(sizeof(int4) * max_pieces),
                     o_row = place(sizeof(int2) * max_long), o_done = place(sizeof(unsigned) * max_long);
        if (t_scratch_device != dev.device || t_scratch_bytes < at) {
            if (t_scratch) cudaFree(t_scratch);
            t_scratch = nullptr;
            t_scratch_bytes = 0;
            t_scratch_clean = false;
            e = device_alloc(&t_scratch, at);
            if (e == cudaSuccess) { t_scratch_bytes = at; t_scratch_device = dev.device; }
        }
        if (e == cudaSuccess && !t_scratch_clean) e = cudaMemsetAsync(t_scratch, 0, t_scratch_bytes, s);
        t_scratch_clean = false;  // until this call has completed
        unsigned char* base = static_cast<unsigned char*>(t_scratch);
        w.ctl = reinterpret_cast<FeatCtl*>(base + o_ctl);
        w.piece = reinterpret_cast<int4*>(base + o_piece);
        w.row = reinterpret_cast<int2*>(base + o_row);
        w.done = reinterpret_cast<unsigned*>(base + o_done);
        w.max_long = (unsigned)max_long;
        w.max_pieces = (unsigned)max_pieces;
        if (e == cudaSuccess) {
            if (features) k_feature_pass<true><<<blocks, kFT, 0, s>>>(A->n_rows, A->n_cols, A->nnz, A->rowptr, A->colind, line_bytes, w, t_host_acc);
            else k_feature_pass<false><<<blocks, kFT, 0, s>>>(A->n_rows, A->n_cols, A->nnz, A->rowptr, A->colind, line_bytes, w, t_host_acc);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) {
            if (features) k_feature_long<true><<<lblocks, kFT, 0, s>>>(A->n_cols, A->nnz, A->colind, line_bytes, w, t_host_acc);
            else k_feature_long<false><<<lblocks, kFT, 0, s>>>(A->n_cols, A->nnz, A->colind, line_bytes, w, t_host_acc);
            e = cudaGetLastError();
        }
        if (e != cudaSuccess) return cuda_fail(e, "feature pass");
    } else {
        memset(t_host_acc, 0, sizeof(FeatAcc));
    }
    return SPMV_OK;
}

spmv_status feature_pass_verdict(const spmv_csr_t* A)
{
    t_scratch_clean = true;
    u64 err = t_host_acc->err;
    if (A->n_rows == 0 && A->nnz != 0) err |= 2;
    if (err) {
        std::string m = "invalid CSR:";
        if (err & 1) m += " rowptr[0] != 0;";
        if (err & 2) m += " rowptr[n_rows] != nnz;";
        if (err & 4) m += " rowptr decreasing or out of [0, nnz];";
        if (err & 8) m += " column index out of [0, n_cols);";
        if (err & 16) m += " columns not strictly increasing within a row;";
        return fail(SPMV_ERR_INVALID_CSR, m);
    }
    return SPMV_OK;
}

spmv_status run_feature_pass(const spmv_csr_t* A, int32_t line_bytes, spmv_features_t* out,
                             cudaStream_t s)
{
    if (line_bytes <= 0) line_bytes = 128;
    spmv_status st = feature_pass_enqueue(A, line_bytes, out != nullptr, s);
    if (st != SPMV_OK) return st;
    SPMV_CUDA_TRY(cudaStreamSynchronize(s));
    if ((st = feature_pass_verdict(A)) != SPMV_OK) return st;
    const FeatAcc& h = *t_host_acc;
    DeviceInfo dev;
    if ((st = current_device(&dev)) != SPMV_OK) return st;
    if (!out) return SPMV_OK;

    spmv_features_t f = {};
    const int64_t N = A->n_rows, M = A->n_cols, NNZ = A->nnz;
    f.n_rows = N; f.n_cols = M; f.nnz = NNZ;
    f.line_bytes = line_bytes;
    f.l2_bytes = dev.l2_bytes;
    f.working_set_bytes = 4 * (N + 1) + 12 * NNZ + 8 * M + 8 * N;
    f.nnz_min = N > 0 ? (int64_t)~h.nnz_min_c : 0;
    f.nnz_max = (int64_t)h.nnz_max;
    f.nnz_sum = h.nnz_sum;
    f.nnz_sumsq_lo = h.nnz_sumsq;
    f.nnz_sumsq_hi = 0;
    f.bw_min = N > 0 ? (int64_t)~h.bw_min_c : 0;
    f.bw_max = (int64_t)h.bw_max;
    f.bw_sum = h.bw_sum;
    const u128 bw_s2 = digits(h.bw_sq), dq_s2 = digits(h.disp_sq);
    f.bw_sumsq_lo = (uint64_t)bw_s2;
    f.bw_sumsq_hi = (uint64_t)(bw_s2 >> 64);
    f.disp_sum = h.disp_sum;
    f.disp_sumsq_lo = (uint64_t)dq_s2;
    f.disp_sumsq_hi = (uint64_t)(dq_s2 >> 64);
    f.clust_sum = h.clust_sum;
    f.ngroups_sum = h.ngroups_sum;
    f.misses_sum = h.misses_sum;

    f.size = f.working_set_bytes <= f.l2_bytes ? 1.0 : 0.0;
    if (N > 0 && M > 0) f.density = (double)NNZ / ((double)N * (double)M);
    if (N > 0) {
        const double q32 = 1.0 / 4294967296.0;
        const double dn = (double)N;
        f.nnz_avg = (double)f.nnz_sum / dn;
        f.nnz_sd = sd_from_sums((u64)N, f.nnz_sum, (u128)f.nnz_sumsq_lo);
        f.bw_avg = (double)f.bw_sum / dn;
        f.bw_sd = sd_from_sums((u64)N, f.bw_sum, bw_s2);
        f.disp_avg = ((double)f.disp_sum / dn) * q32;
        f.disp_sd = sd_from_sums((u64)N, f.disp_sum, dq_s2) * q32;
        f.clustering = ((double)f.clust_sum / dn) * q32;
        f.miss_ratio = (double)f.misses_sum / dn;
    }
    const double dens = f.density > 0x1p-64 ? f.density : 0x1p-64;
    f.vec[0] = (float)f.size;
    f.vec[1] = (float)log2(dens);
    f.vec[2] = lg1p((double)f.nnz_min);
    f.vec[3] = lg1p((double)f.nnz_max);
    f.vec[4] = lg1p(f.nnz_avg);
    f.vec[5] = lg1p(f.nnz_sd);
    f.vec[6] = lg1p((double)f.bw_min);
    f.vec[7] = lg1p((double)f.bw_max);
    f.vec[8] = lg1p(f.bw_avg);
    f.vec[9] = lg1p(f.bw_sd);
    f.vec[10] = (float)f.disp_avg;
    f.vec[11] = (float)f.disp_sd;
    f.vec[12] = (float)f.clustering;
    f.vec[13] = lg1p(f.miss_ratio);
    f.vec[14] = lg1p((double)N);
    f.vec[15] = lg1p((double)NNZ);
    *out = f;
    return SPMV_OK;
}

}  // namespace spmvlib
