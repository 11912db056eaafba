// Conjugate gradients around the library's SpMV (Section 1 names iterative
// solvers as the setting in which SpMV's selection overhead is amortised).
//
// Every iteration: q = A p (the inner prepared SpMV, e.g. COMPRESSED with
// FP32 or BF16 values), alpha = rs / (p.q), x += alpha p, r -= alpha q,
// rs' = r.r, beta = rs'/rs, p = r + beta p -- in one cooperative launch for
// the whole loop where the vectors fit the chip's shared memory
// (k_cg_resident), else in three kernels.  Every `refine` iterations the
// residual is instead recomputed in FP64 as r = b - A x with the exact
// prepared SpMV and the search direction restarts from it (p = r): iterative
// refinement with CG sweeps on the low-precision operator.  Vectors,
// dot products and scalars are FP64 and stay on the device: there is no host
// synchronisation inside the loop, so the loop can run from a CUDA graph.
//
// Dot products are deterministic: each block leaves its sum, and the blocks
// of the next kernel add the sums in the same order.
//
// With a SLICED inner matrix without long rows (none above its cap) q = A p and p.q
// are one kernel, and when that matrix sums in FP32 the p update also writes
// p's FP32 copy, so no separate conversion of p runs per iteration.
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "ptx.cuh"
#include "sliced.cuh"

namespace spmvlib {
namespace {

constexpr int kCT = 512;
// The vector kernels give each thread kUnr elements kCT apart per pass of
// the grid-stride loop and load all of them before any arithmetic, so a
// thread keeps several independent loads of every vector in flight.
constexpr int kUnr = 4;

__device__ __forceinline__ int64_t first_index() { return (int64_t)blockIdx.x * kCT * kUnr + threadIdx.x; }
__device__ __forceinline__ int64_t grid_step() { return (int64_t)gridDim.x * kCT * kUnr; }

// rs[t & 1] is r.r after iteration t, so that the kernel that stores one does
// not overwrite the one its other blocks still read.
struct CgState {
    double rs[2];
};

// A dot product is left as one sum per block, and the blocks of the kernel
// that needs it add them for themselves, in the same order (deterministic),
// while their first vector loads are under way.  A last block that adds them
// for everyone costs its kernel a ticket, two fences, the sums' loads and the
// division on top of the slowest block, about 3 us.  Both additions are done
// by one warp per block: a level of an FP64 shuffle tree executed by all eight
// shares the SM's two FP64 lanes with every other block's.
__device__ __forceinline__ double warp_total(double t)
{
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
}

// the block's sum of v to part[blockIdx.x]
__device__ __forceinline__ void leave_sum(double v, double* __restrict__ part)
{
    __shared__ double red[kCT];
    red[threadIdx.x] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        double a[4] = {};
#pragma unroll
        for (int i = 0; i < kCT; i += 128)
#pragma unroll
            for (int u = 0; u < 4; ++u) a[u] += red[i + 32 * u + threadIdx.x];
        const double t = warp_total((a[0] + a[1]) + (a[2] + a[3]));
        if (threadIdx.x == 0) part[blockIdx.x] = t;
    }
}

// the same with a tree in every warp first, for a kernel that wants the L1
// that the other's shared memory takes
__device__ __forceinline__ void leave_sum_small(double v, double* __restrict__ part)
{
    __shared__ double red[kCT / 32];
    v = warp_total(v);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        double t = threadIdx.x < kCT / 32 ? red[threadIdx.x] : 0.0;
        for (int o = kCT / 64; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (threadIdx.x == 0) part[blockIdx.x] = t;
    }
}

// the sum of n sums (valid in the first warp, which alone calls this)
__device__ __forceinline__ double take_sum(const double* __restrict__ part, int n)
{
    constexpr int U = 16;  // sums a lane has in flight: 512 in one go
    double a[4] = {};
    for (int i = threadIdx.x; i < n; i += 32 * U) {
        double w[U];
#pragma unroll
        for (int u = 0; u < U; ++u) w[u] = i + 32 * u < n ? part[i + 32 * u] : 0.0;
#pragma unroll
        for (int u = 0; u < U; ++u) a[u & 3] += w[u];
    }
    return warp_total((a[0] + a[1]) + (a[2] + a[3]));
}

// alpha = rs / p.q, to every thread of the block
__device__ __forceinline__ double take_alpha(const double* __restrict__ part, int n, const CgState* st, int t)
{
    __shared__ double s_alpha;
    if (threadIdx.x < 32) {
        const double pq = take_sum(part, n);
        if (threadIdx.x == 0) s_alpha = st->rs[(t - 1) & 1] / pq;
    }
    __syncthreads();
    return s_alpha;
}

// p.q as the blocks' sums
__global__ void __launch_bounds__(kCT)
k_dot_pq(int64_t n, const double* __restrict__ p, const double* __restrict__ q, double* __restrict__ part)
{
    double v = 0.0;
    for (int64_t i0 = first_index(); i0 < n; i0 += grid_step()) {
        double pv[kUnr], qv[kUnr];
#pragma unroll
        for (int u = 0; u < kUnr; ++u) {
            const int64_t i = i0 + u * kCT;
            pv[u] = i < n ? p[i] : 0.0;
            qv[u] = i < n ? q[i] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < kUnr; ++u) v = fma(pv[u], qv[u], v);
    }
    leave_sum(v, part);
}

// x += alpha p and r -= alpha q (RECOMPUTE = false, alpha from p.q's sums) or r
// = b - q where q holds A x (RECOMPUTE = true); r.r as the blocks' sums.  (x
// updated beside p instead reads p once less, but leaves its dirty lines to
// the next product: no faster.)
template <bool RECOMPUTE>
__global__ void __launch_bounds__(kCT, 2)
k_update(int64_t n, double* __restrict__ x, const double* __restrict__ p, double* __restrict__ r,
         const double* __restrict__ q, const double* __restrict__ b, const double* __restrict__ pq_part, int n_pq,
         double* __restrict__ part, CgState* st, int t)
{
    double rv[kUnr], qv[kUnr], xv[kUnr], pv[kUnr];
    auto load = [&](int64_t i0) {
#pragma unroll
        for (int u = 0; u < kUnr; ++u) {
            const int64_t i = i0 + u * kCT;
            rv[u] = i < n ? (RECOMPUTE ? b[i] : r[i]) : 0.0;
            qv[u] = i < n ? q[i] : 0.0;
            if (!RECOMPUTE) {
                xv[u] = i < n ? x[i] : 0.0;
                pv[u] = i < n ? p[i] : 0.0;
            }
        }
    };
    int64_t i0 = first_index();
    load(i0);
    const double alpha = RECOMPUTE ? 0.0 : take_alpha(pq_part, n_pq, st, t);
    double v = 0.0;
    while (i0 < n) {
#pragma unroll
        for (int u = 0; u < kUnr; ++u) {
            const int64_t i = i0 + u * kCT;
            if (i < n) {
                if (!RECOMPUTE) x[i] = fma(alpha, pv[u], xv[u]);
                const double ri = RECOMPUTE ? rv[u] - qv[u] : fma(-alpha, qv[u], rv[u]);
                r[i] = ri;
                v = fma(ri, ri, v);
            }
        }
        i0 += grid_step();
        load(i0);
    }
    leave_sum(v, part);
}

// x += alpha p only (the refinement step recomputes r from the new x)
__global__ void __launch_bounds__(kCT)
k_axpy_x(int64_t n, double* __restrict__ x, const double* __restrict__ p, const double* __restrict__ pq_part, int n_pq,
         CgState* st, int t)
{
    const double alpha = take_alpha(pq_part, n_pq, st, t);
    for (int64_t i0 = first_index(); i0 < n; i0 += grid_step()) {
        double xv[kUnr], pv[kUnr];
#pragma unroll
        for (int u = 0; u < kUnr; ++u) {
            const int64_t i = i0 + u * kCT;
            xv[u] = i < n ? x[i] : 0.0;
            pv[u] = i < n ? p[i] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < kUnr; ++u)
            if (i0 + u * kCT < n) x[i0 + u * kCT] = fma(alpha, pv[u], xv[u]);
    }
}

// rs = r.r from the blocks' sums, recorded as sqrt(rs) in resid[t], and p = r
// + beta p: kNext beta = rs / rs before; kRestart beta = 0, the search restarts from the recomputed residual; kFirst p = r.
// With p32, also p's FP32 copy for a low-precision inner SpMV that sums in
// FP32 (the same rounding its own conversion of x would apply).
// 128^3 rows with BF16 values: 58.2 us an iteration, against 65.9 with a last
// block after each dot product and the conversions on the FP64 pipe (FP64
// values: 76.8 and 75.6; 72 with four elements in flight in the product, see
// kDotU).  Launched as programmatic dependents of one another
// the three kernels are slower (61.4): blocks that start early take room from
// the ones still running.
enum Step { kFirst, kNext, kRestart };
template <Step STEP>
__global__ void __launch_bounds__(kCT, 2)
k_update_p(int64_t n, double* __restrict__ p, const double* __restrict__ r, const double* __restrict__ rr_part, int n_rr, CgState* st, double* __restrict__ resid, int t,
           float* __restrict__ p32)
{
    __shared__ double s_beta;
    double pv[kUnr], rv[kUnr];
    auto load = [&](int64_t i0) {
#pragma unroll
        for (int u = 0; u < kUnr; ++u) {
            const int64_t i = i0 + u * kCT;
            rv[u] = i < n ? r[i] : 0.0;
            pv[u] = STEP != kFirst && i < n ? p[i] : 0.0;
        }
    };
    int64_t i0 = first_index();
    load(i0);
    if (threadIdx.x < 32 && (STEP == kNext || blockIdx.x == 0)) {
        const double rs = take_sum(rr_part, n_rr);
        if (threadIdx.x == 0) {
            if (STEP == kNext) s_beta = rs / st->rs[(t - 1) & 1];
            if (blockIdx.x == 0) {
                st->rs[t & 1] = rs;
                if (resid) resid[t] = sqrt(rs);
            }
        }
    }
    double beta = 0.0;
    if (STEP == kNext) {
        __syncthreads();
        beta = s_beta;
    }
    while (i0 < n) {
#pragma unroll
        for (int u = 0; u < kUnr; ++u) {
            const int64_t i = i0 + u * kCT;
            if (i < n) {
                const double v = STEP == kFirst ? rv[u] : fma(beta, pv[u], rv[u]);
                p[i] = v;
                if (p32) p32[i] = dev::round_f32(v);
            }
        }
        i0 += grid_step();
        load(i0);
    }
}

// Fused q = A p and p.q for a SLICED inner matrix without long rows: each
// lane computes its row's q_i (dev::slice_value / slice_value_lp, the same
// arithmetic as the SLICED kernels) and adds p_i q_i to its block's sum.
// Resident blocks per SM of the fused kernel: FP64 values fit 4 (32
// registers, four elements in flight per lane as in the SLICED product), the
// low-precision bodies need 40 registers, so 3.  Two elements in flight leave
// the FP64 kernel waiting on its gathers, at the mercy of the order in which
// the compiler places them: an iteration of 128^3 rows takes 200 us (27-point)
// and 78 (7-point), with the row looked up before the loop 182 and 75; four
// take 153 and 72, three 151 and 76, four on 48 warps of 40 registers 172 and 73.
template <typename VT>
constexpr int dot_blocks() { return sizeof(VT) == 8 ? 4 : 3; }
constexpr int kDotU = 4;

struct SlArgs {
    int64_t n_slices;
    const int* rowlen; const int* slice_len; const int64_t* slice_ptr; const int* perm;
    const int* col; const double* val; const uint16_t* off; const int* rowbase; const void* lowval;
    const void* scol;  // FP64 values: stored columns (int, or int16/int8 offsets from the row)
};

template <typename VT, bool OFF16, bool ACC32, typename CT = int>
__global__ void __launch_bounds__(kCT, dot_blocks<VT>())
k_sliced_dot(SlArgs a, const double* __restrict__ p, const float* __restrict__ p32,
             double* __restrict__ q, double* __restrict__ part)
{
    const int lane = threadIdx.x & 31;
    const int64_t n_warps = (int64_t)gridDim.x * (kCT / 32);
    double contrib = 0.0;
    // grid-stride over slices (a few blocks per SM): few sums
    for (int64_t s = ((int64_t)blockIdx.x * kCT + threadIdx.x) >> 5; s < a.n_slices; s += n_warps) {
        int row;
        double v;
        if constexpr (sizeof(VT) == 8)
            v = dev::slice_value<kDotU, CT>(s, lane, a.rowlen, a.slice_len, a.slice_ptr, a.perm,
                                            static_cast<const CT*>(a.scol), a.val, p, &row);
        else
            v = dev::slice_value_lp<OFF16 ? 2 : 1, VT, OFF16, ACC32>(s, lane, a.rowlen, a.slice_len, a.slice_ptr, a.perm,
                                                         a.col, a.off, a.rowbase,
                                                         static_cast<const VT*>(a.lowval), p, p32, &row);
        if (row >= 0) {
            q[row] = v;
            contrib = fma(p[row], v, contrib);
        }
    }
    leave_sum_small(contrib, part);
}

bool fusable(const spmv_prepared* P)
{
    return P->c.variant == SPMV_V7_SLICED && P->sl.n_long == 0 && P->sl.coding == 0 && P->A.n_rows > 0;
}

SlArgs sl_args(const spmv_prepared* P)
{
    const SlicedPlan& d = P->sl;
    return SlArgs{d.n_slices, d.rowlen, d.slice_len, d.slice_ptr, d.sigma > 1 ? d.perm : nullptr,
                  d.col, d.val, d.off, d.rowbase, d.lowval, d.scol};
}

unsigned sliced_dot_grid(const spmv_prepared* P)
{
    const int per_sm = P->sl.value_type == SPMV_VAL_F64 ? dot_blocks<double>() : dot_blocks<float>();
    const int64_t need = (32 * P->sl.n_slices + kCT - 1) / kCT;
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(need, (int64_t)P->sm_count * per_sm));
}

cudaError_t launch_sliced_dot(const spmv_prepared* P, const double* p, double* q, double* part, cudaStream_t s)
{
    const SlicedPlan& d = P->sl;
    const SlArgs a = sl_args(P);
    const unsigned grid = sliced_dot_grid(P);
    if (d.value_type == SPMV_VAL_F64) {
        if (d.cbytes == 1)
            k_sliced_dot<double, false, false, int8_t><<<grid, kCT, 0, s>>>(a, p, nullptr, q, part);
        else if (d.cbytes == 2)
            k_sliced_dot<double, false, false, int16_t><<<grid, kCT, 0, s>>>(a, p, nullptr, q, part);
        else
            k_sliced_dot<double, false, false, int><<<grid, kCT, 0, s>>>(a, p, nullptr, q, part);
    } else {
#define SPMV_CG_SL(VT, O16, A32) k_sliced_dot<VT, O16, A32><<<grid, kCT, 0, s>>>(a, p, d.x32, q, part)
#define SPMV_CG_SL_VT(VT)                                                                  \
    if (d.off16) { if (d.acc32) SPMV_CG_SL(VT, true, true); else SPMV_CG_SL(VT, true, false); } \
    else { if (d.acc32) SPMV_CG_SL(VT, false, true); else SPMV_CG_SL(VT, false, false); }
        if (d.value_type == SPMV_VAL_F32) { SPMV_CG_SL_VT(float) } else { SPMV_CG_SL_VT(__nv_bfloat16) }
#undef SPMV_CG_SL_VT
#undef SPMV_CG_SL
    }
    return cudaGetLastError();
}

// ---- the whole loop in one launch --------------------------------------------
// For small and middle-sized matrices the loop is bound not by memory but by
// launches and latency: three kernels an iteration, each a few microseconds
// of it (15 us an iteration at 36,000 rows).  Here one cooperative launch, one
// block per SM, runs every iteration.  A lane owns the same rows for the whole
// solve and keeps their x, r, p and q in shared memory, so per iteration only p
// (or its FP32 copy) goes through memory, and the blocks meet three times: for
// p.q, for r.r and when p is written.  The slices go round the warps of the
// grid; with up to three per warp their heads stay in registers (RT).
//
// A meeting: the block's first warp adds the block's values, stores the sum,
// arrives at one counter and waits until every block has; then it adds all
// blocks' sums.  Every block adds them in the same order, so alpha and beta
// are the same everywhere and the result is deterministic.  Two sets of sums
// are used in turn: a block that stores for meeting g + 2 has passed g + 1,
// so everyone has read the set of g.  One counter that a single thread per
// block polls costs 1.2 us on 144 blocks (296: 1.5); blocks that read each
// other's slots until all are filled cost 3.3 us (296: 6.0), clusters of 8
// that exchange through their leaders 2.6 us (3.3).  The launch is cooperative
// (all blocks resident), and each wait is bounded all the same: a block that
// gives up sets x and the remaining residuals to NaN and returns.
//
// Measured per iteration, against three launches from a graph, FP64 / BF16
// values: 7-point Laplacians of 33^3 rows 8.6 / 8.8 us against 14.7 / 14.5, 48^3
// 12.0 / 11.0 against 17.0 / 15.6, 64^3 17.5 / 14.9 against 22.1 / 17.8, 90^3
// 28.5 / 23.7 against 36.6 / 27.0, 101^3 36.0 / 28.0 against 44.3 / 33.0;
// 27-point 48^3 17.6 / 14.0 against 25.6 / 20.8, 64^3 34.3 / 22.6 against 36.0 /
// 25.7 (where it ends: resident_choice).  Beyond the shared memory of the chip
// (1.05 M rows) the state would go through memory again, and the three kernels
// with their 64 warps per SM are faster (128^3: 82 / 71 us here against 72 /
// 60).  Registers instead of shared memory for the state of three rows a lane
// are as fast; chunks of the matrix loaded ahead are not faster (64^3 18.7 /
// 16.1).
//
// A solve above 40,000 rows or so takes every SM, so that several on as many
// streams run one after another, where the three kernels of several overlap.
// Two such solves are no slower for it, many of middle size are: 16 of 200
// iterations on 8 streams take 12.5 ms at 33^3 rows (three kernels 20.4), 37.2 at
// 48^3 (22.5), 55 at 64^3 (38.5), 91 at 90^3 (98.7).
//
// The bound is a constant: as an argument of the launch (or a word that the
// waiting thread reads) it made some forms 1.4 % slower by other instruction
// orders.  A wait runs out all the same when the counter starts one short, as
// spmv_cg_wait_check has it.
constexpr uint64_t kMeetLimitNs = 2000000000ull;

struct Meeting {
    double* sums;       // [2][gridDim.x]
    unsigned* arrived;  // 0 at the start
    unsigned turn;
};

// Arrives and waits (one thread); false when the wait gave up.
__device__ __forceinline__ bool arrive_and_wait(Meeting& m)
{
    const unsigned target = m.turn * gridDim.x;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" :: "l"(m.arrived) : "memory");
    uint64_t t0 = 0;
    for (unsigned tries = 1;; ++tries) {
        unsigned v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(m.arrived) : "memory");
        if ((int)(v - target) >= 0) return true;
        if ((tries & 63) == 0) {
            const uint64_t now = ptx::global_ns();
            if (t0 == 0) t0 = now;
            else if (now - t0 > kMeetLimitNs) return false;
        }
    }
}

// What any block wrote before is visible to every block afterwards.
__device__ __forceinline__ bool meet(Meeting& m)
{
    __shared__ bool s_ok;
    ++m.turn;
    __syncthreads();
    if (threadIdx.x == 0) s_ok = arrive_and_wait(m);
    __syncthreads();
    return s_ok;
}

// The sum over all threads of all blocks, and its quotient with rs (ALPHA: rs
// / sum, else sum / rs), to every thread.  A level of an FP64 shuffle tree
// takes 110 clocks, a division 670, and either one executed by every warp
// shares the two FP64 lanes of the SM with all the others: one warp does both
// for its block.
template <bool ALPHA>
__device__ __forceinline__ bool meet_sum(Meeting& m, double v, double rs, double* red, double* total, double* ratio)
{
    __shared__ double s_total, s_ratio;
    __shared__ bool s_ok;
    const unsigned nb = gridDim.x, lane = threadIdx.x;
    ++m.turn;
    red[threadIdx.x] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        double* sums = m.sums + (size_t)(m.turn & 1) * nb;
        double a[4] = {};
        for (unsigned i = lane; i < blockDim.x; i += 128) {
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (i + 32 * u < blockDim.x) a[u] += red[i + 32 * u];
        }
        double t = (a[0] + a[1]) + (a[2] + a[3]);
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        bool ok = true;
        if (lane == 0) {
            asm volatile("st.relaxed.gpu.global.f64 [%0], %1;" :: "l"(sums + blockIdx.x), "d"(t) : "memory");
            ok = arrive_and_wait(m);
        }
        __syncwarp();
        double w[5];  // one block per SM: at most 160 sums are in flight together
        t = 0.0;
        for (unsigned i0 = lane; i0 < nb; i0 += 160) {
#pragma unroll
            for (int u = 0; u < 5; ++u) {
                w[u] = 0.0;
                if (i0 + 32 * u < nb)
                    asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];" : "=d"(w[u]) : "l"(sums + i0 + 32 * u) : "memory");
            }
            t += ((w[0] + w[1]) + (w[2] + w[3])) + w[4];
        }
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) {
            s_total = t;
            s_ratio = ALPHA ? rs / t : t / rs;
            s_ok = ok;
        }
    }
    __syncthreads();
    *total = s_total;
    *ratio = s_ratio;
    return s_ok;
}

// The matrix as its rows are walked: chunks of eight elements of a lane's row,
// loaded undecoded one chunk ahead (the next chunk of the row, or the first of
// the next slice), so that their latency passes behind the gathers, the
// products and, from the last slice to the first, the meetings.
struct SliceHead {
    int len, row, base;
    int64_t q;
};

template <typename CT>
struct ChunkF64 {
    CT c[8];
    double v[8];
    __device__ __forceinline__ void load(const SlArgs& a, const SliceHead& h, int k)
    {
        const CT* cp = static_cast<const CT*>(a.scol) + h.q + (int64_t)k * 32;
        const double* vp = a.val + h.q + (int64_t)k * 32;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const bool ok = k + u < h.len;
            c[u] = ok ? __ldg(cp + u * 32) : CT(0);
            v[u] = ok ? __ldg(vp + u * 32) : 0.0;
        }
    }
    __device__ __forceinline__ int col(int u, const SliceHead& h) const { return dev::column_of(c[u], h.row); }
    __device__ __forceinline__ double wide(int u) const { return v[u]; }
    __device__ __forceinline__ float val32(int u) const { return (float)v[u]; }
};
template <typename VT, bool OFF16>
struct ChunkLp {
    using CW = typename std::conditional<OFF16, uint2, int4>::type;
    using VW = typename std::conditional<sizeof(VT) == 4, float4, uint2>::type;
    CW c[2];
    VW v[2];
    __device__ __forceinline__ void load(const SlArgs& a, const SliceHead& h, int k)
    {
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            c[g] = CW{};
            v[g] = VW{};
            if (k + 4 * g < h.len) {  // a group's four slots are all stored
                const int64_t q = h.q + (int64_t)(k / 4 + g) * 128;
                if constexpr (OFF16) c[g] = __ldg(reinterpret_cast<const uint2*>(a.off + q));
                else c[g] = __ldg(reinterpret_cast<const int4*>(a.col + q));
                v[g] = __ldg(reinterpret_cast<const VW*>(static_cast<const VT*>(a.lowval) + q));
            }
        }
    }
    __device__ __forceinline__ int col(int u, const SliceHead& h) const
    {
        const CW& w = c[u / 4];
        if constexpr (OFF16) {
            const unsigned p = u % 4 < 2 ? w.x : w.y;
            return h.base + (int)(u % 2 == 0 ? p & 0xffffu : p >> 16);
        } else {
            return u % 4 == 0 ? w.x : u % 4 == 1 ? w.y : u % 4 == 2 ? w.z : w.w;
        }
    }
    __device__ __forceinline__ float val32(int u) const
    {
        const VW& w = v[u / 4];
        if constexpr (sizeof(VT) == 4) {
            return u % 4 == 0 ? w.x : u % 4 == 1 ? w.y : u % 4 == 2 ? w.z : w.w;
        } else {
            const unsigned p = u % 4 < 2 ? w.x : w.y;
            return __uint_as_float(u % 2 == 0 ? p << 16 : p & 0xffff0000u);
        }
    }
    __device__ __forceinline__ double wide(int u) const { return dev::widen_f32(val32(u)); }
};

template <typename VT, bool OFF16, typename CT>
using Chunk = typename std::conditional<sizeof(VT) == 8, ChunkF64<CT>, ChunkLp<VT, OFF16>>::type;

struct ResidentArgs {
    SlArgs in, ex;      // the inner matrix and, for refinement, the exact one (FP64)
    int ex_cbytes;
    int64_t n;
    const double* b;
    double* x;
    const double* r0;   // first residual; p (and p32) hold the first direction
    double* p;
    float* p32;
    double* resid;
    const CgState* st;
    double* sums;
    unsigned* arrived;
    int iters, refine;
    int per_warp;       // slices per warp
};

constexpr int kResidentWarps = 24;  // most per block; one block per SM (80 registers)
constexpr int kResidentSmem = 226 * 1024;  // dynamic; the meetings' words are static

template <typename VT, bool OFF16, bool ACC32, typename CT, int RT>
__global__ void __launch_bounds__(32 * kResidentWarps, 1)
k_cg_resident(const ResidentArgs a)
{
    using T = typename std::conditional<ACC32, float, double>::type;
    extern __shared__ double sm[];
    const int BT = blockDim.x, R = RT > 0 ? RT : a.per_warp;
    double* red = sm;  // [BT]
    // the lane's state: element j BT of each array
    const int64_t span = (int64_t)R * BT;
    double* sp = sm + BT + threadIdx.x;
    double* sr = sp + span;
    double* sq = sr + span;
    double* sx = sq + span;
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * BT + threadIdx.x) >> 5, n_warps = (int64_t)gridDim.x * (BT / 32);
    Meeting m{a.sums, a.arrived, 0};
    // row of the lane in the warp's slice j, -1 past the last
    auto row_of = [&](int j) -> int {
        const int64_t p = (warp + j * n_warps) * 32 + lane;
        if (p >= a.n) return -1;
        return a.in.perm ? a.in.perm[p] : (int)p;
    };
    auto head = [&](int j) {
        SliceHead h{0, 0, 0, 0};
        const int64_t s = warp + j * n_warps;
        if (s < a.in.n_slices) {
            const int64_t p = s * 32 + lane;
            h.len = max(a.in.rowlen[p], 0);
            h.q = a.in.slice_ptr[s] + (sizeof(VT) == 8 ? lane : 4 * lane);
            if (sizeof(VT) != 8 && OFF16) h.base = a.in.rowbase[p];
            if (sizeof(CT) != 4) h.row = row_of(j);
        }
        return h;
    };
    for (int j = 0; j < R; ++j) {
        const int row = row_of(j);
        sp[j * BT] = row >= 0 ? a.p[row] : 0.0;
        sr[j * BT] = row >= 0 ? a.r0[row] : 0.0;
        sx[j * BT] = row >= 0 ? a.x[row] : 0.0;
    }
    double rs = a.st->rs[0];
    // a few slices' heads stay in registers; of more, the next one's is loaded ahead
    SliceHead heads[RT > 0 ? RT : 1];
    int longest_of[RT > 0 ? RT : 1];
#pragma unroll
    for (int j = 0; j < (RT > 0 ? RT : 1); ++j) {
        heads[j] = head(j);
        longest_of[j] = __reduce_max_sync(0xffffffffu, heads[j].len);
    }
    bool ok = true;
    int t = 1;
    for (; t <= a.iters && ok; ++t) {
        // q = A p and p.q
        double part = 0.0;
        auto slice = [&](int j, const SliceHead& h, int longest) {
            T acc = T(0);
            for (int k = 0; k < longest; k += 8) {
                Chunk<VT, OFF16, CT> c;
                c.load(a.in, h, k);
                T xv[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    xv[u] = T(0);
                    if (k + u < h.len) {
                        if constexpr (ACC32)
                            asm volatile("ld.global.f32 %0, [%1];" : "=f"(xv[u]) : "l"(a.p32 + c.col(u, h)) : "memory");
                        else
                            xv[u] = dev::ldx_of<true>(a.p + c.col(u, h));
                    }
                }
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (k + u < h.len) {
                        if constexpr (ACC32) acc = fmaf(c.val32(u), xv[u], acc);
                        else acc = fma(c.wide(u), xv[u], acc);
                    }
            }
            double q;
            if constexpr (ACC32) q = dev::widen_f32(acc);
            else q = acc;
            sq[j * BT] = q;
            part = fma(sp[j * BT], q, part);
        };
        if constexpr (RT > 0) {
#pragma unroll
            for (int j = 0; j < RT; ++j) slice(j, heads[j], longest_of[j]);
        } else {
            for (int j = 0; j < R; ++j) {
                const SliceHead h = heads[0];
                heads[0] = head(j + 1 < R ? j + 1 : 0);
                slice(j, h, __reduce_max_sync(0xffffffffu, h.len));
            }
        }
        double pq, rr, alpha, beta;
        if (!(ok = meet_sum<true>(m, part, rs, red, &pq, &alpha))) break;
        const bool restart = a.refine > 0 && t % a.refine == 0;
        part = 0.0;
        if (restart) {
            for (int j = 0; j < R; ++j) {
                const int row = row_of(j);
                const double xj = fma(alpha, sp[j * BT], sx[j * BT]);
                sx[j * BT] = xj;
                if (row >= 0) a.x[row] = xj;
            }
            if (!(ok = meet(m))) break;
            // r = b - A x with the exact matrix: its rows may be placed
            // otherwise, so the product goes through memory (p's array: the
            // direction is about to be replaced)
            for (int64_t s = warp; s < a.ex.n_slices; s += n_warps) {
                int row;
                double v;
                if (a.ex_cbytes == 1)
                    v = dev::slice_value<4, int8_t, true>(s, lane, a.ex.rowlen, a.ex.slice_len, a.ex.slice_ptr, a.ex.perm,
                                                          static_cast<const int8_t*>(a.ex.scol), a.ex.val, a.x, &row);
                else if (a.ex_cbytes == 2)
                    v = dev::slice_value<4, int16_t, true>(s, lane, a.ex.rowlen, a.ex.slice_len, a.ex.slice_ptr, a.ex.perm,
                                                           static_cast<const int16_t*>(a.ex.scol), a.ex.val, a.x, &row);
                else
                    v = dev::slice_value<4, int, true>(s, lane, a.ex.rowlen, a.ex.slice_len, a.ex.slice_ptr, a.ex.perm,
                                                       static_cast<const int*>(a.ex.scol), a.ex.val, a.x, &row);
                if (row >= 0) a.p[row] = v;
            }
            if (!(ok = meet(m))) break;
            for (int j = 0; j < R; ++j) {
                const int row = row_of(j);
                if (row >= 0) {
                    const double rj = a.b[row] - dev::ldx_of<true>(a.p + row);
                    sr[j * BT] = rj;
                    part = fma(rj, rj, part);
                }
            }
        } else {
#pragma unroll 4
            for (int j = 0; j < R; ++j) {
                sx[j * BT] = fma(alpha, sp[j * BT], sx[j * BT]);
                const double rj = fma(-alpha, sq[j * BT], sr[j * BT]);
                sr[j * BT] = rj;
                part = fma(rj, rj, part);
            }
        }
        if (!(ok = meet_sum<false>(m, part, rs, red, &rr, &beta))) break;
        if (restart) beta = 0.0;  // the search restarts from the recomputed residual
        rs = rr;
        if (a.resid && blockIdx.x == 0 && threadIdx.x == 0) a.resid[t] = sqrt(rr);
        if (t == a.iters) break;
#pragma unroll 4
        for (int j = 0; j < R; ++j) {
            const int row = row_of(j);
            const double pj = fma(beta, sp[j * BT], sr[j * BT]);
            sp[j * BT] = pj;
            if (row >= 0) {
                if constexpr (ACC32) a.p32[row] = dev::round_f32(pj);
                else a.p[row] = pj;
            }
        }
        if (!(ok = meet(m))) break;
    }
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    for (int j = 0; j < R; ++j) {
        const int row = row_of(j);
        if (row >= 0) a.x[row] = ok ? sx[j * BT] : nan;
    }
    if (!ok && a.resid && blockIdx.x == 0 && threadIdx.x == 0)
        for (; t <= a.iters; ++t) a.resid[t] = nan;
}

// The launch of the resident kernel for a matrix's form; no kernel where the
// rows do not fit.
struct Resident {
    const void* kernel = nullptr;
    unsigned grid = 0, threads = 0;
    int per_warp = 0;
    size_t smem = 0;
};

template <typename VT, bool OFF16, bool ACC32, typename CT, int RT>
bool resident_form(int64_t n_slices, int sm_count, Resident* out)
{
    const int64_t per_warp = (n_slices + (int64_t)sm_count * kResidentWarps - 1) / ((int64_t)sm_count * kResidentWarps);
    // one slice per warp: at least four warps a block, so that few blocks meet
    const int64_t warps = per_warp > 1 ? kResidentWarps : std::max<int64_t>(4, (n_slices + sm_count - 1) / sm_count);
    const size_t smem = 8 * (size_t)(32 * warps) * (size_t)(1 + 4 * per_warp);
    if (smem > (size_t)kResidentSmem) return false;
    static LaunchCache cache;
    int per_sm = 0;
    if (cached_occupancy(cache, k_cg_resident<VT, OFF16, ACC32, CT, RT>, 32 * kResidentWarps, kResidentSmem, &per_sm) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    out->kernel = reinterpret_cast<const void*>(k_cg_resident<VT, OFF16, ACC32, CT, RT>);
    out->grid = (unsigned)((n_slices + warps * per_warp - 1) / (warps * per_warp));
    out->threads = (unsigned)(32 * warps);
    out->per_warp = (int)per_warp;
    out->smem = smem;
    return true;
}

template <typename VT, bool OFF16, bool ACC32, typename CT>
bool resident_fits(int64_t n_slices, int sm_count, Resident* out)
{
    const int64_t warps = (int64_t)sm_count * kResidentWarps;
    if (n_slices <= warps) return resident_form<VT, OFF16, ACC32, CT, 1>(n_slices, sm_count, out);
    if (n_slices <= 2 * warps) return resident_form<VT, OFF16, ACC32, CT, 2>(n_slices, sm_count, out);
    if (n_slices <= 3 * warps) return resident_form<VT, OFF16, ACC32, CT, 3>(n_slices, sm_count, out);
    return resident_form<VT, OFF16, ACC32, CT, 0>(n_slices, sm_count, out);
}

bool fp64_sliced(const spmv_prepared* P) { return fusable(P) && P->sl.value_type == SPMV_VAL_F64; }

// What a product of P reads every time: elements (padding included), the
// positions' headers and the gathered vector.
int64_t product_bytes(const spmv_prepared* P)
{
    const SlicedPlan& d = P->sl;
    const bool f64 = d.value_type == SPMV_VAL_F64;
    const int vb = f64 ? 8 : d.value_type == SPMV_VAL_F32 ? 4 : 2, cb = f64 ? d.cbytes : d.off16 ? 2 : 4;
    return (vb + cb) * d.tot + (d.off16 ? 268 : 140) * d.n_slices + (d.acc32 ? 4 : 8) * P->A.n_cols;
}

// Whether the whole loop runs in one launch, and with which kernel: a product
// whose operands stay in the L2 from one iteration to the next waits for
// latency, which the one launch has less of; a larger one streams from memory,
// for which 24 warps per SM keep less in flight than the product kernel's 64
// (or 48).  FP32 and BF16 products take little more than their bytes' time:
// the line lies at seven tenths of the L2.  With FP64 values the DFMAs take
// their time either way, and both loops are equal within 6 % up to 1.7 times
// the L2, where the line lies.  An iteration here / in three kernels, us, by
// product_bytes (an L2 of 135.5 MB):
//   FP64  7-point 101^3     99 MB 36 / 46  27-point 72^3    126 MB  47 / 45
//         27-point 80^3    172 MB 57 / 56  band 524288 x 25 164 MB  55 / 57
//         band 1.04 M x 17 225 MB 73 / 68  27-point 90^3    245 MB  74 / 66
//         band 524288 x 41 264 MB 76 / 76  band 1.04 M x 41 525 MB 130 / 115
//     16-bit columns: 524288 x 41 221 MB 72 / 77, 27-point 100^3 277 MB 92 / 84
//   BF16  27-point 80^3     64 MB 31 / 39  27-point 90^3     91 MB  44 / 48
//         band 1.04 M x 17  96 MB 51 / 48  band 524288 x 41  99 MB  51 / 47
//         27-point 100^3   124 MB 75 / 60  band 1.04 M x 41 196 MB  98 / 74
//   FP32  27-point 80^3     92 MB 39 / 45  band 524288 x 25  95 MB  33 / 43
//         band 786432 x 17 104 MB 46 / 46  band 393216 x 41 109 MB  50 / 45
bool resident_choice(const spmv_prepared* Pi, const spmv_prepared* Pe, int refine, const DeviceInfo& dev, Resident* out)
{
    if (!fusable(Pi) || (refine > 0 && !fp64_sliced(Pe))) return false;
    const SlicedPlan& d = Pi->sl;
    const int sm_count = dev.sm_count;
    if (10 * product_bytes(Pi) > (d.value_type == SPMV_VAL_F64 ? 17 : 7) * (int64_t)dev.l2_bytes) return false;
    if (d.value_type == SPMV_VAL_F64) {
        if (d.cbytes == 1) return resident_fits<double, false, false, int8_t>(d.n_slices, sm_count, out);
        if (d.cbytes == 2) return resident_fits<double, false, false, int16_t>(d.n_slices, sm_count, out);
        return resident_fits<double, false, false, int>(d.n_slices, sm_count, out);
    }
#define SPMV_CG_RES(VT, O16, A32) return resident_fits<VT, O16, A32, int>(d.n_slices, sm_count, out)
#define SPMV_CG_RES_VT(VT)                                                               \
    if (d.off16) { if (d.acc32) SPMV_CG_RES(VT, true, true); SPMV_CG_RES(VT, true, false); } \
    if (d.acc32) SPMV_CG_RES(VT, false, true);                                           \
    SPMV_CG_RES(VT, false, false);
    if (d.value_type == SPMV_VAL_F32) { SPMV_CG_RES_VT(float) }
    SPMV_CG_RES_VT(__nv_bfloat16)
#undef SPMV_CG_RES_VT
#undef SPMV_CG_RES
}

struct CgBufs {
    double *r = nullptr, *p = nullptr, *q = nullptr, *pq = nullptr, *rr = nullptr;
    CgState* st = nullptr;
    double* sums = nullptr;
    unsigned* arrived = nullptr;
};

// r0 = b - A x0 (exact), p0 = r0.  A SLICED inner matrix takes the fused q = A
// p, p.q kernel; when it sums in FP32, p's FP32 copy is written by the p
// updates.
float* direction_copy(const spmv_prepared* Pi) { return fusable(Pi) && Pi->sl.acc32 ? Pi->sl.x32 : nullptr; }

spmv_status enqueue_start(const spmv_prepared* Pi, const spmv_prepared* Pe, const double* b, double* x, double* resid,
                          const CgBufs& w, unsigned grid, cudaStream_t s)
{
    const int64_t n = Pi->A.n_rows;
    spmv_status st;
    if ((st = spmv(Pe, x, w.q, reinterpret_cast<spmv_stream_t>(s))) != SPMV_OK) return st;
    k_update<true><<<grid, kCT, 0, s>>>(n, x, w.p, w.r, w.q, b, nullptr, 0, w.rr, w.st, 0);
    k_update_p<kFirst><<<grid, kCT, 0, s>>>(n, w.p, w.r, w.rr, (int)grid, w.st, resid, 0, direction_copy(Pi));
    SPMV_CUDA_TRY(cudaGetLastError());
    return SPMV_OK;
}

// The one launch after enqueue_start.  short_of: arrivals that the meetings are
// short of (none but in the waits' self-test).  *refused: the device does not take it
// (fewer SMs are free to this process than it has, or no cooperative launches):
// nothing was launched.
spmv_status enqueue_resident(const spmv_prepared* Pi, const spmv_prepared* Pe, const double* b, double* x, int iters,
                             int refine, double* resid, const CgBufs& w, const Resident& res, int short_of,
                             bool* refused, cudaStream_t s)
{
    SPMV_CUDA_TRY(cudaMemsetAsync(w.arrived, short_of ? 0xff : 0, sizeof(unsigned), s));  // 0 or -1
    ResidentArgs a{sl_args(Pi), refine > 0 ? sl_args(Pe) : SlArgs{}, refine > 0 ? Pe->sl.cbytes : 4, Pi->A.n_rows, b, x,
                   w.r, w.p, direction_copy(Pi), resid, w.st, w.sums, w.arrived, iters, refine, res.per_warp};
    void* args[] = {&a};
    const cudaError_t e = cudaLaunchCooperativeKernel(res.kernel, dim3(res.grid), dim3(res.threads), args, res.smem, s);
    if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorLaunchOutOfResources || e == cudaErrorNotSupported) {
        cudaGetLastError();
        *refused = true;
        return SPMV_OK;
    }
    if (e != cudaSuccess) return cuda_fail(e, "spmv_cg launch");
    return SPMV_OK;
}

spmv_status enqueue_loop(const spmv_prepared* Pi, const spmv_prepared* Pe, const double* b, double* x, int iters,
                         int refine, double* resid, const CgBufs& w, unsigned grid, cudaStream_t s)
{
    const int64_t n = Pi->A.n_rows;
    spmv_status st;
    if ((st = enqueue_start(Pi, Pe, b, x, resid, w, grid, s)) != SPMV_OK) return st;
    const bool fused = fusable(Pi);
    float* p32 = direction_copy(Pi);
    const int n_pq = (int)(fused ? sliced_dot_grid(Pi) : grid), n_rr = (int)grid;
    for (int t = 1; t <= iters; ++t) {
        if (fused) {
            SPMV_CUDA_TRY(launch_sliced_dot(Pi, w.p, w.q, w.pq, s));
        } else {
            if ((st = spmv(Pi, w.p, w.q, reinterpret_cast<spmv_stream_t>(s))) != SPMV_OK) return st;
            k_dot_pq<<<grid, kCT, 0, s>>>(n, w.p, w.q, w.pq);
        }
        if (refine > 0 && t % refine == 0) {
            k_axpy_x<<<grid, kCT, 0, s>>>(n, x, w.p, w.pq, n_pq, w.st, t);
            if ((st = spmv(Pe, x, w.q, reinterpret_cast<spmv_stream_t>(s))) != SPMV_OK) return st;
            k_update<true><<<grid, kCT, 0, s>>>(n, x, w.p, w.r, w.q, b, nullptr, 0, w.rr, w.st, t);
            k_update_p<kRestart><<<grid, kCT, 0, s>>>(n, w.p, w.r, w.rr, n_rr, w.st, resid, t, p32);
        } else {
            k_update<false><<<grid, kCT, 0, s>>>(n, x, w.p, w.r, w.q, b, w.pq, n_pq, w.rr, w.st, t);
            k_update_p<kNext><<<grid, kCT, 0, s>>>(n, w.p, w.r, w.rr, n_rr, w.st, resid, t, p32);
        }
    }
    SPMV_CUDA_TRY(cudaGetLastError());
    return SPMV_OK;
}

}  // namespace
}  // namespace spmvlib

using namespace spmvlib;

namespace {

// The three-kernel loop from a graph: captured on a private stream (the
// caller's may be the legacy default stream, which cannot be captured), then
// launched on the caller's.
spmv_status launch_graph(const spmv_prepared* Pi, const spmv_prepared* Pe, const double* b, double* x, int iters,
                         int refine, double* resid, const CgBufs& w, unsigned grid, cudaStream_t s)
{
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    cudaStream_t cs = nullptr;
    spmv_status st = SPMV_OK;
    SPMV_CUDA_TRY(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
    cudaError_t e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        st = enqueue_loop(Pi, Pe, b, x, iters, refine, resid, w, grid, cs);
        e = cudaStreamEndCapture(cs, &graph);
    }
    cudaStreamDestroy(cs);
    if (st == SPMV_OK && e == cudaSuccess) e = cudaGraphInstantiate(&exec, graph, 0);
    if (st == SPMV_OK && e == cudaSuccess) e = cudaGraphLaunch(exec, s);
    if (exec) cudaGraphExecDestroy(exec);
    if (graph) cudaGraphDestroy(graph);
    if (st == SPMV_OK && e != cudaSuccess) st = cuda_fail(e, "spmv_cg graph");
    return st;
}

spmv_status enqueue_cg(const spmv_prepared* Pi, const spmv_prepared* Pe, const double* b, double* x, int iters,
                       int refine, double* resid, bool use_graph, const CgBufs& w, unsigned grid, const Resident& res,
                       int short_of, bool one_launch, cudaStream_t s)
{
    spmv_status st;
    SPMV_CUDA_TRY(cudaMemsetAsync(w.st, 0, sizeof(CgState), s));
    if (res.kernel && iters > 0) {
        bool refused = false;
        if ((st = enqueue_start(Pi, Pe, b, x, resid, w, grid, s)) != SPMV_OK) return st;
        st = enqueue_resident(Pi, Pe, b, x, iters, refine, resid, w, res, short_of, &refused, s);
        if (st != SPMV_OK || !refused) return st;
        if (one_launch) return fail(SPMV_ERR_UNSUPPORTED, "this solve does not run as one launch");
    }
    return use_graph ? launch_graph(Pi, Pe, b, x, iters, refine, resid, w, grid, s)
                     : enqueue_loop(Pi, Pe, b, x, iters, refine, resid, w, grid, s);
}

// spmv_cg; one_launch: refuses what does not run as one launch
spmv_status cg_run(const spmv_prepared_t* A_inner, const spmv_prepared_t* A_exact, const double* b, double* x,
                   int32_t iters, int32_t refine_every, double* resid, int32_t use_graph, int short_of, bool one_launch,
                   spmv_stream_t stream)
{
    if (!A_inner || !b || !x || iters < 0 || refine_every < 0)
        return fail(SPMV_ERR_INVALID_ARG, "spmv_cg: bad argument");
    const spmv_prepared* Pi = A_inner;
    const spmv_prepared* Pe = A_exact ? A_exact : A_inner;
    if (Pi->A.n_rows != Pi->A.n_cols || Pe->A.n_rows != Pi->A.n_rows || Pe->A.n_cols != Pi->A.n_cols)
        return fail(SPMV_ERR_INVALID_ARG, "spmv_cg: square matrices of equal size required");
    const int64_t n = Pi->A.n_rows;
    if (n == 0) return SPMV_OK;
    DeviceInfo dev;
    spmv_status st = current_device(&dev);
    if (st != SPMV_OK) return st;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    int64_t g = (n + kCT * kUnr - 1) / (kCT * kUnr);
    if (g > (int64_t)dev.sm_count * 2) g = (int64_t)dev.sm_count * 2;
    const unsigned grid = (unsigned)g;
    Resident res;
    if (!resident_choice(Pi, Pe, refine_every, dev, &res)) res = Resident{};
    if (one_launch && (!res.kernel || iters == 0))
        return fail(SPMV_ERR_UNSUPPORTED, "this solve does not run as one launch");
    // the work vectors in one allocation
    CgBufs w;
    const size_t n_part = std::max<size_t>(grid, fusable(Pi) ? sliced_dot_grid(Pi) : 0);
    auto room = [](size_t bytes) { return (bytes + 255) / 256 * 256; };
    const size_t vec = room(8 * (size_t)n), parts = room(16 * n_part), state = room(sizeof(CgState));
    unsigned char* base = nullptr;
    SPMV_CUDA_TRY(work_alloc(dev.device, reinterpret_cast<void**>(&base),
                             3 * vec + parts + state + room(sizeof(unsigned)) + room(2 * sizeof(double) * res.grid), s));
    w.r = reinterpret_cast<double*>(base);
    w.p = reinterpret_cast<double*>(base + vec);
    w.q = reinterpret_cast<double*>(base + 2 * vec);
    w.pq = reinterpret_cast<double*>(base + 3 * vec);
    w.rr = w.pq + n_part;
    w.st = reinterpret_cast<CgState*>(base + 3 * vec + parts);
    w.arrived = reinterpret_cast<unsigned*>(base + 3 * vec + parts + state);
    w.sums = reinterpret_cast<double*>(base + 3 * vec + parts + state + room(sizeof(unsigned)));
    st = enqueue_cg(Pi, Pe, b, x, iters, refine_every, resid, use_graph != 0, w, grid, res, short_of, one_launch, s);
    cudaFreeAsync(base, s);  // after an error too
    if (st != SPMV_OK) return st;
    SPMV_CUDA_TRY(cudaGetLastError());
    return SPMV_OK;
}

}  // namespace

extern "C" spmv_status spmv_cg(const spmv_prepared_t* A_inner, const spmv_prepared_t* A_exact,
                               const double* b, double* x, int32_t iters, int32_t refine_every,
                               double* resid, int32_t use_graph, spmv_stream_t stream)
{
    clear_error();
    return cg_run(A_inner, A_exact, b, x, iters, refine_every, resid, use_graph, 0, false, stream);
}

extern "C" spmv_status spmv_cg_wait_check(const spmv_prepared_t* A_inner, const spmv_prepared_t* A_exact,
                                          const double* b, double* x, int32_t iters, int32_t refine_every,
                                          double* resid, int32_t arrive, spmv_stream_t stream)
{
    clear_error();
    return cg_run(A_inner, A_exact, b, x, iters, refine_every, resid, 0, arrive ? 0 : 1, true, stream);
}
