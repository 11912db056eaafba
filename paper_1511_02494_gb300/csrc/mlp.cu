// Learned selector: a fully connected 16 -> H1 -> H2 -> K network with ReLU
// that maps the Table 1 feature vector (Section 3.2.2) to a variant.  The
// paper builds its feature-based classifier with a decision tree or naive
// Bayes; this library trains a small MLP on the GPU with the kernels below
// (forward, softmax cross-entropy backward, Adam), and keeps the paper's
// profiling rule (Section 3.2.1) as its fallback when the network's top two
// logits are close.
//
// Parameters are packed row-major as W1[H1][16], b1[H1], W2[H2][H1], b2[H2],
// W3[K][H2], b3[K] (float).  Inputs are standardised as
// z = (v - mean) * istd, each operation rounded to float.  Every dot product
// is a chain of fmaf starting from the bias, inputs in ascending order: the
// same order on the host and the device, so logits agree bit for bit.
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <string>
#include <vector>

#include "common.cuh"

struct spmv_model {
    int32_t h1 = 0, h2 = 0, k = 0;
    float mean[16] = {}, istd[16] = {};
    std::vector<float> params;
    std::vector<int32_t> variants;
    float min_margin = 0.f;
    // optional launch parameters per output: threads_per_row, block_nnz,
    // items_per_warp (a second-level model choosing among one variant's
    // launch configurations); empty when the model names variants only
    std::vector<int32_t> launch;
};

namespace spmvlib {
namespace {

constexpr int kMaxH = 256;       // hidden width limit of the forward kernels
constexpr int kTrainMaxH = 128;  // hidden width limit of training
constexpr int kMaxK = 32;

__host__ __device__ __forceinline__ int64_t n_params(int h1, int h2, int k)
{
    return (int64_t)h1 * 16 + h1 + (int64_t)h2 * h1 + h2 + (int64_t)k * h2 + k;
}

// ---- host forward (spmv_select_model) ---------------------------------------
void host_forward(const spmv_model& m, const float* v, float* logits)
{
    const float* W1 = m.params.data();
    const float* b1 = W1 + m.h1 * 16;
    const float* W2 = b1 + m.h1;
    const float* b2 = W2 + m.h2 * m.h1;
    const float* W3 = b2 + m.h2;
    const float* b3 = W3 + m.k * m.h2;
    float z[16], a1[kMaxH], a2[kMaxH];
    for (int i = 0; i < 16; ++i) {
        volatile float d = v[i] - m.mean[i];  // keep the two roundings separate
        z[i] = d * m.istd[i];
    }
    for (int o = 0; o < m.h1; ++o) {
        float acc = b1[o];
        for (int i = 0; i < 16; ++i) acc = fmaf(W1[o * 16 + i], z[i], acc);
        a1[o] = acc > 0.f ? acc : 0.f;
    }
    for (int o = 0; o < m.h2; ++o) {
        float acc = b2[o];
        for (int i = 0; i < m.h1; ++i) acc = fmaf(W2[o * m.h1 + i], a1[i], acc);
        a2[o] = acc > 0.f ? acc : 0.f;
    }
    for (int o = 0; o < m.k; ++o) {
        float acc = b3[o];
        for (int i = 0; i < m.h2; ++i) acc = fmaf(W3[o * m.h2 + i], a2[i], acc);
        logits[o] = acc;
    }
}

// ---- device kernels -----------------------------------------------------------
struct Net {
    const float *W1, *b1, *W2, *b2, *W3, *b3;
    int h1, h2, k;
};
__device__ __forceinline__ Net unpack(const float* p, int h1, int h2, int k)
{
    Net n;
    n.W1 = p; n.b1 = n.W1 + h1 * 16; n.W2 = n.b1 + h1; n.b2 = n.W2 + h2 * h1;
    n.W3 = n.b2 + h2; n.b3 = n.W3 + k * h2;
    n.h1 = h1; n.h2 = h2; n.k = k;
    return n;
}

// One sample per thread; weights read through the read-only path.
__global__ void k_mlp_forward(const float* __restrict__ params, const float* __restrict__ mean,
                              const float* __restrict__ istd, int h1, int h2, int k,
                              const float* __restrict__ v, int n, float* __restrict__ logits)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    const Net N = unpack(params, h1, h2, k);
    float z[16], a1[kMaxH], a2[kMaxH];
    for (int i = 0; i < 16; ++i) z[i] = __fmul_rn(__fsub_rn(v[s * 16 + i], mean[i]), istd[i]);
    for (int o = 0; o < h1; ++o) {
        float acc = __ldg(N.b1 + o);
        for (int i = 0; i < 16; ++i) acc = __fmaf_rn(__ldg(N.W1 + o * 16 + i), z[i], acc);
        a1[o] = acc > 0.f ? acc : 0.f;
    }
    for (int o = 0; o < h2; ++o) {
        float acc = __ldg(N.b2 + o);
        for (int i = 0; i < h1; ++i) acc = __fmaf_rn(__ldg(N.W2 + o * h1 + i), a1[i], acc);
        a2[o] = acc > 0.f ? acc : 0.f;
    }
    for (int o = 0; o < k; ++o) {
        float acc = __ldg(N.b3 + o);
        for (int i = 0; i < h2; ++i) acc = __fmaf_rn(__ldg(N.W3 + o * h2 + i), a2[i], acc);
        logits[s * k + o] = acc;
    }
}

// Mean softmax cross-entropy over the batch and its gradient.  A CTA of 256
// threads stages the weights in shared memory once (cp.async) and takes
// slices of kSlice samples: forward and backward in shared memory, then the
// slice's gradient in 4 x 4 register tiles, stored to (from the CTA's second
// slice on: added to) the CTA's partial gradient, each entry always by the
// same thread.  k_mlp_reduce sums the partials in a fixed order, so the
// result is deterministic.
//
// The work is small (25 M FMAs for 1600 samples of the 16-64-64-8 network,
// under 1 us of the chip) and the kernel is bound by latency: of the weight
// loads, then of dependent FMA chains of h1 and h2 steps between barriers.
// Hence slices of 8 samples, so that 1600 samples put a CTA on every SM (200
// CTAs; 32 samples a CTA left two thirds of the SMs idle), a thread per
// output and sample pair (each weight read feeds two FMAs; rows padded by
// four floats, so the 16-byte reads are free of bank conflicts), and two to
// four resident CTAs per SM, as many as fit, looping over the slices, which
// bounds the partials to 608 whatever n is.  1600 samples of the 16-64-64-8
// network: 12.2 us, against 99.8 us with 50 CTAs that re-read the weights from
// global memory for every product.  With two CTAs per SM whatever the network,
// the barriers of small ones leave the SM idle: 200,000 samples of 16-7-5-3 take
// 520 us a call in place of 292, of 16-64-64-8 758 in place of 643 (eight: 295,
// 635, and more time in the reduction at 10,000 samples).
constexpr int kSlice = 8;
constexpr int kMT = 256;
static_assert(kMT / 32 == kSlice, "a warp per sample in the softmax");

// Shared memory of the training kernel in floats; every row starts on 16
// bytes.  Rows and columns past h1, h2 and k up to the next multiple of four
// hold zeros.
struct TrainLayout {
    int h1p, h2p, kp, w2s, w3s, as1, as2, ds3;
    int W1, W2, W3, B, z, a1, a2, d1, d2, d3, total;
};
constexpr int kW1s = 20, kZs = 20;  // row strides of W1 and z (16 + 4)
__host__ __device__ __forceinline__ TrainLayout train_layout(int h1, int h2, int k)
{
    TrainLayout L;
    L.h1p = (h1 + 3) & ~3;
    L.h2p = (h2 + 3) & ~3;
    L.kp = (k + 3) & ~3;
    L.w2s = L.as1 = L.h1p + 4;
    L.w3s = L.as2 = L.h2p + 4;
    L.ds3 = L.kp + 4;
    L.W1 = 0;
    L.W2 = L.W1 + L.h1p * kW1s;
    L.W3 = L.W2 + L.h2p * L.w2s;
    L.B = L.W3 + L.kp * L.w3s;  // b1, b2, b3
    L.z = L.B + L.h1p + L.h2p + L.kp;
    L.a1 = L.z + kSlice * kZs;
    L.a2 = L.a1 + kSlice * L.as1;
    L.d1 = L.a2 + kSlice * L.as2;
    L.d2 = L.d1 + kSlice * L.as1;
    L.d3 = L.d2 + kSlice * L.as2;
    L.total = L.d3 + kSlice * L.ds3 + kSlice;  // + the slice's losses
    return L;
}

// CTAs per SM: those that fit its 228 KB of shared memory (1 KB each is the
// system's), at least two (the widest network's) and at most four
inline int train_ctas(size_t smem)
{
    const int fit = (int)((228 << 10) / (smem + (1 << 10)));
    return std::max(2, std::min(4, fit));
}

__device__ __forceinline__ void cp_async4(float* dst, const float* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;"
                 :: "r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

// rows x cols floats, row r at src + r * cols, into rows_p rows of stride
// floats in shared memory, zero-filled past rows and cols; a warp per row
__device__ __forceinline__ void stage_rows(float* dst, const float* __restrict__ src, int rows, int cols,
                                           int rows_p, int stride)
{
    for (int r = threadIdx.x >> 5; r < rows_p; r += kMT / 32)
        for (int c = threadIdx.x & 31; c < stride; c += 32) {
            if (r < rows && c < cols) cp_async4(dst + r * stride + c, src + r * cols + c);
            else dst[r * stride + c] = 0.f;
        }
}

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }

// two dot products of length n4 (a multiple of four) in ascending order,
// each continuing its accumulator
__device__ __forceinline__ void dot2(const float* w, const float* x0, const float* x1, int n4, float& c0,
                                     float& c1)
{
#pragma unroll 4
    for (int i = 0; i < n4; i += 4) {
        const float4 a = ld4(w + i), u = ld4(x0 + i), v = ld4(x1 + i);
        c0 = __fmaf_rn(a.x, u.x, c0); c1 = __fmaf_rn(a.x, v.x, c1);
        c0 = __fmaf_rn(a.y, u.y, c0); c1 = __fmaf_rn(a.y, v.y, c1);
        c0 = __fmaf_rn(a.z, u.z, c0); c1 = __fmaf_rn(a.z, v.z, c1);
        c0 = __fmaf_rn(a.w, u.w, c0); c1 = __fmaf_rn(a.w, v.w, c1);
    }
}

// the same against a column of w (stride ws): the transposed products of
// the backward pass
__device__ __forceinline__ void dot2_col(const float* w, int ws, const float* x0, const float* x1, int n4,
                                         float& c0, float& c1)
{
#pragma unroll 4
    for (int i = 0; i < n4; i += 4) {
        const float4 u = ld4(x0 + i), v = ld4(x1 + i);
        const float a = w[i * ws], b = w[(i + 1) * ws], c = w[(i + 2) * ws], d = w[(i + 3) * ws];
        c0 = __fmaf_rn(a, u.x, c0); c1 = __fmaf_rn(a, v.x, c1);
        c0 = __fmaf_rn(b, u.y, c0); c1 = __fmaf_rn(b, v.y, c1);
        c0 = __fmaf_rn(c, u.z, c0); c1 = __fmaf_rn(c, v.z, c1);
        c0 = __fmaf_rn(d, u.w, c0); c1 = __fmaf_rn(d, v.w, c1);
    }
}

// One 4 x 4 tile of a weight gradient: entry (o, i) = sum over the slice's
// samples of d[s][o] a[s][i], written to (ADD: added to) g[o * cols + i].
template <bool ADD>
__device__ __forceinline__ void grad_tile(const float* d, int ds, const float* a, int as, int ns, int o0, int i0,
                                          int rows, int cols, float* __restrict__ g)
{
    float acc[4][4] = {};
    for (int s = 0; s < ns; ++s) {
        const float4 u = ld4(d + s * ds + o0), v = ld4(a + s * as + i0);
        const float du[4] = {u.x, u.y, u.z, u.w}, av[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[r][c] = __fmaf_rn(du[r], av[c], acc[r][c]);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (o0 + r < rows && i0 + c < cols) {
                float* e = g + (o0 + r) * cols + i0 + c;
                *e = ADD ? *e + acc[r][c] : acc[r][c];
            }
}

template <bool ADD>
__device__ __forceinline__ void bias_entry(const float* d, int ds, int ns, int o, float* __restrict__ g)
{
    float acc = 0.f;
    for (int s = 0; s < ns; ++s) acc += d[s * ds + o];
    g[o] = ADD ? g[o] + acc : acc;
}

// the slice's gradient: the three weight matrices' tiles and the biases in
// one list over the threads
template <bool ADD>
__device__ __forceinline__ void slice_gradient(const TrainLayout& L, const float* sm, int h1, int h2, int k, int ns,
                                               float* __restrict__ g)
{
    float* gW1 = g;
    float* gb1 = gW1 + h1 * 16;
    float* gW2 = gb1 + h1;
    float* gb2 = gW2 + h2 * h1;
    float* gW3 = gb2 + h2;
    float* gb3 = gW3 + k * h2;
    const int c1 = L.h1p / 4, c2 = L.h2p / 4;
    const int n2 = c2 * c1, n1 = n2 + c1 * 4, n3 = n1 + (L.kp / 4) * c2, nb = n3 + h1 + h2 + k;
    for (int t = threadIdx.x; t < nb; t += kMT) {
        if (t < n2) {
            const int ot = t / c1;
            grad_tile<ADD>(sm + L.d2, L.as2, sm + L.a1, L.as1, ns, 4 * ot, 4 * (t - ot * c1), h2, h1, gW2);
        } else if (t < n1) {
            const int q = t - n2;
            grad_tile<ADD>(sm + L.d1, L.as1, sm + L.z, kZs, ns, 4 * (q >> 2), 4 * (q & 3), h1, 16, gW1);
        } else if (t < n3) {
            const int q = t - n1, ot = q / c2;
            grad_tile<ADD>(sm + L.d3, L.ds3, sm + L.a2, L.as2, ns, 4 * ot, 4 * (q - ot * c2), k, h2, gW3);
        } else {
            const int q = t - n3;
            if (q < h1) bias_entry<ADD>(sm + L.d1, L.as1, ns, q, gb1);
            else if (q < h1 + h2) bias_entry<ADD>(sm + L.d2, L.as2, ns, q - h1, gb2);
            else bias_entry<ADD>(sm + L.d3, L.ds3, ns, q - h1 - h2, gb3);
        }
    }
}

__device__ __forceinline__ float warp_sum_f(float v)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL_MASK, v, o);
    return v;
}

__global__ void __launch_bounds__(kMT)
k_mlp_loss_grad(const float* __restrict__ params, int h1, int h2, int k, const float* __restrict__ z,
                const int32_t* __restrict__ labels, const float* __restrict__ q, int n, int64_t part_stride,
                float* __restrict__ part, float* __restrict__ part_loss)
{
    extern __shared__ __align__(16) float sm[];
    const TrainLayout L = train_layout(h1, h2, k);
    const Net N = unpack(params, h1, h2, k);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int n_slices = (n + kSlice - 1) / kSlice;
    stage_rows(sm + L.W1, N.W1, h1, 16, L.h1p, kW1s);
    stage_rows(sm + L.W2, N.W2, h2, h1, L.h2p, L.w2s);
    stage_rows(sm + L.W3, N.W3, k, h2, L.kp, L.w3s);
    float* b1 = sm + L.B;
    float* b2 = b1 + L.h1p;
    float* b3 = b2 + L.h2p;
    for (int t = tid; t < L.h1p; t += kMT) b1[t] = t < h1 ? N.b1[t] : 0.f;
    for (int t = tid; t < L.h2p; t += kMT) b2[t] = t < h2 ? N.b2[t] : 0.f;
    for (int t = tid; t < L.kp; t += kMT) b3[t] = t < k ? N.b3[t] : 0.f;
    float* g = part + (int64_t)blockIdx.x * part_stride;
    float* losses = sm + L.d3 + kSlice * L.ds3;
    float loss_sum = 0.f;  // thread 0
    for (int slice = blockIdx.x; slice < n_slices; slice += gridDim.x) {
        const int s0 = slice * kSlice;
        const int ns = min(kSlice, n - s0);
        for (int t = tid; t < kSlice * 16; t += kMT)
            sm[L.z + (t >> 4) * kZs + (t & 15)] = (t >> 4) < ns ? z[(int64_t)s0 * 16 + t] : 0.f;
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        // item t: unit t / 4 of a layer for the sample pair t % 4
        for (int t = tid; t < 4 * L.h1p; t += kMT) {
            const int o = t >> 2, s = (t & 3) * 2;
            float c0 = b1[o], c1 = c0;
            dot2(sm + L.W1 + o * kW1s, sm + L.z + s * kZs, sm + L.z + (s + 1) * kZs, 16, c0, c1);
            sm[L.a1 + s * L.as1 + o] = c0 > 0.f ? c0 : 0.f;
            sm[L.a1 + (s + 1) * L.as1 + o] = c1 > 0.f ? c1 : 0.f;
        }
        __syncthreads();
        for (int t = tid; t < 4 * L.h2p; t += kMT) {
            const int o = t >> 2, s = (t & 3) * 2;
            float c0 = b2[o], c1 = c0;
            dot2(sm + L.W2 + o * L.w2s, sm + L.a1 + s * L.as1, sm + L.a1 + (s + 1) * L.as1, L.h1p, c0, c1);
            sm[L.a2 + s * L.as2 + o] = c0 > 0.f ? c0 : 0.f;
            sm[L.a2 + (s + 1) * L.as2 + o] = c1 > 0.f ? c1 : 0.f;
        }
        __syncthreads();
        // softmax cross-entropy, a warp per sample and a lane per output;
        // d3 = (p - onehot) / n, or with a target distribution q: loss =
        // -sum q_o log p_o, d3 = (p S - q) / n where S = sum q_o
        {
            const int s = warp;
            const bool in = lane < k;
            float logit = -INFINITY;
            if (in) {
                float c0 = b3[lane], c1 = 0.f;
                dot2(sm + L.W3 + lane * L.w3s, sm + L.a2 + s * L.as2, sm + L.a2 + s * L.as2, L.h2p, c0, c1);
                logit = c0;
            }
            float mx = logit;
            for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(FULL_MASK, mx, o));
            const float den = warp_sum_f(in ? expf(logit - mx) : 0.f);
            float d = 0.f, l = 0.f;
            if (s < ns) {  // whole warps
                if (q == nullptr) {
                    const int y = labels[s0 + s];
                    const float ly = __shfl_sync(FULL_MASK, logit, y & 31);
                    l = -(ly - mx - logf(den));
                    if (in) d = (expf(logit - mx) / den - (lane == y ? 1.f : 0.f)) / (float)n;
                } else {
                    const float lse = mx + logf(den);
                    const float qo = in ? q[(int64_t)(s0 + s) * k + lane] : 0.f;
                    const float S = warp_sum_f(qo);
                    l = -warp_sum_f(in ? qo * (logit - lse) : 0.f);
                    if (in) d = (expf(logit - lse) * S - qo) / (float)n;
                }
            }
            if (lane < L.kp) sm[L.d3 + s * L.ds3 + lane] = d;
            if (lane == 0) losses[s] = l;
        }
        __syncthreads();
        for (int t = tid; t < 4 * L.h2p; t += kMT) {
            const int i = t >> 2, s = (t & 3) * 2;
            float c0 = 0.f, c1 = 0.f;
            dot2_col(sm + L.W3 + i, L.w3s, sm + L.d3 + s * L.ds3, sm + L.d3 + (s + 1) * L.ds3, L.kp, c0, c1);
            sm[L.d2 + s * L.as2 + i] = sm[L.a2 + s * L.as2 + i] > 0.f ? c0 : 0.f;
            sm[L.d2 + (s + 1) * L.as2 + i] = sm[L.a2 + (s + 1) * L.as2 + i] > 0.f ? c1 : 0.f;
        }
        __syncthreads();
        for (int t = tid; t < 4 * L.h1p; t += kMT) {
            const int i = t >> 2, s = (t & 3) * 2;
            float c0 = 0.f, c1 = 0.f;
            dot2_col(sm + L.W2 + i, L.w2s, sm + L.d2 + s * L.as2, sm + L.d2 + (s + 1) * L.as2, L.h2p, c0, c1);
            sm[L.d1 + s * L.as1 + i] = sm[L.a1 + s * L.as1 + i] > 0.f ? c0 : 0.f;
            sm[L.d1 + (s + 1) * L.as1 + i] = sm[L.a1 + (s + 1) * L.as1 + i] > 0.f ? c1 : 0.f;
        }
        if (tid == 0)
            for (int s = 0; s < ns; ++s) loss_sum += losses[s];
        __syncthreads();
        if (slice == blockIdx.x) slice_gradient<false>(L, sm, h1, h2, k, ns, g);
        else slice_gradient<true>(L, sm, h1, h2, k, ns, g);
        __syncthreads();
    }
    if (tid == 0) part_loss[blockIdx.x] = loss_sum;
}

// Sum of the CTAs' partials: a block takes 32 entries, warp w their partials
// w, w + 8, ... in order, a new chain after every 304 partials (38 of the
// warp's; chains of 76 over 608 partials have 10 % more rounding error), and
// the eight sums are added in warp order.  Block 0 also sums the losses.  5768
// entries of 200 partials: 3.7 us on 181 blocks (a thread per entry, 23 blocks,
// took 5.2 us for 50 partials).
constexpr int kRT = 256;
constexpr int kChain = 304;
__global__ void __launch_bounds__(kRT)
k_mlp_reduce(const float* __restrict__ part, const float* __restrict__ part_loss, int n_parts, int64_t part_stride,
             int64_t P, int n, float* __restrict__ grad, float* __restrict__ loss)
{
    __shared__ float sums[kRT / 32][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t e = (int64_t)blockIdx.x * 32 + lane;
    float acc = 0.f;
    if (e < P) {
        for (int c0 = 0; c0 < n_parts; c0 += kChain) {
            float a = 0.f;
#pragma unroll 8
            for (int c = c0 + warp; c < min(n_parts, c0 + kChain); c += kRT / 32) a += __ldcg(part + (int64_t)c * part_stride + e);
            acc = c0 == 0 ? a : acc + a;
        }
    }
    sums[warp][lane] = acc;
    __syncthreads();
    if (warp == 0 && e < P) {
        float t = sums[0][lane];
#pragma unroll
        for (int w = 1; w < kRT / 32; ++w) t += sums[w][lane];
        grad[e] = t;
    }
    if (blockIdx.x == 0 && warp == 1) {
        float l = 0.f;
        for (int c = lane; c < n_parts; c += 32) l += part_loss[c];
        l = warp_sum_f(l);
        if (lane == 0) *loss = l / (float)n;
    }
}

__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, int64_t n, float lr, float b1, float b2, float eps,
                       float wd, float c1, float c2)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    // each operation rounded separately (no contraction), as the definition reads
    const float gi = g[i];
    const float mi = __fadd_rn(__fmul_rn(b1, m[i]), __fmul_rn(__fsub_rn(1.f, b1), gi));
    const float vi = __fadd_rn(__fmul_rn(b2, v[i]), __fmul_rn(__fsub_rn(1.f, b2), __fmul_rn(gi, gi)));
    m[i] = mi;
    v[i] = vi;
    const float mh = __fdiv_rn(mi, c1), vh = __fdiv_rn(vi, c2);
    const float step = __fadd_rn(__fdiv_rn(mh, __fadd_rn(__fsqrt_rn(vh), eps)), __fmul_rn(wd, p[i]));
    p[i] = __fsub_rn(p[i], __fmul_rn(lr, step));
}

}  // namespace
}  // namespace spmvlib

using namespace spmvlib;

namespace {

bool shape_ok(int h1, int h2, int k, int max_h)
{
    return h1 >= 1 && h2 >= 1 && h1 <= max_h && h2 <= max_h && k >= 2 && k <= kMaxK;
}

const char kMagic[8] = {'S', 'P', 'M', 'V', 'M', 'L', 'P', '1'};
const char kMagic2[8] = {'S', 'P', 'M', 'V', 'M', 'L', 'P', '2'};  // + launch parameters

// output o's launch parameters as a choice of its variant (validated)
spmv_status launch_choice(const spmv_model_t* m, int o, spmv_choice_t* c)
{
    c->variant = m->variants[o];
    c->threads_per_row = m->launch[3 * o];
    c->block_nnz = m->launch[3 * o + 1];
    c->items_per_warp = m->launch[3 * o + 2];
    c->value_type = SPMV_VAL_F64;
    return check_choice(c);
}

}  // namespace

extern "C" {

spmv_status spmv_model_create(int32_t h1, int32_t h2, int32_t k, const float* mean,
                              const float* istd, const float* params, const int32_t* variants,
                              float min_margin, spmv_model_t** out)
{
    clear_error();
    if (!out || !mean || !istd || !params || !variants)
        return fail(SPMV_ERR_INVALID_ARG, "spmv_model_create: NULL argument");
    *out = nullptr;
    if (!shape_ok(h1, h2, k, kMaxH)) return fail(SPMV_ERR_MODEL, "model shape out of range");
    for (int o = 0; o < k; ++o)
        if (variants[o] < 0 || variants[o] >= SPMV_NUM_VARIANTS)
            return fail(SPMV_ERR_MODEL, "model names an unknown variant");
    spmv_model* m = new (std::nothrow) spmv_model();
    if (!m) return fail(SPMV_ERR_NOMEM, "host allocation failed");
    m->h1 = h1; m->h2 = h2; m->k = k;
    memcpy(m->mean, mean, sizeof(m->mean));
    memcpy(m->istd, istd, sizeof(m->istd));
    m->params.assign(params, params + n_params(h1, h2, k));
    m->variants.assign(variants, variants + k);
    m->min_margin = min_margin;
    for (float p : m->params)
        if (!isfinite(p)) { delete m; return fail(SPMV_ERR_MODEL, "non-finite model parameter"); }
    *out = m;
    return SPMV_OK;
}

spmv_status spmv_model_set_launch(spmv_model_t* m, const int32_t* launch)
{
    clear_error();
    if (!m || !launch) return fail(SPMV_ERR_INVALID_ARG, "spmv_model_set_launch: NULL argument");
    std::vector<int32_t> keep;
    keep.swap(m->launch);
    m->launch.assign(launch, launch + 3 * m->k);
    for (int o = 0; o < m->k; ++o) {
        spmv_choice_t c = {};
        if (launch_choice(m, o, &c) != SPMV_OK) {
            m->launch.swap(keep);
            return fail(SPMV_ERR_MODEL, "launch parameters not valid for the output's variant");
        }
    }
    return SPMV_OK;
}

spmv_status spmv_model_save(const spmv_model_t* m, const char* path)
{
    clear_error();
    if (!m || !path) return fail(SPMV_ERR_INVALID_ARG, "spmv_model_save: NULL argument");
    FILE* f = fopen(path, "wb");
    if (!f) return fail(SPMV_ERR_INVALID_ARG, std::string("cannot open ") + path);
    const int32_t hdr[3] = {m->h1, m->h2, m->k};
    const bool v2 = !m->launch.empty();
    bool ok = fwrite(v2 ? kMagic2 : kMagic, 1, 8, f) == 8 && fwrite(hdr, 4, 3, f) == 3 &&
              fwrite(m->mean, 4, 16, f) == 16 && fwrite(m->istd, 4, 16, f) == 16 &&
              fwrite(m->params.data(), 4, m->params.size(), f) == m->params.size() &&
              fwrite(m->variants.data(), 4, m->variants.size(), f) == m->variants.size() &&
              fwrite(&m->min_margin, 4, 1, f) == 1;
    if (v2) ok = ok && fwrite(m->launch.data(), 4, m->launch.size(), f) == m->launch.size();
    ok = (fclose(f) == 0) && ok;
    return ok ? SPMV_OK : fail(SPMV_ERR_INVALID_ARG, std::string("write failed: ") + path);
}

spmv_status spmv_model_load(const char* path, spmv_model_t** out)
{
    clear_error();
    if (!path || !out) return fail(SPMV_ERR_INVALID_ARG, "spmv_model_load: NULL argument");
    *out = nullptr;
    FILE* f = fopen(path, "rb");
    if (!f) return fail(SPMV_ERR_MODEL, std::string("cannot open model file ") + path);
    char magic[8];
    int32_t hdr[3];
    float mean[16], istd[16], margin = 0.f;
    std::vector<float> params;
    std::vector<int32_t> variants, launch;
    bool ok = fread(magic, 1, 8, f) == 8 && (memcmp(magic, kMagic, 8) == 0 || memcmp(magic, kMagic2, 8) == 0) &&
              fread(hdr, 4, 3, f) == 3 && shape_ok(hdr[0], hdr[1], hdr[2], kMaxH);
    const bool v2 = ok && memcmp(magic, kMagic2, 8) == 0;
    if (ok) {
        params.resize((size_t)n_params(hdr[0], hdr[1], hdr[2]));
        variants.resize((size_t)hdr[2]);
        ok = fread(mean, 4, 16, f) == 16 && fread(istd, 4, 16, f) == 16 &&
             fread(params.data(), 4, params.size(), f) == params.size() &&
             fread(variants.data(), 4, variants.size(), f) == variants.size() &&
             fread(&margin, 4, 1, f) == 1;
        if (ok && v2) {
            launch.resize(3 * (size_t)hdr[2]);
            ok = fread(launch.data(), 4, launch.size(), f) == launch.size();
        }
        char extra;
        if (ok && fread(&extra, 1, 1, f) != 0) ok = false;  // trailing bytes: corrupt
    }
    fclose(f);
    if (!ok) return fail(SPMV_ERR_MODEL, std::string("corrupt or truncated model file ") + path);
    spmv_status st = spmv_model_create(hdr[0], hdr[1], hdr[2], mean, istd, params.data(), variants.data(),
                                       margin, out);
    if (st != SPMV_OK || !v2) return st;
    if ((st = spmv_model_set_launch(*out, launch.data())) != SPMV_OK) {
        spmv_model_free(*out);
        *out = nullptr;
    }
    return st;
}

void spmv_model_free(spmv_model_t* m) { delete m; }

spmv_status spmv_model_logits(const spmv_model_t* m, const float* vec16, float* logits)
{
    clear_error();
    if (!m || !vec16 || !logits) return fail(SPMV_ERR_INVALID_ARG, "spmv_model_logits: NULL argument");
    host_forward(*m, vec16, logits);
    return SPMV_OK;
}

spmv_status spmv_select_model(const spmv_features_t* f, const spmv_model_t* m,
                              const spmv_profile_t* p, const spmv_thresholds_t* th,
                              spmv_choice_t* out)
{
    clear_error();
    if (!f || !m || !out) return fail(SPMV_ERR_INVALID_ARG, "spmv_select_model: NULL argument");
    float logits[kMaxK];
    host_forward(*m, f->vec, logits);
    int best = 0;
    for (int o = 1; o < m->k; ++o)
        if (logits[o] > logits[best]) best = o;
    float second = -INFINITY;
    for (int o = 0; o < m->k; ++o)
        if (o != best && logits[o] > second) second = logits[o];
    spmv_choice_t c = {};
    c.variant = m->variants[best];
    if (!m->launch.empty()) {
        spmv_status st = launch_choice(m, best, &c);
        if (st != SPMV_OK) return st;
    }
    c.cls = -1;
    c.value_type = SPMV_VAL_F64;
    c.margin = logits[best] - second;
    c.source = 2;
    if (c.margin < m->min_margin && p) {
        int32_t cls = -1;
        spmv_status st = spmv_classify_profile(p, th, &cls);
        if (st != SPMV_OK) return st;
        const float margin = c.margin;
        if ((st = spmv_class_choice(cls, &c)) != SPMV_OK) return st;
        c.margin = margin;
        c.used_fallback = 1;
    }
    *out = c;
    return SPMV_OK;
}

spmv_status spmv_select_model_refined(const spmv_features_t* f, const spmv_model_t* m,
                                      const spmv_model_t* sub, const spmv_profile_t* p,
                                      const spmv_thresholds_t* th, spmv_choice_t* out)
{
    spmv_status st = spmv_select_model(f, m, p, th, out);
    if (st != SPMV_OK || !sub || sub->launch.empty() || out->used_fallback) return st;
    for (int o = 0; o < sub->k; ++o)
        if (sub->variants[o] != out->variant) return SPMV_OK;  // another variant: first level only
    spmv_choice_t c2;
    if ((st = spmv_select_model(f, sub, nullptr, nullptr, &c2)) != SPMV_OK) return st;
    out->threads_per_row = c2.threads_per_row;
    out->block_nnz = c2.block_nnz;
    out->items_per_warp = c2.items_per_warp;
    return SPMV_OK;
}

spmv_status spmv_mlp_forward(const float* params, const float* mean, const float* istd,
                             int32_t h1, int32_t h2, int32_t k, const float* v, int32_t n,
                             float* logits, spmv_stream_t stream)
{
    clear_error();
    if (!shape_ok(h1, h2, k, kMaxH) || n < 0) return fail(SPMV_ERR_INVALID_ARG, "bad MLP shape");
    if (n == 0) return SPMV_OK;
    if (!params || !mean || !istd || !v || !logits)
        return fail(SPMV_ERR_INVALID_ARG, "spmv_mlp_forward: NULL argument");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    k_mlp_forward<<<(n + 63) / 64, 64, 0, s>>>(params, mean, istd, h1, h2, k, v, n, logits);
    SPMV_CUDA_TRY(cudaGetLastError());
    return SPMV_OK;
}

namespace {
spmv_status loss_grad_impl(const float* params, int32_t h1, int32_t h2, int32_t k,
                           const float* z, const int32_t* labels, const float* q, int32_t n,
                           float* grad, float* loss, spmv_stream_t stream)
{
    clear_error();
    if (!shape_ok(h1, h2, k, kTrainMaxH) || n <= 0)
        return fail(SPMV_ERR_INVALID_ARG, "bad MLP training shape (hidden <= 128, k <= 32)");
    if (!params || !z || (!labels && !q) || !grad || !loss)
        return fail(SPMV_ERR_INVALID_ARG, "spmv_mlp_loss_grad: NULL argument");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    DeviceInfo dev;
    spmv_status st = current_device(&dev);
    if (st != SPMV_OK) return st;
    const size_t smem = sizeof(float) * train_layout(h1, h2, k).total;
    const int parts = std::min((n + kSlice - 1) / kSlice, train_ctas(smem) * dev.sm_count);
    const int64_t P = n_params(h1, h2, k);
    const int64_t stride = (P + 31) / 32 * 32;  // partials start on 128-byte lines
    float* part = nullptr;
    SPMV_CUDA_TRY(stream_alloc(reinterpret_cast<void**>(&part), sizeof(float) * ((size_t)parts * stride + parts), s));
    // shared memory for the widest shape is allowed once per device
    static LaunchCache cache;
    int per_sm = 0;
    const TrainLayout widest = train_layout(kTrainMaxH, kTrainMaxH, kMaxK);
    cudaError_t e = cached_occupancy(cache, k_mlp_loss_grad, kMT, sizeof(float) * widest.total, &per_sm);
    if (e == cudaSuccess) {
        k_mlp_loss_grad<<<parts, kMT, smem, s>>>(params, h1, h2, k, z, labels, q, n, stride, part,
                                                 part + (size_t)parts * stride);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) {
        k_mlp_reduce<<<(unsigned)((P + 31) / 32), kRT, 0, s>>>(part, part + (size_t)parts * stride, parts, stride,
                                                               P, n, grad, loss);
        e = cudaGetLastError();
    }
    cudaError_t ef = cudaFreeAsync(part, s);
    if (e == cudaSuccess) e = ef;
    if (e != cudaSuccess) return cuda_fail(e, "spmv_mlp_loss_grad");
    return SPMV_OK;
}
}  // namespace

spmv_status spmv_mlp_loss_grad(const float* params, int32_t h1, int32_t h2, int32_t k,
                               const float* z, const int32_t* labels, int32_t n, float* grad,
                               float* loss, spmv_stream_t stream)
{
    if (!labels) {
        clear_error();
        return fail(SPMV_ERR_INVALID_ARG, "spmv_mlp_loss_grad: NULL argument");
    }
    return loss_grad_impl(params, h1, h2, k, z, labels, nullptr, n, grad, loss, stream);
}

spmv_status spmv_mlp_loss_grad_soft(const float* params, int32_t h1, int32_t h2, int32_t k,
                                    const float* z, const float* q, int32_t n, float* grad,
                                    float* loss, spmv_stream_t stream)
{
    if (!q) {
        clear_error();
        return fail(SPMV_ERR_INVALID_ARG, "spmv_mlp_loss_grad_soft: NULL argument");
    }
    return loss_grad_impl(params, h1, h2, k, z, nullptr, q, n, grad, loss, stream);
}

spmv_status spmv_mlp_adam(float* params, const float* grad, float* m, float* v, int64_t n,
                          int32_t step, float lr, float beta1, float beta2, float eps,
                          float weight_decay, spmv_stream_t stream)
{
    clear_error();
    if (!params || !grad || !m || !v || n < 0 || step < 1)
        return fail(SPMV_ERR_INVALID_ARG, "spmv_mlp_adam: bad argument");
    if (n == 0) return SPMV_OK;
    const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    k_adam<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(params, grad, m, v, n, lr, beta1, beta2, eps,
                                                       weight_decay, c1, c2);
    SPMV_CUDA_TRY(cudaGetLastError());
    return SPMV_OK;
}

}  // extern "C"
