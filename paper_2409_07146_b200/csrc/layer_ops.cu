// Element-wise pre- and post-operations of the GSA layer (Sec. 3.3): the Swish feature map of
// q, k, v (with its derivative for the backward) and the output path Swish -> RMSNorm over all
// heads of a token (forward, and backward with the gradient of the norm's weight).  All of them
// stream their tensors once with 16-byte accesses: HBM-bound.
//
// Why these are kernels of their own and not part of the chunk kernels: a d-sized tile of the
// tensor-core kernels goes from the copy engine straight into the matrix unit; passing it through
// registers for a Swish costs two special-function operations per element -- 2 k cycles per 128 x 128
// tile at 16 per clock and SM, as much as a whole chunk of the scan takes -- and every tile is read by
// three of the eight scans.  Applied once, in a kernel that runs at memory speed on all SMs, the same
// work costs one pass over q, k, v.  The decode kernel, which touches d values per (sequence, head)
// against 2 m d of memory, applies the feature map as it loads.
#include "common.cuh"

namespace gsa {
namespace {

__device__ __forceinline__ float reciprocal_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
// 1 / (1 + exp(-x)); where all results are rounded to bfloat16, by the approximate reciprocal (1 ulp of fp32): the IEEE
// division is half of all instructions of these kernels (training step of the 2.7B model's layer, 4 x 1999 tokens: 736 us
// with it in all of them, 652 without)
template <typename IO>
__device__ __forceinline__ float sigmoidf(float x);
template <>
__device__ __forceinline__ float sigmoidf<float>(float x) { return 1.f / (1.f + exp_neg(x)); }
template <>
__device__ __forceinline__ float sigmoidf<__nv_bfloat16>(float x) { return reciprocal_approx(1.f + exp_neg(x)); }
__device__ __forceinline__ float sigmoid_exact(float x) { return 1.f / (1.f + exp_neg(x)); }
__device__ __forceinline__ float swish_slope(float x, float sigmoid) { return sigmoid * (1.f + x * (1.f - sigmoid)); }

// The feature map of q, k and v in one launch: blocks of kStream vectors a thread, all requested before the first is used
// (one at a time, in a launch per tensor: 20 us for 41 MB in and out, 4.1 TB/s; three tensors of 41 MB, four vectors a thread held
// as fp32 values, 47 us and 83 backward; held as they come, with the sigmoid in four instructions, 44 and 55; eight vectors, a
// training step of the layer 604 -> 592).
constexpr int kStream = 8;
struct SwishSet { const void* in; void* out; size_t nvec; };
struct SwishSets { SwishSet t[3]; };
template <typename IO, bool BWD>
__global__ void __launch_bounds__(256) swish_kernel(const SwishSets sets) {
    follow_previous_grid();
    constexpr int V = IoTraits<IO>::kVec;
    const SwishSet& t = sets.t[blockIdx.y];
    const IO* in = static_cast<const IO*>(t.in);
    IO* out = static_cast<IO*>(t.out);
    const size_t i0 = (size_t)blockIdx.x * (kStream * 256) + threadIdx.x;
    uint4 xv[kStream], gv[BWD ? kStream : 1];         // (as they come: half the registers of their values in fp32)
#pragma unroll
    for (int j = 0; j < kStream; ++j)
        if (i0 + j * 256 < t.nvec) {
            xv[j] = reinterpret_cast<const uint4*>(in)[i0 + j * 256];
            if (BWD) gv[BWD ? j : 0] = reinterpret_cast<const uint4*>(out)[i0 + j * 256];
        }
#pragma unroll
    for (int j = 0; j < kStream; ++j)
        if (i0 + j * 256 < t.nvec) {
            float x[V], g[V];
            load_vec(reinterpret_cast<const IO*>(&xv[j]), x);
            if (BWD) load_vec(reinterpret_cast<const IO*>(&gv[BWD ? j : 0]), g);
#pragma unroll
            for (int e = 0; e < V; ++e) {
                const float s = sigmoidf<IO>(x[e]);
                x[e] = BWD ? g[e] * swish_slope(x[e], s) : x[e] * s;
            }
            store_vec(out + (i0 + j * 256) * V, x);
        }
}

// ---- the output path.  N = H d_v values of a token make up to 512 vectors of 16 bytes: a thread of the CTA owns one of
// them, and kTokens tokens are in flight together, so that their loads overlap and one barrier serves their sums.
constexpr int kTokens = 4;

// sums over the CTA of n values per thread, the same in every thread and run; `scratch` (16 x n floats) is free again at
// the next but one barrier
template <int n>
__device__ __forceinline__ void cta_sums(float (&v)[n], float (*scratch)[n]) {
#pragma unroll
    for (int i = 0; i < n; ++i)
#pragma unroll
        for (int o = 16; o; o >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    if (lane == 0) {
#pragma unroll
        for (int i = 0; i < n; ++i) scratch[warp][i] = v[i];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < n; ++i) v[i] = 0.f;
    for (int w = 0; w < nw; ++w) {
#pragma unroll
        for (int i = 0; i < n; ++i) v[i] += scratch[w][i];
    }
}

// y = w * Swish(o) / sqrt(mean(Swish(o)^2) + eps), kTokens tokens a CTA.  Bound by memory: 82 MB at 8 K tokens of 2560
// values; a CTA of 256 threads a token, two barriers each, took 39 us.
template <typename IO>
__global__ void __launch_bounds__(512) out_norm_fwd_kernel(const IO* o, const float* weight,
                                                           float eps, IO* y, int N, size_t rows) {
    follow_previous_grid();
    constexpr int V = IoTraits<IO>::kVec;
    __shared__ float scratch[16][kTokens];
    const size_t row0 = (size_t)blockIdx.x * kTokens;
    const int c = threadIdx.x * V;
    const bool own = c < N;
    float x[kTokens][V], ss[kTokens];
#pragma unroll
    for (int r = 0; r < kTokens; ++r)
        if (own && row0 + r < rows) load_vec(o + (row0 + r) * N + c, x[r]);
#pragma unroll
    for (int r = 0; r < kTokens; ++r) {
        ss[r] = 0.f;
        if (own && row0 + r < rows) {
#pragma unroll
            for (int e = 0; e < V; ++e) { x[r][e] *= sigmoidf<IO>(x[r][e]); ss[r] += x[r][e] * x[r][e]; }
        }
    }
    cta_sums(ss, scratch);
    if (!own) return;
    float w[V];
#pragma unroll
    for (int e = 0; e < V; ++e) w[e] = weight ? weight[c + e] : 1.f;
#pragma unroll
    for (int r = 0; r < kTokens; ++r)
        if (row0 + r < rows) {
            const float inv = rsqrtf(ss[r] / (float)N + eps);
#pragma unroll
            for (int e = 0; e < V; ++e) x[r][e] *= inv * w[e];
            store_vec(y + (row0 + r) * N + c, x[r]);
        }
}

// Backward: a CTA takes every gridDim.x-th pair of tokens (so that the weight gradient can be summed over
// them in registers, one partial row per CTA; a second kernel adds the partial rows in order).  With x = Swish(o), g = w dy
// and r = 1 / sqrt(mean(x^2) + eps):  d_o = r (g - x r^2 mean(g x)) Swish'(o) -- both means in one pass over the tokens'
// values, which stay in registers as they came, with their sigmoids; these by the exact reciprocal whatever the io type, since
// the weight gradient leaves in fp32.  Bound by instructions and the latency of a pair (loads, sums, barrier): two tokens in 64
// registers let three CTAs of 320 threads share an SM.  8 K tokens of 2560 values (123 MB): one token at a time, two means after
// one another 143 us; four tokens of one CTA per SM, each sigmoid formed twice, 86;
// so, 60 (both kernels).
// A CTA's tokens are as many as the call has for it, so a run of fp32 additions ends after kRunPairs pairs, in an fp64 sum of
// the thread's own: the rounding of 16 additions whatever the batch.  Run and sum stand in shared memory -- in registers the run
// spills the loop (64 K tokens of 4096 values 600 -> 695 us; so, 590; a partial row for every 16 tokens 630).
constexpr int kBwdTokens = 2;
constexpr int kRunPairs = 8;
template <typename IO>
__global__ void __launch_bounds__(512, 2) out_norm_bwd_kernel(const IO* o, const IO* dy,
                                                           const float* weight, float eps, IO* d_o,
                                                           float* __restrict__ dw_part, int N, size_t rows) {
    follow_previous_grid();
    constexpr int V = IoTraits<IO>::kVec;
    __shared__ float scratch[2][16][2 * kBwdTokens];
    extern __shared__ double sums_of_runs[];          // [V][threads], where the weight gradient is wanted
    float4* run = reinterpret_cast<float4*>(sums_of_runs + V * blockDim.x) + threadIdx.x;      // [V / 4][threads]
    const int c = threadIdx.x * V;
    const bool own = c < N;
    if (dw_part != nullptr) {
#pragma unroll
        for (int e = 0; e < V; ++e) sums_of_runs[e * blockDim.x + threadIdx.x] = 0.0;
#pragma unroll
        for (int e = 0; e < V / 4; ++e) run[e * blockDim.x] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    float w[V];
#pragma unroll
    for (int e = 0; e < V; ++e) {
        w[e] = weight && own ? weight[c + e] : 1.f;
    }
    int it = 0;
    for (size_t row0 = (size_t)blockIdx.x * kBwdTokens; row0 < rows; row0 += (size_t)gridDim.x * kBwdTokens, ++it) {
        uint4 ov[kBwdTokens], gv[kBwdTokens];
#pragma unroll
        for (int r = 0; r < kBwdTokens; ++r)
            if (own && row0 + r < rows) {
                ov[r] = *reinterpret_cast<const uint4*>(o + (row0 + r) * N + c);
                gv[r] = *reinterpret_cast<const uint4*>(dy + (row0 + r) * N + c);
            }
        float sums[2 * kBwdTokens], sg[kBwdTokens][V];
#pragma unroll
        for (int r = 0; r < kBwdTokens; ++r) {
            float ss = 0.f, dot = 0.f;
            if (own && row0 + r < rows) {
                float x[V], g[V];
                load_vec(reinterpret_cast<const IO*>(&ov[r]), x);
                load_vec(reinterpret_cast<const IO*>(&gv[r]), g);
#pragma unroll
                for (int e = 0; e < V; ++e) {
                    sg[r][e] = sigmoid_exact(x[e]);
                    x[e] *= sg[r][e];
                    ss += x[e] * x[e];
                    dot += g[e] * w[e] * x[e];
                }
            }
            sums[2 * r] = ss;
            sums[2 * r + 1] = dot;
        }
        cta_sums(sums, scratch[it & 1]);
        float dw[V];
#pragma unroll
        for (int e = 0; e < V; ++e) dw[e] = 0.f;
#pragma unroll
        for (int r = 0; r < kBwdTokens; ++r)
            if (own && row0 + r < rows) {
                const float inv = rsqrtf(sums[2 * r] / (float)N + eps);
                const float mean = sums[2 * r + 1] * inv / (float)N;          // mean of g times x inv
                float x[V], g[V];
                load_vec(reinterpret_cast<const IO*>(&ov[r]), x);
                load_vec(reinterpret_cast<const IO*>(&gv[r]), g);
#pragma unroll
                for (int e = 0; e < V; ++e) {
                    const float s = sg[r][e], xhat = x[e] * s * inv;
                    dw[e] += g[e] * xhat;
                    g[e] = (g[e] * w[e] - xhat * mean) * inv * swish_slope(x[e], s);
                }
                store_vec(d_o + (row0 + r) * N + c, g);
            }
        if (dw_part != nullptr) {
            const bool last = it % kRunPairs == kRunPairs - 1;
#pragma unroll
            for (int e = 0; e < V; e += 4) {
                float4 t = run[e / 4 * blockDim.x];
                t.x += dw[e]; t.y += dw[e + 1]; t.z += dw[e + 2]; t.w += dw[e + 3];
                if (last) {
                    double* sum = sums_of_runs + e * blockDim.x + threadIdx.x;
                    sum[0] += (double)t.x; sum[blockDim.x] += (double)t.y;
                    sum[2 * blockDim.x] += (double)t.z; sum[3 * blockDim.x] += (double)t.w;
                    t = make_float4(0.f, 0.f, 0.f, 0.f);
                }
                run[e / 4 * blockDim.x] = t;
            }
        }
    }
    if (dw_part != nullptr && own) {
#pragma unroll
        for (int e = 0; e < V; e += 4) {
            const float4 t = run[e / 4 * blockDim.x];
            const double* sum = sums_of_runs + e * blockDim.x + threadIdx.x;
            *reinterpret_cast<float4*>(dw_part + (size_t)blockIdx.x * N + c + e) =
                make_float4((float)(sum[0] + (double)t.x), (float)(sum[blockDim.x] + (double)t.y),
                            (float)(sum[2 * blockDim.x] + (double)t.z), (float)(sum[3 * blockDim.x] + (double)t.w));
        }
    }
}
// 32 columns a CTA, the partial rows dealt out over 32 groups of threads, in a fixed order (all of it latency: a thread a
// column 26 us for 500 partial rows of 2560, 16 groups 17, 32
// groups 10)
constexpr int kDwGroups = 32;
__global__ void __launch_bounds__(32 * kDwGroups) out_norm_dw_kernel(const float* dw_part, float* __restrict__ dweight, int N,
                                                          int nparts) {
    follow_previous_grid();
    __shared__ double group[kDwGroups][32];
    const int c = blockIdx.x * 32 + threadIdx.x;
    double acc = 0.0;
    if (c < N) {
#pragma unroll 16
        for (int p = threadIdx.y; p < nparts; p += kDwGroups) acc += (double)dw_part[(size_t)p * N + c];
    }
    group[threadIdx.y][threadIdx.x] = acc;
    __syncthreads();
    if (threadIdx.y != 0 || c >= N) return;
    for (int i = 1; i < kDwGroups; ++i) acc += group[i][threadIdx.x];
    dweight[c] = (float)acc;
}

// threads of a CTA of the output path: one for each vector of a token
unsigned token_threads(int N, int io) { return (unsigned)((N / (io == GSA_BF16 ? 8 : 4) + 31) / 32 * 32); }

template <bool BWD>
cudaError_t launch_swish(SwishSets sets, int io, cudaStream_t st) {
    size_t most = 0;
    for (SwishSet& t : sets.t) {
        t.nvec /= io == GSA_BF16 ? 8 : 4;
        if (t.nvec > most) most = t.nvec;
    }
    const dim3 grid((unsigned)((most + kStream * 256 - 1) / (kStream * 256)), 3);
    if (io == GSA_BF16) launch_after(swish_kernel<__nv_bfloat16, BWD>, grid, 256, 0, st, sets);
    else launch_after(swish_kernel<float, BWD>, grid, 256, 0, st, sets);
    return cudaGetLastError();
}

}  // namespace

// n elements (a multiple of the 16-byte vector) of io type each
cudaError_t launch_swish_fwd(const void* const in[3], void* const out[3], const size_t n[3], int io, cudaStream_t st) {
    return launch_swish<false>({{{in[0], out[0], n[0]}, {in[1], out[1], n[1]}, {in[2], out[2], n[2]}}}, io, st);
}
// d <- d * Swish'(x), in place on the gradients
cudaError_t launch_swish_bwd(const void* const x[3], void* const d[3], const size_t n[3], int io, cudaStream_t st) {
    return launch_swish<true>({{{x[0], d[0], n[0]}, {x[1], d[1], n[1]}, {x[2], d[2], n[2]}}}, io, st);
}
int out_norm_max_width(int io) { return 512 * (io == GSA_BF16 ? 8 : 4); }
// CTAs of the backward, a partial row of the weight gradient each: as many as the GPU holds at 64 registers a thread, up to
// eight per SM, and no more than there are pairs of tokens
size_t out_norm_bwd_parts(size_t rows, int N, int io) {
    const size_t pairs = (rows + kBwdTokens - 1) / kBwdTokens;
    size_t per_sm = 1024 / token_threads(N, io);
    per_sm = per_sm < 1 ? 1 : (per_sm > 8 ? 8 : per_sm);
    return pairs < kSMs * per_sm ? pairs : kSMs * per_sm;
}
cudaError_t launch_out_norm_fwd(const void* o, const float* weight, float eps, void* y, size_t rows, int N, int io,
                                cudaStream_t st) {
    const unsigned ctas = (unsigned)((rows + kTokens - 1) / kTokens), threads = token_threads(N, io);
    if (io == GSA_BF16)
        launch_after(out_norm_fwd_kernel<__nv_bfloat16>, ctas, threads, 0, st, (const __nv_bfloat16*)o, weight, eps,
                     (__nv_bfloat16*)y, N, rows);
    else
        launch_after(out_norm_fwd_kernel<float>, ctas, threads, 0, st, (const float*)o, weight, eps, (float*)y, N, rows);
    return cudaGetLastError();
}
cudaError_t launch_out_norm_bwd(const void* o, const void* dy, const float* weight, float eps, void* d_o, float* dw_part,
                                float* dweight, size_t rows, int N, int io, cudaStream_t st) {
    const unsigned parts = (unsigned)out_norm_bwd_parts(rows, N, io), threads = token_threads(N, io);
    constexpr int kSumBytes = sizeof(double) + sizeof(float);        // of a value: the sum of its runs and the run
    const size_t smem = dweight ? (size_t)kSumBytes * threads * (io == GSA_BF16 ? 8 : 4) : 0;
    const cudaError_t ready =
        io == GSA_BF16
            ? cudaFuncSetAttribute(out_norm_bwd_kernel<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSumBytes * 512 * 8)
            : cudaFuncSetAttribute(out_norm_bwd_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSumBytes * 512 * 4);
    if (ready != cudaSuccess) return ready;
    if (io == GSA_BF16)
        launch_after(out_norm_bwd_kernel<__nv_bfloat16>, parts, threads, smem, st, (const __nv_bfloat16*)o, (const __nv_bfloat16*)dy,
                     weight, eps, (__nv_bfloat16*)d_o, dweight ? dw_part : nullptr, N, rows);
    else
        launch_after(out_norm_bwd_kernel<float>, parts, threads, smem, st, (const float*)o, (const float*)dy, weight, eps, (float*)d_o,
                     dweight ? dw_part : nullptr, N, rows);
    if (dweight != nullptr) launch_after(out_norm_dw_kernel, (N + 31) / 32, dim3(32, kDwGroups), 0, st, dw_part, dweight, N, (int)parts);
    return cudaGetLastError();
}

}  // namespace gsa
