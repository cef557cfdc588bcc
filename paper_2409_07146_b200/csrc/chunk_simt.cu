// fp32 CUDA-core versions of the two chunk primitives of Algorithm 1 (see common.cuh).
//
// They are the kernels of the fp32 io type (whose tolerance bf16 or tf32 tensor-core
// operands cannot meet) and run either io type when asked for (GSA_IMPL_SIMT).  One CTA of
// 256 threads owns one (batch, head) and one 64-wide slice of the head dimension, walks the
// chunks in order with the slice of the state in shared memory, and does every contraction
// of a chunk as a 64 x N x 64 register-tiled product out of shared memory.
//
// Decay handling inside a chunk.  With G the chunk-local cumulative log gate, the decay
// between rows j <= i is exp(G_i - G_j).  When the chunk's total decay is moderate
// (min_s G_C[s] >= kFactorisedDecayMin) it is factorised as exp(G_i) * exp(-G_j) and folded
// into the operands of a plain product; otherwise the differences are formed explicitly
// (all exponents <= 0, nothing can overflow).
#include <type_traits>

#include "common.cuh"

namespace gsa {
namespace {

constexpr int kC = kChunk;      // rows per chunk
constexpr int kDS = 64;         // head-dimension slice per CTA
constexpr int kLd = 68;         // shared-memory pitch of a 64-wide fp32 tile (16-byte aligned rows)

// ---- 64-row register-tiled products out of shared memory; thread (ty, tx) of a 16 x 16 grid.
// NN: acc[ii][jj] += sum_k A[(4 ty + ii)][k] * B[k][NJ tx + jj]
template <int NJ>
__device__ __forceinline__ void mm_nn(const float* A, int lda, const float* B, int ldb, int K,
                                      int ty, int tx, float (&acc)[4][NJ]) {
#pragma unroll 2
    for (int k = 0; k < K; k += 4) {
        float a[4][4];
#pragma unroll
        for (int ii = 0; ii < 4; ++ii) {
            const float4 t = *reinterpret_cast<const float4*>(A + (4 * ty + ii) * lda + k);
            a[ii][0] = t.x; a[ii][1] = t.y; a[ii][2] = t.z; a[ii][3] = t.w;
        }
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
            float b[NJ];
            if constexpr (NJ == 8) {
                const float4 t = *reinterpret_cast<const float4*>(B + (k + kk) * ldb + 8 * tx);
                const float4 t2 = *reinterpret_cast<const float4*>(B + (k + kk) * ldb + 8 * tx + 4);
                b[0] = t.x; b[1] = t.y; b[2] = t.z; b[3] = t.w; b[4] = t2.x; b[5] = t2.y; b[6] = t2.z; b[7] = t2.w;
            } else if constexpr (NJ == 4) {
                const float4 t = *reinterpret_cast<const float4*>(B + (k + kk) * ldb + 4 * tx);
                b[0] = t.x; b[1] = t.y; b[2] = t.z; b[3] = t.w;
            } else {
                const float2 t = *reinterpret_cast<const float2*>(B + (k + kk) * ldb + 2 * tx);
                b[0] = t.x; b[1] = t.y;
            }
#pragma unroll
            for (int ii = 0; ii < 4; ++ii)
#pragma unroll
                for (int jj = 0; jj < NJ; ++jj) acc[ii][jj] = fmaf(a[ii][kk], b[jj], acc[ii][jj]);
        }
    }
}
// TN: acc[ii][jj] += sum_k A[k][4 ty + ii] * B[k][NJ tx + jj]
template <int NJ>
__device__ __forceinline__ void mm_tn(const float* A, int lda, const float* B, int ldb, int K,
                                      int ty, int tx, float (&acc)[4][NJ]) {
#pragma unroll 4
    for (int k = 0; k < K; ++k) {
        const float4 t = *reinterpret_cast<const float4*>(A + k * lda + 4 * ty);
        const float a[4] = {t.x, t.y, t.z, t.w};
        float b[NJ];
        if constexpr (NJ == 8) {
            const float4 u = *reinterpret_cast<const float4*>(B + k * ldb + 8 * tx);
            const float4 u2 = *reinterpret_cast<const float4*>(B + k * ldb + 8 * tx + 4);
            b[0] = u.x; b[1] = u.y; b[2] = u.z; b[3] = u.w; b[4] = u2.x; b[5] = u2.y; b[6] = u2.z; b[7] = u2.w;
        } else if constexpr (NJ == 4) {
            const float4 u = *reinterpret_cast<const float4*>(B + k * ldb + 4 * tx);
            b[0] = u.x; b[1] = u.y; b[2] = u.z; b[3] = u.w;
        } else {
            const float2 u = *reinterpret_cast<const float2*>(B + k * ldb + 2 * tx);
            b[0] = u.x; b[1] = u.y;
        }
#pragma unroll
        for (int ii = 0; ii < 4; ++ii)
#pragma unroll
            for (int jj = 0; jj < NJ; ++jj) acc[ii][jj] = fmaf(a[ii], b[jj], acc[ii][jj]);
    }
}
// NT: acc[ii][jj] += sum_k A[4 ty + ii][k] * B[tx + 16 jj][k]      (16 NB columns)
template <int NB>
__device__ __forceinline__ void mm_nt(const float* A, int lda, const float* B, int ldb, int K,
                                      int ty, int tx, float (&acc)[4][NB]) {
#pragma unroll 2
    for (int k = 0; k < K; k += 4) {
        float4 a[4], b[NB];
#pragma unroll
        for (int ii = 0; ii < 4; ++ii) a[ii] = *reinterpret_cast<const float4*>(A + (4 * ty + ii) * lda + k);
#pragma unroll
        for (int jj = 0; jj < NB; ++jj) b[jj] = *reinterpret_cast<const float4*>(B + (tx + 16 * jj) * ldb + k);
#pragma unroll
        for (int ii = 0; ii < 4; ++ii)
#pragma unroll
            for (int jj = 0; jj < NB; ++jj) {
                acc[ii][jj] = fmaf(a[ii].x, b[jj].x, acc[ii][jj]);
                acc[ii][jj] = fmaf(a[ii].y, b[jj].y, acc[ii][jj]);
                acc[ii][jj] = fmaf(a[ii].z, b[jj].z, acc[ii][jj]);
                acc[ii][jj] = fmaf(a[ii].w, b[jj].w, acc[ii][jj]);
            }
    }
}

// The masked first product of a chunk, P or A [64 x 64] = A B^T over K: a row needs the columns up to its own (reversed: from
// its own on), a warp's eight rows (8 warp ..) the blocks of 16 columns up to theirs.  Only these are formed, and what lies
// between a row and their edge is set to zero; the product with the rows they weigh leaves the others out, too.  A fifth of
// the multiplications of a scan: fp32 training step, B = 2, T = 1024, 4 heads of 256, 397 -> 366 us (a scan 45 -> 41).
template <bool REV>
__device__ __forceinline__ void masked_product(const float* A, int lda, const float* B, int ldb, int K, float* out, int ty, int tx) {
    const int pair = threadIdx.x >> 6, first = REV ? pair : 0, blocks = REV ? 4 - pair : pair + 1;
    auto form = [&](auto nb) {
        constexpr int NB = decltype(nb)::value;
        float acc[4][NB] = {};
        mm_nt<NB>(A, lda, B + 16 * first * ldb, ldb, K, ty, tx, acc);
#pragma unroll
        for (int ii = 0; ii < 4; ++ii)
#pragma unroll
            for (int jj = 0; jj < NB; ++jj) {
                const int i = 4 * ty + ii, j = tx + 16 * (first + jj);
                const bool keep = REV ? (j >= i) : (j <= i);
                out[i * kLd + j] = keep ? acc[ii][jj] : 0.f;
            }
    };
    if (blocks == 4) form(std::integral_constant<int, 4>{});
    else if (blocks == 3) form(std::integral_constant<int, 3>{});
    else if (blocks == 2) form(std::integral_constant<int, 2>{});
    else form(std::integral_constant<int, 1>{});
}
// acc += (masked product) B, from the columns of it that the warp's rows have
template <bool REV, int NJ>
__device__ __forceinline__ void mm_masked(const float* A, const float* B, int ldb, int ty, int tx, float (&acc)[4][NJ]) {
    const int edge = 8 * (threadIdx.x >> 5), k0 = REV ? edge : 0, k1 = REV ? kC : edge + 8;
    mm_nn<NJ>(A + k0, kLd, B + k0 * ldb, ldb, k1 - k0, ty, tx, acc);
}

// ---- tile loads.  fp32 tiles go to shared memory by asynchronous copies: all tiles of a chunk are requested before the
// first is waited for (through registers a tile's copies waited for those of the tile before it: four to five latencies of
// memory a chunk, a third of the kernels' stalls).  With the second scaling pass of a moderate chunk gone, too: a fp32
// training step, B = 2, T = 1024, 4 heads of 256, 586 -> 439 us, a forward over T = 256 53 -> 41 us.
__device__ __forceinline__ void copy16_async(float* dst, const float* src, bool live) {      // (!live: zeros)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
                 "r"(live ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ void copies_landed() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// 64 rows x 64 columns of io type -> fp32 shared (rows >= valid are zero)
template <typename IO>
__device__ __forceinline__ void load_io_tile(float* dst, const IO* src, size_t row_stride, int valid) {
    constexpr int V = IoTraits<IO>::kVec;
    constexpr int PER_ROW = kDS / V;
    if constexpr (V == 4) {
#pragma unroll
        for (int idx = threadIdx.x; idx < kC * PER_ROW; idx += 256) {
            const int r = idx / PER_ROW, c = (idx % PER_ROW) * V;
            copy16_async(dst + r * kLd + c, src + (size_t)min(r, valid - 1) * row_stride + c, r < valid);
        }
    } else {
#pragma unroll
        for (int idx = threadIdx.x; idx < kC * PER_ROW; idx += 256) {
            const int r = idx / PER_ROW, c = (idx % PER_ROW) * V;
            float x[V];
            if (r < valid) {
                load_vec(src + (size_t)r * row_stride + c, x);
            } else {
#pragma unroll
                for (int e = 0; e < V; ++e) x[e] = 0.f;
            }
#pragma unroll
            for (int e = 0; e < V; e += 4)
                *reinterpret_cast<float4*>(dst + r * kLd + c + e) = make_float4(x[e], x[e + 1], x[e + 2], x[e + 3]);
        }
    }
}
// 64 rows x M fp32; rows >= valid get `fill` (0 for weights) or replicate the last valid row (G)
template <int M, bool REPLICATE_LAST>
__device__ __forceinline__ void load_slot_tile(float* dst, const float* src, size_t row_stride, int valid) {
    constexpr int PER_ROW = M / 4;
#pragma unroll
    for (int idx = threadIdx.x; idx < kC * PER_ROW; idx += 256) {
        const int r = idx / PER_ROW, c = (idx % PER_ROW) * 4;
        copy16_async(dst + r * (M + 4) + c, src + (size_t)min(r, valid - 1) * row_stride + c, REPLICATE_LAST || r < valid);
    }
}

// Decide, for the whole CTA, whether this chunk may use the factorised decay.
template <int M>
__device__ __forceinline__ bool chunk_is_moderate(const float* sG, int* flag) {
    if (threadIdx.x == 0) *flag = 1;
    __syncthreads();
    if (threadIdx.x < M && sG[(kC - 1) * (M + 4) + threadIdx.x] < kFactorisedDecayMin) *flag = 0;
    __syncthreads();
    return *flag != 0;
}

// =============================================================== value_side (pass-1 form)
// FLAGGED: the flagged pairs of a tensor-core scan alone (see launch_value_side_simt), whose slices of `out` are 128 wide:
// the two CTAs of a slice add their sums to the zeros that the tensor-core kernel has left there (two addends: the same
// in either order).  One CTA for both, one after the other: a forward over strong gates, B = 4, T = 1024, 4 heads of 512,
// 128 slots, 2395 us, 1464 so.
template <typename IO, int M, bool REV, bool FLAGGED>
__global__ void __launch_bounds__(256, M > 64 ? 1 : 2) value_side_simt_kernel(ValueSideArgs a, const int* strong_flag) {
    follow_previous_grid();
    if (FLAGGED && strong_flag[blockIdx.x] == 0) return;
    constexpr int NJ = M / 16;
    constexpr int LM = M + 4;
    extern __shared__ __align__(16) float smem[];
    float* sXq = smem;                 // [64][68]
    float* sXk = sXq + kC * kLd;       // [64][68]
    float* sP = sXk + kC * kLd;        // [64][68]
    float* sS = sP + kC * kLd;         // [64 (channel)][LM]
    float* sW = sS + kDS * LM;         // [64][LM]
    float* sG = sW + kC * LM;          // [64][LM]
    __shared__ int s_flag;

    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
    const ScanSpan span = scan_span(blockIdx.x, a.H, a.T, a.nseg, a.tseg);
    const int slice = blockIdx.y, bh = blockIdx.x, b = span.b, h = span.h;
    const int d0 = slice * kDS;
    const size_t strideD = (size_t)a.H * a.D, strideM = (size_t)a.H * M;
    const IO* xq = (const IO*)a.xq + ((size_t)b * a.T * a.H + h) * a.D + d0;
    const IO* xk = (const IO*)a.xk + ((size_t)b * a.T * a.H + h) * a.D + d0;
    const float* w = a.w + ((size_t)b * a.T * a.H + h) * M;
    const float* G = a.G + ((size_t)b * a.T * a.H + h) * M;
    float* out = a.out + (size_t)(FLAGGED ? slice / 2 : slice) * a.B * a.T * a.H * M + ((size_t)b * a.T * a.H + h) * M;

    const int nchunks = (span.t_end - span.t0 + kC - 1) / kC;
    const bool states_only = FLAGGED && a.state_only;          // (beside the kernels for 128 slots; other state runs: state_simt_kernel)
    for (int it = 0; it < nchunks; ++it) {
        const int n = REV ? nchunks - 1 - it : it;
        const int t0 = span.t0 + n * kC;
        const int valid = min(kC, span.t_end - t0);
        __syncthreads();
        if (!states_only) load_io_tile<IO>(sXq, xq + (size_t)t0 * strideD, strideD, valid);
        load_io_tile<IO>(sXk, xk + (size_t)t0 * strideD, strideD, valid);
        load_slot_tile<M, false>(sW, w + (size_t)t0 * strideM, strideM, valid);
        load_slot_tile<M, true>(sG, G + (size_t)t0 * strideM, strideM, valid);
        if (it == 0) {       // (behind the first tiles' copies) state slice S[c][s] <- S0[bh][s][d0 + c]
#pragma unroll
            for (int idx = tid; idx < kDS * M; idx += 256) {
                const int s = idx / kDS, c = idx % kDS;
                sS[c * LM + s] = a.S0 ? a.S0[((size_t)bh * M + s) * a.D + d0 + c] : 0.f;
            }
        }
        copies_landed();
        __syncthreads();
        const bool moderate = chunk_is_moderate<M>(sG, &s_flag);
        if (moderate) {
            // W' = W * exp(-G) (forward) or W * exp(G) (reverse)
            for (int idx = tid; idx < kC * M; idx += 256) {
                const int r = idx / M, s = idx % M;
                const float g = sG[r * LM + s];
                sW[r * LM + s] *= __expf(REV ? g : -g);
            }
        }
        // P = Xq Xk^T, masked to the causal (forward) or anti-causal (reverse) triangle
        if (states_only) {
        } else if (moderate) {
            masked_product<REV>(sXq, kLd, sXk, kLd, kDS, sP, ty, tx);
        } else {
            float acc[4][4] = {};
            mm_nt<4>(sXq, kLd, sXk, kLd, kDS, ty, tx, acc);
#pragma unroll
            for (int ii = 0; ii < 4; ++ii)
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) {
                    const int i = 4 * ty + ii, j = tx + 16 * jj;
                    const bool keep = REV ? (j >= i) : (j <= i);
                    sP[i * kLd + j] = keep ? acc[ii][jj] : 0.f;
                }
        }
        __syncthreads();
        // out = rowscale * ( colscale * (Xq S) + P W' )
        if (!states_only) {
            float acc[4][NJ] = {};
            mm_nn<NJ>(sXq, kLd, sS, LM, kDS, ty, tx, acc);
            if (moderate) {
                if (REV) {
#pragma unroll
                    for (int jj = 0; jj < NJ; ++jj) {
                        const float e = __expf(sG[(kC - 1) * LM + NJ * tx + jj]);
#pragma unroll
                        for (int ii = 0; ii < 4; ++ii) acc[ii][jj] *= e;
                    }
                }
                mm_masked<REV, NJ>(sP, sW, LM, ty, tx, acc);
#pragma unroll
                for (int ii = 0; ii < 4; ++ii)
#pragma unroll
                    for (int jj = 0; jj < NJ; ++jj) {
                        const float g = sG[(4 * ty + ii) * LM + NJ * tx + jj];
                        acc[ii][jj] *= __expf(REV ? -g : g);
                    }
            } else {
                float gi[4][NJ];
#pragma unroll
                for (int ii = 0; ii < 4; ++ii)
#pragma unroll
                    for (int jj = 0; jj < NJ; ++jj) {
                        gi[ii][jj] = sG[(4 * ty + ii) * LM + NJ * tx + jj];
                        const float gc = sG[(kC - 1) * LM + NJ * tx + jj];
                        acc[ii][jj] *= __expf(REV ? gc - gi[ii][jj] : gi[ii][jj]);
                    }
                for (int j = 0; j < kC; ++j) {
#pragma unroll
                    for (int jj = 0; jj < NJ; ++jj) {
                        const float gj = sG[j * LM + NJ * tx + jj];
                        const float wj = sW[j * LM + NJ * tx + jj];
#pragma unroll
                        for (int ii = 0; ii < 4; ++ii) {
                            const float pij = sP[(4 * ty + ii) * kLd + j];
                            const float ex = REV ? gj - gi[ii][jj] : gi[ii][jj] - gj;
                            acc[ii][jj] = fmaf(pij * wj, __expf(fminf(ex, 0.f)), acc[ii][jj]);
                        }
                    }
                }
            }
#pragma unroll
            for (int ii = 0; ii < 4; ++ii) {
                const int i = 4 * ty + ii;
                if (i < valid) {
#pragma unroll
                    for (int jj = 0; jj < NJ; ++jj) {
                        float* o = out + (size_t)(t0 + i) * strideM + NJ * tx + jj;
                        if (FLAGGED) atomicAdd(o, acc[ii][jj]);
                        else *o = acc[ii][jj];
                    }
                }
            }
        }
        __syncthreads();
        // W~ for the state update: forward W exp(G_C - G), reverse W exp(G).  A moderate chunk's weights are W exp(-G) and
        // W exp(G): the forward update takes its exp(G_C) with the state, S <- exp(G_C) (S + Xk^T W')
        if (!moderate) {
            for (int idx = tid; idx < kC * M; idx += 256) {
                const int r = idx / M, s = idx % M;
                sW[r * LM + s] *= __expf(REV ? sG[r * LM + s] : sG[(kC - 1) * LM + s] - sG[r * LM + s]);
            }
            __syncthreads();
        }
        // S <- S * exp(G_C) + Xk^T W~
        {
            float acc[4][NJ] = {};
            mm_tn<NJ>(sXk, kLd, sW, LM, kC, ty, tx, acc);
#pragma unroll
            for (int jj = 0; jj < NJ; ++jj) {
                const int s = NJ * tx + jj;
                const float egc = __expf(sG[(kC - 1) * LM + s]);
#pragma unroll
                for (int ii = 0; ii < 4; ++ii) {
                    float& S = sS[(4 * ty + ii) * LM + s];
                    S = !REV && moderate ? (S + acc[ii][jj]) * egc : fmaf(S, egc, acc[ii][jj]);
                }
            }
        }
    }
    __syncthreads();
    if (a.Send) {
        for (int idx = tid; idx < kDS * M; idx += 256) {
            const int s = idx / kDS, c = idx % kDS;
            a.Send[((size_t)bh * M + s) * a.D + d0 + c] = sS[c * LM + s];
        }
    }
}

// =============================================================== state runs
// The end memories of every segment from empty ones, K and V side in one launch (the first slices0 slices of the grid are
// the K side's).  Only X^T W' of a chunk is left of value_side: the tiles of the next chunk are on their way meanwhile, and the
// state stays in registers (thread (ty, tx): channels 4 ty .., slots NJ tx ..).  Against two launches of value_side and one for
// the segments' log-decay: an fp32 training step, B = 2, T = 1024, 4 heads of 256, 439 -> 430 us; a forward over T = 256, 2 heads
// of 64, which is all launches, 41.0 -> 35.7 us.
struct StateSimtArgs {
    ValueSideArgs set[2];             // (xk, w: what enters the state and its weights; Send)
    int slices0;
};
template <int M> constexpr int kStateStage = kC * kLd + 2 * kC * (M + 4);       // floats of a stage: X, W, G

template <typename IO, int M, bool REV>
__global__ void __launch_bounds__(256, M > 64 ? 1 : 2) state_simt_kernel(StateSimtArgs sets) {
    follow_previous_grid();
    constexpr int NJ = M / 16, LM = M + 4;
    extern __shared__ __align__(16) float smem[];
    const bool second = (int)blockIdx.y >= sets.slices0;
    const ValueSideArgs& a = sets.set[second];
    const int slice = second ? blockIdx.y - sets.slices0 : blockIdx.y;
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
    const ScanSpan span = scan_span(blockIdx.x, a.H, a.T, a.nseg, a.tseg);
    const int bh = blockIdx.x, d0 = slice * kDS;
    const size_t strideD = (size_t)a.H * a.D, strideM = (size_t)a.H * M, head = (size_t)span.b * a.T * a.H + span.h;
    const IO* xk = (const IO*)a.xk + head * a.D + d0;
    const float* w = a.w + head * M;
    const float* G = a.G + head * M;
    const int nchunks = (span.t_end - span.t0 + kC - 1) / kC;
    auto request = [&](int it) {
        if (it < nchunks) {
            const int t0 = span.t0 + (REV ? nchunks - 1 - it : it) * kC, valid = min(kC, span.t_end - t0);
            float* stage = smem + (it & 1) * kStateStage<M>;
            load_io_tile<IO>(stage, xk + (size_t)t0 * strideD, strideD, valid);
            load_slot_tile<M, false>(stage + kC * kLd, w + (size_t)t0 * strideM, strideM, valid);
            load_slot_tile<M, true>(stage + kC * kLd + kC * LM, G + (size_t)t0 * strideM, strideM, valid);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float S[4][NJ] = {};
    double decay = 0.0;
    request(0);
    for (int it = 0; it < nchunks; ++it) {
        request(it + 1);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        const float* sX = smem + (it & 1) * kStateStage<M>;
        float* sW = smem + (it & 1) * kStateStage<M> + kC * kLd;
        const float* sG = sW + kC * LM;
        __syncthreads();
        const float gc = tid < M ? sG[(kC - 1) * LM + tid] : 0.f;
        decay += (double)gc;
        const bool moderate = __syncthreads_and(gc >= kFactorisedDecayMin) != 0;
        // forward: W exp(-G), the update taking its exp(G_C) with the state; W exp(G_C - G) where that would overflow;
        // reverse: W exp(G)
        for (int idx = tid; idx < kC * M; idx += 256) {
            const int r = idx / M, c = idx % M;
            const float g = sG[r * LM + c];
            sW[r * LM + c] *= __expf(REV ? g : (moderate ? -g : sG[(kC - 1) * LM + c] - g));
        }
        __syncthreads();
        float acc[4][NJ] = {};
        mm_tn<NJ>(sX, kLd, sW, LM, kC, ty, tx, acc);
#pragma unroll
        for (int jj = 0; jj < NJ; ++jj) {
            const float egc = __expf(sG[(kC - 1) * LM + NJ * tx + jj]);
#pragma unroll
            for (int ii = 0; ii < 4; ++ii)
                S[ii][jj] = !REV && moderate ? (S[ii][jj] + acc[ii][jj]) * egc : fmaf(S[ii][jj], egc, acc[ii][jj]);
        }
        __syncthreads();                      // the stage may be filled again
    }
#pragma unroll
    for (int jj = 0; jj < NJ; ++jj)
        *reinterpret_cast<float4*>(a.Send + ((size_t)bh * M + NJ * tx + jj) * a.D + d0 + 4 * ty) =
            make_float4(S[0][jj], S[1][jj], S[2][jj], S[3][jj]);
    if (a.seg_logdecay != nullptr && slice == 0 && tid < M) a.seg_logdecay[(size_t)bh * M + tid] = (float)decay;
}

// =============================================================== key_side (pass-2 form)
template <typename IO, int M, bool REV, bool FLAGGED>
__global__ void __launch_bounds__(256, M > 64 ? 1 : 2) key_side_simt_kernel(KeySideArgs a, const int* strong_flag) {
    follow_previous_grid();
    if (FLAGGED && strong_flag[blockIdx.x] == 0) return;
    constexpr int LM = M + 4;
    extern __shared__ __align__(16) float smem[];
    float* sQ = smem;                  // [64][LM]  uq (scaled in place)
    float* sK = sQ + kC * LM;          // [64][LM]  uk (scaled in place)
    float* sG = sK + kC * LM;          // [64][LM]
    float* sV = sG + kC * LM;          // [64][68]
    float* sA = sV + kC * kLd;         // [64][68]
    float* sS = sA + kC * kLd;         // [M][68]
    __shared__ int s_flag;

    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
    const ScanSpan span = scan_span(blockIdx.x, a.H, a.T, a.nseg, a.tseg);
    const int slice = blockIdx.y, bh = blockIdx.x, b = span.b, h = span.h;
    const int d0 = slice * kDS;
    const size_t strideD = (size_t)a.H * a.D, strideM = (size_t)a.H * M;
    const float* uq = a.uq + ((size_t)b * a.T * a.H + h) * M;
    const float* uk = a.uk + ((size_t)b * a.T * a.H + h) * M;
    const float* G = a.G + ((size_t)b * a.T * a.H + h) * M;
    const IO* xv = (const IO*)a.xv + ((size_t)b * a.T * a.H + h) * a.D + d0;
    IO* out = (IO*)a.out + ((size_t)b * a.T * a.H + h) * a.D + d0;

    const int nchunks = (span.t_end - span.t0 + kC - 1) / kC;
    for (int it = 0; it < nchunks; ++it) {
        const int n = REV ? nchunks - 1 - it : it;
        const int t0 = span.t0 + n * kC;
        const int valid = min(kC, span.t_end - t0);
        __syncthreads();
        load_slot_tile<M, false>(sQ, uq + (size_t)t0 * strideM, strideM, valid);
        load_slot_tile<M, false>(sK, uk + (size_t)t0 * strideM, strideM, valid);
        load_slot_tile<M, true>(sG, G + (size_t)t0 * strideM, strideM, valid);
        load_io_tile<IO>(sV, xv + (size_t)t0 * strideD, strideD, valid);
        if (it == 0) {       // (behind the first tiles' copies)
#pragma unroll
            for (int idx = tid; idx < M * kDS; idx += 256) {
                const int s = idx / kDS, c = idx % kDS;
                sS[s * kLd + c] = a.S0 ? a.S0[((size_t)bh * M + s) * a.D + d0 + c] : 0.f;
            }
        }
        copies_landed();
        __syncthreads();
        const bool moderate = chunk_is_moderate<M>(sG, &s_flag);
        // A_ij = sum_s uq_i[s] uk_j[s] exp(+-(G_i[s] - G_j[s])) on the kept triangle
        if (moderate) {
            for (int idx = tid; idx < kC * M; idx += 256) {
                const int r = idx / M, s = idx % M;
                const float e = __expf(sG[r * LM + s]);
                const float einv = __expf(-sG[r * LM + s]);
                sQ[r * LM + s] *= REV ? einv : e;
                sK[r * LM + s] *= REV ? e : einv;
            }
            __syncthreads();
            masked_product<REV>(sQ, LM, sK, LM, M, sA, ty, tx);
        } else {
            float acc[4][4] = {};
            for (int s = 0; s < M; ++s) {
                float qi[4], gi[4], kj[4], gj[4];
#pragma unroll
                for (int ii = 0; ii < 4; ++ii) { qi[ii] = sQ[(4 * ty + ii) * LM + s]; gi[ii] = sG[(4 * ty + ii) * LM + s]; }
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) { kj[jj] = sK[(tx + 16 * jj) * LM + s]; gj[jj] = sG[(tx + 16 * jj) * LM + s]; }
#pragma unroll
                for (int ii = 0; ii < 4; ++ii)
#pragma unroll
                    for (int jj = 0; jj < 4; ++jj) {
                        const float ex = REV ? gj[jj] - gi[ii] : gi[ii] - gj[jj];
                        acc[ii][jj] = fmaf(qi[ii] * kj[jj], __expf(fminf(ex, 0.f)), acc[ii][jj]);
                    }
            }
#pragma unroll
            for (int ii = 0; ii < 4; ++ii)
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) {
                    const int i = 4 * ty + ii, j = tx + 16 * jj;
                    const bool keep = REV ? (j >= i) : (j <= i);
                    sA[i * kLd + j] = keep ? acc[ii][jj] : 0.f;
                }
        }
        __syncthreads();
        // bring uq, uk to the scalings of the state terms:
        //   forward: Q- = uq exp(G),        K- = uk exp(G_C - G)
        //   reverse: Q- = uq exp(G_C - G),  K- = uk exp(G)
        // (a moderate chunk has uq exp(G) and uk exp(-G), reversed uq exp(-G) and uk exp(G): forward, the state takes the
        // exp(G_C) of its update, S <- exp(G_C) (S + K-^T Xv))
        if (!moderate || REV) {
            for (int idx = tid; idx < kC * M; idx += 256) {
                const int r = idx / M, s = idx % M;
                const float g = sG[r * LM + s], gc = sG[(kC - 1) * LM + s];
                sQ[r * LM + s] *= __expf(REV ? (moderate ? gc : gc - g) : g);
                if (!moderate) sK[r * LM + s] *= __expf(REV ? g : gc - g);
            }
            __syncthreads();
        }
        // out = Q- S + A Xv
        {
            float acc[4][4] = {};
            mm_nn<4>(sQ, LM, sS, kLd, M, ty, tx, acc);
            mm_masked<REV, 4>(sA, sV, kLd, ty, tx, acc);
#pragma unroll
            for (int ii = 0; ii < 4; ++ii) {
                const int i = 4 * ty + ii;
                if (i < valid) store_vec4(out + (size_t)(t0 + i) * strideD + 4 * tx, acc[ii]);
            }
        }
        __syncthreads();
        // S <- exp(G_C)[:,None] S + K-^T Xv   (thread (ty,tx): slots 4ty.., channels 4tx..)
        // (64 slots per sweep of the 16 x 16 thread grid)
        for (int s0 = 0; s0 < M; s0 += 64) {
            if (s0 + 4 * ty >= M) break;
            float acc[4][4] = {};
            mm_tn<4>(sK + s0, LM, sV, kLd, kC, ty, tx, acc);
#pragma unroll
            for (int ii = 0; ii < 4; ++ii) {
                const int s = s0 + 4 * ty + ii;
                const float e = __expf(sG[(kC - 1) * LM + s]);
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) {
                    float& S = sS[s * kLd + 4 * tx + jj];
                    S = !REV && moderate ? (S + acc[ii][jj]) * e : fmaf(S, e, acc[ii][jj]);
                }
            }
        }
    }
    __syncthreads();
    if (a.Send) {
        for (int idx = tid; idx < M * kDS; idx += 256) {
            const int s = idx / kDS, c = idx % kDS;
            a.Send[((size_t)bh * M + s) * a.D + d0 + c] = sS[s * kLd + c];
        }
    }
}

template <typename K>
cudaError_t set_smem(K kernel, size_t bytes) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <typename IO, int M, bool REV, bool FLAGGED = false>
cudaError_t launch_vs(const ValueSideArgs& a, cudaStream_t st, const int* strong_flag = nullptr) {
    const size_t smem = sizeof(float) * (3 * kC * kLd + (kDS + 2 * kC) * (M + 4));
    cudaError_t e = set_smem(value_side_simt_kernel<IO, M, REV, FLAGGED>, smem);
    if (e != cudaSuccess) return e;
    dim3 grid(a.B * a.nseg * a.H, a.D / kDS);
    // (beside the tensor-core kernels the CTAs usually leave at once: placed early, they would keep SMs from the scans of
    // other streams while they wait, 1220 against 1145 us for a training step with 128 slots)
    if (FLAGGED) value_side_simt_kernel<IO, M, REV, FLAGGED><<<grid, 256, smem, st>>>(a, strong_flag);
    else launch_after(value_side_simt_kernel<IO, M, REV, FLAGGED>, grid, 256, smem, st, a, strong_flag);
    return cudaGetLastError();
}
template <typename IO, int M, bool REV, bool FLAGGED = false>
cudaError_t launch_ks(const KeySideArgs& a, cudaStream_t st, const int* strong_flag = nullptr) {
    const size_t smem = sizeof(float) * (3 * kC * (M + 4) + 2 * kC * kLd + M * kLd);
    cudaError_t e = set_smem(key_side_simt_kernel<IO, M, REV, FLAGGED>, smem);
    if (e != cudaSuccess) return e;
    dim3 grid(a.B * a.nseg * a.H, a.D / kDS);
    if (FLAGGED) key_side_simt_kernel<IO, M, REV, FLAGGED><<<grid, 256, smem, st>>>(a, strong_flag);
    else launch_after(key_side_simt_kernel<IO, M, REV, FLAGGED>, grid, 256, smem, st, a, strong_flag);
    return cudaGetLastError();
}

template <typename IO, int M, bool REV>
cudaError_t launch_states(const StateSimtArgs& sets, cudaStream_t st) {
    const size_t smem = sizeof(float) * 2 * kStateStage<M>;
    cudaError_t e = set_smem(state_simt_kernel<IO, M, REV>, smem);
    if (e != cudaSuccess) return e;
    const ValueSideArgs &k = sets.set[0], &v = sets.set[1];
    launch_after(state_simt_kernel<IO, M, REV>, dim3(k.B * k.nseg * k.H, sets.slices0 + v.D / kDS), 256, smem, st, sets);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_state_scan_simt(const ValueSideArgs& k, const ValueSideArgs& v, int io, int M, int reverse, cudaStream_t st) {
    const StateSimtArgs sets{{k, v}, k.D / kDS};
#define GSA_STATES(IO, MM) return reverse ? launch_states<IO, MM, true>(sets, st) : launch_states<IO, MM, false>(sets, st)
    if (io == GSA_BF16) {
        if (M == 128) { GSA_STATES(__nv_bfloat16, 128); } else if (M == 64) { GSA_STATES(__nv_bfloat16, 64); } else { GSA_STATES(__nv_bfloat16, 32); }
    } else {
        if (M == 128) { GSA_STATES(float, 128); } else if (M == 64) { GSA_STATES(float, 64); } else { GSA_STATES(float, 32); }
    }
#undef GSA_STATES
}

cudaError_t launch_value_side_simt(const ValueSideArgs& a, int io, int M, int reverse, cudaStream_t st, const int* strong_flag) {
    if (strong_flag != nullptr) {        // (beside the kernels for 128 slots)
        if (io != GSA_BF16 || M != 128) return cudaErrorNotSupported;
        return reverse ? launch_vs<__nv_bfloat16, 128, true, true>(a, st, strong_flag)
                       : launch_vs<__nv_bfloat16, 128, false, true>(a, st, strong_flag);
    }
#define GSA_VS(IO, MM)                                                                   \
    return reverse ? launch_vs<IO, MM, true>(a, st) : launch_vs<IO, MM, false>(a, st)
    if (io == GSA_BF16) {
        if (M == 128) { GSA_VS(__nv_bfloat16, 128); } else if (M == 64) { GSA_VS(__nv_bfloat16, 64); } else { GSA_VS(__nv_bfloat16, 32); }
    } else {
        if (M == 128) { GSA_VS(float, 128); } else if (M == 64) { GSA_VS(float, 64); } else { GSA_VS(float, 32); }
    }
#undef GSA_VS
}

cudaError_t launch_key_side_simt(const KeySideArgs& a, int io, int M, int reverse, cudaStream_t st, const int* strong_flag) {
    if (strong_flag != nullptr) {
        if (io != GSA_BF16 || M != 128) return cudaErrorNotSupported;
        return reverse ? launch_ks<__nv_bfloat16, 128, true, true>(a, st, strong_flag)
                       : launch_ks<__nv_bfloat16, 128, false, true>(a, st, strong_flag);
    }
#define GSA_KS(IO, MM)                                                                   \
    return reverse ? launch_ks<IO, MM, true>(a, st) : launch_ks<IO, MM, false>(a, st)
    if (io == GSA_BF16) {
        if (M == 128) { GSA_KS(__nv_bfloat16, 128); } else if (M == 64) { GSA_KS(__nv_bfloat16, 64); } else { GSA_KS(__nv_bfloat16, 32); }
    } else {
        if (M == 128) { GSA_KS(float, 128); } else if (M == 64) { GSA_KS(float, 64); } else { GSA_KS(float, 32); }
    }
#undef GSA_KS
}

}  // namespace gsa
