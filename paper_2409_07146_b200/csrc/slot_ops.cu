// Slot-axis (m-sized) kernels of the GSA layer: the chunk-local log-gate cumulative sum
// (chunk_cumsum of Algorithm 1), the slot softmax between the two passes and its
// backward, and the forget-gate gradient (reversed cumulative sum, App. B).
// All of them stream [B,T,H,m] fp32 tensors once: they are HBM-bound.
#include <type_traits>

#include "common.cuh"
#include "tc_common.cuh"

namespace gsa {

// ------------------------------------------------------------------ chunk_cumsum
// One CTA per (b,h, chunk): M/2 slot pairs x (chunk / 8) row groups.  A thread takes the logs
// of its 8 rows x 2 slots (8 independent 8-byte loads in flight), sums them, the group sums
// are scanned through shared memory, and the thread writes its running sums.  `chunk` is the
// chunk length of the kernels that will consume G (64 or 128).
constexpr int kCumRows = 8;

// (x0, x1) as a packed bf16 pair and the packed rounding residuals: two packed conversions
__device__ __forceinline__ void split_bf16x2(float x0, float x1, uint32_t& hi, uint32_t& lo) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    const __nv_bfloat162 l = __floats2bfloat162_rn(x0 - __uint_as_float(hi << 16), x1 - __uint_as_float(hi & 0xffff0000u));
    lo = *reinterpret_cast<const uint32_t*>(&l);
}
// ... as three parts: bits 0-7, 8-15 and 16-23 of the mantissas
__device__ __forceinline__ void split_bf16x3(float x0, float x1, uint32_t& hi, uint32_t& mid, uint32_t& lo) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    split_bf16x2(x0 - __uint_as_float(hi << 16), x1 - __uint_as_float(hi & 0xffff0000u), mid, lo);
}
template <int M>
__device__ __forceinline__ void store_split2(__nv_bfloat16* row, int c, float x0, float x1) {
    uint32_t hi, lo;
    split_bf16x2(x0, x1, hi, lo);
    *reinterpret_cast<uint32_t*>(row + c) = hi;
    *reinterpret_cast<uint32_t*>(row + M + c) = lo;
}

// Packed sequences: is token t the first token of a sequence other than the first?  cu holds the
// nseq + 1 ascending sequence offsets along T (cu[0] = 0, cu[nseq] = T).
__device__ __forceinline__ bool sequence_starts_at(const int* cu, int nseq, int t) {
    if (cu == nullptr || t == 0) return false;
    int lo = 1, hi = nseq - 1;
    while (lo <= hi) {
        const int mid = (lo + hi) >> 1, v = cu[mid];
        if (v == t) return true;
        if (v < t) lo = mid + 1; else hi = mid - 1;
    }
    return false;
}

// What the first token of a packed sequence does to the running log gate.  The memories must lose all they carried
// there: a log gate of -100, and that is what the CUDA-core kernels get.  On the tensor-core kernels it drops the chunk's
// total below what the factorised decay can represent, and the whole (batch, head, segment) goes to the strong-decay
// kernels: a training step on 8K tokens of 13 sequences, 4 heads of 512, takes 970 us where every chunk with an offset
// goes there, 620 where the segments with two in a chunk do, 330 where none does.  A drop of kReset leaves e^-40 = 4e-18 of the old memories -- less than an fp32 rounding of the new ones
// while the old are not 1e10 times larger, a slot's first write of 1e-4 of the new values and old values 1e6 times as
// large -- and the chunk stays on the pipelined kernels where the decay of every slot leaves room for it: for one start in
// a chunk down to a chunk's own decay of e^-20.  Everywhere else the chunk takes -100 and the strong-decay kernels.
constexpr float kReset = 40.f;

// KIND: gate_kind.  WIDE: the halves of 128 slots as 2 H heads of 64 (see launch_gate_cumsum_wide), which share their
// head's flag.  907 instructions a thread -- the kind asked for at every element, a predicate at every row, a 64-bit address
// for every access -- kept the issue slots as busy as the memory; with the kind a template argument, whole chunks apart from
// ragged ones and 32-bit offsets from a thread's first element: B = 4, T = 4096, 32 heads, 64 slots (0.54 GB) 137 -> 95 us,
// 5.7 TB/s; 128 slots, B = 8, T = 2048, 4 heads 48 -> 39.
template <int M, bool WIDE, int KIND>
__global__ void __launch_bounds__(M * 8 > 1024 ? 1024 : M * 8, M > 64 ? 1 : 2) gate_cumsum_kernel(const float* gate,
                                                            float inv_tau,
                                                            float* __restrict__ G,
                                                            float* __restrict__ I, int T, int H,
                                                            int chunk, int* __restrict__ strong_flag, int nseg, int tseg,
                                                            __nv_bfloat16* __restrict__ decayed, int fast_log,
                                                            const int* cu_seqlens, int nseq,
                                                            float* __restrict__ E, int leave_out, int* __restrict__ large_weight) {
    follow_previous_grid();
    __shared__ double2 group_sum[16][M / 2];
    const int grp = threadIdx.y, s = 2 * threadIdx.x;          // blockDim.y = chunk / 8 <= 16
    const int n = blockIdx.y;
    const int bh = blockIdx.x, b = bh / H, h = bh % H;
    const int t_chunk = n * chunk, rows_here = min(T - t_chunk, chunk);
    const int rows = max(0, min(kCumRows, rows_here - grp * kCumRows));
    // (a thread's first element, and 32-bit offsets from there: eight rows hold less than 2^32 elements, 16 GB of gates; a
    // chunk's 128 need not)
    const size_t first = (((size_t)b * T + t_chunk + grp * kCumRows) * H + h) * M + s;
    const uint32_t stride = (uint32_t)H * M;
    float2 g[kCumRows], inps[kCumRows];
    __shared__ uint32_t starts[4];                // rows of the chunk that begin a packed sequence, one bit each
    if (cu_seqlens != nullptr) {
        const int tid = threadIdx.y * blockDim.x + threadIdx.x;
        if (tid < 4) starts[tid] = 0;
        __syncthreads();
        for (int r = tid; r < rows_here; r += blockDim.x * blockDim.y)
            if (sequence_starts_at(cu_seqlens, nseq, t_chunk + r)) atomicOr(&starts[r >> 5], 1u << (r & 31));
        __syncthreads();
    }
    {
        // (rows past the end: a = 1, log a = 0)
        const float neutral = KIND == GSA_GATE_LOG_A ? 0.f : (KIND == GSA_GATE_LOGITS ? 80.f : 1.f);
        const float* src = gate + first;
        if (rows == kCumRows) {
#pragma unroll
            for (int i = 0; i < kCumRows; ++i) g[i] = *reinterpret_cast<const float2*>(src + i * stride);
        } else {
#pragma unroll
            for (int i = 0; i < kCumRows; ++i)
                g[i] = i < rows ? *reinterpret_cast<const float2*>(src + i * stride) : make_float2(neutral, neutral);
        }
    }
#pragma unroll
    for (int i = 0; i < kCumRows; ++i) {
        float2 x = g[i];
        if (KIND == GSA_GATE_LOGITS) x = make_float2(log_gate_from_logit(x.x, inv_tau), log_gate_from_logit(x.y, inv_tau));
        if (KIND != GSA_GATE_A) {
            inps[i] = make_float2(-expm1f(x.x), -expm1f(x.y));
        } else {
            inps[i] = make_float2(1.f - x.x, 1.f - x.y);
            x = fast_log ? make_float2(__logf(x.x), __logf(x.y)) : make_float2(logf(x.x), logf(x.y));
        }
        g[i] = make_float2(fmaxf(x.x, kLogGateMin), fmaxf(x.y, kLogGateMin));
    }
    const bool owns_flag = !WIDE && strong_flag != nullptr && owns_strong_flag(nseg, (int)gridDim.y);
    // is there a weight that is 2 or more, or no finite number (the exponent's top bit)?  See remembered_steps.  (Here, where nothing
    // of it is kept: behind the sums two registers spill, 32 K tokens of 16 heads 84.6 -> 86.4 us.)
    if (!WIDE && large_weight != nullptr) {
        uint32_t seen = 0;
#pragma unroll
        for (int i = 0; i < kCumRows; ++i) seen |= __float_as_uint(inps[i].x) | __float_as_uint(inps[i].y);
        bool large = (seen & 0x40000000u) != 0;
        if (owns_flag) large = __syncthreads_or(large);
        if (large || (owns_flag && threadIdx.x == 0 && grp == 0))
            large_weight[(b * nseg + (nseg == 1 ? 0 : t_chunk / tseg)) * H + h] = large;
    }
    // the first token of a packed sequence drops what the memories carried; its own write, 1 - a, is untouched
    if (cu_seqlens != nullptr && (starts[0] | starts[1] | starts[2] | starts[3]) != 0) {
        const uint32_t mine = (starts[(grp * kCumRows) >> 5] >> ((grp * kCumRows) & 31)) & ((1u << kCumRows) - 1);
        float reset = kLogGateMin;
        if (decayed != nullptr) {
            // the rest of the chunk's decay, by slot
            float own0 = 0.f, own1 = 0.f;
#pragma unroll
            for (int i = 0; i < kCumRows; ++i)
                if (i < rows && !((mine >> i) & 1)) { own0 += g[i].x; own1 += g[i].y; }
            group_sum[grp][threadIdx.x] = make_double2(own0, own1);
            __syncthreads();
            double all0 = 0.0, all1 = 0.0;
            for (int q = 0; q < (int)blockDim.y; ++q) { all0 += group_sum[q][threadIdx.x].x; all1 += group_sum[q][threadIdx.x].y; }
            const int count = __popc(starts[0]) + __popc(starts[1]) + __popc(starts[2]) + __popc(starts[3]);
            if (__syncthreads_and(fmin(all0, all1) - kReset * count >= (double)kFactorisedDecayMin)) reset = -kReset;
        }
#pragma unroll
        for (int i = 0; i < kCumRows; ++i)
            if ((mine >> i) & 1) g[i] = make_float2(reset, reset);
    }
    // running sums: fp32 inside the thread's 8 rows (g becomes the running sum), fp64 across the
    // row groups -- G stays within an ulp of the exact cumulative sum also where strong decay
    // makes |G| reach the hundreds, without a conversion per element
#pragma unroll
    for (int i = 1; i < kCumRows; ++i) {
        // (a row past the end adds its log a of 0)
        g[i].x += g[i - 1].x;
        g[i].y += g[i - 1].y;
    }
    const double acc0 = (double)g[kCumRows - 1].x, acc1 = (double)g[kCumRows - 1].y;
    group_sum[grp][threadIdx.x] = make_double2(acc0, acc1);
    __syncthreads();
    double before0 = 0.0, before1 = 0.0, half0 = 0.0, half1 = 0.0;       // (half: since the last multiple of 64 tokens)
#pragma unroll 5
    for (int q = 0; q < grp; ++q) {
        const double2 t = group_sum[q][threadIdx.x];
        if (WIDE && q == 64 / kCumRows) half0 = half1 = 0.0;
        before0 += t.x;
        before1 += t.y;
        if (WIDE) {
            half0 += t.x;
            half1 += t.y;
        }
    }
    if (WIDE && grp == 64 / kCumRows) half0 = half1 = 0.0;
    // the chunk's total log-decay decides which of the chunk kernels takes this (b,h)
    // (with segment-parallel scheduling the flags are per (batch, segment, head))
    const bool strong = strong_flag != nullptr && grp == (int)blockDim.y - 1 &&
                        fmin(before0 + acc0, before1 + acc1) < (double)kFactorisedDecayMin;
    // (1 - a left out: of the chunks that do not decide on the general scans by themselves, see InputGate)
    bool any_strong = strong;
    if (owns_flag || leave_out == 1) any_strong = __syncthreads_or(strong);
    const bool put_I = leave_out == 0 || (leave_out == 1 && any_strong);
    if (strong || (owns_flag && threadIdx.x == 0 && grp == 0)) {
        const int seg = nseg == 1 ? 0 : t_chunk / tseg;
        strong_flag[WIDE ? (b * nseg + seg) * (H / 2) + h / 2 : (b * nseg + seg) * H + h] = any_strong;
    }
    // second pass over the same rows: the sums of the groups before as a float pair (value, rest)
    const float b0h = (float)before0, b0l = (float)(before0 - (double)b0h);
    const float b1h = (float)before1, b1l = (float)(before1 - (double)b1h);
    auto write_row = [&](int i) {
        const uint32_t at = i * stride;
        if (put_I) *reinterpret_cast<float2*>(I + first + at) = inps[i];
        const float G0 = b0h + (b0l + g[i].x), G1 = b1h + (b1l + g[i].y);
        if (!WIDE) {
            *reinterpret_cast<float2*>(G + first + at) = make_float2(G0, G1);
            // (meaningful for moderate decay only; pairs with a strong-decay chunk do not read it)
            if (decayed != nullptr)
                store_split2<M>(decayed + 2 * (first - s) + 2 * (size_t)at, s, inps[i].x * exp_neg(G0), inps[i].y * exp_neg(G1));
        } else {
            // G itself is for the CUDA-core kernels, whose chunks have 64 tokens
            *reinterpret_cast<float2*>(G + first + at) =
                make_float2((float)(half0 + (double)g[i].x), (float)(half1 + (double)g[i].y));
            // exp(+-G) from the sum before its rounding to G: G0 + r0 is the sum of the pair and the thread's rows
            const float r0 = (b0l + g[i].x) - (G0 - b0h), r1 = (b1l + g[i].y) - (G1 - b1h);
            const float e0 = expf(G0), e1 = expf(G1), d0 = expf(-G0), d1 = expf(-G1);
            *reinterpret_cast<float2*>(E + first + at) = make_float2(fmaf(e0, r0, e0), fmaf(e1, r1, e1));
            uint32_t hi, mid, lo;
            split_bf16x3(inps[i].x * fmaf(d0, -r0, d0), inps[i].y * fmaf(d1, -r1, d1), hi, mid, lo);
            uint32_t* row = reinterpret_cast<uint32_t*>(decayed + 3 * (first - s) + s + 3 * (size_t)at);
            row[0] = hi;
            row[M / 2] = mid;
            row[M] = lo;
        }
    };
    if (rows == kCumRows) {
#pragma unroll
        for (int i = 0; i < kCumRows; ++i) write_row(i);
    } else {
#pragma unroll
        for (int i = 0; i < kCumRows; ++i)
            if (i < rows) write_row(i);
    }
}

template <int M, bool WIDE, class... A>
void launch_gate_kind(int gate_kind, dim3 grid, dim3 block, cudaStream_t st, const float* gate, A... rest) {
    if (gate_kind == GSA_GATE_A) launch_after(gate_cumsum_kernel<M, WIDE, GSA_GATE_A>, grid, block, 0, st, gate, rest...);
    else if (gate_kind == GSA_GATE_LOG_A) launch_after(gate_cumsum_kernel<M, WIDE, GSA_GATE_LOG_A>, grid, block, 0, st, gate, rest...);
    else launch_after(gate_cumsum_kernel<M, WIDE, GSA_GATE_LOGITS>, grid, block, 0, st, gate, rest...);
}

// a kernel rather than a memset, which the gate kernel could not follow closely (launch_after): a forward over 1431 tokens,
// 4 heads of 512, 50.7 -> 48.0 us; one over 256 tokens in fp32, which needs no flags, 33.7 -> 30.2
__global__ void clear_flags_kernel(int* __restrict__ flags, int* __restrict__ others, size_t n) {
    follow_previous_grid();
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        flags[i] = 0;
        if (others != nullptr) others[i] = 0;
    }
}
cudaError_t launch_clear_flags(int* flags, int* others, size_t n, cudaStream_t st) {
    launch_after(clear_flags_kernel, dim3((unsigned)((n + 255) / 256)), 256, 0, st, flags, others, n);
    return cudaGetLastError();
}

cudaError_t launch_gate_cumsum(const float* gate, int gate_kind, float inv_tau, float* G, float* I, int B,
                               int T, int H, int M, int chunk, int* strong_flag, int nseg, int tseg, void* decayed, int fast_log,
                               cudaStream_t st, const int* cu_seqlens, int nseq, int leave_out, int* large_weight) {
    if (chunk % kCumRows != 0 || chunk / kCumRows > 16 || (M / 2) * (chunk / kCumRows) > 1024) return cudaErrorInvalidValue;
    const int nchunks = (T + chunk - 1) / chunk;
    dim3 block(M / 2, chunk / kCumRows);
    dim3 grid(B * H, nchunks);
    auto launch = [&](auto m) {
        launch_gate_kind<decltype(m)::value, false>(gate_kind, grid, block, st, gate, inv_tau, G, I, T, H, chunk, strong_flag, nseg, tseg,
                                                    static_cast<__nv_bfloat16*>(decayed), fast_log, cu_seqlens, nseq, (float*)nullptr, leave_out, large_weight);
    };
    if (M == 128) launch(std::integral_constant<int, 128>{});
    else if (M == 64) launch(std::integral_constant<int, 64>{});
    else launch(std::integral_constant<int, 32>{});
    return cudaGetLastError();
}

cudaError_t launch_gate_cumsum_wide(const float* gate, int gate_kind, float inv_tau, float* G, float* I, float* E, int B, int T,
                                    int H, int* strong_flag, int nseg, int tseg, void* decayed, cudaStream_t st,
                                    const int* cu_seqlens, int nseq) {
    constexpr int chunk = 128;
    launch_gate_kind<64, true>(gate_kind, dim3(2 * B * H, (T + chunk - 1) / chunk), dim3(32, chunk / kCumRows), st, gate, inv_tau, G, I, T,
                               2 * H, chunk, strong_flag, nseg, tseg, static_cast<__nv_bfloat16*>(decayed), 0, cu_seqlens, nseq, E, 0, (int*)nullptr);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ slot softmax
// M/4 lanes per token-head row of M slots, four adjacent slots per lane (one 16-byte access per
// tensor and lane), 128/M rows per warp; reductions run over the lanes of a row.
constexpr int kSmR = 4;                                  // slots per lane
__device__ __forceinline__ void ld_vec(const float* p, float (&x)[kSmR]) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
}
__device__ __forceinline__ void st_vec(float* p, const float (&x)[kSmR]) {
    *reinterpret_cast<float4*>(p) = make_float4(x[0], x[1], x[2], x[3]);
}
// the lane's slots of a decayed-operand row [hi(M) | lo(M)]
template <int M>
__device__ __forceinline__ void st_split(__nv_bfloat16* row, int c, const float (&x)[kSmR]) {
    uint32_t h0, h1, l0, l1;
    split_bf16x2(x[0], x[1], h0, l0);
    split_bf16x2(x[2], x[3], h1, l1);
    *reinterpret_cast<uint2*>(row + c) = make_uint2(h0, h1);
    *reinterpret_cast<uint2*>(row + M + c) = make_uint2(l0, l1);
}
// ... as that of the operands with 128 slots: [half][high | middle | low] of 64 slots each
__device__ __forceinline__ void st_split3(__nv_bfloat16* row, int c, const float (&x)[kSmR]) {
    uint32_t h0, h1, m0, m1, l0, l1;
    split_bf16x3(x[0], x[1], h0, m0, l0);
    split_bf16x3(x[2], x[3], h1, m1, l1);
    __nv_bfloat16* at = row + 192 * (c >> 6) + (c & 63);
    *reinterpret_cast<uint2*>(at) = make_uint2(h0, h1);
    *reinterpret_cast<uint2*>(at + 64) = make_uint2(m0, m1);
    *reinterpret_cast<uint2*>(at + 128) = make_uint2(l0, l1);
}
template <int LPR>
__device__ __forceinline__ float row_max(float x) {
#pragma unroll
    for (int o = LPR / 2; o; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
    return x;
}
template <int LPR>
__device__ __forceinline__ float row_sum(float x) {
#pragma unroll
    for (int o = LPR / 2; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// A CTA's 256 threads hold 1024 consecutive values, 1024 / M rows.  These kernels move 16 bytes per thread and stream, so the
// instructions around a row count (302 a thread forward, a third of them integer, kept the issue slots busy for 35 of 57 us;
// 64 MB streams): everything that is the same for the CTA is formed from blockIdx alone, a thread adds a 32-bit offset, and
// the row's token and head come from a multiplication (FastDiv).  B = 4, T = 4096, 32 heads of 128: 113 -> 96 us, backward
// 154 -> 138; T = 32768, 16 heads: 113 -> 88.  (Two or four rows a thread instead, to have the same instructions serve more,
// costs occupancy: 127 .. 131 us and 162 .. 199.)
// x / d for x < 2^31: with mul = floor(2^shift / d) + 1, shift = 31 + ceil(log2 d), mul d exceeds 2^shift by at most d, and
// x d < 2^shift, so the quotient is exact; mul < 2^32.
struct FastDiv {
    uint32_t mul, shift;
    FastDiv() = default;
    explicit FastDiv(uint32_t d) : shift(31) {
        while ((1u << (shift - 31)) < d) ++shift;
        mul = (uint32_t)((1ull << shift) / d + 1);
    }
    __device__ __forceinline__ uint32_t operator()(uint32_t x) const { return (uint32_t)(((uint64_t)x * mul) >> shift); }
};
struct RowDivs { FastDiv heads, segment; };       // by H and by the tokens of a segment

template <int M> struct SlotPlace {
    static constexpr int kRows = 256 * kSmR / M;
    size_t cta;            // the CTA's first element
    uint32_t off;          // this thread's first element from there (a row past the end repeats the last one: full-warp shuffles)
    int col;               // ... and in its row
    int rows;              // of a batch element
    bool live, pending;
    __device__ __forceinline__ SlotPlace(int rows_per_batch, const PendingDecay& pend, const RowDivs& div) {
        const uint32_t row0 = blockIdx.x * kRows, left = rows_per_batch - row0, sub = threadIdx.x / (M / kSmR);
        rows = rows_per_batch;
        live = sub < left;
        const uint32_t r = min(sub, left - 1);
        col = (threadIdx.x % (M / kSmR)) * kSmR;
        cta = ((size_t)blockIdx.y * rows_per_batch + row0) * M;
        off = r * M + col;
        pending = false;
        if (pend.G != nullptr) {
            const uint32_t t = div.heads(row0 + r), h = row0 + r - t * pend.H, seg = pend.nseg == 1 ? 0 : div.segment(t);
            pending = pend.strong[(blockIdx.y * pend.nseg + seg) * (uint32_t)(pend.H >> pend.half_heads) + (h >> pend.half_heads)] == 0;
        }
    }
    // of the decayed operand rows, which hold 2 bf16 a slot (128 slots: 3)
    __device__ __forceinline__ size_t decayed() const { return (M == 128 ? 3 : 2) * (cta + (off - col)); }
};
template <int M>
__device__ __forceinline__ void slot_sums(const float* part, int nslice, const SlotPlace<M>& at, float (&x)[kSmR]) {
    ld_vec(part + at.cta + at.off, x);
    if (nslice == 1) return;
    const size_t total = (size_t)gridDim.y * (uint32_t)at.rows * M;
#pragma unroll 3
    for (int sl = 1; sl < nslice; ++sl) {
        float t[kSmR];
        ld_vec(part + (at.cta + sl * total) + at.off, t);
#pragma unroll
        for (int r = 0; r < kSmR; ++r) x[r] += t[r];
    }
}

template <int M>
__global__ void __launch_bounds__(256) slot_softmax_fwd_kernel(const float* part,
                                                               int nslice, float scale, int act,
                                                               float* __restrict__ ok,
                                                               float* __restrict__ p,
                                                               int rows_per_batch, const float* G,
                                                               __nv_bfloat16* __restrict__ p_decayed,
                                                               PendingDecay pend, int m_active, RowDivs div) {
    follow_previous_grid();
    constexpr int R = kSmR, LPR = M / R;       // lanes per row
    const SlotPlace<M> at(rows_per_batch, pend, div);
    const bool live = at.live, pending = at.pending;
    // slots from m_active on are padding (a layer with fewer slots than the kernels' tile): they take no part
    const bool padded = at.col >= m_active;
    // serving the flagged pairs only: a warp none of whose rows is flagged has nothing to do
    const bool skip = pend.strong_only != 0 && pending;
    if (__all_sync(0xffffffffu, skip)) return;
    float z[R], eg[R];
#pragma unroll
    for (int r = 0; r < R; ++r) eg[r] = 1.f;
    slot_sums<M>(part, nslice, at, z);
    if (G != nullptr) {
        ld_vec(G + at.cta + at.off, eg);
#pragma unroll
        for (int r = 0; r < R; ++r) eg[r] = M == 128 ? eg[r] : __expf(eg[r]);      // (128 slots: G holds exp(G) itself)
    }
    float zmax = -INFINITY;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if (pending) z[r] *= eg[r];
        z[r] *= scale;
        if (!padded) zmax = fmaxf(zmax, z[r]);
    }
    float e[R];
    if (act == GSA_ACT_SOFTMAX) {
        zmax = row_max<LPR>(zmax);
        float den = 0.f;
#pragma unroll
        for (int r = 0; r < R; ++r) { e[r] = padded ? 0.f : __expf(z[r] - zmax); den += e[r]; }
        den = row_sum<LPR>(den);
        const float inv = 1.f / den;
#pragma unroll
        for (int r = 0; r < R; ++r) e[r] *= inv;
    } else {               // element-wise replacement of the softmax (uniform over the launch)
#pragma unroll
        for (int r = 0; r < R; ++r) e[r] = padded ? 0.f : slot_act_value(z[r], act);
    }
    if (!live || skip) return;
    if (ok != nullptr) st_vec(ok + at.cta + at.off, z);
    // fp32 p is read by the general chunk kernels and the CUDA-core kernels only: rows of a pair
    // that the pipelined kernels serve (pending) get the decayed bf16 rows alone
    if (!pending) st_vec(p + at.cta + at.off, e);
    if (p_decayed != nullptr) {
#pragma unroll
        for (int r = 0; r < R; ++r) e[r] *= eg[r];
        if (M == 128) st_split3(p_decayed + at.decayed(), at.col, e);
        else st_split<M>(p_decayed + at.decayed(), at.col, e);
    }
}

cudaError_t launch_slot_softmax_fwd(const float* part, int nslice, float scale, int act, float* ok,
                                    float* p, int B, int rows_per_batch, int M, const float* G, void* p_decayed,
                                    PendingDecay pend, cudaStream_t st, int m_active) {
    if (m_active <= 0 || m_active > M) m_active = M;
    const int rpb = 8 * (128 / M);       // rows per block: 8 warps x 128/M rows
    const dim3 grid((unsigned)((rows_per_batch + rpb - 1) / rpb), (unsigned)B);
    const int rows = rows_per_batch;
    const RowDivs div{FastDiv(pend.H), FastDiv(pend.tseg)};
    if (M == 128)
        launch_after(slot_softmax_fwd_kernel<128>, grid, 256, 0, st, part, nslice, scale, act, ok, p, rows, G,
                                                           static_cast<__nv_bfloat16*>(p_decayed), pend, m_active, div);
    else if (M == 64)
        launch_after(slot_softmax_fwd_kernel<64>, grid, 256, 0, st, part, nslice, scale, act, ok, p, rows, G,
                                                          static_cast<__nv_bfloat16*>(p_decayed), pend, m_active, div);
    else
        launch_after(slot_softmax_fwd_kernel<32>, grid, 256, 0, st, part, nslice, scale, act, ok, p, rows, G,
                                                          static_cast<__nv_bfloat16*>(p_decayed), pend, m_active, div);
    return cudaGetLastError();
}

// Softmax backward (dsoftmax of Algorithm 1; f'(ok) dp for an element-wise replacement f): from the scaled logits ok and the gradient dp
// w.r.t. the softmax output (summed over the d_v slices that produced it):
//   p = softmax(ok); dok = p * (dp - <p,dp>); dz = scale * dok (gradient w.r.t. the unscaled
//   pass-1 output); u = p*dp + ok*dok (the two "query x query-gradient" terms of the
//   forget-gate gradient).
template <int M>
__global__ void __launch_bounds__(256) slot_softmax_bwd_kernel(const float* ok,
                                                               const float* dp_part,
                                                               int nslice, float scale, int act,
                                                               float* __restrict__ p,
                                                               float* __restrict__ dz,
                                                               float* __restrict__ u,
                                                               int rows_per_batch, const float* G,
                                                               __nv_bfloat16* __restrict__ p_decayed,
                                                               __nv_bfloat16* __restrict__ dz_decayed,
                                                               PendingDecay pend, int m_active, RowDivs div) {
    follow_previous_grid();
    constexpr int R = kSmR, LPR = M / R;       // lanes per row
    const SlotPlace<M> at(rows_per_batch, pend, div);
    const bool live = at.live, pending = at.pending;
    const bool skip = pend.strong_only != 0 && pending;      // (as in the forward kernel)
    const bool padded = at.col >= m_active;                  // (likewise)
    if (__all_sync(0xffffffffu, skip)) return;
    float z[R], dpv[R], eg[R];
    ld_vec(ok + at.cta + at.off, z);
#pragma unroll
    for (int r = 0; r < R; ++r) eg[r] = 1.f;
    slot_sums<M>(dp_part, nslice, at, dpv);
    if (G != nullptr) {
        ld_vec(G + at.cta + at.off, eg);
#pragma unroll
        for (int r = 0; r < R; ++r) eg[r] = M == 128 ? eg[r] : __expf(eg[r]);      // (128 slots: G holds exp(G) itself)
    }
    float zmax = -INFINITY;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if (pending) dpv[r] *= eg[r];
        if (padded) { z[r] = 0.f; dpv[r] = 0.f; }
        else zmax = fmaxf(zmax, z[r]);
    }
    float e[R], dzv[R], uv[R];
    if (act == GSA_ACT_SOFTMAX) {
        zmax = row_max<LPR>(zmax);
        float den = 0.f;
#pragma unroll
        for (int r = 0; r < R; ++r) { e[r] = padded ? 0.f : __expf(z[r] - zmax); den += e[r]; }
        den = row_sum<LPR>(den);
        const float inv = 1.f / den;
        float pdp = 0.f;
#pragma unroll
        for (int r = 0; r < R; ++r) { e[r] *= inv; pdp += e[r] * dpv[r]; }
        pdp = row_sum<LPR>(pdp);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float dok = e[r] * (dpv[r] - pdp);
            dzv[r] = scale * dok;
            uv[r] = e[r] * dpv[r] + z[r] * dok;
        }
    } else {               // element-wise replacement f of the softmax: dok = f'(ok) dp
#pragma unroll
        for (int r = 0; r < R; ++r) {
            e[r] = padded ? 0.f : slot_act_value(z[r], act);
            const float dok = slot_act_slope(z[r], act) * dpv[r];
            dzv[r] = scale * dok;
            uv[r] = e[r] * dpv[r] + z[r] * dok;
        }
    }
    if (!live || skip) return;
    if (!pending) {       // (as in the forward: fp32 p and dz only where a non-pipelined kernel reads them)
        if (p != nullptr) st_vec(p + at.cta + at.off, e);      // (p == NULL: the forward's p is kept and in use)
        st_vec(dz + at.cta + at.off, dzv);
    }
    st_vec(u + at.cta + at.off, uv);
    if (dz_decayed != nullptr) {
#pragma unroll
        for (int r = 0; r < R; ++r) { e[r] *= eg[r]; dzv[r] *= eg[r]; }
        if (M == 128) {
            if (p_decayed != nullptr) st_split3(p_decayed + at.decayed(), at.col, e);
            st_split3(dz_decayed + at.decayed(), at.col, dzv);
        } else {
            if (p_decayed != nullptr) st_split<M>(p_decayed + at.decayed(), at.col, e);
            st_split<M>(dz_decayed + at.decayed(), at.col, dzv);
        }
    }
}

cudaError_t launch_slot_softmax_bwd(const float* ok, const float* dp_part, int nslice,
                                    float scale, int act, float* p, float* dz, float* u, int B, int rows_per_batch,
                                    int M, const float* G, void* p_decayed, void* dz_decayed,
                                    PendingDecay pend, cudaStream_t st, int m_active) {
    if (m_active <= 0 || m_active > M) m_active = M;
    const int rpb = 8 * (128 / M);       // rows per block: 8 warps x 128/M rows
    const dim3 grid((unsigned)((rows_per_batch + rpb - 1) / rpb), (unsigned)B);
    const int rows = rows_per_batch;
    const RowDivs div{FastDiv(pend.H), FastDiv(pend.tseg)};
    if (M == 128)
        launch_after(slot_softmax_bwd_kernel<128>, grid, 256, 0, st, ok, dp_part, nslice, scale, act, p, dz, u, rows, G,
                                                           static_cast<__nv_bfloat16*>(p_decayed),
                                                           static_cast<__nv_bfloat16*>(dz_decayed), pend, m_active, div);
    else if (M == 64)
        launch_after(slot_softmax_bwd_kernel<64>, grid, 256, 0, st, ok, dp_part, nslice, scale, act, p, dz, u, rows, G,
                                                          static_cast<__nv_bfloat16*>(p_decayed),
                                                          static_cast<__nv_bfloat16*>(dz_decayed), pend, m_active, div);
    else
        launch_after(slot_softmax_bwd_kernel<32>, grid, 256, 0, st, ok, dp_part, nslice, scale, act, p, dz, u, rows, G,
                                                          static_cast<__nv_bfloat16*>(p_decayed),
                                                          static_cast<__nv_bfloat16*>(dz_decayed), pend, m_active, div);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ forget-gate gradient
// d(log a_t)|decay = sum_{i>=t} (u_i - I_i * dI_i) + <dKT, K_T>_rows + <dVT, V_T>_rows
// (the reversed cumulative sum of App. B, taken over the whole sequence), then
//   gate holds a     : dgate = d(log a)|decay / a - dI
//   gate holds log a : dgate = d(log a)|decay - a * dI
// Three steps: block-local reversed sums of 16-row blocks (the only pass over the inputs), an
// exclusive suffix scan over the block totals (fp64), and the addition of each block's carry.

constexpr int kGG = 16;   // rows per thread of the gate-gradient kernels

// Packed sequences: nothing of a later sequence reaches an earlier one, so the running sum restarts at every token
// that begins a sequence.  (The totals of the later sequences vanish exactly, their roundings do not: without the
// restart they are all added to every token before.)  Which of the rows [t0, t0 + rows) begin one, a bit each.  (An
// offset T is that of an empty sequence behind the last token: callers whose sums take terms from behind the last token
// end their rows at T.)
__device__ __forceinline__ uint32_t starts_among(const int* cu, int nseq, int t0, int rows) {
    uint32_t mask = 0;
    if (cu == nullptr) return mask;
    int lo = 1, hi = nseq;                       // the first offset >= max(t0, 1) among cu[1 .. nseq - 1]
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (cu[mid] < max(t0, 1)) lo = mid + 1; else hi = mid;
    }
    for (; lo < nseq && cu[lo] < t0 + rows; ++lo) mask |= 1u << (cu[lo] - t0);
    return mask;
}

// From the decay-path gradient d(log a) (`run`: what this block knows of it) and the input-gate
// gradient dI to the gradient with respect to the gate tensor as passed (`gt`):
//   a       : run / a - dI            (a == 0 leaves no way back from d(log a): only -dI is kept)
//   log a   : run - a dI
//   logits  : (run - a dI) sigmoid(-x) / tau
__device__ __forceinline__ float gate_grad_out(float run, float dI, float gt, int gate_kind, float inv_tau) {
    if (gate_kind == GSA_GATE_A) return (gt > 0.f) ? run / gt - dI : -dI;
    if (gate_kind == GSA_GATE_LOG_A) return run - __expf(fmaxf(gt, kLogGateMin)) * dI;
    const float a = __expf(fmaxf(log_gate_from_logit(gt, inv_tau), kLogGateMin));
    return (run - a * dI) * dlog_gate_dlogit(gt, inv_tau);
}
// the carry of the blocks after this one, in the same units
__device__ __forceinline__ float gate_grad_carry(float carry, float gt, int gate_kind, float inv_tau) {
    if (gate_kind == GSA_GATE_A) return (gt > 0.f) ? carry / gt : 0.f;
    if (gate_kind == GSA_GATE_LOG_A) return carry;
    return carry * dlog_gate_dlogit(gt, inv_tau);
}

// dI[i] = sum over the d_k and d_v slices of the input-gate gradient partial sums, for the
// kGG rows x 2 slots of this thread; the rows of one slice are loaded together (16 loads of 8
// bytes in flight).
__device__ __forceinline__ void load_dI(const float* dIk, int nsk, const float* dIv,
                                        int nsv, size_t base, size_t stride, size_t total, int rows,
                                        float2 (&dI)[kGG]) {
#pragma unroll
    for (int i = 0; i < kGG; ++i) dI[i] = make_float2(0.f, 0.f);
    for (int sl = 0; sl < nsk + nsv; ++sl) {
        const float* src = sl < nsk ? dIk + (size_t)sl * total : dIv + (size_t)(sl - nsk) * total;
        float2 t[kGG];
#pragma unroll
        for (int i = 0; i < kGG; ++i)
            t[i] = (i < rows) ? *reinterpret_cast<const float2*>(src + base + (size_t)i * stride) : make_float2(0.f, 0.f);
#pragma unroll
        for (int i = 0; i < kGG; ++i) { dI[i].x += t[i].x; dI[i].y += t[i].y; }
    }
}

// blk_tot[bh][n][s] <- sum over blocks n' > n of the totals, plus the final-memory term.
// One CTA per (b,h): M slots x 16 segments of consecutive blocks; fp64 running sums.
// Packed sequences: which blocks hold the first token of one stands in a bit each, set from the offsets once: 8192
// tokens of 13 sequences, 4 heads, 36 -> 12 us against searching the offsets for every block, twice.  (Sequences too long for
// the bits are still searched.)
constexpr int kScanBlocks = 1 << 16;
template <int M>
__global__ void __launch_bounds__(M * (M > 64 ? 8 : 16)) gate_grad_scan_kernel(
    float* blk_tot, const float* dKT, const float* KT,
    const float* dVT, const float* VT, int d_k, int d_v, int nblk, int T,
    const int* cu, int nseq) {
    follow_previous_grid();
    constexpr int kSeg = M > 64 ? 8 : 16;       // segments of consecutive blocks (threads: M slots x kSeg)
    __shared__ double seg_sum[kSeg][M];
    const int s = threadIdx.x, seg = threadIdx.y, bh = blockIdx.x;
    const int per = (nblk + kSeg - 1) / kSeg;
    const int lo = seg * per, hi = min(nblk, lo + per);
    __shared__ uint32_t starting[kScanBlocks / 32];
    const bool bits = nblk <= kScanBlocks;
    if (cu != nullptr && bits) {
        const int tid = seg * M + s;
        for (int i = tid; i < (nblk + 31) / 32; i += M * kSeg) starting[i] = 0;
        __syncthreads();
        for (int i = 1 + tid; i < nseq; i += M * kSeg) {
            const int t = cu[i];
            if (t >= 1 && t < T) atomicOr(&starting[t / kGG / 32], 1u << (t / kGG % 32));
        }
        __syncthreads();
    }
    auto starts_in = [&](int n) {
        if (cu == nullptr) return false;
        return bits ? (starting[n >> 5] >> (n & 31) & 1) != 0 : starts_among(cu, nseq, n * kGG, min(kGG, T - n * kGG)) != 0;
    };
    double sum = 0.0;
    __shared__ bool restarts[kSeg];              // does a packed sequence begin in the segment?
    if (cu == nullptr) {
        for (int n = lo; n < hi; ++n) sum += (double)blk_tot[((size_t)bh * nblk + n) * M + s];
    } else {
        bool any = false;
        for (int n = hi - 1; n >= lo; --n) {
            const bool here = starts_in(n);
            sum = (here ? 0.0 : sum) + (double)blk_tot[((size_t)bh * nblk + n) * M + s];
            any = any || here;
        }
        if (s == 0) restarts[seg] = any;
    }
    seg_sum[seg][s] = sum;
    // final-memory term <dK~_T[s], K~_T[s]> + <dV~_T[s], V~_T[s]>: a warp per slot, lanes along the row
    __shared__ double final_term[M];
    const int warp = (seg * M + s) >> 5, lane = (seg * M + s) & 31, nwarp = (M * kSeg) >> 5;
    for (int slot = warp; slot < M; slot += nwarp) {
        double dot = 0.0;
        if (dKT != nullptr) {
            const float* a = dKT + ((size_t)bh * M + slot) * d_k;
            const float* bb = KT + ((size_t)bh * M + slot) * d_k;
            for (int c = lane; c < d_k; c += 32) dot += (double)a[c] * (double)bb[c];
        }
        if (dVT != nullptr) {
            const float* a = dVT + ((size_t)bh * M + slot) * d_v;
            const float* bb = VT + ((size_t)bh * M + slot) * d_v;
            for (int c = lane; c < d_v; c += 32) dot += (double)a[c] * (double)bb[c];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
        if (lane == 0) final_term[slot] = dot;
    }
    __syncthreads();
    double carry = final_term[s];
    if (cu == nullptr) {
        for (int g = seg + 1; g < kSeg; ++g) carry += seg_sum[g][s];
    } else {
        for (int g = kSeg - 1; g > seg; --g) carry = (restarts[g] ? 0.0 : carry) + seg_sum[g][s];
    }
    for (int n = hi - 1; n >= lo; --n) {
        const size_t idx = ((size_t)bh * nblk + n) * M + s;
        const float t = blk_tot[idx];
        blk_tot[idx] = (float)carry;
        if (starts_in(n)) carry = 0.0;
        carry += (double)t;
    }
}

// Block-local pass: for each 16-row block, the reversed running sums of x = u - I dI that start
// at the block's end, turned into the gate gradient as if nothing followed the block, plus
// the block total for the scan.  One read of every input.
template <int M>
__global__ void __launch_bounds__(128) gate_grad_local_kernel(
    const float* u, const float* I, const float* dIk, int nsk,
    const float* dIv, int nsv, const float* gate, int gate_kind, float inv_tau,
    float* __restrict__ blk_tot, float* __restrict__ dgate, int B, int T, int H, int nblk, PendingDecay pend,
    const int* cu, int nseq) {
    follow_previous_grid();
    const int s = 2 * threadIdx.x;                       // this thread's two slots
    const int n = blockIdx.y * blockDim.y + threadIdx.y;
    if (n >= nblk) return;
    const int bh = blockIdx.x, b = bh / H, h = bh % H;
    const int t0 = n * kGG;
    const int rows = min(kGG, T - t0);
    const size_t stride = (size_t)H * M, total = (size_t)B * T * H * M;
    const size_t base = (((size_t)b * T + t0) * H + h) * M + s;
    auto ld2 = [&](const float* p, int i, float fill) {
        return (i < rows) ? *reinterpret_cast<const float2*>(p + base + (size_t)i * stride) : make_float2(fill, fill);
    };
    float2 x[kGG], dI[kGG], gt[kGG];
    load_dI(dIk, nsk, dIv, nsv, base, stride, total, rows, dI);
    if (pend.pending_at(b, t0, h)) {
        // the time-reversed value_side runs left their row factor exp(-G_i) to this kernel
#pragma unroll
        for (int i = 0; i < kGG; ++i) gt[i] = ld2(pend.G, i, 0.f);
#pragma unroll
        for (int i = 0; i < kGG; ++i) { dI[i].x *= pend.reverse_factor(gt[i].x); dI[i].y *= pend.reverse_factor(gt[i].y); }
    }
#pragma unroll
    for (int i = 0; i < kGG; ++i) {
        // (a gate tensor that holds a gives 1 - a as the gate kernel forms it, which may have left it out)
        gt[i] = gate_kind == GSA_GATE_A ? ld2(gate, i, 1.f) : ld2(I, i, 0.f);
        if (gate_kind == GSA_GATE_A) gt[i] = make_float2(1.f - gt[i].x, 1.f - gt[i].y);
    }
#pragma unroll
    for (int i = 0; i < kGG; ++i) x[i] = make_float2(-gt[i].x * dI[i].x, -gt[i].y * dI[i].y);
#pragma unroll
    for (int i = 0; i < kGG; ++i) gt[i] = ld2(u, i, 0.f);
#pragma unroll
    for (int i = 0; i < kGG; ++i) { x[i].x += gt[i].x; x[i].y += gt[i].y; }
#pragma unroll
    for (int i = 0; i < kGG; ++i) gt[i] = ld2(gate, i, 1.f);
    float run0 = 0.f, run1 = 0.f;
    const uint32_t starts = starts_among(cu, nseq, t0, rows);
#pragma unroll
    for (int i = kGG - 1; i >= 0; --i) {
        run0 += x[i].x;
        run1 += x[i].y;
        if ((starts >> i) & 1) run0 = run1 = 0.f;
        if (i < rows) {
            const float2 out = make_float2(gate_grad_out(run0, dI[i].x, gt[i].x, gate_kind, inv_tau),
                                           gate_grad_out(run1, dI[i].y, gt[i].y, gate_kind, inv_tau));
            *reinterpret_cast<float2*>(dgate + base + (size_t)i * stride) = out;
        }
    }
    *reinterpret_cast<float2*>(blk_tot + ((size_t)bh * nblk + n) * M + s) = make_float2(run0, run1);
}

// The same block-local pass with its inputs staged through shared memory by TMA (M = 64): one
// CTA per (b,h) and 32 rows, every tile of every input stream (u, I, gate, G and the n_k + n_v
// slices of the input-gate gradient: 12 x 8 KB at d = 512) requested at once by one thread --
// 96 KB in flight per CTA, two CTAs per SM, several times what registers can hold as landing
// space.  Thread = (slot, 16-row group, early or late half of the group).
constexpr int kGGTmaRows = 32;
constexpr int kGGTmaMaxSlices = 8;
constexpr int kGGTileB = kGGTmaRows * 64 * 4;      // bytes of one [32 x 64] fp32 tile (two swizzled panels)

// A thread's eight rows of a staged tile -- slot tx, 16-row group ty, early (0) or late (1) half hh of it -- and their output.
// The kind of gate is a template argument, every shared-memory address an offset of the row plus a constant of the stream,
// and whole halves are apart from ragged ones: 802 instructions a thread kept the issue slots busy for 47 of 81 us.  With the
// carry kernel treated alike, the gate gradient of B = 4, T = 4096, 32 heads of 128: 231 -> 211 us; B = 8, T = 2048, 4 heads of
// 512: 61 -> 57, with 128 slots 110 -> 96.
constexpr int kGGHalf = kGG / 2;
template <int KIND, bool WIDE> struct GateGradRows {
    float x[kGGHalf], dI[kGGHalf], gt[kGGHalf];       // u - I dI; dI; the gate as passed
    // tiles 0..3 = u, I, gate, G, then the slices of dI; a swizzled panel of 32 slots is half a tile
    __device__ __forceinline__ void read(const unsigned char* tiles, int nslices, int tx, int ty, int hh, bool pending) {
        const unsigned char* row = tiles + (tx >> 5) * (kGGTileB / 2) + (ty * kGG + hh * kGGHalf) * 128 + (tx & 3) * 4;
        const int q = (tx & 31) >> 2;
        int off[kGGHalf];
#pragma unroll
        for (int i = 0; i < kGGHalf; ++i) off[i] = i * 128 + ((q ^ i) << 4);          // (row & 7 == i)
        take([&](int tile, int i) { return *reinterpret_cast<const float*>(row + off[i] + tile * kGGTileB); }, nslices, pending);
    }
    // at(tile, i): row i of a tile
    template <class At> __device__ __forceinline__ void take(At&& at, int nslices, bool pending) {
#pragma unroll
        for (int i = 0; i < kGGHalf; ++i) dI[i] = 0.f;
#pragma unroll
        for (int sl = 0; sl < kGGTmaMaxSlices; ++sl) {
            if (sl >= nslices) break;
#pragma unroll
            for (int i = 0; i < kGGHalf; ++i) dI[i] += at(4 + sl, i);
        }
        if (pending) {
            // the time-reversed value_side runs left their row factor exp(-G_i) to this kernel
#pragma unroll
            for (int i = 0; i < kGGHalf; ++i) {
                const float g = at(3, i);      // (128 slots: exp(G), 0 past the sequence end)
                dI[i] *= WIDE ? (g > 0.f ? 1.f / g : 0.f) : exp_neg(g);
            }
        }
#pragma unroll
        for (int i = 0; i < kGGHalf; ++i) {
            gt[i] = at(2, i);
            const float ii = KIND == GSA_GATE_A ? 1.f - gt[i] : at(1, i);      // 1 - a as the gate kernel formed it
            x[i] = at(0, i) - ii * dI[i];                                      // rows past the end: u = dI = 0
        }
    }
    // sum over the rows, up to the first token that begins a sequence
    __device__ __forceinline__ float total(uint32_t starts) const {
        float tot = 0.f;
        if (starts == 0) {
#pragma unroll
            for (int i = 0; i < kGGHalf; ++i) tot += x[i];
        } else {
#pragma unroll
            for (int i = 0; i < kGGHalf; ++i)
                if ((starts & ((2u << i) - 1)) == 0) tot += x[i];
        }
        return tot;
    }
    // the rows' gradients from the sum `run` of the rows behind them in the group, which becomes theirs too
    __device__ __forceinline__ float write(float run, uint32_t starts, int rows, float* out, uint32_t stride, float inv_tau) const {
        if (starts == 0 && rows >= kGGHalf) {
#pragma unroll
            for (int i = kGGHalf - 1; i >= 0; --i) {
                run += x[i];
                out[i * stride] = gate_grad_out(run, dI[i], gt[i], KIND, inv_tau);
            }
        } else {
#pragma unroll
            for (int i = kGGHalf - 1; i >= 0; --i) {
                run += x[i];
                if ((starts >> i) & 1) run = 0.f;
                if (i < rows) out[i * stride] = gate_grad_out(run, dI[i], gt[i], KIND, inv_tau);
            }
        }
        return run;
    }
};

template <int KIND, bool WIDE>
__global__ void __launch_bounds__(256) gate_grad_local_tma_kernel(
    const __grid_constant__ CUtensorMap mapU, const __grid_constant__ CUtensorMap mapI,
    const __grid_constant__ CUtensorMap mapGate, const __grid_constant__ CUtensorMap mapG,
    const __grid_constant__ CUtensorMap mapDIk, const __grid_constant__ CUtensorMap mapDIv, int nsk, int nsv,
    float inv_tau, float* __restrict__ blk_tot, float* __restrict__ dgate, int T, int H, int nblk,
    PendingDecay pend, const int* cu, int nseq, int32_t* dev_status) {
    follow_previous_grid();
    using namespace tc;
    constexpr int M = 64;
    extern __shared__ unsigned char gg_smem_raw[];
    unsigned char* smem = gg_smem_raw + ((1024u - (smem_u32(gg_smem_raw) & 1023u)) & 1023u);
    __shared__ uint64_t bar;
    __shared__ float late_half[kGGTmaRows / kGG][M];
    // slot, 16-row group, early (0) or late (1) 8 rows of the group
    const int tx = threadIdx.x & 63, ty = (threadIdx.x >> 6) & 1, hh = threadIdx.x >> 7;
    const int bh = blockIdx.x, b = bh / H, h = bh % H;
    const int t0 = blockIdx.y * kGGTmaRows;
    const int nslices = nsk + nsv;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        // tiles 0..3 = u, I, gate, G; I is not read when the gate tensor holds a itself (1 - a is one
        // subtraction), G only when a row factor is pending
        const bool need[4] = {true, KIND != GSA_GATE_A, true, pend.G != nullptr};
        int ntiles = nslices;
        for (int i = 0; i < 4; ++i) ntiles += need[i] ? 1 : 0;
        mbar_expect_tx(&bar, (uint32_t)(ntiles * kGGTileB));
        const CUtensorMap* maps[4] = {&mapU, &mapI, &mapGate, &mapG};
        for (int i = 0; i < 4; ++i) {
            if (!need[i]) continue;
            tma_load_4d(smem + i * kGGTileB, maps[i], &bar, 0, h, t0, b);
            tma_load_4d(smem + i * kGGTileB + kGGTileB / 2, maps[i], &bar, 32, h, t0, b);
        }
        for (int sl = 0; sl < nslices; ++sl) {
            const CUtensorMap* m = sl < nsk ? &mapDIk : &mapDIv;
            const int z = sl < nsk ? sl : sl - nsk;
            tma_load_5d(smem + (4 + sl) * kGGTileB, m, &bar, 0, h, t0, b, z);
            tma_load_5d(smem + (4 + sl) * kGGTileB + kGGTileB / 2, m, &bar, 32, h, t0, b, z);
        }
    }
    __syncthreads();
    const bool landed = mbar_wait(&bar, 0);
    if (!landed && threadIdx.x == 0 && dev_status != nullptr) *dev_status = GSA_ERR_TIMEOUT;
    if (__syncthreads_or(!landed)) return;

    const int n = blockIdx.y * (kGGTmaRows / kGG) + ty;           // 16-row block of the sequence
    const int rows = n < nblk ? T - n * kGG - hh * kGGHalf : 0;   // ... from this thread's first row on
    GateGradRows<KIND, WIDE> r;
    r.read(smem, nslices, tx, ty, hh, pend.pending_at(b, t0, h));
    // the early half starts from the total of the late half of its group
    const uint32_t starts = starts_among(cu, nseq, n * kGG + hh * kGGHalf, kGGHalf);
    if (hh == 1) late_half[ty][tx] = r.total(starts);
    __syncthreads();
    float* out = dgate + (((size_t)b * T + t0 + ty * kGG + hh * kGGHalf) * H + h) * M + tx;
    const float run = r.write(hh == 0 ? late_half[ty][tx] : 0.f, starts, rows, out, (uint32_t)H * M, inv_tau);
    if (hh == 0 && n < nblk) blk_tot[((size_t)bh * nblk + n) * M + tx] = run;
}

// The TMA-staged pass as a ring, for wide heads (n_k + n_v >= 6: a CTA per tile then keeps
// only two tiles per SM in flight and the copies pause while it computes, leaves and the next
// one starts).  A tile is 32 rows of one (b,h) with every input stream (u, I, gate, G and the n_k + n_v slices of the
// input-gate gradient: 12 x 8 KB at d = 512).  One persistent CTA per SM walks the tiles
// blockIdx.x, blockIdx.x + gridDim.x, ... through a ring of 2-4 stages: a ninth warp requests the
// tiles of the stages ahead while the eight compute warps work on the current one, so copies
// are in flight all the time.  Compute thread = (slot, 16-row group, early or late half of it).
constexpr int kGGMaxStages = 4;
constexpr int kGGRingMinSlices = 6;
constexpr int kGGComputeThreads = 256;

template <int KIND, bool WIDE>
__global__ void __launch_bounds__(kGGComputeThreads + 32) gate_grad_local_ring_kernel(
    const __grid_constant__ CUtensorMap mapU, const __grid_constant__ CUtensorMap mapI,
    const __grid_constant__ CUtensorMap mapGate, const __grid_constant__ CUtensorMap mapG,
    const __grid_constant__ CUtensorMap mapDIk, const __grid_constant__ CUtensorMap mapDIv, int nsk, int nsv,
    float inv_tau, float* __restrict__ blk_tot, float* __restrict__ dgate, int T, int H, int BH,
    int ntile, int nstage, int nblk, PendingDecay pend, const int* cu, int nseq, int32_t* dev_status) {
    follow_previous_grid();
    using namespace tc;
    constexpr int M = 64;
    extern __shared__ unsigned char gg_smem_raw[];
    unsigned char* smem0 = gg_smem_raw + ((1024u - (smem_u32(gg_smem_raw) & 1023u)) & 1023u);
    __shared__ uint64_t bar_full[kGGMaxStages], bar_empty[kGGMaxStages];
    __shared__ float late_half[kGGTmaRows / kGG][M];
    __shared__ volatile int failed_s, stop_s;
    const int nslices = nsk + nsv;
    const int stage_bytes = (4 + nslices) * kGGTileB;
    const int total = BH * ntile;
    if (threadIdx.x == 0) {
        failed_s = 0;
        for (int s = 0; s < nstage; ++s) {
            mbar_init(&bar_full[s], 1);
            mbar_init(&bar_empty[s], 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();

    if (threadIdx.x == kGGComputeThreads) {
        // =============================== copy lane
        // tiles 0..3 = u, I, gate, G; I is not read when the gate tensor holds a itself (1 - a is one
        // subtraction), G only when a row factor is pending
        const bool need[4] = {true, KIND != GSA_GATE_A, true, pend.G != nullptr};
        int ntiles = nslices;
        for (int i = 0; i < 4; ++i) ntiles += need[i] ? 1 : 0;
        const CUtensorMap* maps[4] = {&mapU, &mapI, &mapGate, &mapG};
        int it = 0;
        for (int t = blockIdx.x; t < total; t += gridDim.x, ++it) {
            const int s = it % nstage;
            if (it >= nstage && !mbar_wait(&bar_empty[s], ((it / nstage) - 1) & 1)) {
                failed_s = 1;
                break;
            }
            const int bh = t % BH, b = bh / H, h = bh % H, t0 = (t / BH) * kGGTmaRows;
            unsigned char* smem = smem0 + (size_t)s * stage_bytes;
            mbar_expect_tx(&bar_full[s], (uint32_t)(ntiles * kGGTileB));
            for (int i = 0; i < 4; ++i) {
                if (!need[i]) continue;
                tma_load_4d(smem + i * kGGTileB, maps[i], &bar_full[s], 0, h, t0, b);
                tma_load_4d(smem + i * kGGTileB + kGGTileB / 2, maps[i], &bar_full[s], 32, h, t0, b);
            }
            for (int sl = 0; sl < nslices; ++sl) {
                const CUtensorMap* m = sl < nsk ? &mapDIk : &mapDIv;
                const int z = sl < nsk ? sl : sl - nsk;
                tma_load_5d(smem + (4 + sl) * kGGTileB, m, &bar_full[s], 0, h, t0, b, z);
                tma_load_5d(smem + (4 + sl) * kGGTileB + kGGTileB / 2, m, &bar_full[s], 32, h, t0, b, z);
            }
        }
    } else if (threadIdx.x < kGGComputeThreads) {
        // =============================== compute warps
        // slot, 16-row group, early (0) or late (1) 8 rows of the group
        const int tx = threadIdx.x & 63, ty = (threadIdx.x >> 6) & 1, hh = threadIdx.x >> 7;
        auto csync = [] { asm volatile("bar.sync 1, 256;" ::: "memory"); };
        int it = 0;
        for (int t = blockIdx.x; t < total; t += gridDim.x, ++it) {
            const int s = it % nstage;
            const int bh = t % BH, b = bh / H, h = bh % H, ty0 = t / BH, t0 = ty0 * kGGTmaRows;
            const unsigned char* smem = smem0 + (size_t)s * stage_bytes;
            if (!mbar_wait(&bar_full[s], (it / nstage) & 1)) failed_s = 1;     // (what is read then means nothing)
            const int n = ty0 * (kGGTmaRows / kGG) + ty;           // 16-row block of the sequence
            const int rows = n < nblk ? T - n * kGG - hh * kGGHalf : 0;
            GateGradRows<KIND, WIDE> r;
            r.read(smem, nslices, tx, ty, hh, pend.pending_at(b, t0, h));
            // the early half starts from the total of the late half of its group
            const uint32_t starts = starts_among(cu, nseq, n * kGG + hh * kGGHalf, kGGHalf);
            if (hh == 1) late_half[ty][tx] = r.total(starts);
            csync();                              // (also: every thread has read its part of the stage)
            if (threadIdx.x == 0)
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&bar_empty[s])) : "memory");
            float* out = dgate + (((size_t)b * T + t0 + ty * kGG + hh * kGGHalf) * H + h) * M + tx;
            const float run = r.write(hh == 0 ? late_half[ty][tx] : 0.f, starts, rows, out, (uint32_t)H * M, inv_tau);
            if (hh == 0 && n < nblk) blk_tot[((size_t)bh * nblk + n) * M + tx] = run;
            // (one thread reads the flag that the copy lane may raise at any time, so that all leave together)
            if (threadIdx.x == 0) stop_s = failed_s;
            csync();                              // late_half may be rewritten
            if (stop_s) break;
        }
    }
    __syncthreads();
    if (failed_s) {
        if (threadIdx.x == 0 && dev_status != nullptr) *dev_status = GSA_ERR_TIMEOUT;
        // bounded grace period for tile copies still in flight before shared memory goes away
        for (int i = 0; i < 200; ++i) __nanosleep(1000);
    }
}

// The whole gradient in one pass, where (batch, head) pairs are enough: a CTA takes a pair, or a half or a quarter of its slots,
// and walks its tiles from the last to the first, the running sum carried along -- a thread keeps its slot's in fp64 -- so that
// nothing is written twice and no sums of blocks are scanned (3 of 9 streams at one slice a side).  Thread = (slot, group of eight
// rows); a tile is as many rows as the threads have groups; a warp of one active lane copies the tiles of the stages ahead.
// Bound by a tile's chain -- copies seen, eight rows of every stream, two barriers around the scan of the groups' sums by
// shuffles (summed thread by thread it was half of the chain at 32 groups), rows out -- and by HBM where 128 CTAs walk all slots:
// B = 4, T = 4096, 32 heads of 128 (0.8 GB) 212 -> 146 us, 5.5 TB/s; B = 8, T = 2048, 4 heads of 512 59 -> 47.5, with 128 slots
// 98 -> 80.  512 threads, 16 KB a tile, where the slices of dI are few (256: 207); the next tile read ahead of the scan: 144 / 49.5.
template <int KIND, bool WIDE, int NT>
__global__ void __launch_bounds__(NT + 32) gate_grad_walk_kernel(
    const __grid_constant__ CUtensorMap mapU, const __grid_constant__ CUtensorMap mapI,
    const __grid_constant__ CUtensorMap mapGate, const __grid_constant__ CUtensorMap mapG,
    const __grid_constant__ CUtensorMap mapDIk, const __grid_constant__ CUtensorMap mapDIv, int nsk, int nsv,
    float inv_tau, float* __restrict__ dgate, int T, int H, int log_slots, int nstage, const float* dKT, const float* KT,
    const float* dVT, const float* VT, int d_k, int d_v, PendingDecay pend, const int* cu, int nseq, int32_t* dev_status) {
    follow_previous_grid();
    using namespace tc;
    constexpr int M = 64, kTile = NT * kGGHalf;          // elements of a tile
    extern __shared__ unsigned char gg_smem_raw[];
    unsigned char* smem0 = gg_smem_raw + ((128u - (smem_u32(gg_smem_raw) & 127u)) & 127u);
    __shared__ uint64_t bar_full[kGGMaxStages], bar_empty[kGGMaxStages];
    __shared__ float totals[NT + NT / 16], before[NT + NT / 16];      // [group][slot], rows one word longer than the slots
    __shared__ int restarts[NT / 16];                    // does a packed sequence begin in the group?
    __shared__ double final_term[M];
    __shared__ volatile int failed_s;
    const int slots = 1 << log_slots, groups = NT >> log_slots, tile_rows = groups * kGGHalf;
    const int bh = blockIdx.x, b = bh / H, h = bh % H, s0 = blockIdx.y << log_slots;
    const int ntile = (T + tile_rows - 1) / tile_rows;
    // tiles: u, gate, G where a row factor is pending, the slices of dI, 1 - a unless the gate tensor gives it
    const bool factor = pend.G != nullptr;
    const int nslices = nsk + nsv, first_slice = factor ? 3 : 2, ntiles = first_slice + nslices + (KIND != GSA_GATE_A ? 1 : 0);
    if (threadIdx.x == 0) {
        failed_s = 0;
        for (int s = 0; s < nstage; ++s) {
            mbar_init(&bar_full[s], 1);
            mbar_init(&bar_empty[s], NT / 32);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x >= NT) {
        if (elect_one()) {
            // =============================== copy lane
            for (int it = 0; it < ntile; ++it) {
                const int s = it % nstage, t0 = (ntile - 1 - it) * tile_rows;
                if (it >= nstage && !mbar_wait(&bar_empty[s], ((it / nstage) - 1) & 1)) {
                    failed_s = 1;
                    break;
                }
                unsigned char* smem = smem0 + (size_t)s * ntiles * (kTile * 4);
                uint64_t* bar = &bar_full[s];
                mbar_expect_tx(bar, (uint32_t)(ntiles * kTile * 4));
                auto tile = [&](int i) { return smem + i * (kTile * 4); };
                tma_load_4d(tile(0), &mapU, bar, s0, h, t0, b);
                tma_load_4d(tile(1), &mapGate, bar, s0, h, t0, b);
                if (factor) tma_load_4d(tile(2), &mapG, bar, s0, h, t0, b);
                for (int sl = 0; sl < nslices; ++sl)
                    tma_load_5d(tile(first_slice + sl), sl < nsk ? &mapDIk : &mapDIv, bar, s0, h, t0, b, sl < nsk ? sl : sl - nsk);
                if (KIND != GSA_GATE_A) tma_load_4d(tile(ntiles - 1), &mapI, bar, s0, h, t0, b);
            }
        }
    } else {
        // =============================== compute warps
        const int tx = threadIdx.x & (slots - 1), grp = threadIdx.x >> log_slots, mine = grp * (slots + 1) + tx;
        // the groups' sums are scanned by as many lanes to a slot, the last group first: this thread's place there
        const int rank = threadIdx.x & (groups - 1), scanned = (groups - 1 - rank) * (slots + 1) + threadIdx.x / groups;
        auto csync = [] { asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory"); };
        double carry = 0.0;
        if (dKT != nullptr || dVT != nullptr) {
            // final-memory term <dK~_T[s], K~_T[s]> + <dV~_T[s], V~_T[s]>: a warp per slot, lanes along the row
            const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
            for (int slot = warp; slot < slots; slot += NT / 32) {
                double dot = 0.0;
                const size_t row = (size_t)bh * M + s0 + slot;
                if (dKT != nullptr)
                    for (int c = lane; c < d_k; c += 32) dot += (double)dKT[row * d_k + c] * (double)KT[row * d_k + c];
                if (dVT != nullptr)
                    for (int c = lane; c < d_v; c += 32) dot += (double)dVT[row * d_v + c] * (double)VT[row * d_v + c];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
                if (lane == 0) final_term[slot] = dot;
            }
            csync();
            carry = final_term[threadIdx.x / groups];
        }
        for (int it = 0; it < ntile; ++it) {
            const int s = it % nstage, t0 = (ntile - 1 - it) * tile_rows, row0 = t0 + grp * kGGHalf;
            const unsigned char* smem = smem0 + (size_t)s * ntiles * (kTile * 4) + (size_t)((grp * kGGHalf << log_slots) + tx) * 4;
            if (!failed_s && !mbar_wait(&bar_full[s], (it / nstage) & 1)) failed_s = 1;     // (what is read then means nothing)
            GateGradRows<KIND, WIDE> r;
            // (in the order that GateGradRows names them: u, 1 - a, the gate, G, the slices)
            const int place[4] = {0, ntiles - 1, 1, 2};
            // (asked for this thread's eight rows, which lie in one chunk: a tile of 256 may span two segments, a flagged one and
            // another)
            const bool pending = pend.pending_at(b, min(row0, T - 1), h);
            r.take([&](int tile, int i) {
                return *reinterpret_cast<const float*>(smem + (tile < 4 ? place[tile] : first_slice + tile - 4) * (kTile * 4) + ((i * 4) << log_slots));
            }, nslices, pending);
            __syncwarp();
            if ((threadIdx.x & 31) == 0)
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&bar_empty[s])) : "memory");
            const uint32_t starts = starts_among(cu, nseq, row0, kGGHalf);
            totals[mine] = r.total(starts);
            if (cu != nullptr && tx == 0) restarts[grp] = starts != 0;
            csync();
            // a group passes on what it gets and its own sum; if a sequence begins in it, its own sum alone
            double sum = (double)totals[scanned];
            int restart = cu != nullptr ? restarts[groups - 1 - rank] : 0;
            for (int o = 1; o < groups; o <<= 1) {
                const double later = __shfl_up_sync(0xffffffffu, sum, o, groups);
                const int later_restart = cu != nullptr ? __shfl_up_sync(0xffffffffu, restart, o, groups) : 0;
                if (rank >= o) {
                    if (restart == 0) sum += later;
                    restart |= later_restart;
                }
            }
            const double passed = (restart != 0 ? 0.0 : carry) + sum, got = __shfl_up_sync(0xffffffffu, passed, 1, groups);
            before[scanned] = (float)(rank == 0 ? carry : got);
            carry = __shfl_sync(0xffffffffu, passed, groups - 1, groups);
            csync();
            float* out = dgate + (((size_t)b * T + row0) * H + h) * M + s0 + tx;
            r.write(before[mine], starts, T - row0, out, (uint32_t)H * M, inv_tau);
        }
    }
    __syncthreads();
    if (failed_s) {
        if (threadIdx.x == 0 && dev_status != nullptr) *dev_status = GSA_ERR_TIMEOUT;
        // bounded grace period for tile copies still in flight before shared memory goes away
        for (int i = 0; i < 200; ++i) __nanosleep(1000);
    }
}

// Adds what follows the block: dgate += carry (log gate) or carry / a (linear gate).  A thread
// takes two slots of eight rows (half a block): threadIdx = (slot pair, block, half).
template <int M, int KIND>
__global__ void __launch_bounds__(256) gate_grad_carry_kernel(
    const float* gate, float inv_tau, const float* blk_carry,
    float* dgate, int T, int H, int nblk, const int* cu, int nseq) {
    follow_previous_grid();
    constexpr int kRows = kGG / 2;
    const int s = 2 * threadIdx.x;
    const int n = blockIdx.y * blockDim.y + threadIdx.y;
    if (n >= nblk) return;
    const int bh = blockIdx.x, b = bh / H, h = bh % H;
    // (a thread's first element, and 32-bit offsets from there)
    const int t0 = n * kGG + threadIdx.z * kRows;
    const size_t first = (((size_t)b * T + t0) * H + h) * M + s;
    const uint32_t stride = (uint32_t)H * M;
    const int rows = T - t0;
    // (what follows the block reaches the rows after its last token that begins a sequence)
    const int from = cu == nullptr ? 0 : 32 - __clz(starts_among(cu, nseq, n * kGG, min(kGG, T - n * kGG))) - (int)threadIdx.z * kRows;
    const float2 carry = *reinterpret_cast<const float2*>(blk_carry + ((size_t)bh * nblk + n) * M + s);
    float* out = dgate + first;
    const float* in = gate + first;
    auto load = [&](const float* p, int i) { return *reinterpret_cast<const float2*>(p + i * stride); };
    auto add = [&](int i, float2 d, float2 gt) {
        *reinterpret_cast<float2*>(out + i * stride) =
            make_float2(d.x + gate_grad_carry(carry.x, gt.x, KIND, inv_tau), d.y + gate_grad_carry(carry.y, gt.y, KIND, inv_tau));
    };
    const float2 unused = make_float2(1.f, 1.f);           // (log gates: the carry goes as it is)
    if (rows >= kRows && from <= 0) {
        float2 d[kRows], gt[kRows];
#pragma unroll
        for (int i = 0; i < kRows; ++i) {
            d[i] = load(out, i);
            gt[i] = KIND != GSA_GATE_LOG_A ? load(in, i) : unused;
        }
#pragma unroll
        for (int i = 0; i < kRows; ++i) add(i, d[i], gt[i]);
        return;
    }
    for (int i = max(from, 0); i < min(rows, kRows); ++i) add(i, load(out, i), KIND != GSA_GATE_LOG_A ? load(in, i) : unused);
}
template <int M, class... A>
void launch_gate_carry(int gate_kind, dim3 grid, dim3 block, cudaStream_t st, const float* gate, A... rest) {
    if (gate_kind == GSA_GATE_A) launch_after(gate_grad_carry_kernel<M, GSA_GATE_A>, grid, block, 0, st, gate, rest...);
    else if (gate_kind == GSA_GATE_LOG_A) launch_after(gate_grad_carry_kernel<M, GSA_GATE_LOG_A>, grid, block, 0, st, gate, rest...);
    else launch_after(gate_grad_carry_kernel<M, GSA_GATE_LOGITS>, grid, block, 0, st, gate, rest...);
}
// f(kind, wide) with both as types
template <class F>
cudaError_t with_gate_kind(int gate_kind, int wide, F&& f) {
    auto kind = [&](auto w) {
        if (gate_kind == GSA_GATE_A) return f(std::integral_constant<int, GSA_GATE_A>{}, w);
        if (gate_kind == GSA_GATE_LOG_A) return f(std::integral_constant<int, GSA_GATE_LOG_A>{}, w);
        return f(std::integral_constant<int, GSA_GATE_LOGITS>{}, w);
    };
    return wide ? kind(std::true_type{}) : kind(std::false_type{});
}

int gate_grad_blocks(int T) { return (T + kGG - 1) / kGG; }

// Does the gradient walk, and with how many slots to a CTA (as a power of two; 0: it takes the three kernels)?  A wave of walks
// takes the same time however many SMs it fills; at a half and a quarter of the slots 0.57 and 0.39 of it.  The three kernels
// take a 95th of it for a pair, and 0.12.  us at 2048 tokens, the three kernels / 16 / 32 / 64 slots: 20 pairs
// (four slices a side) 44 / 44 / 66 / 120, logits 47 / 52 / 82 / 150, 28: 53 / 46 / 66 / 121, 40: 71 / 84 / 68 / 121, logits 75 / 97 /
// 82 / 152, 72: 108 / 97 / 86 / 138; (one) 28: 36 / 31 / 46 / 80, 48: 53 / 56 / 47 / 80, 80: 75 / 76 / 80 / 76, 112: 100 / 117 / 82 / 78,
// 160: 133 / 168 / 119 / 148, logits 151 / 199 / 156 / 195, 256: 219 / 256 / 160 / 152.  From 16 tokens to 8192 it holds, the walk being
// ahead by its two launches less at short lengths, but for logits, whose walk takes more to a row: at 8192 tokens, one slice,
// 48 pairs 184 / 234 / 207 / 394, 96: 357 / 408 / 395 / 399, four slices, 28 pairs 174 / 185 / 342 / 590.
constexpr int kWalkWideSlices = 3, kWalkSmem = 200 << 10;
int walk_slots(int pairs, int nslices, int gate_kind, int T) {
    if (nslices > kGGTmaMaxSlices) return 0;
    const float wave[3] = {0.39f, 0.57f, 1.f}, more = gate_kind == GSA_GATE_LOGITS && T > 3072 ? 1.09f : 1.f;
    float best = 0.95f * ((float)pairs / 95.f + 0.12f);
    int log_slots = 0;
    for (int i = 0; i < 3; ++i) {
        const float cost = more * wave[i] * (float)((((long long)pairs << (2 - i)) + kSMs - 1) / kSMs);
        if (cost < best) { best = cost; log_slots = 4 + i; }
    }
    return log_slots;
}

int gate_grad_kernels(int pairs, int M, bool wide, int nslices, int gate_kind, int T) {
    if (!wide && M != 64) return 3;
    return walk_slots(wide ? 2 * pairs : pairs, nslices, gate_kind, T) != 0 ? 1 : 3;
}

cudaError_t launch_gate_grad(const float* u, const float* I, const float* dIk_part, int nsk,
                             const float* dIv_part, int nsv, const float* gate,
                             int gate_kind, float inv_tau, const float* dKT, const float* KT,
                             const float* dVT, const float* VT, int d_k, int d_v,
                             float* blk_tot, float* dgate, int B, int T, int H, int M,
                             PendingDecay pend, cudaStream_t st, int32_t* dev_status, const int* cu_seqlens, int nseq) {
    if (pend.wide && M == 128) {       // as 2 H heads of 64 slots: the kernels that stage their tiles
        pend.half_heads = 1;
        pend.H = 2 * H;
        return launch_gate_grad(u, I, dIk_part, nsk, dIv_part, nsv, gate, gate_kind, inv_tau, dKT, KT, dVT, VT, d_k, d_v, blk_tot,
                                dgate, B, T, 2 * H, 64, pend, st, dev_status, cu_seqlens, nseq);
    }
    if (gate_grad_kernels(B * H, M, false, nsk + nsv, gate_kind, T) == 1) {
        const int log_slots = walk_slots(B * H, nsk + nsv, gate_kind, T);
        const int BH = B * H, nsl = nsk + nsv, cols = 1 << log_slots;
        return with_gate_kind(gate_kind, pend.wide, [&](auto kind, auto wide) {
            auto launch = [&](auto threads) {
                constexpr int NT = decltype(threads)::value;
                constexpr auto kernel = gate_grad_walk_kernel<decltype(kind)::value, decltype(wide)::value, NT>;
                const int rows = NT / cols * kGGHalf;
                const int ntiles = 2 + (pend.G != nullptr) + nsl + (gate_kind != GSA_GATE_A);
                const int stage_bytes = ntiles * NT * kGGHalf * 4;
                int nstage = (kWalkSmem - 128) / stage_bytes;
                if (nstage > kGGMaxStages) nstage = kGGMaxStages;
                CUtensorMap mu, mi, mg, mG, mk, mv;
                const float* Gp = pend.G != nullptr ? pend.G : u;      // (unused without a pending factor)
                cudaError_t e = make_tensor_map_sliced(&mu, u, 0, B, T, H, M, rows, 4, cols);
                if (e == cudaSuccess) e = make_tensor_map_sliced(&mi, I, 0, B, T, H, M, rows, 4, cols);
                if (e == cudaSuccess) e = make_tensor_map_sliced(&mg, gate, 0, B, T, H, M, rows, 4, cols);
                if (e == cudaSuccess) e = make_tensor_map_sliced(&mG, Gp, 0, B, T, H, M, rows, 4, cols);
                if (e == cudaSuccess) e = make_tensor_map_sliced(&mk, dIk_part, nsk, B, T, H, M, rows, 4, cols);
                if (e == cudaSuccess) e = make_tensor_map_sliced(&mv, dIv_part, nsv, B, T, H, M, rows, 4, cols);
                const size_t smem = 128 + (size_t)nstage * stage_bytes;
                if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kWalkSmem);
                if (e != cudaSuccess) return e;
                return launch_after(gate_grad_walk_kernel<decltype(kind)::value, decltype(wide)::value, NT>, dim3(BH, M >> log_slots), NT + 32, smem, st, mu, mi, mg, mG, mk, mv, nsk, nsv,
                                    inv_tau, dgate, T, H, log_slots, nstage, dKT, KT, dVT, VT, d_k, d_v, pend, cu_seqlens, nseq, dev_status);
            };
            // (wide heads: 96 KB of tiles a stage as it is)
            if (nsl > kWalkWideSlices) return launch(std::integral_constant<int, 256>{});
            return launch(std::integral_constant<int, 512>{});
        });
    }
    const int nblk = gate_grad_blocks(T);
    dim3 block(M / 2, 256 / M);      // 128 threads: M/2 slot pairs x 16-row blocks
    dim3 grid(B * H, (nblk + block.y - 1) / block.y);
    if (M == 64) {
        const int nsl = nsk + nsv;
        bool staged = nsl <= kGGTmaMaxSlices;
        CUtensorMap mu, mi, mg, mG, mk, mv;
        if (staged) {
            const float* Gp = pend.G != nullptr ? pend.G : u;      // (unused without a pending factor)
            cudaError_t e = make_tensor_map_bthd(&mu, u, B, T, H, M, kGGTmaRows, 4);
            if (e == cudaSuccess) e = make_tensor_map_bthd(&mi, I, B, T, H, M, kGGTmaRows, 4);
            if (e == cudaSuccess) e = make_tensor_map_bthd(&mg, gate, B, T, H, M, kGGTmaRows, 4);
            if (e == cudaSuccess) e = make_tensor_map_bthd(&mG, Gp, B, T, H, M, kGGTmaRows, 4);
            if (e == cudaSuccess) e = make_tensor_map_sliced(&mk, dIk_part, nsk, B, T, H, M, kGGTmaRows, 4);
            if (e == cudaSuccess) e = make_tensor_map_sliced(&mv, dIv_part, nsv, B, T, H, M, kGGTmaRows, 4);
            staged = e == cudaSuccess;
        }
        if (staged && nsl >= kGGRingMinSlices) {
            const int stage_bytes = (4 + nsl) * kGGTileB;
            const int nstage = 2;
            const size_t smem = 1024 + (size_t)nstage * stage_bytes;
            static int sm_count = 0;
            if (sm_count == 0) {
                int dev = 0;
                if (cudaGetDevice(&dev) != cudaSuccess ||
                    cudaDeviceGetAttribute(&sm_count, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sm_count <= 0)
                    return cudaErrorUnknown;
            }
            const int BH = B * H, ntile = (T + kGGTmaRows - 1) / kGGTmaRows;
            const long long total = (long long)BH * ntile;
            const int ctas = (int)(total < sm_count ? total : sm_count);      // one persistent CTA per SM
            const cudaError_t e = with_gate_kind(gate_kind, pend.wide, [&](auto k, auto w) {
                constexpr auto kernel = gate_grad_local_ring_kernel<decltype(k)::value, decltype(w)::value>;
                const cudaError_t ready = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
                if (ready != cudaSuccess) return ready;
                return launch_after(gate_grad_local_ring_kernel<decltype(k)::value, decltype(w)::value>, ctas, kGGComputeThreads + 32, smem, st, mu, mi, mg, mG, mk, mv, nsk, nsv, inv_tau, blk_tot, dgate,
                                    T, H, BH, ntile, nstage, nblk, pend, cu_seqlens, nseq, dev_status);
            });
            if (e != cudaSuccess) return e;
        } else if (staged) {
            const size_t smem = 1024 + (size_t)(4 + nsl) * kGGTileB;
            dim3 tgrid(B * H, (T + kGGTmaRows - 1) / kGGTmaRows);
            const cudaError_t e = with_gate_kind(gate_kind, pend.wide, [&](auto k, auto w) {
                constexpr auto kernel = gate_grad_local_tma_kernel<decltype(k)::value, decltype(w)::value>;
                const cudaError_t ready = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
                if (ready != cudaSuccess) return ready;
                return launch_after(gate_grad_local_tma_kernel<decltype(k)::value, decltype(w)::value>, tgrid, 256, smem, st, mu, mi, mg, mG, mk, mv, nsk, nsv, inv_tau, blk_tot, dgate, T, H, nblk, pend,
                                    cu_seqlens, nseq, dev_status);
            });
            if (e != cudaSuccess) return e;
        } else {
            launch_after(gate_grad_local_kernel<64>, grid, block, 0, st, u, I, dIk_part, nsk, dIv_part, nsv, gate, gate_kind, inv_tau,
                                                               blk_tot, dgate, B, T, H, nblk, pend, cu_seqlens, nseq);
        }
        launch_after(gate_grad_scan_kernel<64>, B * H, dim3(64, 16), 0, st, blk_tot, dKT, KT, dVT, VT, d_k, d_v, nblk, T, cu_seqlens, nseq);
        launch_gate_carry<64>(gate_kind, grid, dim3(block.x, block.y, 2), st, gate, inv_tau, blk_tot, dgate, T, H, nblk, cu_seqlens, nseq);
    } else if (M == 128) {
        launch_after(gate_grad_local_kernel<128>, grid, block, 0, st, u, I, dIk_part, nsk, dIv_part, nsv, gate, gate_kind, inv_tau,
                                                            blk_tot, dgate, B, T, H, nblk, pend, cu_seqlens, nseq);
        launch_after(gate_grad_scan_kernel<128>, B * H, dim3(128, 8), 0, st, blk_tot, dKT, KT, dVT, VT, d_k, d_v, nblk, T, cu_seqlens, nseq);
        launch_gate_carry<128>(gate_kind, grid, dim3(block.x, block.y, 2), st, gate, inv_tau, blk_tot, dgate, T, H, nblk, cu_seqlens, nseq);
    } else {
        launch_after(gate_grad_local_kernel<32>, grid, block, 0, st, u, I, dIk_part, nsk, dIv_part, nsv, gate, gate_kind, inv_tau,
                                                           blk_tot, dgate, B, T, H, nblk, pend, cu_seqlens, nseq);
        launch_after(gate_grad_scan_kernel<32>, B * H, dim3(32, 16), 0, st, blk_tot, dKT, KT, dVT, VT, d_k, d_v, nblk, T, cu_seqlens, nseq);
        launch_gate_carry<32>(gate_kind, grid, dim3(block.x, block.y, 2), st, gate, inv_tau, blk_tot, dgate, T, H, nblk, cu_seqlens, nseq);
    }
    return cudaGetLastError();
}

// ------------------------------------------------------------------ ABC: no decay, cumulative-softmax write weights
// Eq. 3-4 (the ungated ancestor of GSA, the "no decay" row of the ablations): the memories only
// accumulate, K~_t = K~_{t-1} + phi_t (x) k_t, with write weights phi_t = exp(s_t) / sum_{j<=t} exp(s_j)
// per slot.  In the layer's terms: log a = 0 everywhere and the input gate is phi.  The cumulative
// softmax over time is a scan per (batch, head, slot): one thread each, the rows of eight time steps
// requested together so that the loads overlap; running maximum and rescaled running sum as in any
// streaming softmax.  The decayed bf16 rows of the tensor-core kernels are phi itself (exp(-G) = 1).
constexpr int kAbcBatch = 8;

template <int M>
__global__ void __launch_bounds__(M) abc_write_kernel(const float* s_in, float* __restrict__ G,
                                                      float* __restrict__ I, __nv_bfloat16* __restrict__ decayed, int T,
                                                      int H) {
    follow_previous_grid();
    const int bh = blockIdx.x, b = bh / H, h = bh % H, s = threadIdx.x;
    const size_t stride = (size_t)H * M;
    size_t idx = ((size_t)b * T * H + h) * M + s;
    float mx = -INFINITY, z = 0.f;
    for (int t0 = 0; t0 < T; t0 += kAbcBatch) {
        float x[kAbcBatch];
#pragma unroll
        for (int i = 0; i < kAbcBatch; ++i) x[i] = (t0 + i < T) ? s_in[idx + (size_t)i * stride] : 0.f;
#pragma unroll
        for (int i = 0; i < kAbcBatch; ++i) {
            if (t0 + i >= T) break;
            const float nm = fmaxf(mx, x[i]);
            const float e = __expf(x[i] - nm);
            z = z * __expf(mx - nm) + e;
            mx = nm;
            const float phi = e / z;
            const size_t at = idx + (size_t)i * stride;
            G[at] = 0.f;
            I[at] = phi;
            if (decayed != nullptr) {
                const __nv_bfloat16 hi = __float2bfloat16_rn(phi);
                __nv_bfloat16* row = decayed + 2 * (at - s);
                row[s] = hi;
                row[M + s] = __float2bfloat16_rn(phi - __bfloat162float(hi));
            }
        }
        idx += (size_t)kAbcBatch * stride;
    }
}

// Gradient w.r.t. the scores: with dphi_t the gradient w.r.t. the write weights (the sum of the input-gate
// gradient partial sums of both passes),
//     ds_j = phi_j (dphi_j - R_j),   R_j = dphi_j phi_j + (1 - phi_{j+1}) R_{j+1}
// (Z_j / Z_t = prod_{r=j+1..t} (1 - phi_r): nothing but phi is needed).  A reverse scan, same thread layout.
template <int M>
__global__ void __launch_bounds__(M) abc_grad_kernel(const float* phi_in, const float* dIk, int nsk,
                                                     const float* dIv, int nsv, float* __restrict__ ds, int T,
                                                     int H, size_t total) {
    follow_previous_grid();
    const int bh = blockIdx.x, b = bh / H, h = bh % H, s = threadIdx.x;
    const size_t stride = (size_t)H * M;
    const size_t base = ((size_t)b * T * H + h) * M + s;
    float R = 0.f, phi_next = 0.f;          // (1 - phi_{T}) R_{T} = 0
    for (int t1 = T; t1 > 0; t1 -= kAbcBatch) {
        float phi[kAbcBatch], dphi[kAbcBatch];
#pragma unroll
        for (int i = 0; i < kAbcBatch; ++i) {
            const int t = t1 - 1 - i;
            phi[i] = 0.f; dphi[i] = 0.f;
            if (t >= 0) {
                const size_t at = base + (size_t)t * stride;
                phi[i] = phi_in[at];
                for (int sl = 0; sl < nsk; ++sl) dphi[i] += dIk[at + (size_t)sl * total];
                for (int sl = 0; sl < nsv; ++sl) dphi[i] += dIv[at + (size_t)sl * total];
            }
        }
#pragma unroll
        for (int i = 0; i < kAbcBatch; ++i) {
            const int t = t1 - 1 - i;
            if (t < 0) break;
            R = dphi[i] * phi[i] + (1.f - phi_next) * R;
            ds[base + (size_t)t * stride] = phi[i] * (dphi[i] - R);
            phi_next = phi[i];
        }
    }
}

cudaError_t launch_abc_write(const float* s_in, float* G, float* I, void* decayed, int B, int T, int H, int M, cudaStream_t st) {
    if (M == 128) launch_after(abc_write_kernel<128>, B * H, 128, 0, st, s_in, G, I, static_cast<__nv_bfloat16*>(decayed), T, H);
    else if (M == 64) launch_after(abc_write_kernel<64>, B * H, 64, 0, st, s_in, G, I, static_cast<__nv_bfloat16*>(decayed), T, H);
    else launch_after(abc_write_kernel<32>, B * H, 32, 0, st, s_in, G, I, static_cast<__nv_bfloat16*>(decayed), T, H);
    return cudaGetLastError();
}
cudaError_t launch_abc_grad(const float* phi, const float* dIk, int nsk, const float* dIv, int nsv, float* ds, int B, int T,
                            int H, int M, cudaStream_t st) {
    const size_t total = (size_t)B * T * H * M;
    if (M == 128) launch_after(abc_grad_kernel<128>, B * H, 128, 0, st, phi, dIk, nsk, dIv, nsv, ds, T, H, total);
    else if (M == 64) launch_after(abc_grad_kernel<64>, B * H, 64, 0, st, phi, dIk, nsk, dIv, nsv, ds, T, H, total);
    else launch_after(abc_grad_kernel<32>, B * H, 32, 0, st, phi, dIk, nsk, dIv, nsv, ds, T, H, total);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ data-independent decay
// A gate that does not depend on the input (the "data-independent decay" row of the ablations) is one
// row [H, M] for all tokens: it is spread over [B,T,H,M] on the way in, and the gate gradient is
// summed over the tokens on the way out (partial sums per block of rows, added in order).
__global__ void broadcast_rows_kernel(const float* row, float* __restrict__ out, size_t rows, int n) {
    follow_previous_grid();
    const size_t total = rows * (size_t)n;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x)
        out[i] = row[i % n];
}
constexpr int kColSumRows = 256;
__global__ void column_partial_kernel(const float* in, float* __restrict__ part, size_t rows, int n) {
    follow_previous_grid();
    const int c = blockIdx.y * blockDim.x + threadIdx.x;
    if (c >= n) return;
    const size_t r0 = (size_t)blockIdx.x * kColSumRows;
    const size_t r1 = r0 + kColSumRows < rows ? r0 + kColSumRows : rows;
    float acc = 0.f;
    for (size_t r = r0; r < r1; ++r) acc += in[r * n + c];
    part[(size_t)blockIdx.x * n + c] = acc;
}
__global__ void column_final_kernel(const float* part, float* __restrict__ out, int nparts, int n) {
    follow_previous_grid();
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n) return;
    double acc = 0.0;
    for (int p = 0; p < nparts; ++p) acc += (double)part[(size_t)p * n + c];
    out[c] = (float)acc;
}
cudaError_t launch_broadcast_rows(const float* row, float* out, size_t rows, int n, cudaStream_t st) {
    const size_t total = rows * (size_t)n;
    const unsigned blocks = (unsigned)((total + 255) / 256 < 148 * 32 ? (total + 255) / 256 : 148 * 32);
    launch_after(broadcast_rows_kernel, blocks ? blocks : 1, 256, 0, st, row, out, rows, n);
    return cudaGetLastError();
}
size_t column_sum_parts(size_t rows) { return (rows + kColSumRows - 1) / kColSumRows; }
// out[c] = sum over rows of in[r][c]; part: column_sum_parts(rows) * n floats of scratch
cudaError_t launch_column_sum(const float* in, float* part, float* out, size_t rows, int n, cudaStream_t st) {
    const unsigned parts = (unsigned)column_sum_parts(rows);
    launch_after(column_partial_kernel, dim3(parts, (n + 127) / 128), 128, 0, st, in, part, rows, n);
    launch_after(column_final_kernel, (n + 127) / 128, 128, 0, st, part, out, (int)parts, n);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ gate tensor in bfloat16
// eight values a thread (both tensors start on 16 bytes); two at a time, 15 MB took 8.7 us
__global__ void __launch_bounds__(256) widen_bf16_kernel(const __nv_bfloat16* in, float* __restrict__ out, size_t n) {
    follow_previous_grid();
    const size_t i = ((size_t)blockIdx.x * 256 + threadIdx.x) * 8;
    if (i + 8 <= n) {
        float x[8];
        load_vec(in + i, x);
        *reinterpret_cast<float4*>(out + i) = make_float4(x[0], x[1], x[2], x[3]);
        *reinterpret_cast<float4*>(out + i + 4) = make_float4(x[4], x[5], x[6], x[7]);
    } else {
        for (size_t j = i; j < n; ++j) out[j] = __bfloat162float(in[j]);
    }
}
cudaError_t launch_widen_bf16(const void* in, float* out, size_t n, cudaStream_t st) {
    launch_after(widen_bf16_kernel, (unsigned)((n + 2047) / 2048), 256, 0, st, static_cast<const __nv_bfloat16*>(in), out, n);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ slot padding
// Rows of n_in floats copied into rows of n_out floats: widened rows get `fill` in their tail,
// narrowed rows lose theirs.  Used when a layer with 32 slots runs on the 64-slot tiles of the
// tensor-core kernels: gate rows are widened with a neutral gate, memories with empty slots.
__global__ void resize_rows_kernel(const float* in, float* __restrict__ out, size_t rows, int n_in, int n_out,
                                   float fill) {
    follow_previous_grid();
    const size_t total = rows * (size_t)n_out;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const size_t r = i / n_out;
        const int c = (int)(i - r * n_out);
        out[i] = c < n_in ? in[r * n_in + c] : fill;
    }
}
cudaError_t launch_resize_rows(const float* in, float* out, size_t rows, int n_in, int n_out, float fill, cudaStream_t st) {
    const size_t total = rows * (size_t)n_out;
    const unsigned blocks = (unsigned)((total + 255) / 256 < 148 * 32 ? (total + 255) / 256 : 148 * 32);
    launch_after(resize_rows_kernel, blocks ? blocks : 1, 256, 0, st, in, out, rows, n_in, n_out, fill);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ segment-parallel scheduling
// The memories are linear in (k, v): K~ after a segment = D * K~ before + (K~ of the segment run
// from empty memories), D = product of the gates over the segment.  A sequence cut into nseg
// segments can therefore run as nseg independent sequences once every segment's start
// memories are known.
//
// seg_logdecay[b][r][h][s] = sum over the chunks of segment r of G at the chunk's last row.
// (128 slots on the tensor cores; other calls have it from their state runs)
__global__ void segment_logdecay_kernel(const float* G, float* __restrict__ seg_logdecay, int T, int H,
                                        int nseg, int tseg, int chunk) {
    follow_previous_grid();
    constexpr int M = 128;
    const int s = threadIdx.x, h = blockIdx.y;
    const int b = blockIdx.x / nseg, r = blockIdx.x % nseg;
    const int t_begin = r * tseg, t_end = min(T, t_begin + tseg);
    double acc = 0.0;
    for (int t = t_begin; t < t_end; t += chunk)      // (the last chunk of the sequence may be a ragged one)
        acc += (double)G[(((size_t)b * T + min(t + chunk, t_end) - 1) * H + h) * M + s];
    seg_logdecay[(((size_t)b * nseg + r) * H + h) * M + s] = (float)acc;
}

// start[b][r] = D[r-1] start[b][r-1] + local_end[b][r-1], start[b][0] = S0[b] (or 0); the memory
// after the last segment goes to final (nullable).  Memories [.., H, M, D]; one thread per (s, c).
// reverse: the same from the last segment down (time-reversed scans: start[r] is the state that
// enters segment r from the right, S0 the one after the last token, final the one before the first).
template <int M>
__global__ void segment_combine_kernel(const float* seg_logdecay, CombineSet k, CombineSet v, int H, int nseg,
                                       int reverse) {
    follow_previous_grid();
    const int b = blockIdx.x / H, h = blockIdx.x % H;
    int idx = blockIdx.y * blockDim.x + threadIdx.x;
    const bool second = idx >= M * k.D;
    if (second) idx -= M * k.D;
    const CombineSet& a = second ? v : k;
    if (idx < M * a.D) {
        const int s = idx / a.D;
        float cur = a.S0 ? a.S0[((size_t)(b * H + h)) * M * a.D + idx] : 0.f;
#pragma unroll 4
        for (int i = 0; i < nseg; ++i) {
            const int r = reverse ? nseg - 1 - i : i;
            const size_t pair = ((size_t)b * nseg + r) * H + h;
            a.start[pair * M * a.D + idx] = cur;
            cur = fmaf(cur, expf(seg_logdecay[pair * M + s]), a.local_end[pair * M * a.D + idx]);
        }
        if (a.final_state) a.final_state[((size_t)(b * H + h)) * M * a.D + idx] = cur;
    }
}

// Sequence sharding across GPUs (same linearity): the gathered per-shard log-decays [R,B,H,M] and
// local end memories [R,B,H,M,D] of all R shards -> the memories entering shard `rank` (from the left;
// reverse: from the right, for the reversed scans of the backward) and, optionally, the memories after
// the last shard (reverse: before the first).  S0: what enters the first shard (reverse: the last).
__global__ void shard_combine_kernel(const float* logdecay_all, const float* local_all,
                                     const float* S0, float* __restrict__ start, float* __restrict__ final_state,
                                     int BH, int M, int D, int nshard, int rank, int reverse) {
    follow_previous_grid();
    const int bh = blockIdx.x;
    const int idx = blockIdx.y * blockDim.x + threadIdx.x;
    if (idx >= M * D) return;
    const int s = idx / D;
    float cur = S0 ? S0[(size_t)bh * M * D + idx] : 0.f;
    for (int i = 0; i < nshard; ++i) {
        const int r = reverse ? nshard - 1 - i : i;
        if (r == rank && start != nullptr) start[(size_t)bh * M * D + idx] = cur;
        const size_t pair = (size_t)r * BH + bh;
        cur = fmaf(cur, __expf(logdecay_all[pair * M + s]), local_all[pair * M * D + idx]);
    }
    if (final_state != nullptr) final_state[(size_t)bh * M * D + idx] = cur;
}
cudaError_t launch_shard_combine(const float* logdecay_all, const float* local_all, const float* S0, float* start,
                                 float* final_state, int B, int H, int M, int D, int nshard, int rank, int reverse,
                                 cudaStream_t st) {
    dim3 grid(B * H, (M * D + 255) / 256);
    launch_after(shard_combine_kernel, grid, 256, 0, st, logdecay_all, local_all, S0, start, final_state, B * H, M, D, nshard, rank, reverse);
    return cudaGetLastError();
}

cudaError_t launch_segment_logdecay(const float* G, float* seg_logdecay, int B, int T, int H, int nseg, int tseg, int chunk,
                                    cudaStream_t st) {
    launch_after(segment_logdecay_kernel, dim3(B * nseg, H), 128, 0, st, G, seg_logdecay, T, H, nseg, tseg, chunk);
    return cudaGetLastError();
}

cudaError_t launch_segment_combine(const float* seg_logdecay, CombineSet k, CombineSet v, int B, int H, int M, int nseg,
                                   int reverse, cudaStream_t st) {
    dim3 grid(B * H, (M * (k.D + v.D) + 255) / 256);
    if (M == 128) launch_after(segment_combine_kernel<128>, grid, 256, 0, st, seg_logdecay, k, v, H, nseg, reverse);
    else if (M == 64) launch_after(segment_combine_kernel<64>, grid, 256, 0, st, seg_logdecay, k, v, H, nseg, reverse);
    else launch_after(segment_combine_kernel<32>, grid, 256, 0, st, seg_logdecay, k, v, H, nseg, reverse);
    return cudaGetLastError();
}

}  // namespace gsa
