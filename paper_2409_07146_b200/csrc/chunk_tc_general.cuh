// The general tcgen05 (bf16 tensor-core) versions of the two chunk primitives of Algorithm 1, for the (batch, head)
// pairs that hold a strong-decay chunk.  They are device functions: every scan is ONE launch of a pipelined kernel
// (chunk_tc_lean.cu, chunk_tc_pair.cu) whose CTAs come here when their pair is flagged.  As launches of their own
// they cost every scan a second launch, a side stream and four events, which is what bounded short calls: a forward over
// T = 300, 16 heads of 128, 59 us with them and 42 without; a training step of the 1.3B model's layer 481 and 466.
//
// One CTA owns one (batch, head) and one 128-wide slice of the head dimension and walks the
// chunks (128 tokens each) in order.  It has 256 compute threads and one issuing warp.
// Compute threads r and r + 128 share row r of the chunk, which is channel r of the state
// slice and TMEM lane r of every accumulator; the first works on slots (or columns) 0..31
// (0..63), the second on the rest.  One lane of the issuing warp requests every tile copy
// and issues every MMA, running ahead of the compute threads; the two sides meet on
// mbarriers only.
// Per chunk:
//   * every tile -- the d-sized ones (xq, xk / xv, bf16) and the slot-sized ones (weights,
//     cumulative log gate G, fp32) -- arrives by TMA with the 128-byte swizzle, requested as
//     soon as the buffer it lands in has been consumed by the previous chunk, so the copy of
//     chunk n+1 runs under the computation of chunk n;
//   * each thread reads its own row of the slot-sized tiles (conflict-free under the
//     swizzle), scales it by the decay factors and writes bf16 operand rows;
//   * all contractions run as tcgen05.mma (M = 128) with fp32 accumulators in tensor
//     memory, committed to mbarriers that the compute threads wait on;
//   * the fp32 master copy of the state slice stays in registers (32 per thread); its bf16
//     copy for the next chunk's state product is rewritten every chunk.
// Decay inside a chunk is factorised as exp(G_i) * exp(-G_j) while the chunk's total
// log-decay stays above kFactorisedDecayMin; a chunk that forgets harder computes its
// intra-chunk term with explicit exponent differences on the CUDA cores instead.
// Every wait is bounded: on expiry the CTA flags dev_status, frees its tensor memory and
// returns.
#pragma once
#include "chunk_tc_shared.cuh"

namespace gsa {
namespace {
using namespace tc;
using namespace tcchunk;

// The rows of 1 - a of a flagged pair's moderate chunks, as the gate kernel forms them, where it has left them out
// (InputGate).  Every CTA that is about to read them writes them all -- the same values -- and reads its own.  A warp a chunk.
// (All chunks, strong ones too: 32 K tokens of strong gates, 16 heads, 1279 -> 1517 us.)
// Not inlined: within the pipelined kernels it costs the scan beside it registers (value_side of B = 8, T = 2048, 4 heads of 512,
// 55 -> 64 us).
__device__ __noinline__ void write_input_gate(const ValueSideArgs& a) {
    if (a.input_gate.gate == nullptr) return;
    constexpr int kBatch = 8;
    const ScanSpan span = scan_span(blockIdx.x, a.H, a.T, a.nseg, a.tseg);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const size_t stride = (size_t)a.H * kM;
    for (int t0 = span.t0 + warp * kCT; t0 < span.t_end; t0 += (int)(blockDim.x >> 5) * kCT) {
        const int rows = min(kCT, span.t_end - t0);
        const size_t first = (((size_t)span.b * a.T + t0) * a.H + span.h) * kM;
        // (clearly below the bound that the gate kernel compared the exact sum with: G is that sum to an ulp)
        const float2 g = *reinterpret_cast<const float2*>(a.G + first + (rows - 1) * stride + 2 * lane);
        if (__any_sync(0xffffffffu, fminf(g.x, g.y) < kFactorisedDecayMin - 0.01f)) continue;
        const float* gate = a.input_gate.gate + first + (lane & 15) * 4;
        float* out = const_cast<float*>(a.w) + first + (lane & 15) * 4;
        for (int r0 = lane >> 4; r0 < rows; r0 += 2 * kBatch) {
            float4 x[kBatch];
#pragma unroll
            for (int q = 0; q < kBatch; ++q)
                if (r0 + 2 * q < rows) x[q] = *reinterpret_cast<const float4*>(gate + (r0 + 2 * q) * stride);
#pragma unroll
            for (int q = 0; q < kBatch; ++q) {
                if (r0 + 2 * q >= rows) break;
                float y[4] = {x[q].x, x[q].y, x[q].z, x[q].w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    if (a.input_gate.kind == GSA_GATE_A) { y[e] = 1.f - y[e]; continue; }
                    if (a.input_gate.kind == GSA_GATE_LOGITS) y[e] = log_gate_from_logit(y[e], a.input_gate.inv_tau);
                    y[e] = -expm1f(y[e]);
                }
                *reinterpret_cast<float4*>(out + (r0 + 2 * q) * stride) = make_float4(y[0], y[1], y[2], y[3]);
            }
        }
    }
    __threadfence();
    asm volatile("fence.proxy.async;" ::: "memory");      // (the copy engine reads them next)
    __syncthreads();
}

struct Ctl {
    // filled by TMA
    uint64_t bar_x;        // d-sized tiles of the current chunk
    uint64_t bar_g[2];     // value_side: G tile, two stages; key_side: [0] = uk + G tiles
    uint64_t bar_w;        // value_side: weight tile; key_side: uq tile
    // signalled by tcgen05.commit
    uint64_t bar_p;        // first product of the chunk (P or A) complete
    uint64_t bar_mma1;     // state and inter-chunk products complete
    uint64_t bar_mma2;     // intra-chunk product complete
    // signalled by the compute threads (one arrival after their barrier)
    uint64_t bar_ops;      // operand rows of the chunk are in shared memory
    uint64_t bar_pm;       // masked P / A rows are in shared memory
    uint64_t bar_out;      // output rows are staged (or the chunk is otherwise done)
    uint64_t bar_sb;       // value_side: the state copy for the next chunk is written
                           // key_side: (issuing warp ->) the output staging buffer is free again
    uint32_t tmem_slot;
    volatile int abort;
    volatile int moderate[2];   // decision of the chunk, by chunk parity
    alignas(16) float gc[kM];    // G of the chunk's last valid row
    alignas(16) float egc[kM];   // exp(gc)
};

// Publish the G row of the chunk's last valid token, its exponential and decide whether the
// chunk's decay is moderate.  One compute-thread barrier inside; the result is uniform.
__device__ __forceinline__ bool publish_chunk_decay(Ctl* ctl, int tid, const unsigned char* gtile, int last_row) {
    bool fine = true;
    if (tid < kM) {
        const float g = tile_elem(gtile, last_row, tid);
        ctl->gc[tid] = g;
        ctl->egc[tid] = __expf(g);
        fine = g >= kFactorisedDecayMin;
    }
    return compute_sync_and(fine);
}

// FIRST: this is the CTA's first scan, which allocates its tensor memory (a CTA may do that once: the allocation gives
// up the right to another one); a second scan takes over the barriers' memory and tmem_slot of the first.
template <bool FIRST>
__device__ __forceinline__ void ctl_init(Ctl* ctl, int tid, int warp) {
    if (tid == 0) {
        if (!FIRST) {
            uint64_t* bars[] = {&ctl->bar_x, &ctl->bar_g[0], &ctl->bar_g[1], &ctl->bar_w, &ctl->bar_p, &ctl->bar_mma1,
                                &ctl->bar_mma2, &ctl->bar_ops, &ctl->bar_pm, &ctl->bar_out, &ctl->bar_sb};
            for (uint64_t* b : bars) mbar_inval(b);
        }
        mbar_init(&ctl->bar_x, 1);
        mbar_init(&ctl->bar_g[0], 1);
        mbar_init(&ctl->bar_g[1], 1);
        mbar_init(&ctl->bar_w, 1);
        mbar_init(&ctl->bar_p, 1);
        mbar_init(&ctl->bar_mma1, 1);
        mbar_init(&ctl->bar_mma2, 1);
        mbar_init(&ctl->bar_ops, 1);
        mbar_init(&ctl->bar_pm, 1);
        mbar_init(&ctl->bar_out, 1);
        mbar_init(&ctl->bar_sb, 1);
        ctl->abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (FIRST && warp == 0) {
        __syncwarp();
        tmem_alloc(&ctl->tmem_slot, kTmemCols);
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
}

// Strong-decay chunks (App. A: a decay too strong for one reference point per chunk).  The decay
// between two rows of a chunk is a product of per-step gates, prod_{r=j+1..i} a_r[s], every factor
// <= 1: walking j away from the target row i, the product is carried along by ONE multiplication
// per step and slot -- no exponential in the loop, nothing can overflow -- and the walk stops as
// soon as the product has fallen below 2^-40 for all slots of the thread (what is left of the sum is
// then below 1e-12 of its leading terms).  With strong forgetting that is after a dozen steps.
// The per-step gates a_j = exp(G_j - G_{j-1}) are formed once per chunk, in place of the G tile.
constexpr float kDecayFloor = 9.094947e-13f;      // 2^-40

// Replace the G tile by the per-step gates (rows past the end: 1).  Two compute-thread barriers inside.
__device__ __forceinline__ void gates_in_place(unsigned char* gt, int row, int half, int sb, int valid) {
    const int grow = min(row, valid - 1);
    float aj[kHS];
#pragma unroll
    for (int c = 0; c < kHS / 8; ++c) {
        float g[8], gp[8];
        tile_row8(gt, grow, sb + 8 * c, g);
        if (row > 0 && row < valid) tile_row8(gt, row - 1, sb + 8 * c, gp);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            aj[8 * c + e] = row >= valid ? 1.f : __expf(row > 0 ? g[e] - gp[e] : g[e]);
        }
    }
    compute_sync();           // every thread has read what it needs of G
    unsigned char* panel = gt + half * kPanelB;
#pragma unroll
    for (int c = 0; c < kHS / 4; ++c)
        *reinterpret_cast<float4*>(panel + swz128(row, c)) = make_float4(aj[4 * c], aj[4 * c + 1], aj[4 * c + 2], aj[4 * c + 3]);
    compute_sync();
}

// The walks go by distance: at step d every row i of the chunk is at j = i - d (time-reversed: i + d), so that all lanes of a
// warp are at work until their products have died out.  (By absolute columns, as the accumulator is read, a warp repeats
// the walk for the different rows of its lanes, a third of them live at a time.  32 K tokens, 16 heads of 128, gates that forget
// within a dozen tokens: value_side 615 -> 488 us, key_side 678 -> 408.  What is left is the shared memory's rate: two rows of
// 64 slots a step for each of 128 rows, 8 k cycles a chunk at a dozen steps, beside 8 k of the scan around it.)  The
// accumulator's columns are turned into distances through a band in shared memory, kBand distances at a time, stored
// [distance][row]: the chunk's 128 rows are then 128 consecutive words.
constexpr int kBand = 32;
static_assert(kBand * kCT * 4 == kPanelB, "a band is one operand panel");

// Which 32 accumulator columns of the warp's rows the threads of `half` turn into distances of band k: a row's band lies in
// two adjacent blocks of 32 columns.  (-1: outside the chunk)
template <bool REV> __device__ __forceinline__ int band_block(int wq, int half, int k) {
    const int blk = REV ? wq + k + half : wq - k - half;
    return blk >= 0 && blk < kCT / 32 ? blk : -1;
}
// The gate between j and the next row of the walk: prod_{r=j+1..i} becomes prod_{r=j..i}, reversed prod_{r=i+1..j}
// prod_{r=i+1..j+1}.
template <bool REV> __device__ __forceinline__ int next_gate_row(int j) { return REV ? min(j + 1, kCT - 1) : j; }
template <bool REV> __device__ __forceinline__ int distance(int row, int j) { return REV ? j - row : row - j; }

// Strong-decay chunk of value_side: this thread's 32 output slots of row `row`,
//   out[s] = exp(+-..) * inter[s] + sum_j P_ij w_j[s] prod a_r[s]   (j <= i forward, j >= i reverse),
// P and the inter-chunk product are read from the accumulators; the row goes straight to global
// memory.  `gt` holds the per-step gates (gates_in_place), g_row this row's G; `band`: a panel nobody else uses.  Sixteen slots
// at a time: with 32 at a time the scan around the walk spills, and every chunk of a flagged pair pays for it (the state
// runs of 32 K tokens of strong gates 222 -> 277 us).
template <bool REV>
__device__ __forceinline__ void value_side_explicit_rows(const unsigned char* gt, const unsigned char* sW, float* band,
                                                      const float* gc, const float* g_row, uint32_t tmem, int wq,
                                                      int row, int half, int sb, int valid, float* out_row) {
    const unsigned char* ga = gt + half * kPanelB;           // this thread's 32 slots of the gates and of the weights
    const unsigned char* wa = sW + half * kPanelB;
#pragma unroll 1
    for (int c0 = 0; c0 < kHS / 4; c0 += 4) {
        float acc[16], dec[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) { acc[e] = 0.f; dec[e] = 1.f; }
        bool live = row < valid;
#pragma unroll 1
        for (int k = 0; k < kCT / kBand; ++k) {
            const int blk = band_block<REV>(wq, half, k);
            if (blk >= 0) {
#pragma unroll
                for (int q = 0; q < 32; q += 16) {
                    float v[16];
                    tmem_ld16(tmem_row_addr(tmem, wq, kColP + 32 * blk + q), v);
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        const int d = distance<REV>(row, 32 * blk + q + e) - kBand * k;
                        if (d >= 0 && d < kBand) band[d * kCT + row] = v[e];
                    }
                }
            }
            compute_sync();
#pragma unroll 1
            for (int d0 = 0; d0 < kBand; d0 += 4) {
                if (!__any_sync(0xffffffffu, live)) break;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int d = kBand * k + d0 + u, j = REV ? row + d : row - d;
                    live = live && (REV ? j < valid : j >= 0);
                    if (!live) continue;
                    const float p = band[(d0 + u) * kCT + row];
                    const int jg = next_gate_row<REV>(j);
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const float4 a4 = *reinterpret_cast<const float4*>(ga + swz128(jg, c0 + c));
                        const float4 w4 = *reinterpret_cast<const float4*>(wa + swz128(j, c0 + c));
                        const float aj[4] = {a4.x, a4.y, a4.z, a4.w}, wj[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            float& x = dec[4 * c + e];
                            acc[4 * c + e] = fmaf(p * wj[e], x, acc[4 * c + e]);
                            x *= aj[e];
                        }
                    }
                }
                float top = 0.f;
#pragma unroll
                for (int e = 0; e < 16; ++e) top = fmaxf(top, dec[e]);
                live = live && top >= kDecayFloor;
            }
            if (!compute_sync_or(live)) break;       // (the barrier also covers: the band may be written again)
        }
        float vi[16], vj[16];
        const int s0 = sb + 4 * c0;
        tmem_ld16(tmem_row_addr(tmem, wq, kColO + s0), vi);
        tmem_ld16(tmem_row_addr(tmem, wq, kColO + kM + s0), vj);       // (the state copy is a high/low pair)
        if (row < valid) {
#pragma unroll
            for (int e = 0; e < 16; e += 4) {
                const float4 g4 = *reinterpret_cast<const float4*>(g_row + s0 + e);
                const float g[4] = {g4.x, g4.y, g4.z, g4.w};
                float r[4];
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    r[u] = fmaf(vi[e + u] + vj[e + u], __expf(REV ? gc[s0 + e + u] - g[u] : g[u]), acc[e + u]);
                *reinterpret_cast<float4*>(out_row + s0 + e) = make_float4(r[0], r[1], r[2], r[3]);
            }
        }
    }
}

// ======================================================================================
// value_side: out_i[s] = sum_{j<=i} <xq_i, xk_j> w_j[s] decay_ij[s]  + decayed (xq_i S)[s]
// ======================================================================================
// LAST = false: another scan of this CTA follows, which takes over the tensor memory.  Returns whether all went well
// (the same for every thread); otherwise the tensor memory is freed and nothing may follow.
// STATES: end memories only; of a chunk's products the state's alone is formed.
template <bool REV, bool LAST = true, bool STATES = false>
__device__ __noinline__ bool value_side_general(const CUtensorMap& mapQ, const CUtensorMap& mapK,
                       const CUtensorMap& mapW, const CUtensorMap& mapG,
                       const CUtensorMap& mapO, const ValueSideArgs& args,
                       int32_t* dev_status,
                       int slice) {
    // (a copy: through the reference every field would be read again after each barrier)
    const ValueSideArgs a = args;
    extern __shared__ unsigned char smem_raw[];
    // align by pointer arithmetic (not an integer round trip) so accesses stay in the shared window
    unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    unsigned char* sXq = smem;                       // 2 panels                                  (32 KB)
    unsigned char* sXk = sXq + 2 * kPanelB;          // 2 panels                                  (32 KB)
    unsigned char* sG = sXk + 2 * kPanelB;           // G tile fp32, [2 stages][2 panels]         (64 KB)
    unsigned char* sW = sG + 4 * kPanelB;            // weight tile fp32, 2 panels                (32 KB)
    unsigned char* sWa = sW + 2 * kPanelB;           // decayed weights, bf16 high part, MN-major B [128][64] (16 KB)
    unsigned char* sWb = sWa + kPanelB;              // ... their bf16 rounding residual (low part)           (16 KB)
    unsigned char* sSb = sWb + kPanelB;              // state copy, MN-major B [128][hi 64 | lo 64]  (32 KB)
    Ctl* ctl = reinterpret_cast<Ctl*>(sSb + 2 * kPanelB);
    // (the masked P never goes through shared memory: it is rewritten in place in tensor memory as a bf16
    // high/low pair and read from there as the A operand of the intra-chunk product)

    const int tid = threadIdx.x, warp = tid >> 5, wq = warp & 3, half = (tid >> 7) & 1, row = tid & 127;
    const int sb = kHS * half;          // this thread's first slot
    const ScanSpan span = scan_span(blockIdx.x, a.H, a.T, a.nseg, a.tseg);
    const int bh = blockIdx.x, b = span.b, h = span.h;
    const int d0 = slice * kDST;
    const size_t strideM = (size_t)a.H * kM;
    float* obase = a.out + (size_t)slice * a.B * a.T * a.H * kM + ((size_t)b * a.T * a.H + h) * kM;

    ctl_init<true>(ctl, tid, warp);
    const uint32_t tmem = ctl->tmem_slot;
    const int nchunks = (span.t_end - span.t0 + kCT - 1) / kCT;
    auto chunk_t0 = [&](int it) { return span.t0 + (REV ? nchunks - 1 - it : it) * kCT; };

    if (warp == kComputeThreads / 32) {
        // =============================== issuing warp: TMA loads / stores and all MMAs
        if (elect_one()) {
            auto load_x = [&](int it) {
                const int t = chunk_t0(it);
                mbar_expect_tx(&ctl->bar_x, (STATES ? 2 : 4) * kPanelB);
                if (!STATES) {
                    tma_load_4d(sXq, &mapQ, &ctl->bar_x, d0, h, t, b);
                    tma_load_4d(sXq + kPanelB, &mapQ, &ctl->bar_x, d0 + 64, h, t, b);
                }
                tma_load_4d(sXk, &mapK, &ctl->bar_x, d0, h, t, b);
                tma_load_4d(sXk + kPanelB, &mapK, &ctl->bar_x, d0 + 64, h, t, b);
            };
            auto load_g = [&](int it) {
                const int t = chunk_t0(it), st = it & 1;
                mbar_expect_tx(&ctl->bar_g[st], 2 * kPanelB);
                tma_load_4d(sG + (2 * st) * kPanelB, &mapG, &ctl->bar_g[st], 0, h, t, b);
                tma_load_4d(sG + (2 * st + 1) * kPanelB, &mapG, &ctl->bar_g[st], 32, h, t, b);
            };
            auto load_w = [&](int it) {
                const int t = chunk_t0(it);
                mbar_expect_tx(&ctl->bar_w, 2 * kPanelB);
                tma_load_4d(sW, &mapW, &ctl->bar_w, 0, h, t, b);
                tma_load_4d(sW + kPanelB, &mapW, &ctl->bar_w, 32, h, t, b);
            };
            prefetch_tmap(&mapQ); prefetch_tmap(&mapK); prefetch_tmap(&mapW); prefetch_tmap(&mapG); prefetch_tmap(&mapO);
            load_g(0);
            load_w(0);
            load_x(0);
            constexpr uint32_t idescP = make_idesc(128, 128, false, false);  // xq xk^T
            constexpr uint32_t idescO = make_idesc(128, 2 * kM, false, true);  // xq x state copy [S_hi | S_lo] (MN-major B)
            // the high and the low part of the weights are two adjacent 64-column panels of ONE
            // MN-major B operand (N = 128): one product yields [.. W_hi | .. W_lo]
            constexpr uint32_t idescU = make_idesc(128, 2 * kM, true, true);   // xk^T (MN-major A) x [W_hi | W_lo]
            constexpr uint32_t idescI = make_idesc(128, 2 * kM, false, true);  // masked P (tensor memory) x [W_hi | W_lo]
            // base descriptors of every operand (K step 0); advancing along K is one add each
            const uint64_t dQk = desc_kmajor(smem_u32(sXq), 0), dKk = desc_kmajor(smem_u32(sXk), 0);
            const uint64_t dKm = desc_mnmajor(smem_u32(sXk), 0, kPanelB), dWa = desc_mnmajor(smem_u32(sWa), 0, kPanelB);
            const uint64_t dS = desc_mnmajor(smem_u32(sSb), 0, kPanelB);
            // byte offset of K step kk: K-major operands walk 32 bytes inside a 64-column panel,
            // MN-major operands walk 16 rows (2048 bytes)
            auto kmaj = [](int kk) { return (uint32_t)((kk >> 2) * kPanelB + (kk & 3) * 32); };
            auto mnmaj = [](int kk) { return (uint32_t)(kk * 2048); };
            int n_mod = 0;      // moderate chunks so far (phases of bar_pm / bar_mma2)
            PROF_DECL
            for (int it = 0; it < nchunks && !ctl->abort; ++it) {
                const int t0 = chunk_t0(it);
                PROF_MARK();
                const unsigned char* gt = sG + (2 * (it & 1)) * kPanelB;
                // P = xq xk^T needs nothing but the d-sized tiles: it runs under the operand build
                WAIT_OR_ABORT(&ctl->bar_x, it & 1);
                tc_fence_after_sync();
                PROF_MARK();
                if (!STATES) {
#pragma unroll
                    for (int kk = 0; kk < kDST / 16; ++kk)
                        mma_bf16(tmem + kColP, desc_advance(dQk, kmaj(kk)), desc_advance(dKk, kmaj(kk)), idescP, kk > 0);
                    mma_commit(&ctl->bar_p);
                }
                // so does the inter-chunk product O = xq S: the state copy was written at the end
                // of the previous chunk
                WAIT_OR_ABORT(&ctl->bar_sb, it & 1);
                tc_fence_after_sync();
                if (!STATES) {
#pragma unroll
                    for (int kk = 0; kk < kDST / 16; ++kk)
                        mma_bf16(tmem + kColO, desc_advance(dQk, kmaj(kk)), desc_advance(dS, mnmaj(kk)), idescO, kk > 0);
                }
                PROF_MARK();
                if (it + 1 < nchunks) {
                    bulk_wait_read();     // the output rows staged in that G buffer one chunk ago have left
                    load_g(it + 1);
                }
                // U = xk^T W (high + low part of the weights) once the operand rows are there
                PROF_MARK();
                WAIT_OR_ABORT(&ctl->bar_ops, it & 1);
                tc_fence_after_sync();
                PROF_MARK();
                const bool moderate = !STATES && ctl->moderate[it & 1] != 0;       // (... has an intra-chunk product)
#pragma unroll
                for (int kk = 0; kk < kCT / 16; ++kk)
                    mma_bf16(tmem + kColU, desc_advance(dKm, mnmaj(kk)), desc_advance(dWa, mnmaj(kk)), idescU, kk > 0);
                mma_commit(&ctl->bar_mma1);
                PROF_MARK();
                if (moderate) {
                    WAIT_OR_ABORT(&ctl->bar_pm, n_mod & 1);
                    tc_fence_after_sync();
                    PROF_MARK();
#pragma unroll
                    for (int kk = 0; kk < kCT / 16; ++kk)
                        mma_bf16_ta(tmem + kColO2, tmem + kColP + 64 * (kk >> 2) + 8 * (kk & 3), desc_advance(dWa, mnmaj(kk)),
                                    idescI, kk > 0);
#pragma unroll
                    for (int kk = 0; kk < kCT / 16; ++kk)      // ... and the rounding residual of the masked P
                        mma_bf16_ta(tmem + kColO2, tmem + kColP + 64 * (kk >> 2) + 32 + 8 * (kk & 3),
                                    desc_advance(dWa, mnmaj(kk)), idescI, true);
                    mma_commit(&ctl->bar_mma2);
                    PROF_MARK();
                }
                // the d-sized tiles are consumed once U and O are done: request the next chunk's
                WAIT_OR_ABORT(&ctl->bar_mma1, it & 1);
                PROF_MARK();
                if (it + 1 < nchunks) load_x(it + 1);
                if (moderate) {
                    // the masked P is consumed: its buffer takes the next chunk's weight tile
                    WAIT_OR_ABORT(&ctl->bar_mma2, n_mod & 1);
                    ++n_mod;
                    if (it + 1 < nchunks) load_w(it + 1);
                }
                PROF_MARK();
                WAIT_OR_ABORT(&ctl->bar_out, it & 1);
                PROF_MARK();
                PROF_DUMP("value_side issue");
                if (ctl->abort) break;
                if (moderate) {
                    tma_store_5d(&mapO, gt, 0, h, t0, b, slice);
                    tma_store_5d(&mapO, gt + kPanelB, 32, h, t0, b, slice);
                    bulk_commit();
                } else if (!moderate && it + 1 < nchunks) {
                    load_w(it + 1);       // a strong-decay chunk read the weight tile until now
                }
            }
            bulk_wait_read();      // staged output rows must have left before shared memory goes away
        }
    } else if (tid < kComputeThreads) {
        // =============================== compute threads
        // state slice: S[c = row][s], slots sb .. sb+31
        float S[kHS];
#pragma unroll
        for (int s = 0; s < kHS; ++s) S[s] = (a.S0 && d0 + row < a.D) ? a.S0[((size_t)bh * kM + sb + s) * a.D + d0 + row] : 0.f;

        // bf16 copy of the state (value + rounding residual) for the first chunk's inter-chunk product
        store_state_row_split<false>(sSb, sSb + kPanelB, row, sb, S, nullptr);
        fence_async_smem();
        compute_sync();
        if (tid == 0) mbar_arrive(&ctl->bar_sb);

        int n_mod = 0;
        PROF_DECL
        for (int it = 0; it < nchunks; ++it) {
            const int t0 = chunk_t0(it);
            const int valid = min(kCT, span.t_end - t0);
            PROF_MARK();
            const unsigned char* gt = sG + (2 * (it & 1)) * kPanelB;
            WAIT_OR_ABORT(&ctl->bar_g[it & 1], (it >> 1) & 1);
            WAIT_OR_ABORT(&ctl->bar_w, it & 1);
            PROF_MARK();
            const bool moderate = publish_chunk_decay(ctl, tid, gt, valid - 1);
            if (ctl->abort) break;
            PROF_MARK();

            // ---- this token's slot rows -> operand rows (rows past the end: zero weights)
            const int grow = min(row, valid - 1);
            const float strong = moderate ? 0.f : 1.f;      // adds G_C to the exponent of a strong-decay chunk
#pragma unroll
            for (int s0 = sb; s0 < sb + kHS; s0 += 8) {
                float g[8], w[8], wd[8];
                tile_row8(gt, grow, s0, g);
                tile_row8(sW, row, s0, w);
                // ONE set of decayed weights serves the intra-chunk product and the state update,
                // branch-free over the elements (a branch per element would serialise the exps):
                //   reverse           : w exp(G)
                //   forward, moderate : w exp(-G); the state update gets its exp(G_C) afterwards,
                //                       S <- exp(G_C) (S + xk^T W)
                //   forward, strong   : w exp(G_C - G) (state update only; no intra product)
                // They are stored as a bf16 pair (value + rounding residual): the weights multiply
                // sums that cancel in the gate gradient, where a plain bf16 rounding is too coarse.
                const float4 gc0 = *reinterpret_cast<const float4*>(&ctl->gc[s0]);
                const float4 gc1 = *reinterpret_cast<const float4*>(&ctl->gc[s0 + 4]);
                const float gcv[8] = {gc0.x, gc0.y, gc0.z, gc0.w, gc1.x, gc1.y, gc1.z, gc1.w};
#pragma unroll
                for (int e = 0; e < 8; ++e) wd[e] = w[e] * __expf(REV ? g[e] : fmaf(strong, gcv[e], -g[e]));
                store_chunk_split(sWa, sWb, row, s0 >> 3, wd);
            }
            fence_async_smem();
            if (tid == 0) ctl->moderate[it & 1] = moderate;
            compute_sync();                     // every row is written and the weight tile is read
            if (tid == 0) mbar_arrive(&ctl->bar_ops);
            PROF_MARK();

            if (!STATES) {
                WAIT_OR_ABORT(&ctl->bar_p, it & 1);
                tc_fence_after_sync();
            }
            PROF_MARK();
            if (STATES) {
            } else if (moderate) {
                mask_row_in_tmem<REV, true>(tmem, wq, row, half, kColP);
                tc_fence_before_sync();
                compute_sync();
                if (tid == 0) mbar_arrive(&ctl->bar_pm);
            } else {
                // strong decay: the intra-chunk term by the walk over the per-step gates
                WAIT_OR_ABORT(&ctl->bar_mma1, it & 1);    // the inter-chunk product
                tc_fence_after_sync();
                {
                    gates_in_place(const_cast<unsigned char*>(gt), row, half, sb, valid);
                    // (the band: the weights' operand rows, which the state product, complete, was the last to read)
                    value_side_explicit_rows<REV>(gt, sW, reinterpret_cast<float*>(sWa), ctl->gc,
                                                  a.G + (((size_t)b * a.T + t0 + row) * a.H + h) * kM, tmem, wq, row, half, sb, valid,
                                                  obase + (size_t)(t0 + row) * strideM);
                }
            }

            // ---- state update from U: S <- S exp(G_C) + U  (forward moderate chunk: exp(G_C) (S + U))
            PROF_MARK();
            WAIT_OR_ABORT(&ctl->bar_mma1, it & 1);
            tc_fence_after_sync();
            PROF_MARK();
            {
                float v[kHS], vl[kHS];
                tmem_ld32(tmem_row_addr(tmem, wq, kColU + sb), v);
                tmem_ld32(tmem_row_addr(tmem, wq, kColU + kM + sb), vl);
#pragma unroll
                for (int e = 0; e < kHS; e += 4) {
                    const float4 ec = *reinterpret_cast<const float4*>(&ctl->egc[sb + e]);
                    const float ecv[4] = {ec.x, ec.y, ec.z, ec.w};
#pragma unroll
                    for (int t = 0; t < 4; ++t) {
                        const float u = v[e + t] + vl[e + t];
                        S[e + t] = (!REV && moderate) ? (S[e + t] + u) * ecv[t] : fmaf(S[e + t], ecv[t], u);
                    }
                }
            }
            // its bf16 copy feeds the next chunk's inter-chunk product (issued as soon as the next
            // tiles are there); the product of this chunk that read the old copy is complete
            if (!STATES) store_state_row_split<false>(sSb, sSb + kPanelB, row, sb, S, nullptr);

            // ---- output rows of a moderate chunk: exp(+-G_i) * (inter + intra)
            PROF_MARK();
            if (!STATES && moderate) {
                WAIT_OR_ABORT(&ctl->bar_mma2, n_mod & 1);
                ++n_mod;
                tc_fence_after_sync();
                PROF_MARK();
                // the scaled rows replace this chunk's G rows in place (each thread reads and rewrites
                // only its own 32 slots) and leave as one tiled store, clipped at the sequence end
                float vo[kHS], vi[kHS];
                tmem_ld32(tmem_row_addr(tmem, wq, kColO2 + sb), vo);
                tmem_ld32(tmem_row_addr(tmem, wq, kColO2 + kM + sb), vi);
#pragma unroll
                for (int e = 0; e < kHS; ++e) vo[e] += vi[e];          // high + low weight parts
                {
                    float vj[kHS];
                    tmem_ld32(tmem_row_addr(tmem, wq, kColO + sb), vi);
                    tmem_ld32(tmem_row_addr(tmem, wq, kColO + kM + sb), vj);
#pragma unroll
                    for (int e = 0; e < kHS; ++e) vi[e] += vj[e];      // high + low state parts
                }
                // forward: exp(G) (inter + intra); reverse: exp(-G) (exp(G_C) inter + intra)
#pragma unroll
                for (int e = 0; e < kHS; ++e) vo[e] = REV ? fmaf(vi[e], ctl->egc[sb + e], vo[e]) : vo[e] + vi[e];
                if (row < valid) {
                    unsigned char* panel = const_cast<unsigned char*>(gt) + half * kPanelB;
#pragma unroll
                    for (int c = 0; c < kHS / 4; ++c) {
                        float4* cell = reinterpret_cast<float4*>(panel + swz128(row, c));
                        const float4 g = *cell;
                        *cell = make_float4(vo[4 * c] * __expf(REV ? -g.x : g.x), vo[4 * c + 1] * __expf(REV ? -g.y : g.y),
                                            vo[4 * c + 2] * __expf(REV ? -g.z : g.z), vo[4 * c + 3] * __expf(REV ? -g.w : g.w));
                    }
                }
            }
            fence_async_smem();
            tc_fence_before_sync();
            compute_sync();                 // rows staged; gc / egc and the accumulators may be reused
            if (tid == 0) {
                mbar_arrive(&ctl->bar_sb);
                mbar_arrive(&ctl->bar_out);
            }
            PROF_MARK();
            PROF_DUMP("value_side compute");
            if (ctl->abort) break;
        }
        if (!ctl->abort && a.Send && d0 + row < a.D) {
#pragma unroll
            for (int s = 0; s < kHS; ++s) a.Send[((size_t)bh * kM + sb + s) * a.D + d0 + row] = S[s];
        }
    }

    tc_fence_before_sync();
    __syncthreads();
    if (ctl->abort) {
        if (tid == 0 && dev_status != nullptr) *dev_status = GSA_ERR_TIMEOUT;
        // bounded grace period for tile copies still in flight before shared memory goes away
        for (int i = 0; i < 200; ++i) __nanosleep(1000);
    }
    const bool fine = ctl->abort == 0;
    __syncthreads();
    if ((LAST || !fine) && warp == 0) {
        __syncwarp();
        tmem_dealloc(tmem, kTmemCols);
    }
    return fine;
}

// Strong-decay chunk of key_side: A_ij = sum_s uq_i[s] uk_j[s] prod a_r[s] on the kept triangle, by
// the same walk: the thread carries uq_i[s] times the running decay product for its 32 slots, one
// multiplication per step and slot, and stops once every product is below 2^-40 of the largest it began with.  The two
// threads of a row meet in two bands (over the uq rows, which are in registers by then); the sums go to the
// accumulator's fp32 columns and from there, like those of a moderate chunk, into the masked bf16 operand rows.
// `sG` is replaced by the per-step gates on the way.
template <bool REV>
__device__ __forceinline__ void key_side_explicit_rows(unsigned char* sG, unsigned char* sUq,
                                                    const unsigned char* sUk, uint32_t tmem, int wq, int row, int half,
                                                    int sb, int valid) {
    float qd[kHS];
#pragma unroll
    for (int s0 = 0; s0 < kHS; s0 += 8) {
        float uq[8];
        tile_row8(sUq, row, sb + s0, uq);
#pragma unroll
        for (int e = 0; e < 8; ++e) qd[s0 + e] = uq[e];
    }
    gates_in_place(sG, row, half, sb, valid);       // (its barriers also cover: every uq row is in registers)
    {
        uint32_t zero[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) zero[e] = 0u;
#pragma unroll
        for (int q = 0; q < 4; ++q) tmem_st16(tmem_row_addr(tmem, wq, kColP + 64 * half + 16 * q), zero);
        tmem_st_wait();
        tc_fence_before_sync();
    }
    float* band = reinterpret_cast<float*>(sUq + half * kPanelB);
    const float *band0 = reinterpret_cast<const float*>(sUq), *band1 = reinterpret_cast<const float*>(sUq + kPanelB);
    const unsigned char* ga = sG + half * kPanelB;
    const unsigned char* ka = sUk + half * kPanelB;
    float start = 0.f;
#pragma unroll
    for (int e = 0; e < kHS; ++e) start = fmaxf(start, fabsf(qd[e]));
    const float floor_ = start * kDecayFloor;
    bool live = start > 0.f;
#pragma unroll 1
    for (int k = 0; k < kCT / kBand; ++k) {
#pragma unroll 1
        for (int d0 = 0; d0 < kBand; d0 += 4) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int d = kBand * k + d0 + u, j = REV ? row + d : row - d;
                live = live && (REV ? j < valid : j >= 0);
                float sum[4] = {0.f, 0.f, 0.f, 0.f};
                if (live) {
                    const int jg = next_gate_row<REV>(j);
#pragma unroll
                    for (int c = 0; c < kHS / 4; ++c) {
                        const float4 a4 = *reinterpret_cast<const float4*>(ga + swz128(jg, c));
                        const float4 k4 = *reinterpret_cast<const float4*>(ka + swz128(j, c));
                        const float aj[4] = {a4.x, a4.y, a4.z, a4.w}, uk[4] = {k4.x, k4.y, k4.z, k4.w};
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            float& x = qd[4 * c + e];
                            sum[e] = fmaf(x, uk[e], sum[e]);
                            x *= aj[e];
                        }
                    }
                }
                band[(d0 + u) * kCT + row] = (sum[0] + sum[1]) + (sum[2] + sum[3]);
            }
            float top = 0.f;
#pragma unroll
            for (int e = 0; e < kHS; ++e) top = fmaxf(top, fabsf(qd[e]));
            live = live && top > floor_;
        }
        compute_sync();
        tc_fence_after_sync();
        const int blk = band_block<REV>(wq, half, k);
        if (blk >= 0) {
            float v[32];
            tmem_ld32(tmem_row_addr(tmem, wq, kColP + 32 * blk), v);
            uint32_t out[2][16];
#pragma unroll
            for (int e = 0; e < 32; ++e) {
                const int d = distance<REV>(row, 32 * blk + e) - kBand * k;
                if (d >= 0 && d < kBand) v[e] = band0[d * kCT + row] + band1[d * kCT + row];
                out[e >> 4][e & 15] = __float_as_uint(v[e]);
            }
            tmem_st16(tmem_row_addr(tmem, wq, kColP + 32 * blk), out[0]);
            tmem_st16(tmem_row_addr(tmem, wq, kColP + 32 * blk + 16), out[1]);
            tmem_st_wait();
        }
        tc_fence_before_sync();
        const bool more = compute_sync_or(live);     // (the barrier also covers: the bands may be written again)
        tc_fence_after_sync();
        if (!more) break;
    }
    mask_row_in_tmem<REV, true>(tmem, wq, row, half, kColP);
}

// ======================================================================================
// key_side: out_i = (uq_i * qscale_i) S + sum_j A_ij xv_j,  A_ij = sum_s uq_i[s] uk_j[s] decay_ij[s]
// ======================================================================================
template <bool REV, bool FIRST = true>
__device__ __noinline__ void key_side_general(const CUtensorMap& mapV, const CUtensorMap& mapUq,
                       const CUtensorMap& mapUk, const CUtensorMap& mapG,
                       const CUtensorMap& mapO, const KeySideArgs& args,
                       int32_t* dev_status) {
    // (a copy: through the reference every field would be read again after each barrier)
    const KeySideArgs a = args;
    extern __shared__ unsigned char smem_raw[];
    // align by pointer arithmetic (not an integer round trip) so accesses stay in the shared window
    unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    unsigned char* sXv = smem;                       // 2 panels                                   (32 KB)
    unsigned char* sUk = sXv + 2 * kPanelB;          // uk tile fp32, 2 panels                     (32 KB)
    unsigned char* sG = sUk + 2 * kPanelB;           // G tile fp32, 2 panels                      (32 KB)
    unsigned char* sUq = sG + 2 * kPanelB;           // uq tile fp32, 2 panels                     (32 KB)
    unsigned char* sQt = sUq + 2 * kPanelB;          // decayed uq, K-major A [128][64]: value, rounding residual (32 KB)
                                                     //   ... they also stage the output rows
    unsigned char* sKt = sQt + 2 * kPanelB;          // decayed uk, K-major / MN-major B [128][64]: value, residual (32 KB)
    unsigned char* sSb = sKt + 2 * kPanelB;          // state copy, K-major B [128 (channel)][64]: value, residual  (32 KB)
    Ctl* ctl = reinterpret_cast<Ctl*>(sSb + 2 * kPanelB);
    // (the masked A never goes through shared memory: it is rewritten in place in tensor memory as a bf16
    // high/low pair and read from there as the A operand of the intra-chunk product)

    const int tid = threadIdx.x, warp = tid >> 5, wq = warp & 3, half = (tid >> 7) & 1, row = tid & 127;
    const int sb = kHS * half;          // this thread's first slot
    const ScanSpan span = scan_span(blockIdx.x, a.H, a.T, a.nseg, a.tseg);
    const int bh = blockIdx.x, slice = blockIdx.y, b = span.b, h = span.h;
    const int d0 = slice * kDST;

    ctl_init<FIRST>(ctl, tid, warp);
    const uint32_t tmem = ctl->tmem_slot;
    const int nchunks = (span.t_end - span.t0 + kCT - 1) / kCT;
    auto chunk_t0 = [&](int it) { return span.t0 + (REV ? nchunks - 1 - it : it) * kCT; };

    if (warp == kComputeThreads / 32) {
        // =============================== issuing warp: TMA loads / stores and all MMAs
        if (elect_one()) {
            auto load_v = [&](int it) {
                const int t = chunk_t0(it);
                mbar_expect_tx(&ctl->bar_x, 2 * kPanelB);
                tma_load_4d(sXv, &mapV, &ctl->bar_x, d0, h, t, b);
                tma_load_4d(sXv + kPanelB, &mapV, &ctl->bar_x, d0 + 64, h, t, b);
            };
            auto load_kg = [&](int it) {
                const int t = chunk_t0(it);
                mbar_expect_tx(&ctl->bar_g[0], 4 * kPanelB);
                tma_load_4d(sUk, &mapUk, &ctl->bar_g[0], 0, h, t, b);
                tma_load_4d(sUk + kPanelB, &mapUk, &ctl->bar_g[0], 32, h, t, b);
                tma_load_4d(sG, &mapG, &ctl->bar_g[0], 0, h, t, b);
                tma_load_4d(sG + kPanelB, &mapG, &ctl->bar_g[0], 32, h, t, b);
            };
            auto load_q = [&](int it) {
                const int t = chunk_t0(it);
                mbar_expect_tx(&ctl->bar_w, 2 * kPanelB);
                tma_load_4d(sUq, &mapUq, &ctl->bar_w, 0, h, t, b);
                tma_load_4d(sUq + kPanelB, &mapUq, &ctl->bar_w, 32, h, t, b);
            };
            prefetch_tmap(&mapV); prefetch_tmap(&mapUq); prefetch_tmap(&mapUk); prefetch_tmap(&mapG); prefetch_tmap(&mapO);
            load_kg(0);
            load_q(0);
            load_v(0);
            constexpr uint32_t idescA = make_idesc(128, 128, false, false);   // Q~ K~^T
            constexpr uint32_t idescO = make_idesc(128, kDST, false, false);  // Q- x state copy (K-major B)
            constexpr uint32_t idescU = make_idesc(128, 2 * kM, true, true);  // xv^T (MN-major A) x [K-_hi | K-_lo] (MN-major B)
            constexpr uint32_t idescV = make_idesc(128, kDST, false, true);   // masked A (tensor memory) x xv (MN-major B)
            // base descriptors of every operand (K step 0); advancing along K is one add each
            const uint64_t dV = desc_mnmajor(smem_u32(sXv), 0, kPanelB);
            const uint64_t dQt = desc_kmajor(smem_u32(sQt), 0), dKt = desc_kmajor(smem_u32(sKt), 0);
            const uint64_t dQl = desc_kmajor(smem_u32(sQt + kPanelB), 0), dKl = desc_kmajor(smem_u32(sKt + kPanelB), 0);
            const uint64_t dS = desc_kmajor(smem_u32(sSb), 0), dSl = desc_kmajor(smem_u32(sSb + kPanelB), 0);
            // the decayed uk read MN-major, its value and residual as one N = 128 operand
            const uint64_t dKtm = desc_mnmajor(smem_u32(sKt), 0, kPanelB);
            auto kmaj = [](int kk) { return (uint32_t)((kk >> 2) * kPanelB + (kk & 3) * 32); };
            auto mnmaj = [](int kk) { return (uint32_t)(kk * 2048); };
            for (int it = 0; it < nchunks && !ctl->abort; ++it) {
                const int t0 = chunk_t0(it);
                WAIT_OR_ABORT(&ctl->bar_ops, it & 1);
                WAIT_OR_ABORT(&ctl->bar_x, it & 1);
                tc_fence_after_sync();
                const bool moderate = ctl->moderate[it & 1] != 0;
                if (moderate) {
                    // A = Q- K-^T with both factors as bf16 high/low pairs (the low x low term is dropped)
#pragma unroll
                    for (int kk = 0; kk < kM / 16; ++kk)
                        mma_bf16(tmem + kColP, desc_advance(dQt, kmaj(kk)), desc_advance(dKt, kmaj(kk)), idescA, kk > 0);
#pragma unroll
                    for (int kk = 0; kk < kM / 16; ++kk)
                        mma_bf16(tmem + kColP, desc_advance(dQl, kmaj(kk)), desc_advance(dKt, kmaj(kk)), idescA, true);
#pragma unroll
                    for (int kk = 0; kk < kM / 16; ++kk)
                        mma_bf16(tmem + kColP, desc_advance(dQt, kmaj(kk)), desc_advance(dKl, kmaj(kk)), idescA, true);
                    mma_commit(&ctl->bar_p);     // the state products below run under the read-out of A
                }
                // the decayed uk is read K-major by the intra product and MN-major by the state update
#pragma unroll
                for (int kk = 0; kk < kCT / 16; ++kk)
                    mma_bf16(tmem + kColU, desc_advance(dV, mnmaj(kk)), desc_advance(dKtm, mnmaj(kk)), idescU, kk > 0);
#pragma unroll
                for (int kk = 0; kk < kM / 16; ++kk)
                    mma_bf16(tmem + kColO, desc_advance(dQt, kmaj(kk)), desc_advance(dS, kmaj(kk)), idescO, kk > 0);
#pragma unroll
                for (int kk = 0; kk < kM / 16; ++kk)
                    mma_bf16(tmem + kColO, desc_advance(dQl, kmaj(kk)), desc_advance(dS, kmaj(kk)), idescO, true);
#pragma unroll
                for (int kk = 0; kk < kM / 16; ++kk)
                    mma_bf16(tmem + kColO, desc_advance(dQt, kmaj(kk)), desc_advance(dSl, kmaj(kk)), idescO, true);
                mma_commit(&ctl->bar_mma1);
                // a moderate chunk is done with the uk and G tiles: request the next chunk's
                if (moderate && it + 1 < nchunks) load_kg(it + 1);
                WAIT_OR_ABORT(&ctl->bar_pm, it & 1);
                tc_fence_after_sync();
#pragma unroll
                for (int kk = 0; kk < kCT / 16; ++kk)
                    mma_bf16_ta(tmem + kColO, tmem + kColP + 64 * (kk >> 2) + 8 * (kk & 3), desc_advance(dV, mnmaj(kk)), idescV,
                                true);
#pragma unroll
                for (int kk = 0; kk < kCT / 16; ++kk)      // ... and the rounding residual of A
                    mma_bf16_ta(tmem + kColO, tmem + kColP + 64 * (kk >> 2) + 32 + 8 * (kk & 3), desc_advance(dV, mnmaj(kk)),
                                idescV, true);
                mma_commit(&ctl->bar_mma2);
                if (!moderate && it + 1 < nchunks) load_kg(it + 1);
                // every product of the chunk is done: the uq and xv tiles may be refilled
                WAIT_OR_ABORT(&ctl->bar_mma2, it & 1);
                if (it + 1 < nchunks) {
                    load_q(it + 1);
                    load_v(it + 1);
                }
                // the output rows are staged over the intra operands: store them, then tell the
                // compute threads that those buffers may be rewritten
                WAIT_OR_ABORT(&ctl->bar_out, it & 1);
                if (ctl->abort) break;
                tma_store_4d(&mapO, sQt, d0, h, t0, b);
                if (d0 + 64 < a.D) tma_store_4d(&mapO, sQt + kPanelB, d0 + 64, h, t0, b);
                bulk_commit();
                bulk_wait_read();
                mbar_arrive(&ctl->bar_sb);
            }
        }
    } else if (tid < kComputeThreads) {
        // =============================== compute threads
        // state slice, transposed: S[c = row][s], slots sb .. sb+31
        float S[kHS];
#pragma unroll
        for (int s = 0; s < kHS; ++s) S[s] = (a.S0 && d0 + row < a.D) ? a.S0[((size_t)bh * kM + sb + s) * a.D + d0 + row] : 0.f;

        int n_mod = 0;     // moderate chunks so far (phases of bar_p)
        PROF_DECL
        for (int it = 0; it < nchunks; ++it) {
            const int t0 = chunk_t0(it);
            const int valid = min(kCT, span.t_end - t0);
            (void)t0;
            PROF_MARK();
            WAIT_OR_ABORT(&ctl->bar_g[0], it & 1);
            PROF_MARK();
            const bool moderate = publish_chunk_decay(ctl, tid, sG, valid - 1);
            if (ctl->abort) break;
            PROF_MARK();

            const int grow = min(row, valid - 1);
            // the previous chunk's output rows must have left sQt / sKt before they are rewritten
            if (it > 0) WAIT_OR_ABORT(&ctl->bar_sb, (it - 1) & 1);
            // key side first: it needs the uk and G tiles only; the uq tile (which shares its buffer
            // with the previous chunk's masked A) arrives last
#pragma unroll
            for (int s0 = sb; s0 < sb + kHS; s0 += 8) {
                float g[8], uk[8], kd[8], gcv[8];
                tile_row8(sG, grow, s0, g);
                tile_row8(sUk, row, s0, uk);
                // ONE decayed copy of uk serves the intra product and the state update, with one
                // exponential per element (the SFU is the scarce unit here) and no branch:
                //   reverse           : uk exp(G)
                //   forward, moderate : uk exp(-G); the state update gets its exp(G_C) afterwards,
                //                       S <- exp(G_C) (S + xv^T K)
                //   forward, strong   : uk exp(G_C - G) (state update only)
#pragma unroll
                for (int e = 0; e < 8; ++e) gcv[e] = 0.f;
                if (!REV && !moderate) tile_free_row8(&ctl->gc[s0], gcv);
#pragma unroll
                for (int e = 0; e < 8; ++e) kd[e] = uk[e] * __expf(REV ? g[e] : gcv[e] - g[e]);
                store_chunk_split(sKt, sKt + kPanelB, row, s0 >> 3, kd);
            }
            PROF_MARK();
            WAIT_OR_ABORT(&ctl->bar_w, it & 1);
            PROF_MARK();
#pragma unroll
            for (int s0 = sb; s0 < sb + kHS; s0 += 8) {
                float g[8], uq[8], qd[8], gcv[8];
                tile_row8(sG, grow, s0, g);
                tile_row8(sUq, row, s0, uq);
                // likewise ONE decayed copy of uq:
                //   forward           : uq exp(G)
                //   reverse, moderate : uq exp(-G); the inter-chunk product gets its exp(G_C) through
                //                       the state copy, which is scaled per slot
                //   reverse, strong   : uq exp(G_C - G)
#pragma unroll
                for (int e = 0; e < 8; ++e) gcv[e] = 0.f;
                if (REV && !moderate) tile_free_row8(&ctl->gc[s0], gcv);
#pragma unroll
                for (int e = 0; e < 8; ++e) qd[e] = uq[e] * __expf(REV ? gcv[e] - g[e] : g[e]);
                store_chunk_split(sQt, sQt + kPanelB, row, s0 >> 3, qd);
            }
            if (REV && moderate) store_state_row_split<true>(sSb, sSb + kPanelB, row, sb, S, ctl->egc);
            else store_state_row_split<false>(sSb, sSb + kPanelB, row, sb, S, nullptr);
            fence_async_smem();
            if (tid == 0) ctl->moderate[it & 1] = moderate;
            compute_sync();
            if (tid == 0) mbar_arrive(&ctl->bar_ops);
            PROF_MARK();

            if (moderate) {
                WAIT_OR_ABORT(&ctl->bar_p, n_mod & 1);
                ++n_mod;
                tc_fence_after_sync();
                PROF_MARK();
                mask_row_in_tmem<REV, true>(tmem, wq, row, half, kColP);
            } else {
                // strong decay: A_ij by the walk over the per-step gates
                key_side_explicit_rows<REV>(sG, sUq, sUk, tmem, wq, row, half, sb, valid);
                fence_async_smem();     // (gates and bands were written where the next tiles land)
            }
            tc_fence_before_sync();
            compute_sync();
            if (tid == 0) mbar_arrive(&ctl->bar_pm);
            PROF_MARK();

            // ---- state update from U^T: S <- exp(G_C) S + U^T  (forward moderate chunk: exp(G_C) (S + U^T))
            WAIT_OR_ABORT(&ctl->bar_mma1, it & 1);
            tc_fence_after_sync();
            PROF_MARK();
            {
                float v[kHS], vl[kHS];
                tmem_ld32(tmem_row_addr(tmem, wq, kColU + sb), v);
                tmem_ld32(tmem_row_addr(tmem, wq, kColU + kM + sb), vl);
#pragma unroll
                for (int e = 0; e < kHS; ++e) v[e] += vl[e];          // value + residual of the decayed uk
#pragma unroll
                for (int e = 0; e < kHS; e += 4) {
                    const float4 ec = *reinterpret_cast<const float4*>(&ctl->egc[sb + e]);
                    const float ecv[4] = {ec.x, ec.y, ec.z, ec.w};
#pragma unroll
                    for (int t = 0; t < 4; ++t)
                        S[e + t] = (!REV && moderate) ? (S[e + t] + v[e + t]) * ecv[t] : fmaf(S[e + t], ecv[t], v[e + t]);
                }
            }

            // ---- output rows -> bf16, staged over the intra operands (consumed since bar_p), stored
            // by the issuing warp, clipped at the sequence end
            PROF_MARK();
            WAIT_OR_ABORT(&ctl->bar_mma2, it & 1);
            tc_fence_after_sync();
            PROF_MARK();
#pragma unroll 1
            for (int c0 = 0; c0 < 64; c0 += 32) {
                float v[32];
                tmem_ld32(tmem_row_addr(tmem, wq, kColO + 64 * half + c0), v);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const float x[8] = {v[8 * c], v[8 * c + 1], v[8 * c + 2], v[8 * c + 3],
                                        v[8 * c + 4], v[8 * c + 5], v[8 * c + 6], v[8 * c + 7]};
                    store_chunk(sQt + half * kPanelB, row, (c0 >> 3) + c, x);
                }
            }
            fence_async_smem();
            tc_fence_before_sync();
            compute_sync();
            if (tid == 0) mbar_arrive(&ctl->bar_out);
            PROF_MARK();
            PROF_DUMP("key_side compute");
            if (ctl->abort) break;
        }
        if (!ctl->abort && a.Send && d0 + row < a.D) {
#pragma unroll
            for (int s = 0; s < kHS; ++s) a.Send[((size_t)bh * kM + sb + s) * a.D + d0 + row] = S[s];
        }
    }

    tc_fence_before_sync();
    __syncthreads();
    if (ctl->abort) {
        if (tid == 0 && dev_status != nullptr) *dev_status = GSA_ERR_TIMEOUT;
        for (int i = 0; i < 200; ++i) __nanosleep(1000);
    }
    __syncthreads();
    if (warp == 0) {
        __syncwarp();
        tmem_dealloc(tmem, kTmemCols);
    }
}

constexpr size_t kSmemGeneral = 1024 + 14 * kPanelB + sizeof(Ctl);

}  // namespace
}  // namespace gsa
