// The general versions of the two chunk primitives of Algorithm 1, for the (batch, head) pairs that hold a strong-decay
// chunk: any gates, from a = 1 to a = 0.  They are device functions: every scan is ONE launch of a pipelined kernel
// (chunk_tc_lean.cu, chunk_tc_pair.cu) whose CTAs come here when their pair is flagged.  As launches of their own
// they cost every scan a second launch, a side stream and four events, which is what bounded short calls: a forward over
// T = 300, 16 heads of 128, 59 us with them and 42 without; a training step of the 1.3B model's layer 481 and 466.
//
// The decay between two tokens of a 128-token chunk does not factorise around one reference point where the chunk forgets
// more than e^-60 (App. A: secondary chunking).  Here a CTA walks its scan in steps of kSub = 16 tokens, each with the state
// carried across it, and every decay factor that it forms is at most 1:
//   value side   out_i = e_i (xq_i S) + sum_j P_ij w_j prod a_r,      S <- e_last S + xk^T (w_j s_j)
//   key side     out_i = (uq_i e_i) S + sum_j A_ij xv_j,              S <- e_last S + (uk_j s_j)^T xv
// with e_i the decay from the step's start through token i and s_j that from j to its end (time-reversed: e and s swap).  (On the key
// side one operand of A is lifted by up to e^60, see step_weights; slots that keep most of a chunk take the decay once a
// chunk, with factors of up to e^0.5 on the rows until then, see step_frame.)
// tcgen05, whose products have 128 (64) rows, would do four times the work of a 16-token step and a commit and a wait per
// step on top, so the products are warp-level ones (mma.sync m16n8k16: 8.3 cycles each; 96 a state warp and step on the value
// side, 88 on the key side).  What bounds it: a state warp's chain of splits and products, 2300 and 1760 cycles a step of which it
// waits for 180 and 100 (the slot warps are ahead; the tensor pipe is 35 and 40% active, 0.40 and 0.38 instructions a cycle
// and scheduler).  32 K tokens, 16 heads of 128, a = sigmoid(N(-2, 1)): pass 1 486 -> 290 us, pass 2 410 -> 237 (HBM's share of either:
// 105), state runs 205 -> 82, the forward 1285 -> 763.  The scans before these took 128-token chunks on tcgen05 and walked the
// decay row by row, 28 k cycles a chunk.
//
// Warps of two roles, meeting on mbarriers only:
//   * four slot warps take the steps in turn: a step's rows by TMA, asked for one of a warp's steps ahead (by 16-byte asynchronous
//     copies of all lanes the warps were held up for 40 cycles a copy, 1400 a step); decay factors, a lane two slots; decayed
//     operand rows as three bf16 parts (value side, whose outputs are fp32) or high/low pairs; the intra-step term (value side: P by mma, then running decay products in fp32; key
//     side: A by mma); at the end the output rows;
//   * four state warps take every step: the state (value side: 16 slots x 128 channels a warp, key side: 32 channels x
//     64 slots) stays in registers in fp32, in the fragment layout that serves as the next product's operand as it stands.  On the
//     value side in packed sequences eight, half of the channels each: 1830 cycles a step, a training step on 8 K tokens of 13
//     sequences, 4 heads of 512, 663 -> 624 us.  All calls with twelve warps: the forward above 716 us, but calls without a flagged
//     pair are slower (see kPackedThreads).  Six, the last quarter of the channels by two warps that are idle otherwise: 780, their schedulers
//     hold the others up.  (With high/low pairs, 208 us, and on the key side, 252, eight were no faster than four; splits
//     and decays moved by hand behind other blocks' products: 209 and 250.)
// Every wait is bounded: on expiry the CTA flags dev_status, runs out without waiting and returns.
#pragma once
#include "chunk_tc_shared.cuh"

namespace gsa {
namespace {
using namespace tc;
using namespace tcchunk;

// The rows of 1 - a of a flagged pair's moderate chunks, as the gate kernel forms them, where it has left them out
// (InputGate).  Every CTA that is about to read them writes them all -- the same values -- and reads its own.  A warp a chunk.
// (All chunks, strong ones too: 32 K tokens of strong logits, 16 heads, 806 -> 948 us, of log gates 782 -> 883.)
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

constexpr int kSub = 16;               // tokens of a step
constexpr int kStages = 8;             // steps whose rows are on their way or in use
constexpr int kStateWarps = 4, kSlotWarps = 4;       // one of each to a scheduler (value side, kPackedThreads: two and one)
static_assert(kScanThreads >= 32 * (kStateWarps + kSlotWarps) && kPackedThreads == 32 * (2 * kStateWarps + kSlotWarps) && kStages == 2 * kSlotWarps, "");
// tiles of a step, by TMA: two panels of [16 rows][128 bytes] with the 128-byte swizzle (128 channels in bf16, 64 slots in fp32)
constexpr int kStepPanel = kSub * 128, kXTile = 2 * kStepPanel, kSlotTile = 2 * kStepPanel;
// rows that the warps write, in bytes: eight rows 16 bytes apart modulo 128 meet in no bank
constexpr int kDecRow = 2 * kM + 16;   // 64 slots, bf16
constexpr int kORow = 4 * kM + 16;     // 64 slots, fp32, written by columns
constexpr int kOutRow = 2 * kDST + 16; // 128 channels, bf16
constexpr int kDecTile = kSub * kDecRow;
constexpr int kPRow = 8 * kSub + 16;   // value side: a row of P, every value twice (both slots of a lane)
constexpr int kARow = 2 * kSub + 16;   // key side: a row of A, bf16

struct GeneralCtl {
    uint64_t full[kStages];            // (TMA) the rows of a step have landed
    uint64_t ready[kSlotWarps];        // (slot warp) decayed rows and total decay of its step are in shared memory, key side: and A
    uint64_t done[kSlotWarps];         // (state warps) a slot warp's step has been taken: all its rows may be written again,
                                       // value side: the inter-step product is in shared memory, key side: the output rows
    volatile int abort;
};

// A wait that expires flags the CTA; once flagged, later waits that are not over return at once and the roles run out.
__device__ __forceinline__ void general_wait(GeneralCtl* ctl, uint64_t* bar, uint32_t parity) {
    if (!mbar_try(bar, parity) && !ctl->abort && !mbar_wait(bar, parity)) ctl->abort = 1;
    __syncwarp();
}

__device__ __forceinline__ void general_ctl_init(GeneralCtl* ctl, int tid, int state_warps) {
    if (tid == 0) {
        for (int i = 0; i < kStages; ++i) mbar_init(&ctl->full[i], 1);
        for (int i = 0; i < kSlotWarps; ++i) {
            mbar_init(&ctl->ready[i], 1);
            mbar_init(&ctl->done[i], state_warps);
        }
        ctl->abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
}
// Ends a scan: its barriers' memory may be used again.  Returns whether all went well.
__device__ __forceinline__ bool general_finish(GeneralCtl* ctl, int tid, int32_t* dev_status) {
    __syncthreads();
    const bool fine = ctl->abort == 0;
    if (!fine)         // bounded grace period for tile copies still in flight before shared memory goes away
        for (int i = 0; i < 200; ++i) __nanosleep(1000);
    if (tid == 0) {
        if (!fine && dev_status != nullptr) *dev_status = GSA_ERR_TIMEOUT;
        for (int i = 0; i < kStages; ++i) mbar_inval(&ctl->full[i]);
        for (int i = 0; i < kSlotWarps; ++i) { mbar_inval(&ctl->ready[i]); mbar_inval(&ctl->done[i]); }
    }
    __syncthreads();
    return fine;
}
__device__ __forceinline__ void warp_arrive(uint64_t* bar, int lane) {
    __syncwarp();
    if (lane == 0) mbar_arrive(bar);
}

// ---- warp-level building blocks
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldsm4_trans(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void stsm4_trans(uint32_t addr, uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3) {
    asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(r0), "r"(r1), "r"(r2), "r"(r3)
                 : "memory");
}
// c += a b: m16n8k16
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// a lane's two slots: packed fp32 arithmetic (half the issue slots)
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float x, float y) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ f32x2 both(float x) { return pack2(x, x); }
__device__ __forceinline__ float2 unpack2(f32x2 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
// two values as a bf16 high/low pair
__device__ __forceinline__ void split_pair(float x0, float x1, uint32_t& hi, uint32_t& lo) {
    hi = pack_bf16(x0, x1);
    const float2 rest = unpack2(sub2(pack2(x0, x1), pack2(__uint_as_float(hi << 16), __uint_as_float(hi & 0xffff0000u))));
    lo = pack_bf16(rest.x, rest.y);
}
// ... as three bf16 parts by truncation, which hold all 24 bits: no conversions, which go at half the rate
__device__ __forceinline__ uint32_t upper_halves(float x0, float x1) {
    return __byte_perm(__float_as_uint(x0), __float_as_uint(x1), 0x7632);
}
__device__ __forceinline__ f32x2 below_upper_halves(float x0, float x1) {
    return sub2(pack2(x0, x1), pack2(__uint_as_float(__float_as_uint(x0) & 0xffff0000u), __uint_as_float(__float_as_uint(x1) & 0xffff0000u)));
}
__device__ __forceinline__ void split_triple(float x0, float x1, uint32_t (&part)[3]) {
    part[0] = upper_halves(x0, x1);
    float2 r = unpack2(below_upper_halves(x0, x1));
    part[1] = upper_halves(r.x, r.y);
    r = unpack2(below_upper_halves(r.x, r.y));
    part[2] = upper_halves(r.x, r.y);
}
// s = s dec + u of both
__device__ __forceinline__ void decay_add(float& s0, float& s1, f32x2 dec, float u0, float u1) {
    const float2 v = unpack2(fma2(pack2(s0, s1), dec, pack2(u0, u1)));
    s0 = v.x;
    s1 = v.y;
}
// exp of a log-decay difference to - from <= 0 of both slots
__device__ __forceinline__ f32x2 decay2(float2 from, float2 to) { return pack2(exp_neg(from.x - to.x), exp_neg(from.y - to.y)); }
// kBatch tokens at a time, operation by operation: the chains of a token then overlap (token by token the compiler leaves
// them one behind the other, 35 cycles each)
constexpr int kBatch = 8;
// two slots of decayed rows row0 .. row0 + kBatch - 1 as a high/low pair, or as three parts, a tile each
template <int PARTS>
__device__ __forceinline__ void store_parts(unsigned char* tile, int row0, int lane, const f32x2 (&v)[kBatch]) {
    static_assert(PARTS == 2 || PARTS == 3, "");
    uint32_t part[PARTS][kBatch];
    float2 x[kBatch];
#pragma unroll
    for (int j = 0; j < kBatch; ++j) x[j] = unpack2(v[j]);
    if constexpr (PARTS == 2) {
#pragma unroll
        for (int j = 0; j < kBatch; ++j) part[0][j] = pack_bf16(x[j].x, x[j].y);
#pragma unroll
        for (int j = 0; j < kBatch; ++j)
            x[j] = unpack2(sub2(v[j], pack2(__uint_as_float(part[0][j] << 16), __uint_as_float(part[0][j] & 0xffff0000u))));
#pragma unroll
        for (int j = 0; j < kBatch; ++j) part[1][j] = pack_bf16(x[j].x, x[j].y);
    } else {
#pragma unroll
        for (int i = 0; i < PARTS; ++i) {
#pragma unroll
            for (int j = 0; j < kBatch; ++j) part[i][j] = upper_halves(x[j].x, x[j].y);
            if (i + 1 < PARTS) {
#pragma unroll
                for (int j = 0; j < kBatch; ++j) x[j] = unpack2(below_upper_halves(x[j].x, x[j].y));
            }
        }
    }
    uint32_t* p = reinterpret_cast<uint32_t*>(tile + row0 * kDecRow) + lane;
#pragma unroll
    for (int j = 0; j < kBatch; ++j)
#pragma unroll
        for (int i = 0; i < PARTS; ++i) p[j * (kDecRow / 4) + i * (kDecTile / 4)] = part[i][j];
}
// a lane's two slots of a row of a slot-sized tile
__device__ __forceinline__ f32x2 slots2(const unsigned char* tile, int row, int lane) {
    const uint32_t at = (lane >> 4) * kStepPanel + ((lane & 15) >> 1) * 16 + (lane & 1) * 8;
    return *reinterpret_cast<const f32x2*>(tile + row * 128 + (at ^ ((row & 7) << 4)));
}
// ... of one that holds a where 1 - a is meant
__device__ __forceinline__ f32x2 weights2(const unsigned char* tile, int row, int lane, bool keeps) {
    const f32x2 x = slots2(tile, row, lane);
    return keeps ? sub2(pack2(1.f, 1.f), x) : x;
}
// where 8 channels of a row of a d-sized tile are: 16-byte piece `piece` of 16
__device__ __forceinline__ uint32_t x_at(uint32_t tile, int row, int piece) {
    return tile + (piece >> 3) * kStepPanel + row * 128 + (((piece & 7) ^ (row & 7)) << 4);
}

// Which steps a scan takes: step n works on tokens [t, t + 16) from token() on; forward in order, reversed from the last one.
struct Steps {
    int t0, t_end, first, count;       // steps first .. first + count - 1 of the span
    template <bool REV> __device__ __forceinline__ int token(int n) const {
        return t0 + kSub * (first + (REV ? count - 1 - n : n));
    }
    // (a 128-token chunk, which G is local to, begins here)
    __device__ __forceinline__ bool chunk_start(int t) const { return (t - t0) % kCT == 0; }
    // the scan leaves a chunk with this step
    template <bool REV> __device__ __forceinline__ bool chunk_ends(int t) const { return REV ? chunk_start(t) : chunk_start(t + kSub) || t + kSub >= t_end; }
};
__device__ __forceinline__ Steps all_steps(const ScanSpan& s) { return {s.t0, s.t_end, 0, (s.t_end - s.t0 + kSub - 1) / kSub}; }

// End memories need only the chunks from which anything is left: with gates that forget within a dozen tokens, all but one chunk of
// the span.  What every slot's decay carries below 2^-150 on the way to the span's end (reversed: its start) can change nothing
// in fp32, whatever follows.  A memory whose weights are 1 - a is at most as large as the largest row, whose bound is 2^17: e^-130.
// Reversed, with rows and weights below 2^17, it is below 2^65 for any T: e^-150.  An infinity, a NaN or a number beyond the
// bound stays in the memories however hard they forget, or may, so the rows left out are looked through first, and where one of
// them is found nothing is left out.  32 K tokens of such gates, 16 heads of 128, state runs 31 us without the look, 82 with, 220
// walking all.
template <bool REV> constexpr float kForgotten = REV ? -150.f : -130.f;
// Every warp comes to the same result by itself.
template <bool REV> __device__ __forceinline__ Steps last_steps(const ValueSideArgs& a, const ScanSpan& span, int lane) {
    Steps s = all_steps(span);
    const int chunks = (span.t_end - span.t0 + kCT - 1) / kCT;
    constexpr int kBatch = 4;
    float2 sum = make_float2(0.f, 0.f);
    int kept = 0;
    for (int c0 = 0; c0 < chunks && kept == 0; c0 += kBatch) {
        float2 g[kBatch];
#pragma unroll
        for (int q = 0; q < kBatch; ++q) {
            const int c = min(c0 + q, chunks - 1), n = REV ? c : chunks - 1 - c;
            const int last = min(span.t0 + (n + 1) * kCT, span.t_end) - 1;
            g[q] = *reinterpret_cast<const float2*>(a.G + (((size_t)span.b * a.T + last) * a.H + span.h) * kM + 2 * lane);
        }
#pragma unroll
        for (int q = 0; q < kBatch; ++q) {
            if (kept != 0 || c0 + q >= chunks) continue;
            sum.x += g[q].x;
            sum.y += g[q].y;
            if (__all_sync(0xffffffffu, fmaxf(sum.x, sum.y) < kForgotten<REV>)) kept = c0 + q + 1;
        }
    }
    if (kept == 0 || kept == chunks) return s;
    const int steps = kept * (kCT / kSub);
    if (REV) {
        s.count = steps;
    } else {
        s.first = (chunks - kept) * (kCT / kSub);
        s.count -= s.first;
    }
    return s;
}

// (read once: not into the little that is left of L1 beside the scans' shared memory)
__device__ __forceinline__ uint4 load_once(const void* p) {
    uint4 v;
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
// The steps of a state run.  All threads call it; BOTH: of two sets at once.  Whether a weight 1 - a is not below 2 the gate kernel has
// seen (`large`); reversed the weights are looked through here.
template <bool REV, bool BOTH>
__device__ __noinline__ Steps remembered_steps(const ValueSideArgs& a, const ValueSideArgs& b, int slice, bool large) {
    const ScanSpan span = scan_span(blockIdx.x, a.H, a.T, a.nseg, a.tseg);
    const Steps all = all_steps(span), kept = last_steps<REV>(a, span, threadIdx.x & 31);
    if (kept.count == all.count || large) return all;
    // sixteen threads a row: eight channels and four slots each
    constexpr int kBatch = 8, kRows = kScanThreads / 16, kSets = BOTH ? 2 : 1;
    const int t_lo = REV ? span.t0 + kSub * kept.count : span.t0, t_hi = REV ? span.t_end : span.t0 + kSub * kept.first;
    const int piece = threadIdx.x & 15;
    // (a magnitude of 2^17 or more, or no finite number, has bits from 0x4800 on and carries into the place of the sign)
    uint32_t rows_seen = 0, weights_seen = 0;
    for (int t0 = t_lo + (int)(threadIdx.x >> 4); t0 < t_hi; t0 += kBatch * kRows) {
        uint4 x[kSets][kBatch], w[kBatch];
#pragma unroll
        for (int q = 0; q < kBatch; ++q) {
            const size_t row = ((size_t)span.b * a.T + min(t0 + q * kRows, t_hi - 1)) * a.H + span.h;
            w[q] = REV ? load_once(a.w + row * kM + 4 * piece) : make_uint4(0, 0, 0, 0);
#pragma unroll
            for (int i = 0; i < kSets; ++i) {
                const ValueSideArgs& set = i == 0 ? a : b;
                const int c = slice * kDST + 8 * piece;
                x[i][q] = c < set.D ? load_once(static_cast<const __nv_bfloat16*>(set.xk) + row * set.D + c) : make_uint4(0, 0, 0, 0);
            }
        }
#pragma unroll
        for (int q = 0; q < kBatch; ++q) {
            if (REV) {
                const uint32_t words[4] = {w[q].x, w[q].y, w[q].z, w[q].w};
#pragma unroll
                for (int e = 0; e < 4; ++e) weights_seen |= (words[e] & 0x7fffffffu) + 0x38000000u;
            }
#pragma unroll
            for (int i = 0; i < kSets; ++i) {
                const uint32_t pairs[4] = {x[i][q].x, x[i][q].y, x[i][q].z, x[i][q].w};
#pragma unroll
                for (int e = 0; e < 4; ++e) rows_seen |= (pairs[e] & 0x7fff7fffu) + 0x38003800u;
            }
        }
    }
    return __syncthreads_or((rows_seen & 0x80008000u) | (weights_seen & 0x80000000u)) ? all : kept;
}

// A slot warp's copies: the rows of step n into its stage.  A stage's tiles, in this order: NX d-sized ones (128 channels from
// d0 on, those past D zero), NS slot-sized ones, then G.  Rows past the end of T are zeros (a span ends there or at a whole chunk).
struct StepMaps { const CUtensorMap *x[2], *s[2], *G; };
template <bool REV, int NX, int NS>
__device__ __forceinline__ void load_step(GeneralCtl* ctl, unsigned char* ring, const StepMaps& maps, const Steps& steps,
                                          const ScanSpan& span, int d0, int n) {
    if (n >= steps.count) return;
    if (elect_one()) {
        const int st = n % kStages, t = steps.token<REV>(n);
        uint64_t* bar = &ctl->full[st];
        unsigned char* dst = ring + st * (NX * kXTile + (NS + 1) * kSlotTile);
        mbar_expect_tx(bar, NX * kXTile + (NS + 1) * kSlotTile);
#pragma unroll
        for (int i = 0; i < NX; ++i, dst += kXTile) {
            tma_load_4d(dst, maps.x[i], bar, d0, span.h, t, span.b);
            tma_load_4d(dst + kStepPanel, maps.x[i], bar, d0 + 64, span.h, t, span.b);
        }
#pragma unroll
        for (int i = 0; i <= NS; ++i, dst += kSlotTile) {
            const CUtensorMap* map = i < NS ? maps.s[i] : maps.G;
            tma_load_4d(dst, map, bar, 0, span.h, t, span.b);
            tma_load_4d(dst + kStepPanel, map, bar, 32, span.h, t, span.b);
        }
    }
    __syncwarp();
}
// G around step n, this lane's two slots: of the token before it (0 at the start of a 128-token chunk, which G is local to), and of
// the chunk's last one
struct StepBounds { float2 before, chunk_end; };
template <bool REV>
__device__ __forceinline__ StepBounds step_bounds(const float* G, const Steps& steps, const ScanSpan& span, int T, int H, int n, int lane) {
    StepBounds s{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    if (n >= steps.count) return s;
    const int t = steps.token<REV>(n), end = min(t + kCT - (t - span.t0) % kCT, span.t_end) - 1;
    const float* row = G + (((size_t)span.b * T + t) * H + span.h) * kM + 2 * lane;
    if (!steps.chunk_start(t)) s.before = *reinterpret_cast<const float2*>(row - (size_t)H * kM);
    s.chunk_end = *reinterpret_cast<const float2*>(row + (size_t)(end - t) * H * kM);
    return s;
}
// What the state takes once every step it rounds once every step, and for slots that keep nearly all the errors of thousands of steps
// add up; nor are they random: gates near 1 are multiples of 2^-24, and from such a decay rounding always leaves out the same square.
// So the memory of a slot that keeps e^-0.5 of a chunk or more stays in the frame of the chunk's start (reversed: end) and takes the
// decay with the chunk's last step, all of it; until then the factors of the step's rows bridge the difference.  Final memories
// of 16 K tokens, slots that keep e^-0.08 of them, a in fp32, rms error 8.2e-6 without, 8.7e-7 so.
struct StepFrame {
    f32x2 out, weight;                 // on the output's factors (value side: of the inter-step product; key side: of uq), on those of the weights (uk)
    f32x2 total, inverse;              // what the state decays by, and 1 / total
};
__device__ __forceinline__ float frame_decay(float g) {            // exp(g), g <= 0; near 0 a Taylor polynomial (2^-27), 1 at 0
    const float p = fmaf(g, fmaf(g, fmaf(g, fmaf(g, fmaf(g, 1.f / 120.f, 1.f / 24.f), 1.f / 6.f), 0.5f), 1.f), 1.f);
    return g > -0.125f ? p : exp_neg(-g);
}
template <bool REV>
__device__ __forceinline__ StepFrame step_frame(const StepBounds& s, float2 last, bool chunk_ends) {
    float out[2], weight[2], total[2], inverse[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const float before = e ? s.before.y : s.before.x, l = e ? last.y : last.x, end = e ? s.chunk_end.y : s.chunk_end.x;
        const bool framed = end > -0.5f;
        const float lt = framed ? (chunk_ends ? end : 0.f) : l - before;
        out[e] = exp_neg(framed ? (REV ? l - end : -before) : 0.f);
        weight[e] = exp_neg(framed && !chunk_ends ? (REV ? end - before : l) : 0.f);
        total[e] = frame_decay(lt);
        inverse[e] = exp_neg(lt);
    }
    return {pack2(out[0], out[1]), pack2(weight[0], weight[1]), pack2(total[0], total[1]), pack2(inverse[0], inverse[1])};
}
// this lane's two slots of G on the step's rows; past the end as on the last row (a gate of 1)
__device__ __forceinline__ void step_gates(float2 (&g)[kSub], const unsigned char* tile, int rows, int lane) {
#pragma unroll
    for (int j = 0; j < kSub; ++j) g[j] = unpack2(slots2(tile, j, lane));
    if (rows < kSub) {
#pragma unroll
        for (int j = 1; j < kSub; ++j) g[j] = j < rows ? g[j] : g[j - 1];
    }
}

// ======================================================================================
// value_side: out_i[s] = sum_{j<=i} <xq_i, xk_j> w_j[s] decay_ij[s]  + decayed (xq_i S)[s]
// ======================================================================================
// A slot warp's shared memory: the decayed weights w_j s_j [16][64] in three parts, the step's total decay, the inter-step
// product [16][64] from the state warps (two sums), P.  (The outputs are fp32, and what a step takes from the one before it is not small beside
// its own: with high/low pairs of the weights and of the state the gate gradient of gates sigmoid(N(0, 1)), 2048 tokens, is 2.0e-5 off
// (rms), with three parts 3.5e-6; of sigmoid(N(-2, 1)) 2.1e-5 and 1.0e-5.  Pass 1 of the 32 K tokens above takes 208 us with pairs.)
constexpr int kParts = 3;              // of the decayed weights, and of the state as the output's operand
constexpr int kValueTotal = kParts * kDecTile, kValueO = kValueTotal + 4 * kM, kValueP = kValueO + 2 * kSub * kORow;
constexpr int kValueSlotB = kValueP + kSub * kPRow;
constexpr int kValueStageB = 2 * kXTile + 2 * kSlotTile, kValueStateStageB = kXTile + 2 * kSlotTile;

// P = xq xk^T of a step, every value twice, into `out` (rows of kPRow bytes)
__device__ __forceinline__ void step_scores(uint32_t xq, uint32_t xk, unsigned char* out, int lane) {
    float p[2][2][4] = {};             // [keys 8 n ..][channels: even, odd blocks of 16]
    const int q = lane >> 3, r = lane & 7;
#pragma unroll
    for (int kk = 0; kk < kDST / 16; ++kk) {
        uint32_t fa[4], fb[4];
        // A: rows 0-7, 8-15 of both channel halves; B: both channel halves of keys 0-7, 8-15
        ldsm4(fa, x_at(xq, (q & 1) * 8 + r, 2 * kk + (q >> 1)));
        ldsm4(fb, x_at(xk, (q >> 1) * 8 + r, 2 * kk + (q & 1)));
        mma16816(p[0][kk & 1], fa, fb[0], fb[1]);
        mma16816(p[1][kk & 1], fa, fb[2], fb[3]);
    }
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int e = 0; e < 4; e += 2) {
            const float x = p[n][0][e] + p[n][1][e], y = p[n][0][e + 1] + p[n][1][e + 1];
            *reinterpret_cast<float4*>(out + (g + 4 * e) * kPRow + 64 * n + 16 * t) = make_float4(x, x, y, y);
        }
}

// A state warp: 16 slots, of the channels of NKB blocks of 16 (all, or half number `half`), as accumulator tiles S^T [16 slots][8
// channels].
template <bool STATES, int NKB>
__device__ __forceinline__ void value_state_warp(GeneralCtl* ctl, unsigned char* ring, unsigned char* slots, const ValueSideArgs& a, const Steps& steps, int d0,
                                                 int group, int half, int lane) {
    constexpr int kTiles = 2 * NKB, kStageB = STATES ? kValueStateStageB : kValueStageB;
    const int s0 = 16 * group, c0 = d0 + 16 * NKB * half, g = lane >> 2, t = lane & 3, q = lane >> 3, r = lane & 7;
    const size_t state = ((size_t)blockIdx.x * kM + s0 + g) * a.D + c0 + 2 * t;
    float S[kTiles][4];
#pragma unroll
    for (int nt = 0; nt < kTiles; ++nt)
#pragma unroll
        for (int e = 0; e < 4; e += 2) {
            float2 x = make_float2(0.f, 0.f);
            if (!STATES && c0 + 8 * nt < a.D && a.S0 != nullptr) x = *reinterpret_cast<const float2*>(a.S0 + state + (size_t)4 * e * a.D + 8 * nt);
            S[nt][e] = x.x;
            S[nt][e + 1] = x.y;
        }
    // the fragments' places in the tiles: channels 16 kb, 16 kb + 8
    uint32_t at_q[NKB], at_k[NKB];
#pragma unroll
    for (int kb = 0; kb < NKB; ++kb) {
        at_q[kb] = x_at(0, (q >> 1) * 8 + r, 2 * (NKB * half + kb) + (q & 1));
        at_k[kb] = x_at(0, (q & 1) * 8 + r, 2 * (NKB * half + kb) + (q >> 1));
    }
    bool ready = false;
    for (int n = 0; n < steps.count; ++n) {
        const int st = n % kStages, w = n % kSlotWarps;
        unsigned char* tile = ring + st * kStageB;
        unsigned char* theirs = slots + w * kValueSlotB;
        // (the slot warp has seen the rows land before it says that its own are ready)
        if (!ready) general_wait(ctl, &ctl->ready[w], (n / kSlotWarps) & 1);
        // W^T (rows: slots, k: tokens); xq (k: channels, columns: tokens); xk (k: tokens, columns: channels)
        uint32_t wp[kParts][4], x[2][4], y[2][4];
        const uint32_t wa = smem_u32(theirs) + ((q >> 1) * 8 + r) * kDecRow + 2 * (s0 + (q & 1) * 8);
        const uint32_t qa = smem_u32(tile), ka = smem_u32(tile + (STATES ? 0 : kXTile));
        if (!STATES) ldsm4(x[0], qa + at_q[0]);
        ldsm4_trans(y[0], ka + at_k[0]);
#pragma unroll
        for (int i = kParts - 1; i >= 0; --i) ldsm4_trans(wp[i], wa + i * kDecTile);
        const float* total = reinterpret_cast<const float*>(theirs + kValueTotal) + s0 + g;
        const f32x2 dec[2] = {both(total[0]), both(total[8])};
        float O[2][2][4] = {};     // [tokens 8 n ..][upper part of the state, the others]
#pragma unroll
        for (int kb = 0; kb < NKB; ++kb) {
            const uint32_t (&xb)[4] = x[kb & 1], (&yb)[4] = y[kb & 1];
            uint32_t sp[kParts][4];
            if (!STATES) {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float (&f)[4] = S[2 * kb + (e >> 1)];
                    uint32_t part[kParts];
                    split_triple(f[2 * (e & 1)], f[2 * (e & 1) + 1], part);
#pragma unroll
                    for (int i = 0; i < kParts; ++i) sp[i][e] = part[i];
                }
            }
            if (kb + 1 < NKB) {
                if (!STATES) ldsm4(x[(kb + 1) & 1], qa + at_q[kb + 1]);
                ldsm4_trans(y[(kb + 1) & 1], ka + at_k[kb + 1]);
            }
            float U[2][4] = {};
#pragma unroll
            for (int i = kParts - 1; i >= 0; --i) {
                mma16816(U[0], wp[i], yb[0], yb[1]);
                mma16816(U[1], wp[i], yb[2], yb[3]);
                if (!STATES) {
                    mma16816(O[0][i > 0], sp[i], xb[0], xb[1]);
                    mma16816(O[1][i > 0], sp[i], xb[2], xb[3]);
                }
            }
            // (is the next step's there? asked while the products run)
            if (kb == 2) ready = n + 1 < steps.count && __all_sync(0xffffffffu, mbar_try(&ctl->ready[(n + 1) % kSlotWarps], ((n + 1) / kSlotWarps) & 1));
#pragma unroll
            for (int nn = 0; nn < 2; ++nn)
#pragma unroll
                for (int e = 0; e < 4; e += 2) decay_add(S[2 * kb + nn][e], S[2 * kb + nn][e + 1], dec[e >> 1], U[nn][e], U[nn][e + 1]);
        }
        if (!STATES) {
            // (columns of the product are tokens: rows of kORow bytes 8 banks apart)
            float* o = reinterpret_cast<float*>(theirs + kValueO + half * kSub * kORow) + s0 + g;
#pragma unroll
            for (int nn = 0; nn < 2; ++nn)
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    o[(8 * nn + 2 * t + (e & 1)) * (kORow / 4) + 8 * (e >> 1)] = O[nn][0][e] + O[nn][1][e];
        }
        warp_arrive(&ctl->done[w], lane);
    }
    if (!ctl->abort && a.Send != nullptr) {           // (channels past D are zeros throughout and not written)
#pragma unroll
        for (int nt = 0; nt < kTiles; ++nt)
#pragma unroll
            for (int e = 0; e < 4; e += 2)
                if (c0 + 8 * nt < a.D) *reinterpret_cast<float2*>(a.Send + state + (size_t)4 * e * a.D + 8 * nt) = make_float2(S[nt][e], S[nt][e + 1]);
    }
}

// STATES: end memories only (from empty ones), of the steps given.
template <bool REV, bool STATES = false>
__device__ __noinline__ bool value_side_general(const StepMaps maps, const ValueSideArgs& args, int32_t* dev_status, int slice, Steps given = {}) {
    // (a copy: through the reference every field would be read again after each barrier)
    const ValueSideArgs a = args;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* ring = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    constexpr int kStageB = STATES ? kValueStateStageB : kValueStageB;
    unsigned char* slots = ring + kStages * kStageB;                  // of the slot warps
    GeneralCtl* ctl = reinterpret_cast<GeneralCtl*>(slots + kSlotWarps * kValueSlotB);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const ScanSpan span = scan_span(blockIdx.x, a.H, a.T, a.nseg, a.tseg);
    const int d0 = slice * kDST;
    const Steps steps = STATES ? given : all_steps(span);
    // twice the state warps, half of the channels each
    const bool halves = !STATES && blockDim.x == kPackedThreads;
    general_ctl_init(ctl, tid, halves ? 2 * kStateWarps : kStateWarps);

    if (warp >= kStateWarps && warp < kStateWarps + kSlotWarps) {
        // =============================== slot warps: lane l has slots 2 l and 2 l + 1
        const int w = warp - kStateWarps;
        unsigned char* mine = slots + w * kValueSlotB;
        float* obase = STATES ? nullptr : a.out + (size_t)slice * a.B * a.T * a.H * kM + 2 * lane;
        load_step<REV, STATES ? 1 : 2, 1>(ctl, ring, maps, steps, span, d0, w);
        StepBounds next = step_bounds<REV>(a.G, steps, span, a.T, a.H, w, lane);
        for (int n = w; n < steps.count; n += kSlotWarps) {
            const int st = n % kStages, use = n / kSlotWarps;
            unsigned char* tile = ring + st * kStageB;
            const unsigned char *weights = tile + (STATES ? 1 : 2) * kXTile, *gates = weights + kSlotTile;
            general_wait(ctl, &ctl->full[st], (n / kStages) & 1);
            f32x2 E[kSub];                                           // w_j, later times the decay between j and i
            float2 g[kSub];
            const float2 before = next.before;
            step_gates(g, gates, span.t_end - steps.token<REV>(n), lane);
            const StepFrame frame = step_frame<REV>(next, g[kSub - 1], steps.chunk_ends<REV>(steps.token<REV>(n)));
#pragma unroll
            for (int j = 0; j < kSub; ++j) E[j] = weights2(weights, j, lane, a.w_keeps != 0);
            // decayed weights, total decay: what the state warps wait for
            f32x2 gate[kSub];                                        // the gates, whose products the factors within a step are
#pragma unroll
            for (int j = 0; j < kSub; ++j) gate[j] = decay2(j > 0 ? g[j - 1] : before, g[j]);
            f32x2 run = REV ? mul2(gate[0], frame.weight) : frame.weight;
#pragma unroll
            for (int i0 = 0; i0 < kSub; i0 += kBatch) {
                const int j0 = REV ? i0 : kSub - kBatch - i0;
                f32x2 f[kBatch];
#pragma unroll
                for (int i = 0; i < kBatch; ++i) {
                    const int j = REV ? i : kBatch - 1 - i, next = REV ? j0 + j + 1 : j0 + j;
                    f[j] = run;
                    if (next < kSub) run = mul2(run, gate[next]);
                }
#pragma unroll
                for (int j = 0; j < kBatch; ++j) f[j] = mul2(E[j0 + j], f[j]);
                store_parts<kParts>(mine, j0, lane, f);
            }
            *reinterpret_cast<f32x2*>(mine + kValueTotal + 8 * lane) = frame.total;
            warp_arrive(&ctl->ready[w], lane);
            // (the stage of this warp's next step: all are done with the step that it held, the one before this)
            load_step<REV, STATES ? 1 : 2, 1>(ctl, ring, maps, steps, span, d0, n + kSlotWarps);
            next = step_bounds<REV>(a.G, steps, span, a.T, a.H, n + kSlotWarps, lane);
            if (STATES) {
                general_wait(ctl, &ctl->done[w], use & 1);
                continue;
            }
            step_scores(smem_u32(tile), smem_u32(tile + kXTile), mine + kValueP, lane);
            __syncwarp();
            f32x2 acc[kSub];
            // intra-step rows: the products prod a_r are carried along by one multiplication a token, every factor <= 1
            const unsigned char* scores = mine + kValueP;
#pragma unroll
            for (int ii = 0; ii < kSub; ++ii) {
                const int i = REV ? kSub - 1 - ii : ii;
                if (ii > 0) {
                    const f32x2 x = gate[REV ? i + 1 : i];
#pragma unroll
                    for (int jj = 0; jj < ii; ++jj) E[REV ? kSub - 1 - jj : jj] = mul2(E[REV ? kSub - 1 - jj : jj], x);
                }
                f32x2 sum[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) sum[u] = pack2(0.f, 0.f);
#pragma unroll
                for (int j0 = 0; j0 < kSub; j0 += 2) {
                    const bool one = REV ? j0 >= i : j0 <= i, two = REV ? j0 + 1 >= i : j0 + 1 <= i;
                    if (!one && !two) continue;
                    const ulonglong2 p = *reinterpret_cast<const ulonglong2*>(scores + i * kPRow + 8 * j0);
                    if (one) sum[j0 & 2] = fma2(p.x, E[j0], sum[j0 & 2]);
                    if (two) sum[(j0 & 2) + 1] = fma2(p.y, E[j0 + 1], sum[(j0 & 2) + 1]);
                }
                acc[i] = add2(add2(sum[0], sum[1]), add2(sum[2], sum[3]));
            }
            // + the row factor times the inter-step product
            f32x2 f[kSub];
            run = REV ? frame.out : mul2(gate[0], frame.out);
#pragma unroll
            for (int i = 0; i < kSub; ++i) {
                const int j = REV ? kSub - 1 - i : i;
                f[j] = run;
                if (i + 1 < kSub) run = mul2(run, gate[REV ? j : j + 1]);
            }
            general_wait(ctl, &ctl->done[w], use & 1);
            const int t = steps.token<REV>(n);
            float* row = obase + (((size_t)span.b * a.T + t) * a.H + span.h) * kM;
            const unsigned char* inter = mine + kValueO + 8 * lane;
#pragma unroll
            for (int j = 0; j < kSub; ++j) {
                f32x2 sum = *reinterpret_cast<const f32x2*>(inter + j * kORow);
                if (halves) sum = add2(sum, *reinterpret_cast<const f32x2*>(inter + (kSub + j) * kORow));
                f[j] = fma2(f[j], sum, acc[j]);
            }
#pragma unroll
            for (int j = 0; j < kSub; ++j)
                if (t + j < span.t_end) *reinterpret_cast<f32x2*>(row + (size_t)j * a.H * kM) = f[j];
            __syncwarp();
        }
    } else if (!halves) {
        if (warp < kStateWarps) value_state_warp<STATES, kDST / 16>(ctl, ring, slots, a, steps, d0, warp, 0, lane);
    } else if (!STATES) {
        value_state_warp<STATES, kDST / 32>(ctl, ring, slots, a, steps, d0, warp & 3, warp >= kStateWarps ? 1 : 0, lane);
    }
    return general_finish(ctl, tid, dev_status);
}

// ======================================================================================
// key_side: out_i = (uq_i * qscale_i) S + sum_j A_ij xv_j,  A_ij = sum_s uq_i[s] uk_j[s] decay_ij[s]
// ======================================================================================
// A slot warp's shared memory: decayed uq and uk [16][64], each a high/low pair; a third pair for A (see step_weights); A as
// a high/low pair [16 (i)][16 (j)]; the step's total decay
constexpr int kKeyUk = 2 * kDecTile, kKeyZ = 4 * kDecTile, kKeyA = 6 * kDecTile, kKeyTotal = kKeyA + 2 * kSub * kARow;
constexpr int kKeyOut = kKeyTotal + 4 * kM;          // ... and the output rows [16][128 channels]
constexpr int kKeySlotB = kKeyOut + kSub * kOutRow;
constexpr int kKeyStageB = kXTile + 3 * kSlotTile;

// c = X Y^T [16 x 16] over the 64 slots, both as high/low pairs (the low x low term is dropped)
__device__ __forceinline__ void step_product(float (&c)[2][4], uint32_t x, uint32_t y, int lane) {
    const int q = lane >> 3, r = lane & 7;
    const uint32_t xa = x + ((q & 1) * 8 + r) * kDecRow + (q >> 1) * 16, ya = y + ((q >> 1) * 8 + r) * kDecRow + (q & 1) * 16;
    float part[3][2][4] = {};
#pragma unroll
    for (int kk = 0; kk < kM / 16; ++kk) {
        uint32_t xh[4], xl[4], yh[4], yl[4];
        ldsm4(xh, xa + 32 * kk);
        ldsm4(xl, xa + kDecTile + 32 * kk);
        ldsm4(yh, ya + 32 * kk);
        ldsm4(yl, ya + kDecTile + 32 * kk);
#pragma unroll
        for (int nn = 0; nn < 2; ++nn) {
            mma16816(part[0][nn], xl, yh[2 * nn], yh[2 * nn + 1]);
            mma16816(part[1][nn], xh, yl[2 * nn], yl[2 * nn + 1]);
            mma16816(part[2][nn], xh, yh[2 * nn], yh[2 * nn + 1]);
        }
    }
#pragma unroll
    for (int nn = 0; nn < 2; ++nn)
#pragma unroll
        for (int e = 0; e < 4; ++e) c[nn][e] = part[2][nn][e] + (part[0][nn][e] + part[1][nn][e]);
}

// A_ij = sum_s uq_i[s] uk_j[s] prod a_r[s] of a step, on the kept triangle, as accumulator fragments.  While no slot's decay
// over the step is below e^-60 (kFactorisedDecayMin is the bound of the pipelined kernels' chunks, too): a product of decayed rows,
//   forward  (uq_i e_i / e_last) (uk_j s_j),     reversed  (uq_i s_i) (uk_j e_j / e_last),
// one side as it is and the other divided by the step's total decay (in the frame of step_frame, where its factors cancel): the side that may hold a gradient of any size (dz), beside
// the input gate.  Its rows with e, up to 2^-87, come 2^kLift larger (`lifted`) and the quotient 2^-kLift smaller, so that both stay
// within fp32 for gradients of 1e-23 to 1e23.  (With the input gate's rows divided, and the gradient's as small as e makes them,
// gradients of 1e-17 came out as what subnormal numbers leave of them.)
// Otherwise by halves: i and j in the two halves of a block of 2 L tokens meet
// at the block's middle, to which both decay by factors <= 1; four levels L = 8, 4, 2, 1, of which a token plays one part in
// each -- one pair of rows Z serves both sides -- and the diagonal.
constexpr int kLift = 43;              // half of -kFactorisedDecayMin log2 e
constexpr float kLifted = (float)(1ull << kLift), kLowered = 1.f / kLifted;
template <bool REV>
__device__ __forceinline__ void step_weights(float (&c)[2][4], const f32x2 (&lifted)[kSub], const unsigned char* uq, const unsigned char* uk, const unsigned char* gates,
                                             const float2 (&g)[kSub], float2 before, f32x2 inverse, int rows, bool uq_keeps, bool uk_keeps, unsigned char* mine, int lane) {
    unsigned char* Z = mine + kKeyZ;
    const float2 whole = make_float2(g[kSub - 1].x - before.x, g[kSub - 1].y - before.y);
    if (__all_sync(0xffffffffu, fminf(whole.x, whole.y) >= kFactorisedDecayMin)) {
        const f32x2 quotient = mul2(inverse, both(kLowered * kLowered));
#pragma unroll
        for (int j0 = 0; j0 < kSub; j0 += kBatch) {
            f32x2 f[kBatch];
#pragma unroll
            for (int j = 0; j < kBatch; ++j) f[j] = mul2(lifted[j0 + j], quotient);
            store_parts<2>(Z, j0, lane, f);
        }
        __syncwarp();
        if (REV) step_product(c, smem_u32(mine), smem_u32(Z), lane);
        else step_product(c, smem_u32(Z), smem_u32(mine + kKeyUk), lane);
#pragma unroll
        for (int nn = 0; nn < 2; ++nn)
#pragma unroll
            for (int e = 0; e < 4; ++e) c[nn][e] *= kLifted;
        return;
    }
    // (rolled loops: few registers, little code beside the usual case)
    const int gr = lane >> 2, t = lane & 3;
    auto gate = [&](int j) { return unpack2(slots2(gates, min(j, rows - 1), lane)); };
#pragma unroll 1
    for (int L = kSub / 2; L > 0; L >>= 1) {
#pragma unroll 1
        for (int j0 = 0; j0 < kSub; j0 += kBatch) {
            f32x2 f[kBatch];
#pragma unroll
            for (int j = 0; j < kBatch; ++j) {
                const int at = j0 + j, mid = (at & ~(2 * L - 1)) + L;         // the first token of the block's second half
                const bool later = (at & L) != 0;
                const float2 g0 = gate(mid - 1), g1 = gate(at);
                f[j] = mul2(weights2(later != REV ? uq : uk, at, lane, later != REV ? uq_keeps : uk_keeps), later ? decay2(g0, g1) : decay2(g1, g0));
            }
            store_parts<2>(Z, j0, lane, f);
        }
        __syncwarp();
        float part[2][4];
        step_product(part, smem_u32(Z), smem_u32(Z), lane);
        __syncwarp();
#pragma unroll
        for (int nn = 0; nn < 2; ++nn)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int d = (gr + 8 * (e >> 1)) ^ (8 * nn + 2 * t + (e & 1));
                if (L == kSub / 2 || (d >= L && d < 2 * L)) c[nn][e] = part[nn][e];
            }
    }
#pragma unroll 1
    for (int j = 0; j < kSub; ++j) {
        const float2 x = unpack2(mul2(weights2(uq, j, lane, uq_keeps), weights2(uk, j, lane, uk_keeps)));
        float sum = x.x + x.y;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
#pragma unroll
        for (int nn = 0; nn < 2; ++nn)
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (gr + 8 * (e >> 1) == j && 8 * nn + 2 * t + (e & 1) == j) c[nn][e] = sum;
    }
}

template <bool REV>
__device__ __noinline__ bool key_side_general(const StepMaps maps, const KeySideArgs& args, int32_t* dev_status, int slice) {
    const KeySideArgs a = args;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* ring = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    unsigned char* slots = ring + kStages * kKeyStageB;
    GeneralCtl* ctl = reinterpret_cast<GeneralCtl*>(slots + kSlotWarps * kKeySlotB);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const ScanSpan span = scan_span(blockIdx.x, a.H, a.T, a.nseg, a.tseg);
    const int d0 = slice * kDST;
    const Steps steps = all_steps(span);
    general_ctl_init(ctl, tid, kStateWarps);

    if (warp >= kStateWarps && warp < kStateWarps + kSlotWarps) {
        // =============================== slot warps: lane l has slots 2 l and 2 l + 1
        const int w = warp - kStateWarps, gr = lane >> 2, t = lane & 3;
        unsigned char* mine = slots + w * kKeySlotB;
        load_step<REV, 1, 2>(ctl, ring, maps, steps, span, d0, w);
        StepBounds next = step_bounds<REV>(a.G, steps, span, a.T, a.H, w, lane);
        for (int n = w; n < steps.count; n += kSlotWarps) {
            const int st = n % kStages, use = n / kSlotWarps;
            const unsigned char *queries = ring + st * kKeyStageB + kXTile, *keys = queries + kSlotTile, *gates = keys + kSlotTile;
            general_wait(ctl, &ctl->full[st], (n / kStages) & 1);
            float2 g[kSub];
            const float2 before = next.before;
            const int rows = min(kSub, span.t_end - steps.token<REV>(n));
            step_gates(g, gates, rows, lane);
            const StepFrame frame = step_frame<REV>(next, g[kSub - 1], steps.chunk_ends<REV>(steps.token<REV>(n)));
            // (the stage of this warp's next step: all are done with the step that it held, the one before this)
            load_step<REV, 1, 2>(ctl, ring, maps, steps, span, d0, n + kSlotWarps);
            next = step_bounds<REV>(a.G, steps, span, a.T, a.H, n + kSlotWarps, lane);
            f32x2 gate[kSub], lifted[kSub];                          // the gates, whose products the factors are; see step_weights
#pragma unroll
            for (int j = 0; j < kSub; ++j) gate[j] = decay2(j > 0 ? g[j - 1] : before, g[j]);
#pragma unroll
            for (int side = 0; side < 2; ++side) {         // uq, then uk
                // the products of the gates from the step's start through a token, and from behind it to the end
                const bool from_start = (side != 0) == REV;
                f32x2 run = side != 0 ? frame.weight : frame.out;
                if (from_start) run = mul2(run, mul2(gate[0], both(kLifted)));
#pragma unroll
                for (int i0 = 0; i0 < kSub; i0 += kBatch) {
                    const int j0 = from_start ? i0 : kSub - kBatch - i0;
                    f32x2 f[kBatch];
#pragma unroll
                    for (int i = 0; i < kBatch; ++i) {
                        const int j = from_start ? i : kBatch - 1 - i, next = from_start ? j0 + j + 1 : j0 + j;
                        f[j] = run;
                        if (next < kSub) run = mul2(run, gate[next]);
                    }
#pragma unroll
                    for (int j = 0; j < kBatch; ++j) {
                        f[j] = mul2(weights2(side != 0 ? keys : queries, j0 + j, lane, (side != 0 ? a.uk_keeps : a.uq_keeps) != 0), f[j]);
                        if (!from_start) continue;
                        lifted[j0 + j] = f[j];
                        f[j] = mul2(f[j], both(kLowered));
                    }
                    store_parts<2>(mine + (side != 0 ? kKeyUk : 0), j0, lane, f);
                }
            }
            *reinterpret_cast<f32x2*>(mine + kKeyTotal + 8 * lane) = frame.total;
            __syncwarp();
            float c[2][4];
            step_weights<REV>(c, lifted, queries, keys, gates, g, before, frame.inverse, rows, a.uq_keeps != 0, a.uk_keeps != 0, mine, lane);
            unsigned char* A = mine + kKeyA;
#pragma unroll
            for (int nn = 0; nn < 2; ++nn)
#pragma unroll
                for (int e = 0; e < 4; e += 2) {
                    const int i = gr + 4 * e, j = 8 * nn + 2 * t;
                    uint32_t hi, lo;
                    split_pair((REV ? j >= i : j <= i) ? c[nn][e] : 0.f, (REV ? j + 1 >= i : j + 1 <= i) ? c[nn][e + 1] : 0.f, hi, lo);
                    uint32_t* p = reinterpret_cast<uint32_t*>(A + i * kARow + 2 * j);
                    p[0] = hi;
                    p[kSub * kARow / 4] = lo;
                }
            warp_arrive(&ctl->ready[w], lane);
            // the step's output rows
            general_wait(ctl, &ctl->done[w], use & 1);
            const int tok = steps.token<REV>(n) + (lane >> 4);
            __nv_bfloat16* out = static_cast<__nv_bfloat16*>(a.out) + (((size_t)span.b * a.T + tok) * a.H + span.h) * a.D + d0 + 8 * (lane & 15);
            const unsigned char* o_rows = mine + kKeyOut + (lane >> 4) * kOutRow + 16 * (lane & 15);
            if (d0 + 8 * (lane & 15) < a.D) {
#pragma unroll
                for (int j = 0; j < kSub; j += 2)
                    if (tok + j < span.t_end) *reinterpret_cast<uint4*>(out + (size_t)j * a.H * a.D) = *reinterpret_cast<const uint4*>(o_rows + j * kOutRow);
            }
            __syncwarp();
        }
    } else if (warp < kStateWarps) {
        // =============================== state warps: S^T[32 channels][64 slots] as accumulator tiles [16 channels][8 slots]
        constexpr int kMt = 2;
        const int c0 = 16 * kMt * warp, g = lane >> 2, t = lane & 3, q = lane >> 3, r = lane & 7;
        const bool live = d0 + c0 < a.D;           // (channels past D are zeros throughout and not written)
        const size_t state = ((size_t)blockIdx.x * kM + 2 * t) * a.D + d0 + c0 + g;
        float S[kMt][kM / 8][4];
#pragma unroll
        for (int mt = 0; mt < kMt; ++mt)
#pragma unroll
            for (int nt = 0; nt < kM / 8; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    S[mt][nt][e] = live && a.S0 != nullptr ? a.S0[state + (size_t)(8 * nt + (e & 1)) * a.D + 16 * mt + 8 * (e >> 1)] : 0.f;
        uint32_t at_v[kMt];
#pragma unroll
        for (int mt = 0; mt < kMt; ++mt) at_v[mt] = x_at(0, (q >> 1) * 8 + r, c0 / 8 + 2 * mt + (q & 1));
        bool ready = false;
        for (int n = 0; n < steps.count; ++n) {
            const int st = n % kStages, w = n % kSlotWarps;
            unsigned char* theirs = slots + w * kKeySlotB;
            // (the slot warp has seen the rows land before it says that its own are ready)
            if (!ready) general_wait(ctl, &ctl->ready[w], (n / kSlotWarps) & 1);
            // xv^T (rows: channels, k: tokens); uq (k: slots, columns: tokens); uk (k: tokens, columns: slots)
            uint32_t x[kMt][4], ah[4], al[4], qh[2][4], ql[2][4], kh[2][4], kl[2][4];
            const uint32_t va = smem_u32(ring + st * kKeyStageB);
            const uint32_t qa = smem_u32(theirs) + ((q >> 1) * 8 + r) * kDecRow + (q & 1) * 16;
            const uint32_t ka = smem_u32(theirs + kKeyUk) + ((q & 1) * 8 + r) * kDecRow + (q >> 1) * 16;
            const uint32_t aa = smem_u32(theirs + kKeyA) + ((q >> 1) * 8 + r) * kARow + (q & 1) * 16;
#pragma unroll
            for (int mt = 0; mt < kMt; ++mt) ldsm4_trans(x[mt], va + at_v[mt]);
            ldsm4_trans(kl[0], ka + kDecTile);
            ldsm4(qh[0], qa);
            ldsm4_trans(kh[0], ka);
            ldsm4(ql[0], qa + kDecTile);
            const float* total = reinterpret_cast<const float*>(theirs + kKeyTotal) + 2 * t;
            float O[kMt][2][4] = {};     // [channels 16 mt ..][tokens 8 nn ..]
#pragma unroll
            for (int ks = 0; ks < kM / 16; ++ks) {
                const int b = ks & 1;
                uint32_t sh[kMt][4], sl[kMt][4];
#pragma unroll
                for (int mt = 0; mt < kMt; ++mt)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float (&f)[4] = S[mt][2 * ks + (e >> 1)];
                        split_pair(f[2 * (e & 1)], f[2 * (e & 1) + 1], sh[mt][e], sl[mt][e]);
                    }
                const f32x2 dec[2] = {*reinterpret_cast<const f32x2*>(total + 16 * ks), *reinterpret_cast<const f32x2*>(total + 16 * ks + 8)};
                if (ks + 1 < kM / 16) {
                    ldsm4_trans(kl[b ^ 1], ka + kDecTile + 32 * (ks + 1));
                    ldsm4(qh[b ^ 1], qa + 32 * (ks + 1));
                    ldsm4_trans(kh[b ^ 1], ka + 32 * (ks + 1));
                    ldsm4(ql[b ^ 1], qa + kDecTile + 32 * (ks + 1));
                } else {
                    ldsm4(al, aa + kSub * kARow);
                    ldsm4(ah, aa);
                }
                float U[kMt][2][4] = {};
#pragma unroll
                for (int mt = 0; mt < kMt; ++mt)
#pragma unroll
                    for (int nn = 0; nn < 2; ++nn) mma16816(U[mt][nn], x[mt], kl[b][2 * nn], kl[b][2 * nn + 1]);
#pragma unroll
                for (int mt = 0; mt < kMt; ++mt)
#pragma unroll
                    for (int nn = 0; nn < 2; ++nn) mma16816(O[mt][nn], sl[mt], qh[b][2 * nn], qh[b][2 * nn + 1]);
#pragma unroll
                for (int mt = 0; mt < kMt; ++mt)
#pragma unroll
                    for (int nn = 0; nn < 2; ++nn) mma16816(U[mt][nn], x[mt], kh[b][2 * nn], kh[b][2 * nn + 1]);
#pragma unroll
                for (int mt = 0; mt < kMt; ++mt)
#pragma unroll
                    for (int nn = 0; nn < 2; ++nn) mma16816(O[mt][nn], sh[mt], ql[b][2 * nn], ql[b][2 * nn + 1]);
#pragma unroll
                for (int mt = 0; mt < kMt; ++mt)
#pragma unroll
                    for (int nn = 0; nn < 2; ++nn) {
                        float (&f)[4] = S[mt][2 * ks + nn];
#pragma unroll
                        for (int e = 0; e < 4; e += 2) decay_add(f[e], f[e + 1], dec[nn], U[mt][nn][e], U[mt][nn][e + 1]);
                    }
#pragma unroll
                for (int mt = 0; mt < kMt; ++mt)
#pragma unroll
                    for (int nn = 0; nn < 2; ++nn) mma16816(O[mt][nn], sh[mt], qh[b][2 * nn], qh[b][2 * nn + 1]);
                // (is the next step's there? asked while the products run)
                if (ks == 2) ready = n + 1 < steps.count && __all_sync(0xffffffffu, mbar_try(&ctl->ready[(n + 1) % kSlotWarps], ((n + 1) / kSlotWarps) & 1));
            }
            // intra-step rows, xv^T A^T
#pragma unroll
            for (int mt = 0; mt < kMt; ++mt)
#pragma unroll
                for (int nn = 0; nn < 2; ++nn) mma16816(O[mt][nn], x[mt], al[2 * nn], al[2 * nn + 1]);
#pragma unroll
            for (int mt = 0; mt < kMt; ++mt)
#pragma unroll
                for (int nn = 0; nn < 2; ++nn) mma16816(O[mt][nn], x[mt], ah[2 * nn], ah[2 * nn + 1]);
            // output rows, token-major, for the slot warp to store
            const uint32_t oa = smem_u32(theirs + kKeyOut) + ((q >> 1) * 8 + r) * kOutRow + 2 * c0 + (q & 1) * 16;
#pragma unroll
            for (int mt = 0; mt < kMt; ++mt)
                stsm4_trans(oa + 32 * mt, pack_bf16(O[mt][0][0], O[mt][0][1]), pack_bf16(O[mt][0][2], O[mt][0][3]),
                            pack_bf16(O[mt][1][0], O[mt][1][1]), pack_bf16(O[mt][1][2], O[mt][1][3]));
            warp_arrive(&ctl->done[w], lane);
        }
        if (!ctl->abort && a.Send != nullptr && live) {
#pragma unroll
            for (int mt = 0; mt < kMt; ++mt)
#pragma unroll
                for (int nt = 0; nt < kM / 8; ++nt)
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        a.Send[state + (size_t)(8 * nt + (e & 1)) * a.D + 16 * mt + 8 * (e >> 1)] = S[mt][nt][e];
        }
    }
    return general_finish(ctl, tid, dev_status);
}

// the tensor maps of the scans' steps
inline cudaError_t step_map(CUtensorMap* map, const void* base, int B, int T, int H, int D, int elem_bytes) {
    return make_tensor_map_bthd(map, base, B, T, H, D, kSub, elem_bytes);
}
struct GeneralValueMaps {
    CUtensorMap q, k, w, G;
    __device__ __forceinline__ StepMaps steps() const { return {{&q, &k}, {&w, nullptr}, &G}; }
};
struct GeneralKeyMaps {
    CUtensorMap v, uq, uk, G;
    __device__ __forceinline__ StepMaps steps() const { return {{&v, nullptr}, {&uq, &uk}, &G}; }
};
inline cudaError_t make_general_maps(GeneralValueMaps* m, const ValueSideArgs& a) {
    cudaError_t e = step_map(&m->q, a.xq, a.B, a.T, a.H, a.D, 2);
    if (e == cudaSuccess) e = step_map(&m->k, a.xk, a.B, a.T, a.H, a.D, 2);
    if (e == cudaSuccess) e = step_map(&m->w, a.w, a.B, a.T, a.H, kM, 4);
    if (e == cudaSuccess) e = step_map(&m->G, a.G, a.B, a.T, a.H, kM, 4);
    return e;
}
inline cudaError_t make_general_maps(GeneralKeyMaps* m, const KeySideArgs& a) {
    cudaError_t e = step_map(&m->v, a.xv, a.B, a.T, a.H, a.D, 2);
    if (e == cudaSuccess) e = step_map(&m->uq, a.uq, a.B, a.T, a.H, kM, 4);
    if (e == cudaSuccess) e = step_map(&m->uk, a.uk, a.B, a.T, a.H, kM, 4);
    if (e == cudaSuccess) e = step_map(&m->G, a.G, a.B, a.T, a.H, kM, 4);
    return e;
}

constexpr size_t kSmemGeneralValue = kStages * kValueStageB + kSlotWarps * kValueSlotB;
constexpr size_t kSmemGeneralKey = kStages * kKeyStageB + kSlotWarps * kKeySlotB;
constexpr size_t kSmemGeneral = 1024 + (kSmemGeneralValue > kSmemGeneralKey ? kSmemGeneralValue : kSmemGeneralKey) + sizeof(GeneralCtl);

}  // namespace
}  // namespace gsa
