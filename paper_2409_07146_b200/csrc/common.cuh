// Shared declarations of the GSA CUDA library (internal; the public surface is include/gsa.h).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "gsa.h"

namespace gsa {

constexpr int kChunk = 64;            // C of the chunkwise form, fp32 CUDA-core kernels (tensor-core kernels: 128)
constexpr float kLogGateMin = -100.f; // clamp of log a (exp(-100) == 0 in fp32)
// A chunk whose total log-decay stays above this bound uses the factorised
// decay exp(G_i) * exp(-G_j) (one reference point per chunk); below it the
// exponent differences are taken explicitly so nothing can overflow.
constexpr float kFactorisedDecayMin = -60.f;
constexpr int kSMs = 148;              // B200

template <typename T> struct IoTraits;
template <> struct IoTraits<float> {
    static constexpr int kVec = 4;  // elements per 16-byte access
};
template <> struct IoTraits<__nv_bfloat16> {
    static constexpr int kVec = 8;
};

// 16-byte global load of kVec consecutive elements, widened to fp32.
__device__ __forceinline__ void load_vec(const float* p, float (&out)[4]) {
    float4 v = *reinterpret_cast<const float4*>(p);
    out[0] = v.x; out[1] = v.y; out[2] = v.z; out[3] = v.w;
}
__device__ __forceinline__ void load_vec(const __nv_bfloat16* p, float (&out)[8]) {
    uint4 v = *reinterpret_cast<const uint4*>(p);
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float2 f = __bfloat1622float2(h[i]);
        out[2 * i] = f.x; out[2 * i + 1] = f.y;
    }
}
__device__ __forceinline__ void store_vec(float* p, const float (&in)[4]) {
    *reinterpret_cast<float4*>(p) = make_float4(in[0], in[1], in[2], in[3]);
}
__device__ __forceinline__ void store_vec(__nv_bfloat16* p, const float (&in)[8]) {
    uint4 v;
    __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&v);
#pragma unroll
    for (int i = 0; i < 4; ++i) h[i] = __floats2bfloat162_rn(in[2 * i], in[2 * i + 1]);
    *reinterpret_cast<uint4*>(p) = v;
}
__device__ __forceinline__ void store_vec4(float* p, const float (&in)[4]) {
    *reinterpret_cast<float4*>(p) = make_float4(in[0], in[1], in[2], in[3]);
}
__device__ __forceinline__ void store_vec4(__nv_bfloat16* p, const float (&in)[4]) {
    uint2 v;
    __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&v);
    h[0] = __floats2bfloat162_rn(in[0], in[1]);
    h[1] = __floats2bfloat162_rn(in[2], in[3]);
    *reinterpret_cast<uint2*>(p) = v;
}

// Kernels of a call follow one another closely: each is launched with launch_after, may be placed on the GPU as soon as
// every CTA of the kernel before it in the stream has started, and waits, first thing, until that kernel is complete and its
// memory is visible (follow_previous_grid).  As every kernel waits, what is complete for one is complete for all after it.
// The gaps between the 8 kernels of a forward over 1431 tokens, 2.4 us each, take 17 of its 67 us without; 56 us with it.
// (A CTA that waits holds its SM's resources: not for kernels whose CTAs usually leave at once while another stream works.)
// What such a kernel reads may be written while the kernel is already resident, so no pointer it reads through carries
// __restrict__: the qualifier lets the compiler take the data for unchanging over the kernel's whole life, load it by the
// read-only path and move the load above the wait.  Pointers that are only written through may have it (and should where
// loads and stores alternate: the loads then need not wait for the stores).
__device__ __forceinline__ void follow_previous_grid() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
struct ClusterGrid { dim3 grid, cluster; };
template <typename... P, typename... A>
cudaError_t launch_after(void (*kernel)(P...), ClusterGrid in, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = in.grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = in.cluster.x;
    attr[1].val.clusterDim.y = in.cluster.y;
    attr[1].val.clusterDim.z = in.cluster.z;
    cfg.attrs = attr;
    cfg.numAttrs = in.cluster.x * in.cluster.y * in.cluster.z > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
template <typename... P, typename... A>
cudaError_t launch_after(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
    return launch_after(kernel, ClusterGrid{grid, dim3(1, 1, 1)}, block, smem, st, static_cast<A&&>(args)...);
}

// ---- arguments of the two chunk primitives (both passes, forward and time-reversed) ----
//
// value_side ("gsa_fwd" of Algorithm 1 with GATE_K = False, the pass-1 form):
//     out_i[s] = sum_{j<=i} <xq_i, xk_j> w_j[s] prod_{r=j+1..i} a_r[s]   (+ state term)
//   xq, xk: [B,T,H,D] io; w, G: [B,T,H,M] fp32; state S (D x M), given/returned in the
//   memory layout [B,H,M,D].  The contraction over D is split into `nslice` slices of
//   width D/nslice; slice z writes its partial sums to out + z * B*T*H*M.
//
// key_side ("gsa_fwd" with GATE_K = True, the pass-2 form):
//     out_i = sum_{j<=i} (sum_s uq_i[s] uk_j[s] prod_{r=j+1..i} a_r[s]) xv_j   (+ state term)
//   uq, uk, G: [B,T,H,M] fp32; xv, out: [B,T,H,D] io; state S (M x D) in [B,H,M,D].
//
// reverse = 1 sums over i >= j instead (same decay product): the gradients w.r.t. keys,
// values and the input gate are such time-reversed runs.
// Where w is the input gate 1 - a and only the flagged pairs read it in fp32 (the general scans): a gate tensor that holds a
// takes its place (w_keeps).  Otherwise the gate kernel leaves it out but of the chunks that flag their pair, and the scans form
// the other rows of a flagged pair from the gate before they go on (write_input_gate).
struct InputGate { const float* gate = nullptr; int kind = 0; float inv_tau = 0.f; };
struct ValueSideArgs {
    const void* xq; const void* xk;   // io
    const float* w; const float* G;
    const float* S0;                  // nullable
    float* Send;                      // nullable
    float* out;                       // [nslice][B,T,H,M]
    int B, T, H, D;
    // tensor-core path: the weights already multiplied by their decay factor, bf16 rows of 2M
    // [high part | rounding residual] of w exp(-G) (forward) or w exp(G) (reverse); nullable
    const void* wd;
    // only the end state matters to the caller (the state runs of segment-parallel scheduling): `out` is not written
    int state_only;
    int single;                       // tensor-core kernels: derived operands as one bf16 value (GSA_TC_SINGLE)
    // T runs as nseg segments of tseg tokens (the last one shorter), each an independent scan: S0, Send and the
    // strong-decay flags are then [B, nseg, H, ..]
    int nseg = 1, tseg = 0;
    const float* E = nullptr;         // kernels for 128 slots: exp(G), see launch_gate_cumsum_wide
    InputGate input_gate;             // forward-direction runs on the tensor cores; gate null: w is there
    int w_keeps = 0;                  // general scans: w holds a, the weights are 1 - a
    int packed = 0;                   // tensor-core kernels: of packed sequences (how many warps the general scans get)
    float* seg_logdecay = nullptr;    // state runs, forward, K side: receives the segments' log-decay (launch_segment_logdecay)
};
struct KeySideArgs {
    const float* uq; const float* uk; const float* G;
    const void* xv;                   // io
    const float* S0;                  // nullable
    float* Send;                      // nullable
    void* out;                        // io [B,T,H,D]
    int B, T, H, D;
    // tensor-core path: decayed bf16 rows of 2M (the first M are used): forward uq exp(G) and
    // uk exp(-G), reverse uq exp(-G) and uk exp(G); nullable (both or neither)
    const void* uq_d; const void* uk_d;
    int single;                       // as in ValueSideArgs
    int nseg = 1, tseg = 0;           // likewise
    const float* E = nullptr;         // likewise
    int uq_keeps = 0, uk_keeps = 0;   // general scans: uq, uk hold a and stand for 1 - a
};

// What scan `bhs` of a launch over B * nseg * H scans works on: batch element, head and the tokens [t0, t_end).
struct ScanSpan { int b, h, t0, t_end; };
__host__ __device__ inline ScanSpan scan_span(int bhs, int H, int T, int nseg, int tseg) {
    const int bs = bhs / H, b = bs / nseg, t0 = (bs - b * nseg) * tseg;
    return {b, bhs - bs * H, t0, nseg == 1 ? T : (t0 + tseg < T ? t0 + tseg : T)};
}

// Element-wise replacements of the slot softmax (gsa_act_t other than GSA_ACT_SOFTMAX): f(z) and f'(z).
__device__ __forceinline__ float slot_act_value(float z, int act) {
    const float r = fmaxf(z, 0.f);
    if (act == GSA_ACT_NONE) return z;
    if (act == GSA_ACT_RELU) return r;
    if (act == GSA_ACT_SWISH) return z / (1.f + __expf(-z));
    return r * r;
}
__device__ __forceinline__ float slot_act_slope(float z, int act) {
    if (act == GSA_ACT_NONE) return 1.f;
    if (act == GSA_ACT_RELU) return z > 0.f ? 1.f : 0.f;
    if (act == GSA_ACT_SWISH) {
        const float sg = 1.f / (1.f + __expf(-z));
        return sg * (1.f + z * (1.f - sg));
    }
    return 2.f * fmaxf(z, 0.f);
}

// exp(-x) = 2^(-x log2 e) in two instructions, zero where that is below 2^-126; infinite x give 0 and infinity.  Relative
// error: 2^-21 and, for the rounding of the exponent, |x| 2^-23.
__device__ __forceinline__ float exp_neg(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x * -1.4426950408889634f));
    return r;
}

// GSA_GATE_LOGITS: log a = -softplus(-x) / tau (a = sigmoid(x)^(1/tau), Sec. 3.3) and the factor
// d(log a)/dx = sigmoid(-x) / tau of the gate gradient.
__device__ __forceinline__ float log_gate_from_logit(float x, float inv_tau) {
    return -(fmaxf(-x, 0.f) + log1pf(__expf(-fabsf(x)))) * inv_tau;
}
__device__ __forceinline__ float dlog_gate_dlogit(float x, float inv_tau) {
    return inv_tau / (1.f + __expf(x));
}

// The pipelined tensor-core value_side kernel leaves the row factor of its partial sums --
// exp(G_i) of a forward run, exp(-G_i) of a time-reversed one -- to the element-wise kernel that
// consumes them (slot softmax forward / backward, gate gradient), which sums the D/128 slices
// anyway.  strong[(b * nseg + segment) * H + h] != 0 marks the (batch, head) pairs that the general
// kernel wrote, with the factor already applied.  G == nullptr: nothing is pending.
struct PendingDecay {
    const float* G;
    const int* strong;
    int T, H, nseg, tseg;             // (tseg: tokens per segment, see ValueSideArgs)
    // != 0: the slot kernel serves ONLY the pairs flagged in `strong` (the fused chunk kernel has done
    // the others on chip): rows with a pending factor are skipped
    int strong_only;
    // 128 slots on the tensor-core kernels: G holds exp(G) itself, and a kernel may see the tensors as H = 2 x heads of
    // 64 slots (half_heads), both of which have the flag of their head
    int wide = 0, half_heads = 0;
    // the answer for token t is that for all rows of its 128-token chunk, and not beyond: the next chunk may be another segment's
    __host__ __device__ bool pending_at(int b, int t, int h) const {
        if (G == nullptr) return false;
        const int seg = nseg == 1 ? 0 : t / tseg;
        return strong[(b * nseg + seg) * (H >> half_heads) + (h >> half_heads)] == 0;
    }
    // the factor exp(-G_i) left out of the time-reversed partial sums, from an element of G (0 past the sequence end)
    __device__ float reverse_factor(float g) const { return wide ? (g > 0.f ? 1.f / g : 0.f) : __expf(-g); }
};

// launchers (definitions in the .cu files); all return cudaGetLastError() of the launch
// n of each (others nullable)
cudaError_t launch_clear_flags(int* flags, int* others, size_t n, cudaStream_t st);
// Is a strong-decay flag written by one CTA of the gate kernel alone (64-slot tiles)?  It then needs no clearing, which is a launch
// of a short call's five: pairs or segments of a single chunk (a forward over 114 tokens, 8 heads of 256: 29.8 -> 27.0 us).
// (Up to eight chunks, their CTAs a cluster whose first one collects: the cluster's launch and barriers cost more than the clearing,
// in a graph 24.6 -> 25.8 us at 130 tokens, 56 -> 60 at B = 2, T = 1024, 16 heads of 128.)
__host__ __device__ inline bool owns_strong_flag(int nseg, int nchunks) { return nseg == nchunks; }
// strong_flag (nullable, [B*H] ints, zeroed by launch_clear_flags, but see owns_strong_flag): set to 1 for every (b,h) that has a
// chunk whose total log-decay is below kFactorisedDecayMin (nseg > 1: [B*nseg*H], per segment).  large_weight (with strong_flag
// only, as many, alike): one with a weight 1 - a that is 2 or more or no finite number.
// decayed (nullable, bf16 [B,T,H,2M]): rows [high part | rounding residual] of I exp(-G), the
// input-gate operand of the pipelined tensor-core kernels.  leave_out: I only of the chunks that decay
// below kFactorisedDecayMin (1, see InputGate), or not at all (2).  fast_log: take log a with the
// hardware base-2 logarithm (absolute error 2^-21.4 for a in [0.5, 1], 3 ulp below), for bf16 io.
// gate_kind: gsa_gate_t (a, log a, or logits with inv_tau = 1/tau)
cudaError_t launch_gate_cumsum(const float* gate, int gate_kind, float inv_tau, float* G, float* I,
                               int B, int T, int H, int M, int chunk, int* strong_flag, int nseg, int tseg,
                               void* decayed, int fast_log, cudaStream_t st, const int* cu_seqlens = nullptr,
                               int nseq = 0, int leave_out = 0, int* large_weight = nullptr);
// The same for the tensor-core kernels with 128 slots, M = 2 x 64: `decayed` are bf16 [B,T,2H,192] rows [high | middle |
// low part] of I exp(-G), E = exp(G), local to chunks of 128 tokens; both, and log a, to fp32 accuracy whatever the io
// type.  G is local to 64 tokens, the chunks of the CUDA-core kernels that take the flagged pairs.
cudaError_t launch_gate_cumsum_wide(const float* gate, int gate_kind, float inv_tau, float* G, float* I, float* E, int B, int T,
                                    int H, int* strong_flag, int nseg, int tseg, void* decayed, cudaStream_t st,
                                    const int* cu_seqlens, int nseq);
// ABC (Eq. 3-4): write weights phi (cumulative softmax over time of the scores) into I, zeros into G, phi as the
// decayed bf16 rows; and the gradient w.r.t. the scores from phi and the input-gate gradient partial sums
cudaError_t launch_abc_write(const float* s_in, float* G, float* I, void* decayed, int B, int T, int H, int M, cudaStream_t st);
cudaError_t launch_abc_grad(const float* phi, const float* dIk, int nsk, const float* dIv, int nsv, float* ds, int B, int T,
                            int H, int M, cudaStream_t st);
// a gate row [n] spread over `rows` rows; column sums of [rows, n] (scratch: column_sum_parts(rows) * n floats)
cudaError_t launch_broadcast_rows(const float* row, float* out, size_t rows, int n, cudaStream_t st);
size_t column_sum_parts(size_t rows);
cudaError_t launch_column_sum(const float* in, float* part, float* out, size_t rows, int n, cudaStream_t st);
// n bfloat16 values -> fp32 (a gate tensor given in bfloat16)
cudaError_t launch_widen_bf16(const void* in, float* out, size_t n, cudaStream_t st);
// Segment-parallel scheduling (T cut into nseg segments run as independent sequences): per-segment
// log-decay [B,nseg,H,128] from G (128 slots on the tensor cores; the other state runs leave it themselves, which spares
// every segmented call a launch), and the start memories [B,nseg,H,M,D] of every segment from the
// end memories of the segments run from empty memories.
cudaError_t launch_segment_logdecay(const float* G, float* seg_logdecay, int B, int T, int H, int nseg, int tseg, int chunk,
                                    cudaStream_t st);
// one side's memories in launch_segment_combine (S0 and final_state nullable); the K and the V side go in one launch
struct CombineSet { const float* local_end; const float* S0; float* start; float* final_state; int D; };
cudaError_t launch_segment_combine(const float* seg_logdecay, CombineSet k, CombineSet v, int B, int H, int M, int nseg,
                                   int reverse, cudaStream_t st);
cudaError_t launch_shard_combine(const float* logdecay_all, const float* local_all, const float* S0, float* start,
                                 float* final_state, int B, int H, int M, int D, int nshard, int rank, int reverse,
                                 cudaStream_t st);
// G, p_decayed / dz_decayed (nullable together; bf16 [rows, 2M]): rows [high | residual] of
// p exp(G) and dz exp(G), operands of the pipelined tensor-core kernels.
// (tensors [B, rows_per_batch = T*H, M])
// act: gsa_act_t (the softmax over the slots or an element-wise replacement)
cudaError_t launch_slot_softmax_fwd(const float* part, int nslice, float scale, int act, float* ok,
                                    float* p, int B, int rows_per_batch, int M, const float* G, void* p_decayed,
                                    PendingDecay pend, cudaStream_t st, int m_active = 0);
cudaError_t launch_slot_softmax_bwd(const float* ok, const float* dp_part, int nslice,
                                    float scale, int act, float* p, float* dz, float* u, int B, int rows_per_batch,
                                    int M, const float* G, void* p_decayed, void* dz_decayed,
                                    PendingDecay pend, cudaStream_t st, int m_active = 0);
// m_active (0 = all M): slots from m_active on are padding and take no part in the non-linearity.
// rows of n_in floats -> rows of n_out floats (tail filled with `fill`, or cut)
cudaError_t launch_resize_rows(const float* in, float* out, size_t rows, int n_in, int n_out, float fill, cudaStream_t st);
cudaError_t launch_gate_grad(const float* u, const float* I, const float* dIk_part, int nsk,
                             const float* dIv_part, int nsv, const float* gate,
                             int gate_kind, float inv_tau, const float* dKT, const float* KT,
                             const float* dVT, const float* VT, int d_k, int d_v,
                             float* chunk_tot, float* dgate, int B, int T, int H, int M,
                             PendingDecay pend, cudaStream_t st, int32_t* dev_status, const int* cu_seqlens = nullptr,
                             int nseq = 0);
int gate_grad_blocks(int T);       // entries per (b,h,slot) of launch_gate_grad's scratch
int gate_grad_kernels(int pairs, int M, bool wide, int nslices, int gate_kind, int T);      // how many kernels it is
// strong_flag != NULL: after the tensor-core kernels, for the flagged (batch, head) pairs alone; value_side then adds its
// slices to their 128-wide ones, which those have zeroed
cudaError_t launch_value_side_simt(const ValueSideArgs& a, int io, int M, int reverse,
                                   cudaStream_t st, const int* strong_flag = nullptr);
// state runs (end memories only, from empty ones) of the K and the V side in one launch; k also takes seg_logdecay
cudaError_t launch_state_scan_simt(const ValueSideArgs& k, const ValueSideArgs& v, int io, int M, int reverse, cudaStream_t st);
cudaError_t launch_key_side_simt(const KeySideArgs& a, int io, int M, int reverse,
                                 cudaStream_t st, const int* strong_flag = nullptr);
// tcgen05 (bf16 tensor-core) versions of the two primitives; bf16 io only.
bool tc_supported(int d_k, int d_v, int M);
bool tc_dim_ok(int D);
int tc_value_side_slices(int D);
int tc_chunk();                    // chunk length of the tensor-core kernels   // how many partial-sum slices value_side writes for width D
cudaError_t launch_value_side_tc(const ValueSideArgs& a, int M, int reverse, const int* strong_flag,
                                 cudaStream_t st, int32_t* dev_status);
cudaError_t launch_key_side_tc(const KeySideArgs& a, int M, int reverse, const int* strong_flag,
                               cudaStream_t st, int32_t* dev_status);
// 128 slots (chunk_tc_wide.cu): the slot tensors as above, the decayed rows as launch_gate_cumsum_wide writes them
cudaError_t launch_value_side_wide(const ValueSideArgs& a, int reverse, const int* strong_flag, cudaStream_t st,
                                   int32_t* dev_status);
cudaError_t launch_key_side_wide(const KeySideArgs& a, int reverse, const int* strong_flag, cudaStream_t st,
                                 int32_t* dev_status);
cudaError_t launch_state_scans_wide(const ValueSideArgs& k, const ValueSideArgs& v, int reverse, const int* strong_flag,
                                    cudaStream_t st, int32_t* dev_status);
// the general scan as a launch of its own, for the flagged pairs (beside the fused kernel; forward direction)
cudaError_t launch_value_side_general(const ValueSideArgs& a, const int* strong_flag, cudaStream_t st, int32_t* dev_status);
cudaError_t launch_key_side_general(const KeySideArgs& a, const int* strong_flag, cudaStream_t st, int32_t* dev_status);
// end memories only, from empty ones, of the K and the V side in one launch: xk, w and wd of each set are the tile that
// enters the state and its weights (key_side: xv, uk, uk_d)
cudaError_t launch_state_scan_tc(const ValueSideArgs& k, const ValueSideArgs& v, int reverse, const int* strong_flag,
                                 const int* large_weight, cudaStream_t st, int32_t* dev_status);
// The two reversed scans that share a state (dv with dI^v, dk with dI^k) as one kernel
// (chunk_tc_pair.cu): av / ak are the arguments the single reversed scans would get.
bool rev_pair_supported(const ValueSideArgs& av, const KeySideArgs& ak, int M);
cudaError_t launch_rev_pair_tc(const ValueSideArgs& av, const KeySideArgs& ak, int M, const int* strong_flag, bool packed,
                               cudaStream_t st, int32_t* dev_status);
// the side stream of the calling host thread on the current device, with its fork / join events
struct SideLane {
    cudaStream_t stream = nullptr;
    cudaEvent_t fork = nullptr, join = nullptr;
};
cudaError_t side_lane(SideLane** out);
cudaError_t side_lane_release();
// Fused chunk kernel: value_side scan -> slot non-linearity -> key_side scan in one kernel, for the
// (batch, head) pairs without a strong-decay chunk (chunk_tc_fused.cu).
//   mode 0 (forward):  xq1 = q,  xk1 = k, xv = v, out = o;   ok (nullable) receives the scaled logits
//   mode 1 (backward): xq1 = dO, xk1 = v, xv = k, out = dq;  ok holds the scaled logits; u, Pd, Zd are written
bool fused_pair_supported(int d_k, int d_v, int M);
cudaError_t launch_fused_pair(int mode, const void* xq1, const void* xk1, const void* wd, const void* xv, void* out,
                              const float* G, const float* S1_0, const float* S2_0, float* S1_end, float* S2_end, int B,
                              int T, int H, int D1, int D2, float scale, int act, float* ok, float* u, void* Pd,
                              void* Zd, const int* strong_flag, cudaStream_t st, int32_t* dev_status);
// layer pre- and post-operations (layer_ops.cu)
// (q, k and v, or their gradients, in one launch)
cudaError_t launch_swish_fwd(const void* const in[3], void* const out[3], const size_t n[3], int io, cudaStream_t st);
cudaError_t launch_swish_bwd(const void* const x[3], void* const d[3], const size_t n[3], int io, cudaStream_t st);
int out_norm_max_width(int io);
size_t out_norm_bwd_parts(size_t rows, int N, int io);
cudaError_t launch_out_norm_fwd(const void* o, const float* weight, float eps, void* y, size_t rows, int N, int io,
                                cudaStream_t st);
cudaError_t launch_out_norm_bwd(const void* o, const void* dy, const float* weight, float eps, void* d_o, float* dw_part,
                                float* dweight, size_t rows, int N, int io, cudaStream_t st);
// gsa_fwd in a scratch memory of a fixed size (api.cu)
gsa_status_t fwd_within(const gsa_params_t* params, const void* q, const void* k, const void* v, const float* gate,
                        const float* K0, const float* V0, void* o, float* ok_save, float* KT, float* VT, void* ws,
                        size_t ws_bytes, void* stream, int32_t* dev_status);
cudaError_t launch_decode(const gsa_params_t& p, const void* q, const void* k, const void* v,
                          const float* gate, float* Ks, float* Vs, void* o, cudaStream_t st);

}  // namespace gsa
