// Recurrent decode step of Gated Slot Attention: one iteration of Eq. 6 per (sequence, head).
//
// Per pair the kernel reads and rewrites both slot memories once (m*(d_k+d_v) fp32 each
// way) and does about one FMA per two bytes moved, so it is a pure HBM stream.  One CTA of
// 8 warps owns one pair; a warp owns a memory row at a time, with 16-byte accesses that
// cover the row contiguously (coalesced); rows are loaded in batches before any is used so
// that several 512-byte requests per warp are in flight.  The key memory is updated and
// read first (slot logits), then the softmax, then the value memory is updated and summed.  A step is placed while the launch
// before it drains: 24 layers of one sequence, 32 heads of 128, 148 -> 105 us as calls; 256 sequences, one layer 165.5 -> 163.1.
#include "common.cuh"

namespace gsa {

template <typename IO>
__device__ __forceinline__ float io_to_float(IO x);
template <>
__device__ __forceinline__ float io_to_float<float>(float x) { return x; }
template <>
__device__ __forceinline__ float io_to_float<__nv_bfloat16>(__nv_bfloat16 x) { return __bfloat162float(x); }
template <typename IO>
__device__ __forceinline__ IO float_to_io(float x);
template <>
__device__ __forceinline__ float float_to_io<float>(float x) { return x; }
template <>
__device__ __forceinline__ __nv_bfloat16 float_to_io<__nv_bfloat16>(float x) { return __float2bfloat16_rn(x); }

constexpr int kDecodeWarps = 8;

// One memory row of D floats per warp: lane l owns the float4s l, l+32, ... (D >= 128) or
// one float2 (D == 64).
template <int D>
struct RowVec {
    static constexpr int kW = (D >= 128) ? 4 : 2;      // floats per access
    static constexpr int kN = D / (32 * kW);           // accesses per lane
    float v[kN][kW];
    __device__ __forceinline__ void load(const float* row, int lane) {
#pragma unroll
        for (int r = 0; r < kN; ++r) {
            if constexpr (kW == 4) {
                float4 t = *reinterpret_cast<const float4*>(row + (lane + 32 * r) * 4);
                v[r][0] = t.x; v[r][1] = t.y; v[r][2] = t.z; v[r][3] = t.w;
            } else {
                float2 t = *reinterpret_cast<const float2*>(row + (lane + 32 * r) * 2);
                v[r][0] = t.x; v[r][1] = t.y;
            }
        }
    }
    __device__ __forceinline__ void store(float* row, int lane) const {
#pragma unroll
        for (int r = 0; r < kN; ++r) {
            if constexpr (kW == 4)
                *reinterpret_cast<float4*>(row + (lane + 32 * r) * 4) = make_float4(v[r][0], v[r][1], v[r][2], v[r][3]);
            else
                *reinterpret_cast<float2*>(row + (lane + 32 * r) * 2) = make_float2(v[r][0], v[r][1]);
        }
    }
    // The token's q, k, v.  Heads of 256 and more: an access of kW values, as a row's; value by value they are 48 loads a warp at
    // D = 512 (24 layers of one sequence, 4 heads of 512, 115 us value by value, so 109; 8 layers of 8, 8 heads of 256, 56 / 51).
    // Narrow heads value by value: 8 layers of 100, 12 heads of 64, 148 / 161; 24 of one, 16 heads of 128, 104 / 106.
    template <typename IO>
    __device__ __forceinline__ void load_io(const IO* row, int lane) {
#pragma unroll
        for (int r = 0; r < kN; ++r) {
            if constexpr (D >= 256) {
                struct alignas(sizeof(IO) * kW) Values { IO x[kW]; };
                const Values t = *reinterpret_cast<const Values*>(row + (lane + 32 * r) * kW);
#pragma unroll
                for (int w = 0; w < kW; ++w) v[r][w] = io_to_float<IO>(t.x[w]);
            } else {
#pragma unroll
                for (int w = 0; w < kW; ++w) v[r][w] = io_to_float<IO>(row[(lane + 32 * r) * kW + w]);
            }
        }
    }
    // the layer's feature map (Sec. 3.3), applied as the token's q, k, v are loaded
    __device__ __forceinline__ void swish() {
#pragma unroll
        for (int r = 0; r < kN; ++r)
#pragma unroll
            for (int w = 0; w < kW; ++w) v[r][w] = v[r][w] / (1.f + __expf(-v[r][w]));
    }
};

// a and 1 - a from element gi of the gate tensor
__device__ __forceinline__ void decode_gate(const void* gate_raw, size_t gi, int gate_bf16, int gate_kind, float inv_tau,
                                            float& a, float& ia) {
    float gt = gate_bf16 ? __bfloat162float(static_cast<const __nv_bfloat16*>(gate_raw)[gi])
                         : static_cast<const float*>(gate_raw)[gi];
    if (gate_kind == GSA_GATE_LOGITS) gt = log_gate_from_logit(gt, inv_tau);
    if (gate_kind != GSA_GATE_A) { a = __expf(gt); ia = -expm1f(gt); }
    else { a = gt; ia = 1.f - gt; }
}

template <typename IO, int DK, int DV, int M>
__global__ void __launch_bounds__(kDecodeWarps * 32)
decode_step_kernel(const IO* q, const IO* k, const IO* v,
                   const void* gate_raw, int gate_bf16, int gate_row_of_head, int feature_map, int gate_kind, float inv_tau, float scale, int act,
                   float* Ks, float* Vs, IO* __restrict__ o) {
    follow_previous_grid();
    constexpr int RPW = M / kDecodeWarps;  // memory rows per warp
    const size_t pair = blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __shared__ float s_z[M];
    __shared__ float s_p[M];
    __shared__ float s_o[kDecodeWarps][DV];

    float* Kp = Ks + pair * (size_t)M * DK;
    float* Vp = Vs + pair * (size_t)M * DV;

    RowVec<DK> qv, kv;
    RowVec<DV> vv;
    qv.load_io(q + pair * DK, lane);
    kv.load_io(k + pair * DK, lane);
    vv.load_io(v + pair * DV, lane);
    if (feature_map == GSA_FEAT_SWISH) { qv.swish(); kv.swish(); vv.swish(); }
    float a[RPW], ia[RPW];
#pragma unroll
    for (int r = 0; r < RPW; ++r) {
        // (data-independent decay: one gate row per head, shared by all sequences; gate_row_of_head = H then)
        const size_t gi = (gate_row_of_head ? pair % gate_row_of_head : pair) * M + warp * RPW + r;
        decode_gate(gate_raw, gi, gate_bf16, gate_kind, inv_tau, a[r], ia[r]);
    }

    // K~ <- a K~ + (1-a) k ; z = scale * K~ q.  Rows go through registers in batches whose
    // loads are all issued before the first use.
    constexpr int KB = (RPW * (DK / 32) <= 32) ? RPW : (32 / (DK / 32));
#pragma unroll
    for (int r0 = 0; r0 < RPW; r0 += KB) {
        RowVec<DK> kr[KB];
#pragma unroll
        for (int r = 0; r < KB; ++r) kr[r].load(Kp + (size_t)(warp * RPW + r0 + r) * DK, lane);
#pragma unroll
        for (int r = 0; r < KB; ++r) {
            float dot = 0.f;
#pragma unroll
            for (int i = 0; i < RowVec<DK>::kN; ++i)
#pragma unroll
                for (int w = 0; w < RowVec<DK>::kW; ++w) {
                    const float x = fmaf(a[r0 + r], kr[r].v[i][w], ia[r0 + r] * kv.v[i][w]);
                    kr[r].v[i][w] = x;
                    dot = fmaf(x, qv.v[i][w], dot);
                }
            kr[r].store(Kp + (size_t)(warp * RPW + r0 + r) * DK, lane);
#pragma unroll
            for (int off = 16; off; off >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, off);
            if (lane == 0) s_z[warp * RPW + r0 + r] = dot * scale;
        }
    }
    __syncthreads();
    // softmax over the m slots, or its element-wise replacement
    if (warp == 0 && act != GSA_ACT_SOFTMAX) {
#pragma unroll
        for (int r = 0; r < M / 32; ++r) s_p[lane + 32 * r] = slot_act_value(s_z[lane + 32 * r], act);
    } else if (warp == 0) {
        float z[M / 32], zmax = -INFINITY;
#pragma unroll
        for (int r = 0; r < M / 32; ++r) { z[r] = s_z[lane + 32 * r]; zmax = fmaxf(zmax, z[r]); }
#pragma unroll
        for (int off = 16; off; off >>= 1) zmax = fmaxf(zmax, __shfl_xor_sync(0xffffffffu, zmax, off));
        float den = 0.f;
#pragma unroll
        for (int r = 0; r < M / 32; ++r) { z[r] = __expf(z[r] - zmax); den += z[r]; }
#pragma unroll
        for (int off = 16; off; off >>= 1) den += __shfl_xor_sync(0xffffffffu, den, off);
        const float inv = 1.f / den;
#pragma unroll
        for (int r = 0; r < M / 32; ++r) s_p[lane + 32 * r] = z[r] * inv;
    }
    __syncthreads();
    // V~ <- a V~ + (1-a) v ; o = V~^T p: each warp sums its rows, then the 8 partial rows
    // are added in a fixed order
    RowVec<DV> acc;
#pragma unroll
    for (int i = 0; i < RowVec<DV>::kN; ++i)
#pragma unroll
        for (int w = 0; w < RowVec<DV>::kW; ++w) acc.v[i][w] = 0.f;
    constexpr int VB = (RPW * (DV / 32) <= 32) ? RPW : (32 / (DV / 32));
#pragma unroll
    for (int r0 = 0; r0 < RPW; r0 += VB) {
        RowVec<DV> vr[VB];
#pragma unroll
        for (int r = 0; r < VB; ++r) vr[r].load(Vp + (size_t)(warp * RPW + r0 + r) * DV, lane);
#pragma unroll
        for (int r = 0; r < VB; ++r) {
            const float pr = s_p[warp * RPW + r0 + r];
#pragma unroll
            for (int i = 0; i < RowVec<DV>::kN; ++i)
#pragma unroll
                for (int w = 0; w < RowVec<DV>::kW; ++w) {
                    const float x = fmaf(a[r0 + r], vr[r].v[i][w], ia[r0 + r] * vv.v[i][w]);
                    vr[r].v[i][w] = x;
                    acc.v[i][w] = fmaf(pr, x, acc.v[i][w]);
                }
            vr[r].store(Vp + (size_t)(warp * RPW + r0 + r) * DV, lane);
        }
    }
    acc.store(&s_o[warp][0], lane);
    __syncthreads();
    for (int c = threadIdx.x; c < DV; c += kDecodeWarps * 32) {
        float sum = 0.f;
#pragma unroll
        for (int w = 0; w < kDecodeWarps; ++w) sum += s_o[w][c];
        o[pair * DV + c] = float_to_io<IO>(sum);
    }
}

// Few (sequence, head) pairs: a pair is dealt out over a cluster of M / (8 RPW) CTAs, so that one sequence uses more than H SMs:
// RPW rows of the key memory to a warp, and of the value memory a CTA's share of the channels, all slots of them.  A step of one
// CTA per pair is bound by the latency of its chain -- K rows in
// batches, logits, softmax, V rows in batches, sums -- and by what one SM can pull: 512 KB at d = 512, 9.6 us a launch
// where 4 pairs keep 4 SMs busy.  Here all of both memories is requested at once, before anything is used; the CTAs
// exchange the M logits through distributed shared memory and nothing else (two cluster barriers; with rows of the value memory
// to a warp, too, the output's partial sums took a third: 24 layers of 4 pairs of d = 512, 109 us, so 88).  The steps
// of a stack of layers follow one another: each is placed while the one before it drains (150 -> 118 us as calls then).
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// the word at the same place of CTA `rank`'s shared memory <- x
__device__ __forceinline__ void store_to_rank(float* local, unsigned rank, float x) {
    uint32_t at, remote;
    at = (uint32_t)__cvta_generic_to_shared(local);
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(at), "r"(rank));
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(remote), "f"(x) : "memory");
}

template <int n> struct alignas(n * sizeof(float)) Floats { float x[n]; };

template <typename IO, int DK, int DV, int M, int RPW>
__global__ void __launch_bounds__(kDecodeWarps * 32)
decode_split_kernel(const IO* q, const IO* k, const IO* v,
                    const void* gate_raw, int gate_bf16, int gate_row_of_head, int feature_map,
                    int gate_kind, float inv_tau, float scale, int act, float* Ks, float* Vs,
                    IO* __restrict__ o) {
    follow_previous_grid();
    constexpr int C = M / (kDecodeWarps * RPW);                 // CTAs of the cluster
    constexpr int kOwn = DV / C, W = kOwn < 32 ? 1 : kOwn / 32; // channels of the value memory a CTA, a lane
    constexpr int kRows = M / kDecodeWarps;                     // rows of it a warp
    static_assert(C <= 8 && (W == 1 || W == 2 || W == 4), "");
    const size_t pair = blockIdx.x / C;
    const int rank = blockIdx.x % C, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int row0 = (rank * kDecodeWarps + warp) * RPW;        // this warp's rows of the key memory
    const int vrow0 = warp * kRows, c0 = rank * kOwn + W * lane;
    const bool live = kOwn >= 32 || lane < kOwn;                // (narrow values: lanes without a channel)
    __shared__ float s_z[M];
    __shared__ Floats<W> s_o[kDecodeWarps][32];
    cluster_arrive();                       // (every CTA runs before another one writes to it)

    float* Kp = Ks + (pair * M + row0) * DK;
    float* Vp = Vs + (pair * M + vrow0) * DV + c0;
    RowVec<DK> kr[RPW], qv, kv;
    Floats<W> vr[kRows];
#pragma unroll
    for (int r = 0; r < RPW; ++r) kr[r].load(Kp + (size_t)r * DK, lane);
#pragma unroll
    for (int r = 0; r < kRows; ++r)
        if (live) vr[r] = *reinterpret_cast<const Floats<W>*>(Vp + (size_t)r * DV);
    qv.load_io(q + pair * DK, lane);
    kv.load_io(k + pair * DK, lane);
    float vv[W];
#pragma unroll
    for (int w = 0; w < W; ++w) vv[w] = live ? io_to_float<IO>(v[pair * DV + c0 + w]) : 0.f;
    const size_t gates = (gate_row_of_head ? pair % gate_row_of_head : pair) * M;
    float a[RPW], ia[RPW], va, via;
#pragma unroll
    for (int r = 0; r < RPW; ++r) decode_gate(gate_raw, gates + row0 + r, gate_bf16, gate_kind, inv_tau, a[r], ia[r]);
    decode_gate(gate_raw, gates + vrow0 + lane % kRows, gate_bf16, gate_kind, inv_tau, va, via);      // (lane r: the warp's row r)
    if (feature_map == GSA_FEAT_SWISH) {
        qv.swish(); kv.swish();
#pragma unroll
        for (int w = 0; w < W; ++w) vv[w] = vv[w] / (1.f + __expf(-vv[w]));
    }
    float z[RPW];
#pragma unroll
    for (int r = 0; r < RPW; ++r) {
        float dot = 0.f;
#pragma unroll
        for (int i = 0; i < RowVec<DK>::kN; ++i)
#pragma unroll
            for (int w = 0; w < RowVec<DK>::kW; ++w) {
                const float x = fmaf(a[r], kr[r].v[i][w], ia[r] * kv.v[i][w]);
                kr[r].v[i][w] = x;
                dot = fmaf(x, qv.v[i][w], dot);
            }
#pragma unroll
        for (int off = 16; off; off >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, off);
        z[r] = dot * scale;
    }
    cluster_wait();
#pragma unroll
    for (int r = 0; r < RPW; ++r)
        if (lane < C) store_to_rank(&s_z[row0 + r], lane, z[r]);
    cluster_arrive();
    // (the memories leave while the logits travel)
#pragma unroll
    for (int r = 0; r < RPW; ++r) kr[r].store(Kp + (size_t)r * DK, lane);
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
        const float ar = __shfl_sync(0xffffffffu, va, r), ir = __shfl_sync(0xffffffffu, via, r);
#pragma unroll
        for (int w = 0; w < W; ++w) vr[r].x[w] = fmaf(ar, vr[r].x[w], ir * vv[w]);
        if (live) *reinterpret_cast<Floats<W>*>(Vp + (size_t)r * DV) = vr[r];
    }
    cluster_wait();
    // slot weights of this warp's rows of the value memory, each warp by itself (lane r: row r)
    float p = s_z[vrow0 + lane % kRows];
    if (act != GSA_ACT_SOFTMAX) {
        p = slot_act_value(p, act);
    } else {
        float zmax = -INFINITY, den = 0.f;
#pragma unroll
        for (int s = lane; s < M; s += 32) zmax = fmaxf(zmax, s_z[s]);
#pragma unroll
        for (int off = 16; off; off >>= 1) zmax = fmaxf(zmax, __shfl_xor_sync(0xffffffffu, zmax, off));
#pragma unroll
        for (int s = lane; s < M; s += 32) den += __expf(s_z[s] - zmax);
#pragma unroll
        for (int off = 16; off; off >>= 1) den += __shfl_xor_sync(0xffffffffu, den, off);
        p = __expf(p - zmax) * (1.f / den);
    }
    Floats<W> acc;
#pragma unroll
    for (int w = 0; w < W; ++w) acc.x[w] = 0.f;
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
        const float pr = __shfl_sync(0xffffffffu, p, r);
#pragma unroll
        for (int w = 0; w < W; ++w) acc.x[w] = fmaf(pr, vr[r].x[w], acc.x[w]);
    }
    s_o[warp][lane] = acc;
    __syncthreads();
    for (int c = threadIdx.x; c < kOwn; c += kDecodeWarps * 32) {
        float sum = 0.f;
#pragma unroll
        for (int w = 0; w < kDecodeWarps; ++w) sum += s_o[w][c / W].x[c % W];
        o[pair * DV + rank * kOwn + c] = float_to_io<IO>(sum);
    }
}

template <typename IO, int DK, int DV, int M, int RPW>
static cudaError_t launch_decode_split(const gsa_params_t& p, const IO* q, const IO* k, const IO* v, const float* gate,
                                       float* Ks, float* Vs, IO* o, cudaStream_t st) {
    constexpr unsigned C = M / (kDecodeWarps * RPW);
    return launch_after(decode_split_kernel<IO, DK, DV, M, RPW>, ClusterGrid{dim3((unsigned)p.B * (unsigned)p.H * C), dim3(C, 1, 1)},
                        dim3(kDecodeWarps * 32), 0, st, q, k, v, static_cast<const void*>(gate),
                              (int)(p.gate_dtype == GSA_BF16), (int)(p.gate_broadcast ? p.H : 0), (int)p.feature_map,
                              (int)p.gate_kind, p.tau > 0.f ? 1.f / p.tau : 0.f, p.scale, (int)p.slot_act, Ks, Vs, o);
}

// One CTA a pair.  A step placed while the one before it runs takes what that leaves: where the GPU holds one step's CTAs but not
// two steps', the CTAs left over come last, to whichever SMs are free first, five to some while others have one.  With three a
// balanced share and five held, that costs more than the early launch gives: shared memory then limits an SM to three.  384
// pairs of d = 64, us a step of one layer / of 8 layers, logits: early 9.3 / 11.1, plain 8.2 / 11.1, so 7.2 / 9.8; 444 pairs alike;
// at four a balanced share early 8.7 (456 pairs, 8 layers), so 9.6.  Four held (d = 128, 304 pairs): early 8.9 / 10.4, plain 8.2 /
// 12.3, so 8.6 / 11.9: left as it is.
constexpr int kShare = 3, kHeldMin = 5;
template <auto kernel, typename... A>
static cudaError_t launch_step(unsigned pairs, cudaStream_t st, A&&... args) {
    size_t smem = 0;
    if (pairs > 2 * kSMs && pairs <= kShare * kSMs) {
        struct Held { int ctas; size_t smem; };
        static const Held held = [] {
            Held h{0, 0};
            cudaFuncAttributes at;
            // (an SM has 228 KB, a CTA takes 1 KB beside its own)
            if (cudaFuncGetAttributes(&at, kernel) == cudaSuccess) h.smem = ((228 << 10) / kShare - (1 << 10) - at.sharedSizeBytes) & ~(size_t)127;
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&h.ctas, kernel, kDecodeWarps * 32, 0) != cudaSuccess) h.ctas = 0;
            return h;
        }();
        if (held.ctas >= kHeldMin && 2 * (long long)pairs > (long long)held.ctas * kSMs) {
            smem = held.smem;
            const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
        }
    }
    return launch_after(kernel, pairs, kDecodeWarps * 32, smem, st, static_cast<A&&>(args)...);
}

template <typename IO, int DK, int DV>
static cudaError_t launch_decode_m(const gsa_params_t& p, const IO* q, const IO* k, const IO* v,
                                   const float* gate, float* Ks, float* Vs, IO* o, cudaStream_t st) {
    const unsigned pairs = (unsigned)p.B * (unsigned)p.H;
    // The line between the kernels, us a step of one layer / of a layer of eight: one CTA a pair, against a row a warp or (from 19
    // pairs on) two.  64 slots, d = 64: 12 pairs 4.2 / 3.8, 3.1 / 2.9; 48: 4.2 / 3.8, 3.3 / 3.3; 96: 4.5 / 3.9, 4.7 / 4.7.  128: 4 pairs
    // 4.4 / 4.3, 3.1 / 2.9; 32: 4.5 / 4.4, 3.1 / 3.4; 64: 4.6 / 4.4, 4.6 / 4.0; 96: 5.1 / 4.5, 5.0 / 4.9.  256: 8 pairs 6.3 / 5.8, 3.1 /
    // 3.1; 64: 6.6 / 6.4, 5.6 / 5.3; 96: 6.6 / 10.6, 5.4 / 7.0; 128: 6.3 / 12.1, 9.2 / 11.5.  512: 4 pairs 10.2 / 10.2, 3.5 / 3.4; 64: 11.9 /
    // 19.0, 6.4 / 9.0; 96: 12.0 / 20.4, 10.9 / 14.6; 128: 10.9 / 22.1, 11.4 / 16.2.  32 slots, a row a warp: d = 64: 12 pairs 3.1 / 3.0, 3.0 /
    // 2.8, 96: 3.0 / 3.2, 3.3 / 3.4; 128: 64 pairs 4.1 / 3.5, 3.1 / 3.1, 96: 4.2 / 3.5, 4.1 / 4.2; 512: 64 pairs 6.3 / 6.4, 4.3 / 4.6, 80:
    // 6.4 / 8.3, 7.6 / 8.7.  128 slots, two rows a warp or four: d = 128: 4 pairs 7.2 / 7.2, 3.2 / 3.2, 64: 7.9 / 7.8, 6.2 / 6.1, 128: 7.6 /
    // 12.3, 9.2 / 11.9; 512: 16 pairs 15.5 / 15.4, 5.8 / 5.7, 64: 15.9 / 21.7, 12.3 / 17.3, 96: 17.2 / 24.9, 17.7 / 24.7.
    const long long eighths = 8LL * pairs, quarters = 4LL * pairs;           // CTAs of the clusters
    constexpr int kTwice = 2 * kSMs, kSome = DK + DV >= 512 ? 400 : (DK + DV >= 256 ? kTwice : 3 * kSMs / 2);
    if (p.m == 32 && quarters <= (DK + DV >= 256 ? kTwice : kSMs)) return launch_decode_split<IO, DK, DV, 32, 1>(p, q, k, v, gate, Ks, Vs, o, st);
    if (p.m == 64 && eighths <= kSMs) return launch_decode_split<IO, DK, DV, 64, 1>(p, q, k, v, gate, Ks, Vs, o, st);
    if (p.m == 64 && quarters <= kSome) return launch_decode_split<IO, DK, DV, 64, 2>(p, q, k, v, gate, Ks, Vs, o, st);
    if constexpr (DK + DV >= 256) {
        if (p.m == 128 && eighths <= kSMs) return launch_decode_split<IO, DK, DV, 128, 2>(p, q, k, v, gate, Ks, Vs, o, st);
        if (p.m == 128 && quarters <= kTwice) return launch_decode_split<IO, DK, DV, 128, 4>(p, q, k, v, gate, Ks, Vs, o, st);
    }
    const int is_log = p.gate_kind;
    const float inv_tau = p.tau > 0.f ? 1.f / p.tau : 0.f;
    if (p.m == 128)
        return launch_step<decode_step_kernel<IO, DK, DV, 128>>(pairs, st, q, k, v, gate, p.gate_dtype == GSA_BF16, p.gate_broadcast ? p.H : 0, p.feature_map, is_log, inv_tau, p.scale, p.slot_act, Ks, Vs, o);
    if (p.m == 64)
        return launch_step<decode_step_kernel<IO, DK, DV, 64>>(pairs, st, q, k, v, gate, p.gate_dtype == GSA_BF16, p.gate_broadcast ? p.H : 0, p.feature_map, is_log, inv_tau, p.scale, p.slot_act, Ks, Vs, o);
    return launch_step<decode_step_kernel<IO, DK, DV, 32>>(pairs, st, q, k, v, gate, p.gate_dtype == GSA_BF16, p.gate_broadcast ? p.H : 0, p.feature_map, is_log, inv_tau, p.scale, p.slot_act, Ks, Vs, o);
}

template <typename IO, int DK>
static cudaError_t launch_decode_dv(const gsa_params_t& p, const IO* q, const IO* k, const IO* v,
                                    const float* gate, float* Ks, float* Vs, IO* o, cudaStream_t st) {
    switch (p.d_v) {
        case 64: return launch_decode_m<IO, DK, 64>(p, q, k, v, gate, Ks, Vs, o, st);
        case 128: return launch_decode_m<IO, DK, 128>(p, q, k, v, gate, Ks, Vs, o, st);
        case 256: return launch_decode_m<IO, DK, 256>(p, q, k, v, gate, Ks, Vs, o, st);
        default: return launch_decode_m<IO, DK, 512>(p, q, k, v, gate, Ks, Vs, o, st);
    }
}

template <typename IO>
static cudaError_t launch_decode_io(const gsa_params_t& p, const void* q, const void* k, const void* v,
                                    const float* gate, float* Ks, float* Vs, void* o, cudaStream_t st) {
    const IO* q_ = (const IO*)q; const IO* k_ = (const IO*)k; const IO* v_ = (const IO*)v; IO* o_ = (IO*)o;
    switch (p.d_k) {
        case 64: return launch_decode_dv<IO, 64>(p, q_, k_, v_, gate, Ks, Vs, o_, st);
        case 128: return launch_decode_dv<IO, 128>(p, q_, k_, v_, gate, Ks, Vs, o_, st);
        case 256: return launch_decode_dv<IO, 256>(p, q_, k_, v_, gate, Ks, Vs, o_, st);
        default: return launch_decode_dv<IO, 512>(p, q_, k_, v_, gate, Ks, Vs, o_, st);
    }
}

cudaError_t launch_decode(const gsa_params_t& p, const void* q, const void* k, const void* v,
                          const float* gate, float* Ks, float* Vs, void* o, cudaStream_t st) {
    if (p.io == GSA_BF16) return launch_decode_io<__nv_bfloat16>(p, q, k, v, gate, Ks, Vs, o, st);
    return launch_decode_io<float>(p, q, k, v, gate, Ks, Vs, o, st);
}

}  // namespace gsa
