// Host side of the tensor-core scans that is common to the kernels, and the general kernels as launches of their own,
// for the fused kernel (chunk_tc_fused.cu), which does not carry them.
#include "chunk_tc_general.cuh"

namespace gsa {
namespace {

__global__ void __launch_bounds__(kScanThreads, 1)
value_side_general_kernel(const __grid_constant__ GeneralValueMaps maps, const __grid_constant__ ValueSideArgs a, const int* __restrict__ strong_flag, int32_t* dev_status) {
    if (strong_flag[blockIdx.x] == 0) return;
    write_input_gate(a);
    value_side_general<false>(maps.steps(), a, dev_status, blockIdx.y);
}
__global__ void __launch_bounds__(kScanThreads, 1)
key_side_general_kernel(const __grid_constant__ GeneralKeyMaps maps, const __grid_constant__ KeySideArgs a, const int* __restrict__ strong_flag, int32_t* dev_status) {
    if (strong_flag[blockIdx.x] != 0) key_side_general<false>(maps.steps(), a, dev_status, blockIdx.y);
}

}  // namespace

// The fused kernel serves the pairs without a strong-decay chunk only; the flagged ones run on a side stream of the
// calling host thread, beside it.  fork: the side stream waits for what precedes on the caller's stream; join: the
// caller's stream waits for the side stream.
namespace {
constexpr int kMaxLaneDevices = 64;
thread_local SideLane g_side_lanes[kMaxLaneDevices];
}  // namespace

cudaError_t side_lane(SideLane** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxLaneDevices) return cudaErrorInvalidDevice;
    SideLane& l = g_side_lanes[dev];
    if (l.stream == nullptr) {
        e = cudaStreamCreateWithFlags(&l.stream, cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&l.fork, cudaEventDisableTiming);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&l.join, cudaEventDisableTiming);
        if (e != cudaSuccess) return e;
    }
    *out = &l;
    return cudaSuccess;
}

// destroys the calling thread's side stream and events on the current device (created again on demand)
cudaError_t side_lane_release() {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxLaneDevices) return cudaErrorInvalidDevice;
    SideLane& l = g_side_lanes[dev];
    if (l.stream != nullptr) {
        cudaStreamDestroy(l.stream);
        if (l.fork != nullptr) cudaEventDestroy(l.fork);
        if (l.join != nullptr) cudaEventDestroy(l.join);
        l = SideLane{};
    }
    return cudaSuccess;
}

// Head dimensions the tensor-core kernels serve: multiples of the 128-wide slice, and 64 (half a
// slice: the tile copies zero-fill the channels beyond the head, stores are clipped).
bool tc_dim_ok(int D) { return D == 64 || (D > 0 && D % kDST == 0); }
bool tc_supported(int d_k, int d_v, int M) {
    return M == kM && tc_dim_ok(d_k) && tc_dim_ok(d_v);
}
int tc_value_side_slices(int D) { return (D + kDST - 1) / kDST; }
int tc_chunk() { return kCT; }

cudaError_t launch_value_side_general(const ValueSideArgs& a, const int* strong_flag, cudaStream_t st, int32_t* dev_status) {
    GeneralValueMaps maps;
    cudaError_t e = make_general_maps(&maps, a);
    if (e == cudaSuccess) e = prepare<value_side_general_kernel>(kSmemGeneral);
    if (e != cudaSuccess) return e;
    const dim3 grid(a.B * a.nseg * a.H, tc_value_side_slices(a.D));
    value_side_general_kernel<<<grid, kScanThreads, kSmemGeneral, st>>>(maps, a, strong_flag, dev_status);
    return cudaGetLastError();
}

cudaError_t launch_key_side_general(const KeySideArgs& a, const int* strong_flag, cudaStream_t st, int32_t* dev_status) {
    GeneralKeyMaps maps;
    cudaError_t e = make_general_maps(&maps, a);
    if (e == cudaSuccess) e = prepare<key_side_general_kernel>(kSmemGeneral);
    if (e != cudaSuccess) return e;
    const dim3 grid(a.B * a.nseg * a.H, tc_value_side_slices(a.D));
    key_side_general_kernel<<<grid, kScanThreads, kSmemGeneral, st>>>(maps, a, strong_flag, dev_status);
    return cudaGetLastError();
}

}  // namespace gsa
