// A product launched behind a kernel that lets it start at once and then takes its time: its activation copies wait for that
// kernel, so every wait on them runs out at the short limit handed in. No access or barrier depends on which wait it is.
#include "../paper_2312_05693_b200/csrc/aq_common.cuh"

namespace {
__device__ unsigned long long now_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}
__global__ void busy_kernel(unsigned long long ns) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const unsigned long long t0 = now_ns();
    for (int i = 0; i < 100000000 && now_ns() - t0 < ns; ++i) {}
}
}  // namespace

// ms: from the start of the kernel ahead to the end of the product. Returns a CUDA error code.
extern "C" int starved_product(int device, int M, int K, int N, const void* codes, const void* packed, const void* scales, void* y,
                               void* ctl, void* scratch, size_t scratch_bytes, unsigned long long busy_ns, unsigned long long wait_cycles,
                               float* ms) {
    aq::DeviceInfo dev = {};
    dev.device = device;
    cudaDriverEntryPointQueryResult found;
    cudaError_t e = cudaSetDevice(device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&dev.sm_count, cudaDevAttrMultiProcessorCount, device);
    if (e == cudaSuccess) e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &dev.encode_tiled, cudaEnableDefault, &found);
    cudaStream_t stream = nullptr;
    cudaEvent_t begin = nullptr, end = nullptr;
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&stream, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreate(&begin);
    if (e == cudaSuccess) e = cudaEventCreate(&end);
    if (e != cudaSuccess) return (int)e;
    aq::GemmArgs a = {};
    a.q = static_cast<const int8_t*>(codes);
    a.M = M; a.K = K; a.N = N; a.group = 128;
    a.w_packed = static_cast<const uint8_t*>(packed);
    a.w_scales = static_cast<const __half*>(scales);
    a.ctl = static_cast<aq::Control*>(ctl);
    a.scale_exp = &a.ctl->scale_exp;
    a.y = static_cast<__half*>(y);
    a.split_scratch = static_cast<float*>(scratch);
    a.split_bytes = scratch_bytes;
    a.after_quantize = true;                       // may start while the kernel ahead runs
    a.wait_cycles = wait_cycles;
    cudaEventRecord(begin, stream);
    busy_kernel<<<1, 32, 0, stream>>>(busy_ns);
    e = aq::launch_gemm_tensor(a, dev, stream);
    cudaEventRecord(end, stream);
    const cudaError_t done = cudaStreamSynchronize(stream);
    if (e == cudaSuccess) e = done;
    if (e == cudaSuccess) e = cudaEventElapsedTime(ms, begin, end);
    cudaEventDestroy(begin);
    cudaEventDestroy(end);
    cudaStreamDestroy(stream);
    return (int)e;
}
