// Version and status strings, the status-word read-back and the message byte count of the lpdt library.
#include "common.cuh"

extern "C" const char *lpdt_version(void) { return "lpdt 0.1 (sm_100a)"; }

extern "C" const char *lpdt_last_kernel(void) { return lpdt::g_last_kernel; }
extern "C" uint64_t lpdt_launch_count(void) { return lpdt::g_launch_count; }

namespace lpdt {

// ResNet-20 on 40 nodes (sums of 0.2 to 2.9 MB beside the main stream): 2895 us a step, 2938 with kernels for those as well.
constexpr size_t kZeroByCopyEngine = 64u << 10;

__global__ void __launch_bounds__(256) zero_kernel(uint32_t *__restrict__ p, int n, int head /*words before a 16-byte boundary*/) {
    pdl_enter();
    const int t = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
    uint4 *p4 = reinterpret_cast<uint4 *>(p + head);
    const int n4 = (n - head) / 4;
    for (int i = t; i < n4; i += nth) p4[i] = make_uint4(0u, 0u, 0u, 0u);
    if (t < head) p[t] = 0u;
    if (t < n - head - 4 * n4) p[head + 4 * n4 + t] = 0u;
}

cudaError_t zero_async(void *p, size_t bytes, cudaStream_t st) {
    if (bytes == 0) return cudaSuccess;
    if (bytes >= kZeroByCopyEngine || bytes % 4 || !aligned(p, 4)) return cudaMemsetAsync(p, 0, bytes, st);
    const int n = (int)(bytes / 4);
    int head = (int)((16 - (uintptr_t)p % 16) % 16 / 4);
    if (head > n) head = n;
    const int64_t blocks = ceil_div(n, 1024);
    return launch_k(zero_kernel, (unsigned)(blocks < kNumSMs * 8 ? blocks : kNumSMs * 8), 256, 0, st, (uint32_t *)p, n, head);
}

// Whether the byte at p is memory of the current device.
static bool on_device(const void *p) {
    cudaPointerAttributes a;
    int dev;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) { (void)cudaGetLastError(); return false; }
    return a.type == cudaMemoryTypeDevice && cudaGetDevice(&dev) == cudaSuccess && a.device == dev;
}

}  // namespace lpdt

// (Anything but memory of this device, first byte and last, is for the runtime's fill to take or to refuse: a kernel would fault.)
extern "C" lpdt_status lpdt_fill_zero(void *p, size_t bytes, void *stream) {
    if (bytes == 0) return LPDT_OK;
    LPDT_CHECK_ARG(p != nullptr);
    const bool ours = lpdt::on_device(p) && lpdt::on_device((const char *)p + bytes - 1);
    LPDT_CUDA(ours ? lpdt::zero_async(p, bytes, lpdt::as_stream(stream)) : cudaMemsetAsync(p, 0, bytes, lpdt::as_stream(stream)));
    return LPDT_OK;
}

extern "C" const char *lpdt_status_string(lpdt_status s) {
    switch (s) {
        case LPDT_OK: return "ok";
        case LPDT_ERR_INVALID_ARG: return "invalid argument";
        case LPDT_ERR_UNSUPPORTED: return "unsupported shape or mode";
        case LPDT_ERR_WORKSPACE: return "workspace missing or too small";
        case LPDT_ERR_CUDA: return "CUDA call failed";
        case LPDT_ERR_TIMEOUT: return "device-side wait timed out";
        case LPDT_ERR_OVERFLOW: return "integer overflow";
        default: return "unknown status";
    }
}

// The one call of the library that waits: everything enqueued on `stream` so far has finished when it
// returns, and the value of the status word at that moment is the result.
extern "C" lpdt_status lpdt_check_status(const int32_t *dev_status, void *stream) {
    LPDT_CHECK_ARG(dev_status != nullptr);
    int32_t host = 0;
    cudaStream_t st = lpdt::as_stream(stream);
    LPDT_CUDA(cudaMemcpyAsync(&host, dev_status, sizeof(host), cudaMemcpyDeviceToHost, st));
    LPDT_CUDA(cudaStreamSynchronize(st));
    return (host >= LPDT_OK && host <= LPDT_ERR_OVERFLOW) ? (lpdt_status)host : LPDT_ERR_CUDA;
}

// Host arithmetic only: the size of what one node hands to each neighbour in one gossip step.
extern "C" int64_t lpdt_message_bytes(int64_t d, int32_t n_segments, const int64_t *seg_offsets,
                                      const int64_t *seg_k, int32_t value_bits, int32_t index_bits) {
    if (d < 0 || n_segments < 1 || !seg_offsets || !seg_k) return -1;
    if ((value_bits != 8 && value_bits != 16 && value_bits != 32) || index_bits < 0 || index_bits > 64) return -1;
    if (seg_offsets[0] != 0 || seg_offsets[n_segments] != d) return -1;
    int64_t bits = 0;
    for (int s = 0; s < n_segments; ++s) {
        const int64_t len = seg_offsets[s + 1] - seg_offsets[s];
        if (len < 0 || seg_k[s] < 0) return -1;
        const int64_t k = seg_k[s] < len ? seg_k[s] : len;
        bits += k * value_bits;
        if (k < len) bits += k * index_bits;          // a dense segment needs no positions
        if (value_bits == 8 && k > 0) bits += 32;      // the fp32 step of the segment's 8-bit codes
    }
    return (bits + 7) / 8;
}
