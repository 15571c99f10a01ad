// Per-tensor, per-node 8-bit quantizer: a range reduction followed by a
// scale-and-round pass (Section 3, "Low Precision Training").  Both passes are
// HBM-bound streaming kernels: 16-byte loads, warp-shuffle reduction of the
// range, one atomic per block; the second pass stores 4 codes per thread.
#include <atomic>
#include <type_traits>
#include "common.cuh"

namespace lpdt {

// ---- Philox4x32-10 (Salmon et al., SC'11), from the published round function.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
        uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
        c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
        k.x += 0x9E3779B9u;
        k.y += 0xBB67AE85u;
    }
    return c;
}
// (r >> 8) * 2^-24 without the conversion unit: the bits of a 24-bit integer m, read as a float, are m * 2^-149 (below 2^23
// a denormal, from there on the first normal binade, which has the same spacing), and the scaling is exact.
__device__ __forceinline__ float u24(uint32_t r) { return __fmul_rn(__uint_as_float(r >> 8), 0x1p125f); }
// Rounding to integers by adding 1.5 * 2^23 (nearest-even, exact for |t| < 2^22): the conversion unit, which rintf,
// floorf and (int) use, runs at an eighth of the adders' rate (stochastic quantizer, 8 x 4.2 M values: 52.8 -> 50.1 us
// together with the range; without it 47.6, and 41.1 with the shorter u24 and q_sym_sr below and a 32-bit Philox counter).  The low byte of the biased sum is the two's-complement code.
constexpr float kRoundBias = 12582912.f;
__device__ __forceinline__ float clamp127(float r) { return fminf(fmaxf(r, -127.f), 127.f); }
__device__ __forceinline__ uint32_t biased(float r) { return __float_as_uint(__fadd_rn(r, kRoundBias)); }
__device__ __forceinline__ uint32_t pack_low_bytes(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    return __byte_perm(__byte_perm(a, b, 0x0040), __byte_perm(c, d, 0x0040), 0x5410);
}

// ws[2*node] = bits of max(0, max x) or of max|x|; ws[2*node+1] = bits of -min(0, min x).
// Non-negative floats order like their bit patterns, so atomicMax on uint works.
// (eight blocks an SM, which the grid is made for, leave 32 registers; with 33 it ran in two waves: 8 x 4.2 M values, range
// and nearest codes 47.4 us, 42.0 with one)
template <bool AFFINE, bool VEC>
__global__ void __launch_bounds__(256, 8)
range_kernel(const float *__restrict__ x, int64_t n, int64_t stride,
                             uint32_t *__restrict__ ws) {
    pdl_enter();
    const int node = blockIdx.y;
    const float *xn = x + (int64_t)node * stride;
    float hi = 0.f, nlo = 0.f;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t nth = (int64_t)gridDim.x * blockDim.x;
    if (VEC) {
        const float4 *x4 = reinterpret_cast<const float4 *>(xn);
        for (int64_t i = tid; i < n / 4; i += nth) {
            float4 v = __ldg(x4 + i);
            if (AFFINE) {
                hi = fmaxf(hi, fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w)));
                nlo = fmaxf(nlo, -fminf(fminf(v.x, v.y), fminf(v.z, v.w)));
            } else {
                hi = fmaxf(hi, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
            }
        }
    } else {
        for (int64_t i = tid; i < n; i += nth) {
            float v = xn[i];
            if (AFFINE) { hi = fmaxf(hi, v); nlo = fmaxf(nlo, -v); }
            else hi = fmaxf(hi, fabsf(v));
        }
    }
    hi = warp_max(hi);
    if (AFFINE) nlo = warp_max(nlo);
    __shared__ float s_hi[32], s_lo[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) { s_hi[warp] = hi; s_lo[warp] = nlo; }
    __syncthreads();
    if (warp == 0) {
        const int nw = blockDim.x >> 5;
        hi = lane < nw ? s_hi[lane] : 0.f;
        nlo = lane < nw ? s_lo[lane] : 0.f;
        hi = warp_max(hi);
        if (AFFINE) nlo = warp_max(nlo);
        if (lane == 0) {
            if (gridDim.x == 1) {            // nobody else has a part of this node: the words need not be cleared before
                ws[2 * node] = __float_as_uint(hi);
                ws[2 * node + 1] = AFFINE ? __float_as_uint(nlo) : 0u;
            } else {
                atomicMax(ws + 2 * node, __float_as_uint(hi));
                if (AFFINE) atomicMax(ws + 2 * node + 1, __float_as_uint(nlo));
            }
        }
    }
}

// Codes as the low byte of a word; +-127 are integers, so clamping before the rounding gives the same code.
__device__ __forceinline__ uint32_t q_sym_rne(float x, float inv) { return biased(clamp127(__fmul_rn(x, inv))); }
// The sum rounded down is floor(t) + bias; beyond 2^22 (a caller's range below max|x|) it may be off by the float's spacing,
// and the clamp, on the biased sum, decides.
__device__ __forceinline__ uint32_t q_sym_sr(float x, float inv, float u) {
    const float t = __fmul_rn(x, inv), fl = __fadd_rd(t, kRoundBias);
    const float f = __fsub_rn(t, __fsub_rn(fl, kRoundBias));
    const float r = u < f ? __fadd_rn(fl, 1.f) : fl;
    return __float_as_uint(fminf(fmaxf(r, kRoundBias - 127.f), kRoundBias + 127.f));
}
__device__ __forceinline__ uint32_t q_affine(float x, float s, float zf) {
    const float r = __fadd_rn(rintf(__fdiv_rn(x, s)), zf);
    return biased(fminf(fmaxf(r, 0.f), 255.f));
}

// The range pass before this one went upwards, so the last values of every node are the ones that L2 still holds: this
// pass goes downwards (8 x 4.2 M values, with the range: nearest 53.1 -> 47.4 us, affine 64.4 -> 58.8).  Stochastic codes are
// bound by Philox's wide multiplies and the rounding's instructions, not by memory: as many registers as it likes, 41.1 us
// without the range, 47.1 at 32 registers and eight blocks an SM.
template <int MODE /*0 sym rne, 1 sym stochastic, 2 affine*/, bool VEC>
__global__ void __launch_bounds__(256, MODE == 1 ? 4 : 8)
quantize_kernel(const float *__restrict__ x, int64_t n, int64_t stride,
                                const uint32_t *__restrict__ ws, int8_t *__restrict__ q,
                                float *__restrict__ scale, int32_t *__restrict__ zero_point,
                                uint2 key, uint32_t ctr_offset, int wstride) {
    pdl_enter();
    const int node = blockIdx.y;
    const float *xn = x + (int64_t)node * stride;
    int8_t *qn = q + (int64_t)node * n;
    float s, inv = 0.f, zf = 0.f;
    if (MODE == 2) {
        const float hi = __uint_as_float(ws[wstride * node]);
        const float lo = -__uint_as_float(ws[wstride * node + 1]);
        s = (hi == lo) ? 1.f : __fdiv_rn(__fsub_rn(hi, lo), 255.f);
        zf = rintf(__fdiv_rn(-lo, s));
        zf = fminf(fmaxf(zf, 0.f), 255.f);
    } else {
        const float amax = __uint_as_float(ws[wstride * node]);
        if (amax == 0.f) { s = 1.f; inv = 0.f; }
        else { s = __fdiv_rn(amax, 127.f); inv = __fdiv_rn(127.f, amax); }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        scale[node] = s;
        if (MODE == 2) zero_point[node] = (int)zf;
    }
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t nth = (int64_t)gridDim.x * blockDim.x;
    if (VEC) {
        const float4 *x4 = reinterpret_cast<const float4 *>(xn);
        uint32_t *q4 = reinterpret_cast<uint32_t *>(qn);
        auto walk = [&](auto wide) {
#pragma unroll 4
        for (int64_t i = n / 4 - 1 - tid; i >= 0; i -= nth) {
            const float4 v = __ldg(x4 + i);
            uint32_t a, b, c, d;
            if (MODE == 0) {
                a = q_sym_rne(v.x, inv); b = q_sym_rne(v.y, inv);
                c = q_sym_rne(v.z, inv); d = q_sym_rne(v.w, inv);
            } else if (MODE == 1) {
                uint4 r = philox4x32_10(make_uint4((uint32_t)i, decltype(wide)::value ? (uint32_t)((uint64_t)i >> 32) : 0u,
                                                   (uint32_t)node, ctr_offset), key);
                a = q_sym_sr(v.x, inv, u24(r.x)); b = q_sym_sr(v.y, inv, u24(r.y));
                c = q_sym_sr(v.z, inv, u24(r.z)); d = q_sym_sr(v.w, inv, u24(r.w));
            } else {
                a = q_affine(v.x, s, zf); b = q_affine(v.y, s, zf);
                c = q_affine(v.z, s, zf); d = q_affine(v.w, s, zf);
            }
            q4[i] = pack_low_bytes(a, b, c, d);
        }
        };
        // (a counter whose upper word is known to be zero saves two of the twenty wide multiplies)
        if (MODE == 1 && n / 4 > (int64_t)0xffffffff) walk(std::true_type{});
        else walk(std::false_type{});
    } else {
        for (int64_t i = tid; i < n; i += nth) {
            float v = xn[i];
            uint32_t a;
            if (MODE == 0) a = q_sym_rne(v, inv);
            else if (MODE == 1) {
                uint4 r = philox4x32_10(make_uint4((uint32_t)(i >> 2), (uint32_t)((uint64_t)i >> 34),
                                                   (uint32_t)node, ctr_offset), key);
                uint32_t w = (i & 3) == 0 ? r.x : (i & 3) == 1 ? r.y : (i & 3) == 2 ? r.z : r.w;
                a = q_sym_sr(v, inv, u24(w));
            } else a = q_affine(v, s, zf);
            qn[i] = (int8_t)a;
        }
    }
}

// VEC: 4 codes and one 16-byte store per step, four steps in flight (scalar 1-byte loads: 34.4 us for 8 x 4.2 M codes,
// 28.7 us).  A signed code c becomes a float as 2^23 + (c + 128), by its bits, minus 2^23 + 128, both exact.
template <bool AFFINE, bool VEC>
__global__ void __launch_bounds__(256)
dequantize_kernel(const int8_t *__restrict__ q, int64_t n,
                                  const float *__restrict__ scale,
                                  const int32_t *__restrict__ zp, float *__restrict__ y,
                                  int64_t ystride) {
    pdl_enter();
    const int node = blockIdx.y;
    const float s = scale[node];
    const int z = AFFINE ? zp[node] : 0;
    const int64_t base = (int64_t)node * n;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, nth = (int64_t)gridDim.x * blockDim.x;
    if constexpr (VEC) {
        const uint32_t *q4 = reinterpret_cast<const uint32_t *>(q + base);
        float4 *y4 = reinterpret_cast<float4 *>(y + (int64_t)node * ystride);
#pragma unroll 4
        for (int64_t i = tid; i < n / 4; i += nth) {
            const uint32_t c = __ldg(q4 + i) ^ (AFFINE ? 0u : 0x80808080u);
            float f[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (AFFINE) f[k] = __int2float_rn((int)((c >> (8 * k)) & 0xffu) - z);
                else f[k] = __fsub_rn(__uint_as_float(__byte_perm(c, 0x4b000000u, 0x7440 + k)), 8388736.f);
            }
            y4[i] = make_float4(__fmul_rn(f[0], s), __fmul_rn(f[1], s), __fmul_rn(f[2], s), __fmul_rn(f[3], s));
        }
    } else for (int64_t i = tid; i < n; i += nth) {
        int code = AFFINE ? (int)(uint8_t)q[base + i] - z : (int)q[base + i];
        y[(int64_t)node * ystride + i] = __fmul_rn(__int2float_rn(code), s);
    }
}

static int blocks_for(int64_t work_items, int nodes) {
    int64_t b = ceil_div(work_items, 256 * 4);
    int64_t cap = ceil_div((int64_t)kNumSMs * 8, nodes);
    if (b > cap) b = cap;
    if (b < 1) b = 1;
    return (int)b;
}

}  // namespace lpdt

using namespace lpdt;

constexpr int64_t kOneBlock = 4096;      // values of a node whose range one block finds

extern "C" size_t lpdt_quantize_workspace_size(int32_t nodes) {
    return align_up((size_t)(nodes > 0 ? nodes : 1) * 2 * sizeof(uint32_t), 256);
}

extern "C" lpdt_status lpdt_quantize(const float *x, int32_t nodes, int64_t n, int64_t x_node_stride,
                                     lpdt_qmode mode, lpdt_round rounding, uint64_t seed,
                                     uint32_t ctr_offset, int8_t *q, float *scale,
                                     int32_t *zero_point, void *ws, size_t ws_bytes, void *stream) {
    LPDT_CHECK_ARG(nodes >= 0 && n >= 0);
    if (nodes == 0 || n == 0) return LPDT_OK;
    LPDT_CHECK_ARG(x && q && scale);
    LPDT_CHECK_ARG(x_node_stride >= n || nodes == 1);
    LPDT_CHECK_ARG(mode == LPDT_SYM_S8 || mode == LPDT_AFFINE_U8);
    LPDT_CHECK_ARG(rounding == LPDT_ROUND_NEAREST_EVEN || rounding == LPDT_ROUND_STOCHASTIC);
    LPDT_CHECK_ARG(aligned(x, 4) && aligned(scale, 4));
    if (mode == LPDT_AFFINE_U8) {
        LPDT_CHECK_ARG(zero_point != nullptr);
        if (rounding != LPDT_ROUND_NEAREST_EVEN) return LPDT_ERR_UNSUPPORTED;
    }
    if (nodes > 65535) return LPDT_ERR_UNSUPPORTED;
    if (!ws || ws_bytes < lpdt_quantize_workspace_size(nodes)) return LPDT_ERR_WORKSPACE;
    cudaStream_t st = as_stream(stream);
    uint32_t *w = (uint32_t *)ws;
    const bool vec = aligned(x, 16) && (x_node_stride % 4 == 0) && (n % 4 == 0) && aligned(q, 4);
    dim3 grid(blocks_for(vec ? n / 4 : n, nodes), nodes), block(256);
    // the range of a short tensor is one block's work: no words to clear in a launch of their own (9 nodes x 704
    // values, in the step's chain: 1.4 us less)
    const dim3 range_grid(n <= kOneBlock ? 1 : grid.x, nodes);
    if (range_grid.x > 1) LPDT_CUDA(zero_async(w, (size_t)nodes * 2 * sizeof(uint32_t), st));
    const uint2 key = make_uint2((uint32_t)seed, (uint32_t)(seed >> 32));
    if (mode == LPDT_AFFINE_U8) {
        if (vec) launch_k(range_kernel<true, true>, range_grid, block, 0, st, x, n, x_node_stride, w);
        else launch_k(range_kernel<true, false>, range_grid, block, 0, st, x, n, x_node_stride, w);
        LPDT_LAUNCH_CHECK();
        if (vec) launch_k(quantize_kernel<2, true>, grid, block, 0, st, x, n, x_node_stride, w, q, scale, zero_point, key, ctr_offset, 2);
        else launch_k(quantize_kernel<2, false>, grid, block, 0, st, x, n, x_node_stride, w, q, scale, zero_point, key, ctr_offset, 2);
    } else {
        if (vec) launch_k(range_kernel<false, true>, range_grid, block, 0, st, x, n, x_node_stride, w);
        else launch_k(range_kernel<false, false>, range_grid, block, 0, st, x, n, x_node_stride, w);
        LPDT_LAUNCH_CHECK();
        if (rounding == LPDT_ROUND_NEAREST_EVEN) {
            if (vec) launch_k(quantize_kernel<0, true>, grid, block, 0, st, x, n, x_node_stride, w, q, scale, zero_point, key, ctr_offset, 2);
            else launch_k(quantize_kernel<0, false>, grid, block, 0, st, x, n, x_node_stride, w, q, scale, zero_point, key, ctr_offset, 2);
        } else {
            if (vec) launch_k(quantize_kernel<1, true>, grid, block, 0, st, x, n, x_node_stride, w, q, scale, zero_point, key, ctr_offset, 2);
            else launch_k(quantize_kernel<1, false>, grid, block, 0, st, x, n, x_node_stride, w, q, scale, zero_point, key, ctr_offset, 2);
        }
    }
    LPDT_LAUNCH_CHECK();
    return LPDT_OK;
}

extern "C" lpdt_status lpdt_dequantize(const int8_t *q, int32_t nodes, int64_t n, const float *scale,
                                       const int32_t *zero_point, float *y, int64_t y_node_stride,
                                       void *stream) {
    LPDT_CHECK_ARG(nodes >= 0 && n >= 0);
    if (nodes == 0 || n == 0) return LPDT_OK;
    LPDT_CHECK_ARG(q && scale && y && nodes <= 65535 && (y_node_stride >= n || nodes == 1));
    const bool vec = n % 4 == 0 && aligned(q, 4) && aligned(y, 16) && y_node_stride % 4 == 0;
    dim3 grid(blocks_for(vec ? n / 4 : n, nodes), nodes), block(256);
    using Fn = void (*)(const int8_t *, int64_t, const float *, const int32_t *, float *, int64_t);
    static const Fn fns[2][2] = {{dequantize_kernel<false, false>, dequantize_kernel<false, true>},
                                 {dequantize_kernel<true, false>, dequantize_kernel<true, true>}};
    launch_k(fns[zero_point ? 1 : 0][vec ? 1 : 0], grid, block, 0, as_stream(stream), q, n, scale, zero_point, y, y_node_stride);
    LPDT_LAUNCH_CHECK();
    return LPDT_OK;
}

extern "C" lpdt_status lpdt_quantize_with_range(const float *x, int32_t nodes, int64_t n, int64_t x_node_stride,
                                                const float *amax, lpdt_round rounding, uint64_t seed,
                                                uint32_t ctr_offset, int8_t *q, float *scale, void *stream) {
    LPDT_CHECK_ARG(nodes >= 0 && n >= 0);
    if (nodes == 0 || n == 0) return LPDT_OK;
    LPDT_CHECK_ARG(x && q && scale && amax);
    LPDT_CHECK_ARG(x_node_stride >= n || nodes == 1);
    LPDT_CHECK_ARG(rounding == LPDT_ROUND_NEAREST_EVEN || rounding == LPDT_ROUND_STOCHASTIC);
    LPDT_CHECK_ARG(aligned(x, 4) && aligned(scale, 4) && aligned(amax, 4));
    if (nodes > 65535) return LPDT_ERR_UNSUPPORTED;
    cudaStream_t st = as_stream(stream);
    const uint32_t *w = reinterpret_cast<const uint32_t *>(amax);      // non-negative floats, read as bit patterns
    const bool vec = aligned(x, 16) && (x_node_stride % 4 == 0) && (n % 4 == 0) && aligned(q, 4);
    dim3 grid(blocks_for(vec ? n / 4 : n, nodes), nodes), block(256);
    const uint2 key = make_uint2((uint32_t)seed, (uint32_t)(seed >> 32));
    if (rounding == LPDT_ROUND_NEAREST_EVEN) {
        if (vec) launch_k(quantize_kernel<0, true>, grid, block, 0, st, x, n, x_node_stride, w, q, scale, nullptr, key, ctr_offset, 1);
        else launch_k(quantize_kernel<0, false>, grid, block, 0, st, x, n, x_node_stride, w, q, scale, nullptr, key, ctr_offset, 1);
    } else {
        if (vec) launch_k(quantize_kernel<1, true>, grid, block, 0, st, x, n, x_node_stride, w, q, scale, nullptr, key, ctr_offset, 1);
        else launch_k(quantize_kernel<1, false>, grid, block, 0, st, x, n, x_node_stride, w, q, scale, nullptr, key, ctr_offset, 1);
    }
    LPDT_LAUNCH_CHECK();
    return LPDT_OK;
}

// ---------------------------------------------------------------------------
// Quantizer for callers that own no device scratch.
//
// lpdt_quantize needs a few bytes of caller-provided scratch for the per-node
// range words.  Some users of this library cannot supply any: an edge-device
// training loop that was given a fixed set of buffers at start-up and has no
// allocator afterwards, or a plug-in called from a host application whose device
// memory belongs to that application's own pool and which forbids device
// allocation on its hot path (cudaMalloc also synchronises the whole device).
// For them the range words live in the array below, which is part of the loaded
// library image: every GPU that loads the library holds these 8 KB until the
// process exits.
//
// In host code `g_static_range_words` is only a handle for the symbol, not a device
// address, so its address on the current device is looked up once per device with
// cudaGetSymbolAddress and that pointer is what the kernels receive.
constexpr int kStaticMaxNodes = LPDT_QUANTIZE_STATIC_MAX_NODES;
static __device__ __align__(256) uint32_t g_static_range_words[2 * kStaticMaxNodes];

// One cached address per device ordinal.  Two host threads that both make the first call on a device
// look the same address up and store the same value (an atomic pointer store), so the race is benign.
// The cache does not outlive a cudaDeviceReset: after one, the library must be reloaded.
constexpr int kMaxDevices = 64;
static std::atomic<uint32_t *> g_static_range_ptr[kMaxDevices];

static lpdt_status static_range_words(uint32_t **out) {
    int dev = -1;
    LPDT_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return LPDT_ERR_UNSUPPORTED;
    uint32_t *p = g_static_range_ptr[dev].load(std::memory_order_acquire);
    if (!p) {
        if (cudaGetSymbolAddress((void **)&p, g_static_range_words) != cudaSuccess || !p) {
            (void)cudaGetLastError();
            return LPDT_ERR_CUDA;
        }
        g_static_range_ptr[dev].store(p, std::memory_order_release);
    }
    *out = p;
    return LPDT_OK;
}

extern "C" lpdt_status lpdt_quantize_static(const float *x, int32_t nodes, int64_t n_per_node,
                                            int64_t x_node_stride, lpdt_qmode mode, lpdt_round rounding,
                                            uint64_t seed, uint32_t ctr_offset, int8_t *q, float *scale,
                                            int32_t *zero_point, void *stream) {
    LPDT_CHECK_ARG(nodes >= 0 && n_per_node >= 0);
    if (nodes > kStaticMaxNodes) return LPDT_ERR_WORKSPACE;     // the built-in scratch holds 1024 nodes
    if (nodes == 0 || n_per_node == 0) return LPDT_OK;          // nothing to do: no address lookup either
    uint32_t *words = nullptr;
    lpdt_status s = static_range_words(&words);
    if (s != LPDT_OK) return s;
    // Same two passes as lpdt_quantize; the words it uses are zeroed before the range pass, or stored by it,
    // so whatever the previous call left in the array does not matter.
    return lpdt_quantize(x, nodes, n_per_node, x_node_stride, mode, rounding, seed, ctr_offset, q, scale,
                         zero_point, words, sizeof(uint32_t) * 2 * kStaticMaxNodes, stream);
}

// ---------------------------------------------------------------------------
// Batched symmetric quantization of many small tensors that live inside one flat
// per-node parameter vector (all layer weights of a network): two launches in
// total instead of two per tensor.
namespace lpdt {

constexpr int kMaxBatchTensors = 64;
struct QuantBatch {
    int count;
    long long src_off[kMaxBatchTensors];    // element offset inside a node's parameter row
    long long size[kMaxBatchTensors];       // elements per node
    long long dst_off[kMaxBatchTensors];    // byte offset of the tensor's [nodes][size] block in q
};

// Four consecutive floats with the widest loads that the alignment of the tensor allows (16, 8 or 4 bytes): the rows of
// a parameter matrix whose width is even but no multiple of 4 start on 8-byte boundaries only.
__device__ __forceinline__ int load_width(const float *p) { return ((uintptr_t)p & 15) == 0 ? 16 : ((uintptr_t)p & 7) == 0 ? 8 : 4; }
__device__ __forceinline__ float4 load4(const float *p, int width) {
    if (width == 16) return __ldg(reinterpret_cast<const float4 *>(p));
    if (width == 8) {
        const float2 a = __ldg(reinterpret_cast<const float2 *>(p)), b = __ldg(reinterpret_cast<const float2 *>(p) + 1);
        return make_float4(a.x, a.y, b.x, b.y);
    }
    return make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));
}
__device__ __forceinline__ float amax4(float4 v) { return fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))); }

// (The codes are written from the last tensor back: 8 x 9.2 M weights 112.7 -> 102.5 us.)
// grid = (blocks, nodes, tensors); blocks beyond a tensor's length fall through.  Four groups of four values in flight
// per thread (one value per step: 62 + 81 us for the two passes over 8 x 9.2 M weights, 45 + 60 us now).
__global__ void __launch_bounds__(256)
batch_range_kernel(const float *__restrict__ params, long long row_stride, QuantBatch qb, uint32_t *__restrict__ ws) {
    pdl_enter();
    const int t = blockIdx.z, node = blockIdx.y;
    const long long n = qb.size[t], n4 = n / 4;
    const float *x = params + (long long)node * row_stride + qb.src_off[t];
    const int width = load_width(x);
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x, nth = (long long)gridDim.x * blockDim.x;
    if ((long long)blockIdx.x * blockDim.x >= n4 && blockIdx.x > 0) return;      // block 0 takes the last n % 4 values
    float m = 0.f;
    for (long long i = tid; i < n4; i += 4 * nth) {
        float4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = i + u * nth < n4 ? load4(x + 4 * (i + u * nth), width) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < 4; ++u) m = fmaxf(m, amax4(v[u]));
    }
    if (tid < n - 4 * n4) m = fmaxf(m, fabsf(x[4 * n4 + tid]));
    // (a block that has its tensor to itself stores: the words need not be cleared before)
    block_amax_to(m, reinterpret_cast<float *>(ws + (size_t)t * gridDim.y + node), gridDim.x == 1);
}

__global__ void __launch_bounds__(256)
batch_quantize_kernel(const float *__restrict__ params, long long row_stride, QuantBatch qb,
                      const uint32_t *__restrict__ ws, int8_t *__restrict__ q, float *__restrict__ scales) {
    pdl_enter();
    const int nodes = gridDim.y, t = gridDim.z - 1 - blockIdx.z, node = nodes - 1 - blockIdx.y;      // what the range pass read last first
    const long long n = qb.size[t], n4 = n / 4;
    const float *x = params + (long long)node * row_stride + qb.src_off[t];
    int8_t *dst = q + qb.dst_off[t] + (long long)node * n;
    const float amax = __uint_as_float(ws[(size_t)t * nodes + node]);
    float s = 1.f, inv = 0.f;
    if (amax != 0.f) { s = __fdiv_rn(amax, 127.f); inv = __fdiv_rn(127.f, amax); }
    if (blockIdx.x == 0 && threadIdx.x == 0) scales[(size_t)t * nodes + node] = s;
    const int width = load_width(x);
    const bool words = ((uintptr_t)dst & 3) == 0;
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x, nth = (long long)gridDim.x * blockDim.x;
    for (long long i = tid; i < n4; i += 4 * nth) {
        float4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) if (i + u * nth < n4) v[u] = load4(x + 4 * (i + u * nth), width);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const long long at = i + u * nth;
            if (at >= n4) break;
            const uint32_t c = pack_low_bytes(q_sym_rne(v[u].x, inv), q_sym_rne(v[u].y, inv), q_sym_rne(v[u].z, inv), q_sym_rne(v[u].w, inv));
            if (words) reinterpret_cast<uint32_t *>(dst)[at] = c;
            else {
#pragma unroll
                for (int k = 0; k < 4; ++k) dst[4 * at + k] = (int8_t)(c >> (8 * k));
            }
        }
    }
    if (tid < n - 4 * n4) dst[4 * n4 + tid] = (int8_t)q_sym_rne(x[4 * n4 + tid], inv);
}

}  // namespace lpdt

extern "C" size_t lpdt_quantize_batch_workspace_size(int32_t nodes, int32_t n_tensors) {
    return align_up((size_t)(nodes > 0 ? nodes : 1) * (size_t)(n_tensors > 0 ? n_tensors : 1) * sizeof(uint32_t), 256);
}

extern "C" lpdt_status lpdt_quantize_batch(const float *params, int32_t nodes, int64_t row_stride, int32_t n_tensors,
                                           const int64_t *src_offsets, const int64_t *sizes,
                                           const int64_t *dst_offsets, int8_t *q, float *scales, void *ws,
                                           size_t ws_bytes, void *stream) {
    LPDT_CHECK_ARG(nodes >= 0 && n_tensors >= 0);
    if (nodes == 0 || n_tensors == 0) return LPDT_OK;
    LPDT_CHECK_ARG(params && src_offsets && sizes && dst_offsets && q && scales);
    if (n_tensors > kMaxBatchTensors || nodes > 65535) return LPDT_ERR_UNSUPPORTED;
    if (!ws || ws_bytes < lpdt_quantize_batch_workspace_size(nodes, n_tensors)) return LPDT_ERR_WORKSPACE;
    QuantBatch qb;
    qb.count = n_tensors;
    long long longest = 0;
    for (int t = 0; t < n_tensors; ++t) {
        LPDT_CHECK_ARG(src_offsets[t] >= 0 && sizes[t] >= 0 && dst_offsets[t] >= 0 && src_offsets[t] + sizes[t] <= row_stride);
        qb.src_off[t] = src_offsets[t]; qb.size[t] = sizes[t]; qb.dst_off[t] = dst_offsets[t];
        if (sizes[t] > longest) longest = sizes[t];
    }
    if (longest == 0) return LPDT_OK;
    cudaStream_t st = as_stream(stream);
    uint32_t *w = (uint32_t *)ws;
    int bx = (int)ceil_div(longest, 256 * 16);
    if (bx > 64) bx = 64;
    if (bx < 1) bx = 1;
    if (bx > 1) LPDT_CUDA(zero_async(w, (size_t)nodes * n_tensors * sizeof(uint32_t), st));
    dim3 grid(bx, nodes, n_tensors);
    launch_k(batch_range_kernel, grid, 256, 0, st, params, row_stride, qb, w);
    LPDT_LAUNCH_CHECK();
    launch_k(batch_quantize_kernel, grid, 256, 0, st, params, row_stride, qb, w, q, scales);
    LPDT_LAUNCH_CHECK();
    return LPDT_OK;
}
