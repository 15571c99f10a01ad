// Pixel kernel on pairs of SMs: forward and backward-data contractions large enough that every SM has several 128 x 256
// tiles with long K loops (signed codes).  Two CTAs of a cluster work on two pixel tiles of one node and the same 256 channels; the
// leader issues one tcgen05.mma.cta_group::2 of M = 256 for both, each CTA holds its own 128 pixels and half of the
// channels' weights in shared memory, and its 128 rows of the accumulator in its own tensor memory.
//
// What bounds the one-SM kernel there is shared memory: per 128 x 256 x 32-byte step it reads 4 KB of pixels and 8 KB of
// weights and TMA writes as much, 192 bytes a cycle at the tensor cores' full rate, above the 128 it has.  Halving the
// weights leaves 128.  In one run, forward / backward-data: 8192 x 8192 x 8192 0.359 / 0.342 ms against 0.403 / 0.410 on
// one SM, 256 x 56x56 256 -> 256 3x3 0.360 / 0.345 against 0.410 / 0.438 ms, 8192 x 2048 x 2048 31 / 31 against 44 / 45 us.
// (Backward-weight already shares an error tile between two accumulators and stays on one SM.)
//
// Roles per CTA as in the one-SM kernel: warp 0 fetches its own operands and signals the LEADER's full barrier (64 KB a
// stage, both CTAs together), warp 1 of the leader issues the MMAs and commits to the empty and accumulator barriers of
// both CTAs, warps 2-9 run the epilogue and release the accumulator at the leader's barrier.  Every wait is bounded.
#include <stdlib.h>
#include "qconv_internal.cuh"
#include "tc_common.cuh"

namespace lpdt {
namespace tc {

constexpr int kPairThreads = 320, kPairStages = 6, kPairUnit = 16384, kPairBN = 256, kPairRaster = 8;

struct PairParams {
    int mode;
    int nodes, B, Hout, Wout, R, S, pad;
    int Nc, cpt, taps;                        // result channels, 128-byte boxes of summed channels per tap
    int w_rows_per_node;
    int TB, TH, TW, tilesB, tilesH, tilesW, tilesN, pairs;       // pairs of pixel tiles per node (the last may be half empty)
    const float *s1, *s2, *bias; long long bias_stride;
    const float *addend;
    int32_t *dev_status;
};
struct PairCtl {
    unsigned long long full[kPairStages], empty[kPairStages], tmem_full[2], tmem_empty[2];
    uint32_t tmem_base;
    volatile int abort_flag;
};

__device__ __forceinline__ uint32_t cluster_rank() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// shared::cluster address of the same variable in the CTA of rank `rank`
__device__ __forceinline__ uint32_t peer_addr(uint32_t local, uint32_t rank) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(local), "r"(rank));
    return a;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t addr) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
// Loads into this CTA that signal a barrier of the pair's leader (no multicast).
__device__ __forceinline__ void pair_load_3d(uint32_t dst, const CUtensorMap *map, uint32_t bar, int c0, int c1, int c2) {
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2) : "memory");
}
__device__ __forceinline__ void pair_load_5d(uint32_t dst, const CUtensorMap *map, uint32_t bar, int c0, int c1, int c2, int c3, int c4) {
    asm volatile(
        "cp.async.bulk.tensor.5d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6, %7}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4) : "memory");
}
__device__ __forceinline__ void pair_mma_i8(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::i8 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
// arrives at the barrier of this offset in both CTAs once the MMAs issued so far have completed
__device__ __forceinline__ void pair_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(bar), "h"((uint16_t)3) : "memory");
}

struct PairTile { int tw, th, tb, nt, node; };
// Groups of kPairRaster pair rows sweep all N tiles, so that the tiles in flight share operand panels in L2.
__device__ __forceinline__ PairTile pair_tile(const PairParams &p, int tile, int rank) {
    const int rows = p.nodes * p.pairs, per_group = kPairRaster * p.tilesN;
    const int g = tile / per_group, rem = tile - g * per_group;
    int gsize = rows - g * kPairRaster; if (gsize > kPairRaster) gsize = kPairRaster;
    PairTile c;
    c.nt = rem / gsize;
    const int row = g * kPairRaster + (rem - c.nt * gsize);
    c.node = row / p.pairs;
    int m = (row - c.node * p.pairs) * 2 + rank;
    c.tw = m % p.tilesW; m /= p.tilesW;
    c.th = m % p.tilesH; c.tb = m / p.tilesH;          // tb = tilesB: the empty half of the last pair, all out of range
    return c;
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPairThreads, 1)
conv_pair_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapW,
                 const __grid_constant__ CUtensorMap mapY, const PairParams p) {
    extern __shared__ __align__(1024) unsigned char smem[];
    PairCtl *ctl = reinterpret_cast<PairCtl *>(smem);
    unsigned char *data = smem + 1024, *staging = data + kPairStages * 2 * kPairUnit;
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const int total = p.nodes * p.pairs * p.tilesN, first = (int)(blockIdx.x >> 1), step = (int)(gridDim.x >> 1);
    const int iters = p.taps * p.cpt;

    if (threadIdx.x == 0) {
        for (int i = 0; i < kPairStages; ++i) { mbar_init(smem_u32(&ctl->full[i]), 1); mbar_init(smem_u32(&ctl->empty[i]), 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(smem_u32(&ctl->tmem_full[i]), 1); mbar_init(smem_u32(&ctl->tmem_empty[i]), 16); }
        ctl->abort_flag = 0;
        mbar_fence_init();
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem_base)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();           // the other CTA's barriers are initialised
    tc_fence_after();
    pdl_enter();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, ctl->tmem_base, 0);

    if (warp == 0) {
        if (elect_one()) { tma_prefetch_desc(&mapA); tma_prefetch_desc(&mapW); }
        int st = 0; uint32_t ph = 0;
        for (int tile = first; tile < total && !ctl->abort_flag; tile += step) {
            const PairTile c = pair_tile(p, tile, (int)rank);
            const int n0 = c.nt * kPairBN + (int)rank * 128, w0 = c.tw * p.TW, h0 = c.th * p.TH, b0 = c.tb * p.TB;
            const int wrow = c.node * p.w_rows_per_node;
            int chunk = 0, tap = 0, r = 0, s = 0;
            for (int it = 0; it < iters; ++it) {
                if (!mbar_wait(smem_u32(&ctl->empty[st]), ph ^ 1, &ctl->abort_flag, p.dev_status)) break;
                const uint32_t full = peer_addr(smem_u32(&ctl->full[st]), 0);
                const bool leader = elect_one();
                if (leader) {
                    if (rank == 0) mbar_expect_tx(smem_u32(&ctl->full[st]), 4 * kPairUnit);
                    const uint32_t a_dst = smem_u32(data + (size_t)st * 2 * kPairUnit), b_dst = a_dst + kPairUnit;
                    const int dh = p.mode == 0 ? r - p.pad : p.pad - r, dw = p.mode == 0 ? s - p.pad : p.pad - s;
                    pair_load_5d(a_dst, &mapA, full, chunk * 128, w0 + dw, h0 + dh, b0, c.node);
                    if (p.mode == 0) pair_load_3d(b_dst, &mapW, full, chunk * 128, tap, wrow + n0);
                    else pair_load_3d(b_dst, &mapW, full, n0, tap, wrow + chunk * 128);
                }
                __syncwarp();
                if (++chunk == p.cpt) { chunk = 0; ++tap; if (++s == p.S) { s = 0; ++r; } }
                if (++st == kPairStages) { st = 0; ph ^= 1; }
            }
        }
        // the leader's commits reach this CTA's empty barriers from outside: all of them before the CTA may end
        for (int i = 0; i < kPairStages && !ctl->abort_flag; ++i) {
            mbar_wait(smem_u32(&ctl->empty[st]), ph ^ 1, &ctl->abort_flag, p.dev_status);
            if (++st == kPairStages) { st = 0; ph ^= 1; }
        }
    } else if (warp == 1) {
        if (rank == 0) {
            const uint32_t idesc = idesc_i8(256, kPairBN, 0, p.mode == 0 ? 0 : 1, 0);
            const uint64_t a_tpl = smem_desc(0, 16, 1024, 2), b_tpl = p.mode == 0 ? a_tpl : smem_desc(0, kPairUnit, 1024, 2);
            const uint32_t b_step = p.mode == 0 ? 2 : 256;                  // 32 K bytes of a row, or 32 rows of 128 bytes
            int st = 0; uint32_t ph = 0, tcount = 0;
            for (int tile = first; tile < total && !ctl->abort_flag; tile += step, ++tcount) {
                const int acc = tcount & 1;
                if (!mbar_wait(smem_u32(&ctl->tmem_empty[acc]), ((tcount >> 1) & 1) ^ 1, &ctl->abort_flag, p.dev_status)) break;
                tc_fence_after();
                bool ok = true;
                for (int it = 0; it < iters; ++it) {
                    if (!mbar_wait(smem_u32(&ctl->full[st]), ph, &ctl->abort_flag, p.dev_status)) { ok = false; break; }
                    tc_fence_after();
                    if (elect_one()) {
                        uint32_t a_lo = smem_u32(data + (size_t)st * 2 * kPairUnit) >> 4, b_lo = a_lo + (kPairUnit >> 4);
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            pair_mma_i8(tmem_base + acc * kPairBN, a_tpl | (a_lo & 0x3FFFu), b_tpl | (b_lo & 0x3FFFu), idesc, (uint32_t)(it | k));
                            a_lo += 2; b_lo += b_step;
                        }
                        pair_commit(smem_u32(&ctl->empty[st]));
                        if (it == iters - 1) pair_commit(smem_u32(&ctl->tmem_full[acc]));
                    }
                    __syncwarp();
                    if (++st == kPairStages) { st = 0; ph ^= 1; }
                }
                if (!ok) break;
            }
        }
    } else {
        const int q = warp & 3, half = (warp - 2) >> 2, row = q * 32 + lane;
        const int pw = row % p.TW, phh = (row / p.TW) % p.TH, pb = row / (p.TW * p.TH);
        unsigned char *buf = staging + (warp - 2) * 4096;
        const int r0 = q * 32, box_w0 = r0 % p.TW, box_h0 = (r0 / p.TW) % p.TH, box_b0 = r0 / (p.TW * p.TH);
        if (lane == 0) tma_prefetch_desc(&mapY);
        const uint32_t empty0 = peer_addr(smem_u32(&ctl->tmem_empty[0]), 0), sw = (uint32_t)(lane & 7);
        int sc_node = -1; float sc = 0.f;
        uint32_t tcount = 0;
        for (int tile = first; tile < total && !ctl->abort_flag; tile += step, ++tcount) {
            const PairTile c = pair_tile(p, tile, (int)rank);
            const int n0 = c.nt * kPairBN, w = c.tw * p.TW + pw, h = c.th * p.TH + phh, b = c.tb * p.TB + pb;
            const bool some = c.tb < p.tilesB, valid = w < p.Wout && h < p.Hout && b < p.B;
            if (c.node != sc_node) { sc_node = c.node; sc = __fmul_rn(p.s1[c.node], p.s2[c.node]); }
            const int acc = tcount & 1;
            if (!mbar_wait(smem_u32(&ctl->tmem_full[acc]), (tcount >> 1) & 1, &ctl->abort_flag, p.dev_status)) break;
            tc_fence_after();
            const long long pix = (((long long)c.node * p.B + b) * p.Hout + h) * p.Wout + w;
            const uint32_t t_row = tmem_base + ((uint32_t)(q * 32) << 16) + acc * kPairBN;
            // as in the one-SM kernel: 32 channels -> fp32 -> swizzled rows of this warp's buffer -> one bulk store, the
            // next 32 fetched meanwhile
            const int bn = p.Nc - n0 < kPairBN ? p.Nc - n0 : kPairBN;
            uint32_t v[32];
            int cc = half * 32;
            bool have = some && cc < bn;
            if (have) tmem_ld_32x32(t_row + cc, v);
            while (have) {
                tmem_ld_wait();
                float f[32];
#pragma unroll
                for (int k = 0; k < 32; ++k) f[k] = __fmul_rn(__int2float_rn((int)v[k]), sc);
                const int ncc = cc + 64;
                const bool more = ncc < bn;
                if (more) tmem_ld_32x32(t_row + ncc, v);
                if (p.bias) {
#pragma unroll
                    for (int k = 0; k < 32; ++k)
                        if (cc + k < bn) f[k] = __fadd_rn(f[k], p.bias[(long long)c.node * p.bias_stride + n0 + cc + k]);
                }
                if (p.addend && valid) {
                    const float4 *ad = reinterpret_cast<const float4 *>(p.addend + pix * p.Nc + n0 + cc);
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        if (cc + 4 * k >= bn) continue;
                        const float4 a4 = ad[k];
                        f[4 * k] = __fadd_rn(f[4 * k], a4.x); f[4 * k + 1] = __fadd_rn(f[4 * k + 1], a4.y);
                        f[4 * k + 2] = __fadd_rn(f[4 * k + 2], a4.z); f[4 * k + 3] = __fadd_rn(f[4 * k + 3], a4.w);
                    }
                }
                if (lane == 0) tma_store_wait_read<0>();
                __syncwarp();
                float4 *grow = reinterpret_cast<float4 *>(buf + lane * 128);
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    grow[(uint32_t)k ^ sw] = make_float4(f[4 * k], f[4 * k + 1], f[4 * k + 2], f[4 * k + 3]);
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    tma_store_5d(&mapY, smem_u32(buf), n0 + cc, c.tw * p.TW + box_w0, c.th * p.TH + box_h0, c.tb * p.TB + box_b0, c.node);
                    tma_store_commit();
                }
                cc = ncc; have = more;
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(empty0 + acc * 8);
        }
        if (lane == 0) tma_store_wait_all();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();           // neither CTA leaves while the other may still signal it or read its operands
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
    }
}

// LPDT_PIX_PAIR=0: one SM per tile for every shape (A/B timing)
static bool pair_enabled() {
    static int on = -1;
    if (on < 0) { const char *e = getenv("LPDT_PIX_PAIR"); on = (e && e[0] == '0') ? 0 : 1; }
    return on == 1;
}

lpdt_status tc_pix_pair(const lpdt_conv_desc &d, int mode, const PixTile &t, int cpt, const CUtensorMap &mA, const CUtensorMap &mY,
                        const int8_t *Wq, int pitch_w, const float *s1, const float *s2, const float *bias, int64_t bias_stride,
                        int32_t *dev_status, cudaStream_t st, const float *addend) {
    PairParams p = {};
    p.mode = mode; p.nodes = d.nodes; p.B = d.B;
    p.Hout = mode == 0 ? conv_out(d.H, d.pad, d.R, 1) : d.H; p.Wout = mode == 0 ? conv_out(d.W, d.pad, d.S, 1) : d.W;
    p.R = d.R; p.S = d.S; p.pad = d.pad; p.taps = d.R * d.S; p.cpt = cpt;
    p.Nc = mode == 0 ? d.Cout : d.Cin; p.w_rows_per_node = d.Cout;
    p.TB = t.TB; p.TH = t.TH; p.TW = t.TW; p.tilesB = t.tilesB; p.tilesH = t.tilesH; p.tilesW = t.tilesW;
    p.tilesN = (int)ceil_div(p.Nc, kPairBN);
    const long long tiles = (long long)t.tilesB * t.tilesH * t.tilesW;
    const long long total = (long long)p.nodes * ((tiles + 1) / 2) * p.tilesN;
    if (!pair_enabled() || total > 0x3fffffff) return LPDT_ERR_UNSUPPORTED;
    p.pairs = (int)((tiles + 1) / 2);
    p.s1 = s1; p.s2 = s2; p.bias = bias; p.bias_stride = bias_stride; p.addend = addend; p.dev_status = dev_status;
    CUtensorMap mW;
    uint64_t dims[3] = {(uint64_t)d.Cin, (uint64_t)p.taps, (uint64_t)d.nodes * d.Cout};
    uint64_t strides[2] = {(uint64_t)pitch_w, (uint64_t)p.taps * pitch_w};
    uint32_t box[3] = {128, 1, 128};
    if (!make_map_u8(&mW, Wq, 3, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B)) return LPDT_ERR_UNSUPPORTED;
    const size_t smem = 1024 + (size_t)kPairStages * 2 * kPairUnit + 32 * 1024;
    static PerDeviceOnce attr;
    int dev;
    if (attr.pending(&dev)) {
        LPDT_CUDA(cudaFuncSetAttribute(conv_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        attr.mark(dev);
    }
    const long long ctas = 2 * total < kNumSMs ? 2 * total : kNumSMs;
    g_last_kernel = "lpdt::tc::conv_pair_kernel";
    launch_k(conv_pair_kernel, (unsigned)ctas, kPairThreads, smem, st, mA, mW, mY, p);
    LPDT_LAUNCH_CHECK();
    return LPDT_OK;
}

}  // namespace tc
}  // namespace lpdt
