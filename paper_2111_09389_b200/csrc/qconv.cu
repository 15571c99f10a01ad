// Front end of the quantized contractions: argument validation, workspace
// accounting and the choice between the tensor-core engine and the CUDA-core
// kernels.  Operands whose channel count is not a multiple of 16 (the RGB first
// layer, a classifier's class scores) have rows that TMA cannot address; the engine
// reads copies of them in the workspace whose rows are padded with zeros to the next
// multiple: zero channels add nothing to an integer sum, so the result is unchanged.
// Results keep the caller's channel count.
#include <stdlib.h>
#include "common.cuh"
#include "qconv_internal.cuh"

using namespace lpdt;

namespace lpdt {

// dst[row][0..Cp) = src[row][0..C) followed by zeros, Cp the next multiple of 16.  One 16-byte piece of a destination row
// is assembled from the aligned 4-byte words that hold it (rows start at any byte) and written with a single 16-byte
// store; a thread has PIECES of them in flight.  blockIdx.y selects one of up to two tensors: both operands of a product
// in one launch.
struct PadJob { const int8_t *src; int8_t *dst; int64_t rows; int C; };
template <int PIECES>
__global__ void __launch_bounds__(256) pad_channels_kernel(const PadJob j0, const PadJob j1) {
    pdl_enter();
    const PadJob j = blockIdx.y ? j1 : j0;
    const int C = j.C, pieces = (C + 15) / 16, Cp = pieces * 16;
    const int64_t total = j.rows * pieces, bytes = j.rows * C, nth = (int64_t)gridDim.x * blockDim.x;
    const bool words = ((uintptr_t)j.src & 3) == 0;
    for (int64_t o0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; o0 < total; o0 += PIECES * nth) {
        uint32_t w[PIECES][5];
        int64_t row[PIECES];
        int c0[PIECES], n[PIECES];
        bool fits[PIECES];                                           // the piece's last word lies inside the tensor
#pragma unroll
        for (int u = 0; u < PIECES; ++u) {
            const int64_t o = o0 + u * nth;
            row[u] = total <= 0x7fffffff ? (int64_t)((uint32_t)o / (uint32_t)pieces) : o / pieces;
            c0[u] = (int)(o - row[u] * pieces) * 16;
            n[u] = o < total ? (C - c0[u] < 16 ? C - c0[u] : 16) : 0;
            const int64_t off = row[u] * C + c0[u];
            fits[u] = words && ((off + n[u] + 3) & ~(int64_t)3) <= bytes;
            const uint32_t *p = reinterpret_cast<const uint32_t *>(j.src + (off & ~(int64_t)3));
            const int need = n[u] > 0 && fits[u] ? ((int)(off & 3) + n[u] + 3) / 4 : 0;
#pragma unroll
            for (int k = 0; k < 5; ++k) w[u][k] = k < need ? __ldg(p + k) : 0u;
        }
#pragma unroll
        for (int u = 0; u < PIECES; ++u) {
            if (n[u] == 0) continue;
            const int64_t off = row[u] * C + c0[u];
            const int sh = (int)(off & 3);
            uint32_t r[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t x = __funnelshift_r(w[u][k], w[u][k + 1], 8 * sh);
                const int left = n[u] - 4 * k;                       // bytes of this word that exist
                r[k] = left >= 4 ? x : left <= 0 ? 0u : x & ((1u << (8 * left)) - 1u);
            }
            if (!fits[u]) {
                union { int8_t b[16]; uint32_t w[4]; } t;
#pragma unroll
                for (int k = 0; k < 16; ++k) t.b[k] = k < n[u] ? j.src[off + k] : (int8_t)0;
#pragma unroll
                for (int k = 0; k < 4; ++k) r[k] = t.w[k];
            }
            *reinterpret_cast<uint4 *>(j.dst + row[u] * Cp + c0[u]) = make_uint4(r[0], r[1], r[2], r[3]);
        }
    }
}

}  // namespace lpdt

static unsigned grid_for(int64_t n) {
    int64_t b = ceil_div(n, 256), cap = (int64_t)kNumSMs * 32;
    return (unsigned)(b < 1 ? 1 : (b > cap ? cap : b));
}

// LPDT_DISABLE_TC=1 in the environment routes every shape to the CUDA-core kernels.
static bool tc_enabled() {
    static int disabled = -1;
    if (disabled < 0) {
        const char *e = getenv("LPDT_DISABLE_TC");
        disabled = (e && e[0] == '1') ? 1 : 0;
    }
    return !disabled;
}
// LPDT_DISABLE_HALO=1 keeps 16-channel layers on the general tensor-core kernel.
static bool use_halo(const lpdt_conv_desc &d, int mode) {
    static int disabled = -1;
    if (disabled < 0) {
        const char *e = getenv("LPDT_DISABLE_HALO");
        disabled = (e && e[0] == '1') ? 1 : 0;
    }
    return !disabled && tc::halo_supported(d, mode);
}
static int pad16(int c) { return (c + 15) / 16 * 16; }
static tc::Pitches pitches(const lpdt_conv_desc &d) { return {pad16(d.Cin), pad16(d.Cout), pad16(d.Cin)}; }

// Operands in rows of pad16(channels) bytes.
static lpdt_status run_pix(const lpdt_conv_desc &d, int mode, const int8_t *A, const float *s1, const int8_t *Wq,
                           const float *s2, const float *bias, int64_t bias_stride, float *Y, int32_t *Yacc,
                           int32_t *dev_status, cudaStream_t st, bool uns, const float *addend,
                           const tc::AffineArgs *aff) {
    lpdt_conv_desc dh = d;                   // the halo kernel pads the summed side only: its results are whole rows
    if (mode == 0) dh.Cin = pad16(d.Cin);
    if (!aff && use_halo(dh, mode)) {
        lpdt_status r = tc::tc_pix_halo(dh, mode, A, s1, Wq, s2, bias, bias_stride, Y, Yacc, dev_status, st, uns, addend);
        if (r != LPDT_ERR_UNSUPPORTED) return r;
    }
    return tc::tc_pix(d, mode, A, s1, Wq, s2, bias, bias_stride, Y, Yacc, dev_status, st, uns, addend, aff, pitches(d));
}

static lpdt_status check_desc(const lpdt_conv_desc *d) {
    LPDT_CHECK_ARG(d != nullptr);
    LPDT_CHECK_ARG(d->nodes >= 0 && d->B >= 0 && d->H > 0 && d->W > 0 && d->Cin > 0 && d->Cout > 0);
    LPDT_CHECK_ARG(d->R > 0 && d->S > 0 && d->stride > 0 && d->pad >= 0);
    LPDT_CHECK_ARG(d->H + 2 * d->pad >= d->R && d->W + 2 * d->pad >= d->S);
    return LPDT_OK;
}

// Zero-padded copies of the operands whose channel count is no multiple of 16 (0 bytes for the others).
struct PadPlan { size_t in, err, w; };
static PadPlan pad_plan(const lpdt_conv_desc &d) {
    const int Ho = conv_out(d.H, d.pad, d.R, d.stride), Wo = conv_out(d.W, d.pad, d.S, d.stride);
    PadPlan p = {0, 0, 0};
    if (d.Cin % 16) {
        p.in = align_up((size_t)d.nodes * d.B * d.H * d.W * pad16(d.Cin), 256);
        p.w = align_up((size_t)d.nodes * d.Cout * d.R * d.S * pad16(d.Cin), 256);
    }
    if (d.Cout % 16) p.err = align_up((size_t)d.nodes * d.B * Ho * Wo * pad16(d.Cout), 256);
    return p;
}
static PadJob pad_job(const int8_t *src, void *dst, int64_t rows, int C) { return {src, (int8_t *)dst, rows, C}; }
// One launch for up to two tensors (rows = 0: none).
static lpdt_status pad_launch(PadJob a, PadJob b, cudaStream_t st) {
    if (a.rows == 0) { a = b; b.rows = 0; }
    if (a.rows == 0) return LPDT_OK;
    const int64_t na = a.rows * (pad16(a.C) / 16), nb = b.rows ? b.rows * (pad16(b.C) / 16) : 0;
    // four pieces per thread where that leaves the chip full: 16 nodes x 32 x 32x32 x 3 (524 K pieces, 3x3 to 16 channels
    // forward) 18.2 us with four, 20.6 with one; 40 nodes 34.6 and 38.9; a thread with one costs small calls less (1 x 32 x
    // 8x8 x 3, backward-weight: 10.7 us, 12.4 with four)
    const int64_t most = na > nb ? na : nb;
    // (rows of several pieces have four or five words each in flight as it is)
    const bool many = most >= (int64_t)kNumSMs * 2048 && (na > nb ? a.C : b.C) < 16;
    launch_k(many ? pad_channels_kernel<4> : pad_channels_kernel<1>, dim3(grid_for(many ? ceil_div(most, 4) : most), b.rows ? 2 : 1), 256, 0,
             st, a, b);
    LPDT_LAUNCH_CHECK();
    return LPDT_OK;
}

// The least workspace a call is accepted with: [transposed weights] of the CUDA-core backward-data kernel,
// [int32 sums | padded input] of backward-weight.  With less than lpdt_qconv_workspace_size, which adds the padded
// copies that the tensor-core engine reads, a shape that needs them runs on the CUDA cores.
static size_t least_workspace(const lpdt_conv_desc *d, int32_t which) {
    if (!d || d->nodes <= 0 || check_desc(d) != LPDT_OK) return 256;
    const size_t wn = (size_t)d->nodes * d->Cout * d->R * d->S * d->Cin;
    const PadPlan p = pad_plan(*d);
    size_t need = 256;
    if (which == 0 && p.in + p.w > need) need = p.in + p.w;
    if (which == 1) need = align_up(wn, 256);
    if (which == 2) need = align_up(wn * sizeof(int32_t), 256) + p.in;
    return need;
}
extern "C" size_t lpdt_qconv_workspace_size(const lpdt_conv_desc *d, int32_t which) {
    size_t need = least_workspace(d, which);
    if (!d || d->nodes <= 0 || check_desc(d) != LPDT_OK) return need;
    const PadPlan p = pad_plan(*d);
    if (which == 1 && p.err + p.w > need) need = p.err + p.w;
    if (which == 2) need += p.err;
    return need;
}

// Whether the tensor-core engine may take the shape with a workspace of ws_bytes.  Only shapes that need padded
// copies look at the workspace.
static bool use_tc(const lpdt_conv_desc &d, int which, const void *ws, size_t ws_bytes) {
    if (!tc_enabled() || !tc::tc_supported(d)) return false;
    const bool pads = which == 0 ? d.Cin % 16 : (d.Cin % 16 || d.Cout % 16);
    return !pads || (ws && aligned(ws, 256) && ws_bytes >= lpdt_qconv_workspace_size(&d, which));
}
// Products that finish sooner on the CUDA cores although the tensor cores could take them: each result a dot product of a
// few dozen steps, and few steps in all (a classifier's scores and their adjoint, a small first layer).  The tensor-core
// kernel's fixed cost (padded copies, barriers, TMEM, first boxes) is 6-8 us.  Measured, CUDA cores against tensor cores:
// 40 x 32 x 64 -> 10 forward 2.8 / 6.0 us and its adjoint 4.9 / 5.6, 8 x 32 x 512 -> 10 forward 9.9 / 6.7; 3x3 from 3
// channels 5.0 / 7.3 us at 65 K results (1.8 M steps), 9.1 / 7.6 at 131 K, 11.8 / 7.6 at 262 K; zero-point backward-data
// of 7 x 34 rows, 11 -> 751 (2.0 M steps) 16 / 21 us in all, 2 x 113 rows, 12 -> 115 9.5 / 16.5.  Only shapes that need
// padding; the others fill the tiles.
static bool tiny_dot(const lpdt_conv_desc &d, int64_t results, int K, bool vec4) {
    const int steps = vec4 ? K / 4 : K;
    return (d.Cin % 16 || d.Cout % 16) && steps <= 64 && results * steps <= (int64_t)kNumSMs * 16384;
}
static bool tiny_fwd(const lpdt_conv_desc &d, const int8_t *A, const int8_t *Wq) {
    const int64_t results = (int64_t)d.nodes * d.B * conv_out(d.H, d.pad, d.R, d.stride) * conv_out(d.W, d.pad, d.S, d.stride) * d.Cout;
    return tiny_dot(d, results, d.R * d.S * d.Cin, d.Cin % 4 == 0 && aligned(A, 4) && aligned(Wq, 4));
}
static bool tiny_bwd_data(const lpdt_conv_desc &d, const int8_t *E) {
    return tiny_dot(d, (int64_t)d.nodes * d.B * d.H * d.W * d.Cin, d.R * d.S * d.Cout, d.Cout % 4 == 0 && aligned(E, 4));
}
// An operand of `C` channels the engine can read: its padded copy, or itself at a 16-byte boundary.
static bool readable(const void *p, int C) { return C % 16 != 0 || aligned(p, 16); }

// Forward contraction on raw codes (signed, or unsigned when `uns`): kernel choice only.  With `aff` the zero-point
// terms are applied in the epilogue, or UNSUPPORTED is returned.
static lpdt_status fwd_impl(const lpdt_conv_desc *d, const int8_t *A, const float *sA, const int8_t *Wq,
                            const float *sW, const float *bias, int64_t bias_node_stride, float *Y, int32_t *Yacc,
                            void *ws, size_t ws_bytes, int32_t *dev_status, cudaStream_t st, bool uns,
                            const tc::AffineArgs *aff = nullptr) {
    const bool out_ok = (!Y || aligned(Y, 16)) && (!Yacc || aligned(Yacc, 16));
    if (!tiny_fwd(*d, A, Wq) && use_tc(*d, 0, ws, ws_bytes) && readable(A, d->Cin) && readable(Wq, d->Cin) && out_ok) {
        const bool pad = d->Cin % 16 != 0;
        const int8_t *Ae = A, *We = Wq;
        if (pad) {
            const PadPlan pp = pad_plan(*d);
            Ae = (int8_t *)ws; We = Ae + pp.in;
            lpdt_status s = pad_launch(pad_job(A, ws, (int64_t)d->nodes * d->B * d->H * d->W, d->Cin),
                                       pad_job(Wq, (char *)ws + pp.in, (int64_t)d->nodes * d->Cout * d->R * d->S, d->Cin), st);
            if (s != LPDT_OK) return s;
        }
        lpdt_status r = run_pix(*d, 0, Ae, sA, We, sW, bias, bias_node_stride, Y, Yacc, dev_status, st, uns, nullptr, aff);
        if (r != LPDT_ERR_UNSUPPORTED || (!pad && d->Cout % 16 == 0)) return r;
    }
    if (aff) return LPDT_ERR_UNSUPPORTED;
    return generic_fwd(*d, A, sA, Wq, sW, bias, bias_node_stride, Y, Yacc, st, uns);
}

extern "C" lpdt_status lpdt_qconv_fwd(const lpdt_conv_desc *d, const int8_t *A, const float *sA,
                                      const int8_t *Wq, const float *sW, const float *bias,
                                      int64_t bias_node_stride, float *Y, int32_t *Yacc, void *ws,
                                      size_t ws_bytes, int32_t *dev_status, void *stream) {
    lpdt_status s = check_desc(d);
    if (s != LPDT_OK) return s;
    if (d->nodes == 0 || d->B == 0) return LPDT_OK;
    LPDT_CHECK_ARG(A && Wq && (Y || Yacc));
    LPDT_CHECK_ARG(!Y || (sA && sW));
    LPDT_CHECK_ARG(!bias || bias_node_stride >= d->Cout || d->nodes == 1);
    return fwd_impl(d, A, sA, Wq, sW, bias, bias_node_stride, Y, Yacc, ws, ws_bytes, dev_status, as_stream(stream),
                    false);
}

// ---- affine (zero-point) operands -------------------------------------------------------------
// sum (qa - zA)(qw - zW) over the taps inside the image
//   = sum qa*qw  -  zW * sum qa  -  zA * sum qw  +  (taps inside * Cin) * zA * zW.
// The first term is the contraction engine on the unsigned codes (taps outside the image read code 0
// and add nothing); the other three come from per-pixel channel sums of the input and from prefix
// sums over the filter taps of the weights' channel sums (the taps inside the image form a rectangle
// of the filter).  All arithmetic is modulo 2^32, like the accumulators.
namespace lpdt {

// out[row] = sum of the `len` unsigned bytes of row `row`.  A group of G lanes (a power of two up to
// 32, chosen by the launcher from the row length) shares a row: 16-byte loads when the rows allow.
// `block` of `blocks` blocks that share the rows.
struct RowSums { const uint8_t *src; int32_t *out; int64_t rows; int len, G; bool vec16; };
__device__ __forceinline__ void row_sums(const RowSums &rs, unsigned block, unsigned blocks) {
    const int G = rs.G, len = rs.len;
    const int64_t rows = rs.rows;
    const uint8_t *__restrict__ src = rs.src;
    int32_t *__restrict__ out = rs.out;
    const bool vec16 = rs.vec16;
    const int lane_in_group = threadIdx.x & (G - 1);
    const int64_t groups_total = ((int64_t)blocks * blockDim.x) / G;
    for (int64_t row = ((int64_t)block * blockDim.x + threadIdx.x) / G;; row += groups_total) {
        if (row - (int)((threadIdx.x & 31) / G) >= rows) break;      // warp-uniform: the warp's first row is past the end
        const bool valid = row < rows;                               // lanes past the end still take part in the shuffles
        const uint8_t *a = src + (valid ? row : 0) * len;
        unsigned sum = 0;
        if (!valid) {
        } else if (vec16) {
            const uint4 *a16 = reinterpret_cast<const uint4 *>(a);
            for (int i = lane_in_group; i < len / 16; i += G) {
                const uint4 v = __ldg(a16 + i);
                sum = __dp4a(v.x, 0x01010101u, sum); sum = __dp4a(v.y, 0x01010101u, sum);
                sum = __dp4a(v.z, 0x01010101u, sum); sum = __dp4a(v.w, 0x01010101u, sum);
            }
        } else {
            for (int i = lane_in_group; i < len; i += G) sum += a[i];
        }
        for (int o = G >> 1; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (valid && lane_in_group == 0) out[row] = (int32_t)sum;
    }
}
__global__ void row_sum_u8_kernel(RowSums rs) {
    pdl_enter();
    row_sums(rs, blockIdx.x, gridDim.x);
}

// P[n][r][s][co] for 0 <= r <= R, 0 <= s <= S: sum of tapsum[n][co][r'][s'] over r' < r, s' < s.  The output
// channel is the fastest index, so the correction pass reads four neighbours with one 16-byte load.
__global__ void weight_prefix_kernel(const int32_t *__restrict__ tapsum, int nodes, int Cout, int R, int S,
                                     int32_t *__restrict__ P) {
    pdl_enter();
    const int row = blockIdx.x * blockDim.x + threadIdx.x;        // (node, co)
    if (row >= nodes * Cout) return;
    const int n = row / Cout, co = row % Cout, PS = S + 1;
    const int32_t *t = tapsum + (int64_t)row * R * S;
    int32_t *p = P + (int64_t)n * (R + 1) * PS * Cout + co;
    for (int s = 0; s <= S; ++s) p[(int64_t)s * Cout] = 0;
    for (int r = 1; r <= R; ++r) {
        p[(int64_t)(r * PS) * Cout] = 0;
        unsigned run = 0;                                     // taps (r-1, < s)
        for (int s = 1; s <= S; ++s) {
            run += (unsigned)t[(r - 1) * S + (s - 1)];
            p[(int64_t)(r * PS + s) * Cout] = (int32_t)((unsigned)p[(int64_t)((r - 1) * PS + s) * Cout] + run);
        }
    }
}

// The same table in one launch, for both directions and any stride (layout: PixParams in the tensor-core engine):
//   over_cout = 0: t[co][r][s] = sum over ci of W[n][co][r][s][ci], st = 1              (C = Cout)
//   over_cout = 1: t[ci][r][s] = sum over co of W[n][co][r][s][ci], st = the stride     (C = Cin)
// Block (16 result channels, node): tap sums in shared memory, prefix sums over the taps, table written out.  One thread
// per entry with a serial loop over the other channels took 15.9 us at 8 x 128 x 128 x 9 for the sums alone.
constexpr int kTabC = 16;
__host__ __device__ inline int table_lanes(const lpdt_conv_desc &d) {
    return d.R * d.S == 1 && (d.Cin >= 2048 || d.Cin % 16) ? 32 : 8;      // (ragged rows are read byte by byte)
}
// Threads per block: forward, a group of lanes per row, up to 1024 (144 rows of a 3x3 filter in two goes); backward-data,
// whose sums meet in atomics, one per row of 16 bytes, up to 512.  (1024 and 512 throughout: 13 nodes of 512 -> 1536 took
// 17.9 us, four waves of blocks with half of their threads idle, and the whole product 26.8 us; 14.2 now.)
static int table_threads(const lpdt_conv_desc &d, int over_cout) {
    const int64_t rows = over_cout ? (int64_t)d.R * d.S * d.Cout : (int64_t)d.R * d.S * kTabC * table_lanes(d), most = over_cout ? 512 : 1024;
    const int64_t t = (rows + 31) / 32 * 32;
    return (int)(t < 64 ? 64 : t > most ? most : t);
}
// The activations' (or errors') row sums, which the contraction's epilogue reads beside the table, ride in the same launch:
// the blocks behind the `tables` first ones.  The few table blocks, a serial chain each, run beside them
// (8 x 32 x 16x16 128 -> 128 3x3: forward 30.3 us with two launches, 28.6 with one; backward-data 35.9 and 33.1).
__global__ void __launch_bounds__(1024)
weight_table_kernel(lpdt_conv_desc d, const uint8_t *__restrict__ Wq, int over_cout, int st, bool vec16, bool vec4, int32_t *__restrict__ P,
                    unsigned tables, RowSums rs) {
    pdl_enter();
    if (blockIdx.x >= tables) {
        row_sums(rs, blockIdx.x - tables, gridDim.x - tables);
        return;
    }
    extern __shared__ unsigned s_tab[];
    const int taps = d.R * d.S, C = over_cout ? d.Cin : d.Cout, PS = d.S + st, cells = (d.R + st) * PS;
    unsigned *t = s_tab, *pre = s_tab + taps * kTabC;             // [taps][16], [cells][16]
    const unsigned chunks = (C + kTabC - 1) / kTabC;
    const int n = blockIdx.x / chunks, c0 = (blockIdx.x - n * chunks) * kTabC, nc = C - c0 < kTabC ? C - c0 : kTabC, tid = threadIdx.x, T = blockDim.x;
    const uint8_t *w = Wq + (int64_t)n * d.Cout * taps * d.Cin;
    for (int i = tid; i < taps * kTabC; i += T) t[i] = 0;
    __syncthreads();
    if (over_cout) {
        // thread = (tap, every (T / taps)-th output channel), 16 input channels of the row; pairs of bytes are summed
        // in 16-bit halves, at most 256 rows at a time
        const int step = T / taps, tap = tid % taps;
        if (tid < step * taps) {
            int co = tid / taps;
            while (co < d.Cout) {
                unsigned e[4] = {0, 0, 0, 0}, o[4] = {0, 0, 0, 0};
                const int end = co + 256 * step < d.Cout ? co + 256 * step : d.Cout;
#pragma unroll 4
                for (; co < end; co += step) {
                    const uint8_t *row = w + ((int64_t)co * taps + tap) * d.Cin + c0;
                    uint4 q;
                    if (vec16) q = __ldg(reinterpret_cast<const uint4 *>(row));
                    else {
                        unsigned b[4] = {0, 0, 0, 0};
                        if (vec4) {
#pragma unroll
                            for (int k = 0; k < 4; ++k) if (4 * k < nc) b[k] = __ldg(reinterpret_cast<const unsigned *>(row) + k);
                        } else
#pragma unroll
                        for (int k = 0; k < 16; ++k) if (k < nc) b[k >> 2] |= (unsigned)row[k] << (8 * (k & 3));
                        q = make_uint4(b[0], b[1], b[2], b[3]);
                    }
                    const unsigned v[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                    for (int k = 0; k < 4; ++k) { e[k] += v[k] & 0x00ff00ffu; o[k] += (v[k] >> 8) & 0x00ff00ffu; }
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    atomicAdd(t + tap * kTabC + 4 * k, e[k] & 0xffffu); atomicAdd(t + tap * kTabC + 4 * k + 2, e[k] >> 16);
                    atomicAdd(t + tap * kTabC + 4 * k + 1, o[k] & 0xffffu); atomicAdd(t + tap * kTabC + 4 * k + 3, o[k] >> 16);
                }
            }
        }
    } else {
        // eight lanes per row (output channel, tap), 32 where there are few and long ones
        const int G = table_lanes(d), lane = tid & (G - 1);
        for (int row = tid / G; row < taps * kTabC; row += T / G) {
            const int tap = row % taps, c = row / taps;
            unsigned sum = 0;
            if (c < nc) {
                const uint8_t *r = w + ((int64_t)(c0 + c) * taps + tap) * d.Cin;
                if (vec16) {
#pragma unroll 4
                    for (int i = lane; i < d.Cin / 16; i += G) {
                        const uint4 v = __ldg(reinterpret_cast<const uint4 *>(r) + i);
                        sum = __dp4a(v.x, 0x01010101u, sum); sum = __dp4a(v.y, 0x01010101u, sum);
                        sum = __dp4a(v.z, 0x01010101u, sum); sum = __dp4a(v.w, 0x01010101u, sum);
                    }
                } else {
                    for (int i = lane; i < d.Cin; i += G) sum += r[i];
                }
            }
            atomicAdd(t + tap * kTabC + c, sum);
        }
    }
    __syncthreads();
    if (tid < kTabC) {
        for (int r = 0; r < d.R + st; ++r)
            for (int s = 0; s < PS; ++s) {
                unsigned v = 0;
                if (r >= st && s >= st)
                    v = t[((r - st) * d.S + s - st) * kTabC + tid] + pre[((r - st) * PS + s) * kTabC + tid] +
                        pre[(r * PS + s - st) * kTabC + tid] - pre[((r - st) * PS + s - st) * kTabC + tid];
                pre[(r * PS + s) * kTabC + tid] = v;
            }
    }
    __syncthreads();
    for (int i = tid; i < cells * kTabC; i += T)
        if ((i & (kTabC - 1)) < nc) P[((int64_t)n * cells + i / kTabC) * C + c0 + (i & (kTabC - 1))] = (int32_t)pre[i];
}
// Shapes the kernel above takes: a thread per tap, the tables in 48 KB of shared memory, blocks of all nodes and row sums in one grid.
static bool table_fits(const lpdt_conv_desc &d, int st) {
    return d.R * d.S <= 256 && ((int64_t)d.R * d.S + (int64_t)(d.R + st) * (d.S + st)) * kTabC * 4 <= 48 * 1024 && d.nodes <= 65535 &&
           (int64_t)d.nodes * (d.Cin > d.Cout ? d.Cin : d.Cout) <= (int64_t)1 << 30;
}
// rows of `len` bytes -> out[row]; lanes per row grow with the row length
static RowSums row_sums_of(const uint8_t *src, int64_t rows, int len, int32_t *out) {
    const bool vec16 = len % 16 == 0 && aligned(src, 16);
    const int units = vec16 ? len / 16 : len;
    int G = 1;
    while (G < 32 && G * 4 <= units) G <<= 1;             // at least four loads per lane
    return {src, out, rows, len, G, vec16};
}
static unsigned row_sum_blocks(const RowSums &rs, int threads) {
    int64_t blocks = ceil_div(rs.rows * rs.G, threads);
    const int64_t cap = (int64_t)kNumSMs * 32 * 256 / threads;
    if (blocks > cap) blocks = cap;
    return (unsigned)(blocks < 1 ? 1 : blocks);
}
static lpdt_status row_sum_launch(const RowSums &rs, cudaStream_t st) {
    launch_k(row_sum_u8_kernel, row_sum_blocks(rs, 256), 256, 0, st, rs);
    LPDT_LAUNCH_CHECK();
    return LPDT_OK;
}
static lpdt_status weight_table_launch(const lpdt_conv_desc &d, const uint8_t *Wq, int over_cout, int st, int32_t *P, const RowSums &rs,
                                       cudaStream_t stream) {
    const int C = over_cout ? d.Cin : d.Cout, T = table_threads(d, over_cout);
    const size_t smem = ((size_t)d.R * d.S + (size_t)(d.R + st) * (d.S + st)) * kTabC * 4;
    const bool vec16 = d.Cin % 16 == 0 && aligned(Wq, 16);
    const unsigned tables = (unsigned)(ceil_div(C, kTabC) * d.nodes), blocks = tables + row_sum_blocks(rs, T);
    static PerDeviceOnce attr;
    int dev;
    if (attr.pending(&dev)) {
        LPDT_CUDA(cudaFuncSetAttribute(weight_table_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024));
        attr.mark(dev);
    }
    // (2 x 50 x 6x6, 502 -> 42 backward-data behind itself: 30.4 us with the blocks on the first SMs to be free, 27.1 spread)
    launch_k(weight_table_kernel, blocks, T, spread_smem(smem, blocks, 2048 / T), stream, d, Wq, over_cout, st, vec16,
             d.Cin % 4 == 0 && aligned(Wq, 4), P, tables, rs);
    LPDT_LAUNCH_CHECK();
    return LPDT_OK;
}

// One thread per (output pixel, V consecutive output channels); V = 4 with 16-byte accesses when the
// channel count allows, else 1.
template <int V>
__global__ void affine_fix_kernel(lpdt_conv_desc d, int Ho, int Wo, const int32_t *__restrict__ raw,
                                  const int32_t *__restrict__ asum, const int32_t *__restrict__ P,
                                  const int32_t *__restrict__ zA, const int32_t *__restrict__ zW,
                                  const float *__restrict__ sA, const float *__restrict__ sW,
                                  const float *__restrict__ bias, int64_t bias_stride, float *__restrict__ Y,
                                  int32_t *__restrict__ Yacc) {
    pdl_enter();
    const int chunks = d.Cout / V;
    const int64_t total = (int64_t)d.nodes * d.B * Ho * Wo * chunks;
    for (int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; o < total; o += (int64_t)gridDim.x * blockDim.x) {
        const int co0 = (int)(o % chunks) * V;
        const int64_t pix = o / chunks;
        const int ow = (int)(pix % Wo);
        const int oh = (int)((pix / Wo) % Ho);
        const int64_t nb = pix / ((int64_t)Wo * Ho);
        const int n = (int)(nb / d.B);
        // filter rows / columns whose tap lies inside the image
        int r_lo = d.pad - oh * d.stride; if (r_lo < 0) r_lo = 0;
        int r_hi = d.H + d.pad - oh * d.stride; if (r_hi > d.R) r_hi = d.R;
        int s_lo = d.pad - ow * d.stride; if (s_lo < 0) s_lo = 0;
        int s_hi = d.W + d.pad - ow * d.stride; if (s_hi > d.S) s_hi = d.S;
        if (r_hi < r_lo) r_hi = r_lo;
        if (s_hi < s_lo) s_hi = s_lo;
        unsigned ra = 0;
        for (int r = r_lo; r < r_hi; ++r)
            for (int s = s_lo; s < s_hi; ++s)
                ra += (unsigned)__ldg(asum + (nb * d.H + oh * d.stride + r - d.pad) * d.W + ow * d.stride + s - d.pad);
        const unsigned za = (unsigned)zA[n], zw = (unsigned)zW[n];
        const unsigned cnt = (unsigned)((r_hi - r_lo) * (s_hi - s_lo) * d.Cin);
        const unsigned fixed = cnt * za * zw - zw * ra;
        const float sc = Y ? __fmul_rn(sA[n], sW[n]) : 0.f;
        const int PS = d.S + 1;
        const int64_t oi = pix * d.Cout + co0;
        int rawv[V], acc[V];
        if (V == 4) { const int4 t = *reinterpret_cast<const int4 *>(raw + oi); rawv[0] = t.x; rawv[1] = t.y; rawv[2] = t.z; rawv[3] = t.w; }
        else rawv[0] = raw[oi];
        // rectangle sum of the weights' channel sums over the taps inside the image: four corners of the prefix table
        const int32_t *p = P + (int64_t)n * (d.R + 1) * PS * d.Cout + co0;
        int c11[V], c01[V], c10[V], c00[V];
        auto corner = [&](int r, int s2, int (&o)[V]) {
            const int32_t *q = p + (int64_t)(r * PS + s2) * d.Cout;
            if (V == 4) { const int4 t = __ldg(reinterpret_cast<const int4 *>(q)); o[0] = t.x; o[1] = t.y; o[2] = t.z; o[3] = t.w; }
            else o[0] = __ldg(q);
        };
        corner(r_hi, s_hi, c11); corner(r_lo, s_hi, c01); corner(r_hi, s_lo, c10); corner(r_lo, s_lo, c00);
#pragma unroll
        for (int k = 0; k < V; ++k) {
            const unsigned rw = (unsigned)c11[k] - (unsigned)c01[k] - (unsigned)c10[k] + (unsigned)c00[k];
            acc[k] = (int)((unsigned)rawv[k] + fixed - za * rw);
        }
        if (Yacc) {
            if (V == 4) *reinterpret_cast<int4 *>(Yacc + oi) = make_int4(acc[0], acc[1], acc[2], acc[3]);
            else Yacc[oi] = acc[0];
        }
        if (Y) {
            float v[V];
#pragma unroll
            for (int k = 0; k < V; ++k) {
                v[k] = __fmul_rn(__int2float_rn(acc[k]), sc);
                if (bias) v[k] = __fadd_rn(v[k], bias[(int64_t)n * bias_stride + co0 + k]);
            }
            if (V == 4) *reinterpret_cast<float4 *>(Y + oi) = make_float4(v[0], v[1], v[2], v[3]);
            else Y[oi] = v[0];
        }
    }
}

}  // namespace lpdt

// LPDT_AFFINE_SEPARATE=1 keeps the separate correction passes of forward and backward-data on every shape.
static bool affine_separate() {
    static int separate = -1;
    if (separate < 0) { const char *e = getenv("LPDT_AFFINE_SEPARATE"); separate = (e && e[0] == '1') ? 1 : 0; }
    return separate == 1;
}
static size_t affine_raw_bytes(const lpdt_conv_desc *d) {
    const int Ho = conv_out(d->H, d->pad, d->R, d->stride), Wo = conv_out(d->W, d->pad, d->S, d->stride);
    return align_up((size_t)d->nodes * d->B * Ho * Wo * d->Cout * sizeof(int32_t), 256);
}
static size_t affine_asum_bytes(const lpdt_conv_desc *d) {
    return align_up((size_t)d->nodes * d->B * d->H * d->W * sizeof(int32_t), 256);
}
// The prefix table may be read up to 31 entries past its end by the tensor-core epilogue: at least 256 bytes of
// workspace (the contraction's own) follow it.
static size_t affine_prefix_bytes(const lpdt_conv_desc *d) {     // prefix table + per-tap channel sums
    return align_up((size_t)d->nodes * d->Cout * (d->R + 1) * (d->S + 1) * sizeof(int32_t), 256) +
           align_up((size_t)d->nodes * d->Cout * d->R * d->S * sizeof(int32_t), 256);
}

static size_t affine_fwd_own(const lpdt_conv_desc *d) { return affine_raw_bytes(d) + affine_asum_bytes(d) + affine_prefix_bytes(d); }

extern "C" size_t lpdt_qconv_fwd_affine_workspace_size(const lpdt_conv_desc *d) {
    if (!d || d->nodes <= 0 || check_desc(d) != LPDT_OK) return 256;
    return affine_fwd_own(d) + lpdt_qconv_workspace_size(d, 0);
}

extern "C" lpdt_status lpdt_qconv_fwd_affine(const lpdt_conv_desc *d, const uint8_t *A, const float *sA,
                                             const int32_t *zA, const uint8_t *Wq, const float *sW,
                                             const int32_t *zW, const float *bias, int64_t bias_node_stride,
                                             float *Y, int32_t *Yacc, void *ws, size_t ws_bytes,
                                             int32_t *dev_status, void *stream) {
    lpdt_status s = check_desc(d);
    if (s != LPDT_OK) return s;
    if (d->nodes == 0 || d->B == 0) return LPDT_OK;
    LPDT_CHECK_ARG(A && Wq && zA && zW && (Y || Yacc));
    LPDT_CHECK_ARG(!Y || (sA && sW));
    LPDT_CHECK_ARG(!bias || bias_node_stride >= d->Cout || d->nodes == 1);
    if (!ws || !aligned(ws, 256) || ws_bytes < affine_fwd_own(d) + least_workspace(d, 0)) return LPDT_ERR_WORKSPACE;
    cudaStream_t st = as_stream(stream);
    const int Ho = conv_out(d->H, d->pad, d->R, d->stride), Wo = conv_out(d->W, d->pad, d->S, d->stride);
    int32_t *raw = (int32_t *)ws;
    int32_t *asum = (int32_t *)((char *)ws + affine_raw_bytes(d));
    int32_t *P = (int32_t *)((char *)asum + affine_asum_bytes(d));
    void *inner = (char *)P + affine_prefix_bytes(d);
    const int64_t pixels = (int64_t)d->nodes * d->B * d->H * d->W;
    const RowSums sums = row_sums_of(A, pixels, d->Cin, asum);
    const int rows = d->nodes * d->Cout;
    int32_t *tapsum = (int32_t *)((char *)P + align_up((size_t)rows * (d->R + 1) * (d->S + 1) * sizeof(int32_t), 256));
    if (table_fits(*d, 1)) {
        s = weight_table_launch(*d, Wq, 0, 1, P, sums, st);
        if (s != LPDT_OK) return s;
    } else {
        s = row_sum_launch(sums, st);
        if (s == LPDT_OK) s = row_sum_launch(row_sums_of(Wq, (int64_t)rows * d->R * d->S, d->Cin, tapsum), st);
        if (s != LPDT_OK) return s;
        launch_k(weight_prefix_kernel, (rows + 127) / 128, 128, 0, st, tapsum, d->nodes, d->Cout, d->R, d->S, P);
        LPDT_LAUNCH_CHECK();
    }
    // Tensor-core path: the zero-point terms are applied in the contraction's own epilogue (no raw sums in
    // memory, no second pass over the result).
    const size_t inner_bytes = ws_bytes - (size_t)((char *)inner - (char *)ws);
    if (!affine_separate()) {
        const tc::AffineArgs aff = {asum, P, zA, zW};
        lpdt_status r = fwd_impl(d, reinterpret_cast<const int8_t *>(A), sA, reinterpret_cast<const int8_t *>(Wq), sW,
                                 bias, bias_node_stride, Y, Yacc, inner, inner_bytes, dev_status, st, true, &aff);
        if (r != LPDT_ERR_UNSUPPORTED) return r;
    }
    s = fwd_impl(d, reinterpret_cast<const int8_t *>(A), nullptr, reinterpret_cast<const int8_t *>(Wq), nullptr, nullptr,
                 0, nullptr, raw, inner, inner_bytes, dev_status, st, true);
    if (s != LPDT_OK) return s;
    const bool v4 = d->Cout % 4 == 0 && (!Y || aligned(Y, 16)) && (!Yacc || aligned(Yacc, 16));
    const int64_t work = (int64_t)d->nodes * d->B * Ho * Wo * (d->Cout / (v4 ? 4 : 1));
    if (v4)
        launch_k(affine_fix_kernel<4>, grid_for(work), 256, 0, st, *d, Ho, Wo, raw, asum, P, zA, zW, sA, sW, bias,
                                                             bias_node_stride, Y, Yacc);
    else
        launch_k(affine_fix_kernel<1>, grid_for(work), 256, 0, st, *d, Ho, Wo, raw, asum, P, zA, zW, sA, sW, bias,
                                                             bias_node_stride, Y, Yacc);
    LPDT_LAUNCH_CHECK();
    return LPDT_OK;
}

// Backward-data contraction on raw codes (signed, or unsigned when `uns`): kernel choice only; `aff` as in fwd_impl.
static lpdt_status bwd_data_impl(const lpdt_conv_desc *d, const int8_t *E, const float *sE, const int8_t *Wq,
                                 const float *sW, float *dA, int32_t *dAacc, const float *addend, void *ws,
                                 size_t ws_bytes, int32_t *dev_status, cudaStream_t st, bool uns,
                                 const tc::AffineArgs *aff = nullptr) {
    if (!tiny_bwd_data(*d, E) && use_tc(*d, 1, ws, ws_bytes) && readable(E, d->Cout) && readable(Wq, d->Cin) &&
        (!dA || aligned(dA, 16)) && (!dAacc || aligned(dAacc, 16))) {
        const int Ho = conv_out(d->H, d->pad, d->R, d->stride), Wo = conv_out(d->W, d->pad, d->S, d->stride);
        const PadPlan pp = pad_plan(*d);
        void *Ep = ws, *Wp = (char *)ws + pp.err;
        lpdt_status s = pad_launch(pad_job(E, Ep, pp.err ? (int64_t)d->nodes * d->B * Ho * Wo : 0, d->Cout),
                                   pad_job(Wq, Wp, pp.w ? (int64_t)d->nodes * d->Cout * d->R * d->S : 0, d->Cin), st);
        if (s != LPDT_OK) return s;
        lpdt_status r = run_pix(*d, 1, pp.err ? (int8_t *)Ep : E, sE, pp.w ? (int8_t *)Wp : Wq, sW, nullptr, 0, dA, dAacc,
                                dev_status, st, uns, addend, aff);
        if (r != LPDT_ERR_UNSUPPORTED || (!pp.err && !pp.w)) return r;
    }
    if (aff) return LPDT_ERR_UNSUPPORTED;
    return generic_bwd_data(*d, E, sE, Wq, sW, dA, dAacc, addend, ws, st, uns);
}

extern "C" lpdt_status lpdt_qconv_bwd_data(const lpdt_conv_desc *d, const int8_t *E, const float *sE,
                                           const int8_t *Wq, const float *sW, float *dA, int32_t *dAacc,
                                           const float *addend, void *ws, size_t ws_bytes, int32_t *dev_status,
                                           void *stream) {
    lpdt_status s = check_desc(d);
    if (s != LPDT_OK) return s;
    if (d->nodes == 0 || d->B == 0) return LPDT_OK;
    LPDT_CHECK_ARG(E && Wq && (dA || dAacc));
    LPDT_CHECK_ARG(!dA || (sE && sW));
    LPDT_CHECK_ARG(!addend || (dA && addend != dA && aligned(addend, 16)));
    if (!ws || ws_bytes < least_workspace(d, 1)) return LPDT_ERR_WORKSPACE;
    return bwd_data_impl(d, E, sE, Wq, sW, dA, dAacc, addend, ws, ws_bytes, dev_status, as_stream(stream), false);
}

// Backward-weight contraction on raw codes.  Workspace: [int32 sums (used unless the caller gave dWacc) |
// padded input | padded layer gradient].  `more_clear` as in tc_wgrad.
static lpdt_status bwd_weight_impl(const lpdt_conv_desc *d, const int8_t *E, const float *sE, const int8_t *A,
                                   const float *sA, float *dW, int64_t dw_node_stride, int32_t *dWacc, void *ws,
                                   size_t ws_bytes, int32_t *dev_status, cudaStream_t st, bool uns, size_t *more_clear = nullptr) {
    const size_t acc_bytes = align_up((size_t)d->nodes * d->Cout * d->R * d->S * d->Cin * sizeof(int32_t), 256);
    int32_t *acc_ws = (int32_t *)ws;
    if (use_tc(*d, 2, ws, ws_bytes) && d->B > 0 && readable(E, d->Cout) && readable(A, d->Cin)) {
        const int Ho = conv_out(d->H, d->pad, d->R, d->stride), Wo = conv_out(d->W, d->pad, d->S, d->stride);
        const PadPlan pp = pad_plan(*d);
        void *Ap = (char *)ws + acc_bytes, *Ep = (char *)Ap + pp.in;
        lpdt_status s = pad_launch(pad_job(A, Ap, pp.in ? (int64_t)d->nodes * d->B * d->H * d->W : 0, d->Cin),
                                   pad_job(E, Ep, pp.err ? (int64_t)d->nodes * d->B * Ho * Wo : 0, d->Cout), st);
        if (s != LPDT_OK) return s;
        lpdt_status r = tc::tc_wgrad(*d, pp.err ? (int8_t *)Ep : E, sE, pp.in ? (int8_t *)Ap : A, sA, dWacc, acc_ws, dW,
                                     dw_node_stride, dev_status, st, uns, pitches(*d), more_clear);
        if (r != LPDT_ERR_UNSUPPORTED) return r;
    }
    return generic_bwd_weight(*d, E, sE, A, sA, dW, dw_node_stride, dWacc, acc_ws, st, uns);
}

extern "C" lpdt_status lpdt_qconv_bwd_weight(const lpdt_conv_desc *d, const int8_t *E, const float *sE,
                                             const int8_t *A, const float *sA, float *dW,
                                             int64_t dw_node_stride, int32_t *dWacc, void *ws,
                                             size_t ws_bytes, int32_t *dev_status, void *stream) {
    lpdt_status s = check_desc(d);
    if (s != LPDT_OK) return s;
    if (d->nodes == 0) return LPDT_OK;
    LPDT_CHECK_ARG((d->B == 0 || (E && A)) && (dW || dWacc));      // an empty batch has no operands to point at
    LPDT_CHECK_ARG(!dW || (sE && sA));
    LPDT_CHECK_ARG(!dW || dw_node_stride >= (int64_t)d->Cout * d->R * d->S * d->Cin || d->nodes == 1);
    if (!ws || ws_bytes < least_workspace(d, 2) || !aligned(ws, 256)) return LPDT_ERR_WORKSPACE;
    return bwd_weight_impl(d, E, sE, A, sA, dW, dw_node_stride, dWacc, ws, ws_bytes, dev_status, as_stream(stream), false);
}

extern "C" int32_t lpdt_qconv_bwd_weight_direct(const lpdt_conv_desc *d) {
    if (check_desc(d) != LPDT_OK || d->nodes == 0 || d->B == 0 || d->Cin % 16 || d->Cout % 16) return 0;
    return tc_enabled() && tc::tc_shape(*d) && tc::wgrad_direct(*d, pitches(*d)) ? 1 : 0;      // else the CUDA cores add in memory
}

// ---- backward products on affine (zero-point) operands -----------------------------------------
// With e' = qe - zE, w' = qw - zW, a' = qa - zA and the sums running over the taps that exist,
//   sum e'w' = sum qe*qw - zW * sum qe - zE * sum qw + (terms) * zE*zW          (backward-data)
//   sum e'a' = sum qe*qa - zA * sum qe - zE * sum qa + (terms) * zE*zA          (backward-weight)
// the first term is the contraction engine on the unsigned codes; the others come from channel sums
// of the operands, gathered over the same taps.  All arithmetic is modulo 2^32.
namespace lpdt {

// wsum[n][r][s][ci] = sum over co of W[n][co][r][s][ci]; one thread per output, ci fastest.
__global__ void weight_cout_sum_kernel(lpdt_conv_desc d, const uint8_t *__restrict__ Wq, int32_t *__restrict__ wsum) {
    pdl_enter();
    const int per = d.R * d.S * d.Cin;
    const int64_t total = (int64_t)d.nodes * per;
    for (int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; o < total; o += (int64_t)gridDim.x * blockDim.x) {
        const int n = (int)(o / per), i = (int)(o % per);
        const uint8_t *w = Wq + (int64_t)n * d.Cout * per + i;
        unsigned sum = 0;
        for (int co = 0; co < d.Cout; ++co) sum += w[(int64_t)co * per];
        wsum[o] = (int32_t)sum;
    }
}

// One thread per (input pixel, V consecutive input channels).
template <int V>
__global__ void affine_fix_bwd_data_kernel(lpdt_conv_desc d, int Ho, int Wo, const int32_t *__restrict__ raw,
                                           const int32_t *__restrict__ esum, const int32_t *__restrict__ wsum,
                                           const int32_t *__restrict__ zE, const int32_t *__restrict__ zW,
                                           const float *__restrict__ sE, const float *__restrict__ sW,
                                           float *__restrict__ dA, int32_t *__restrict__ dAacc) {
    pdl_enter();
    const int chunks = d.Cin / V;
    const int64_t total = (int64_t)d.nodes * d.B * d.H * d.W * chunks;
    for (int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; o < total; o += (int64_t)gridDim.x * blockDim.x) {
        const int ci0 = (int)(o % chunks) * V;
        const int64_t pix = o / chunks;
        const int iw = (int)(pix % d.W);
        const int ih = (int)((pix / d.W) % d.H);
        const int64_t nb = pix / ((int64_t)d.W * d.H);
        const int n = (int)(nb / d.B);
        unsigned es = 0, cnt = 0, ws_[V];
#pragma unroll
        for (int k = 0; k < V; ++k) ws_[k] = 0;
        for (int r = 0; r < d.R; ++r) {
            const int th = ih + d.pad - r;
            if (th < 0 || th % d.stride) continue;
            const int oh = th / d.stride;
            if (oh >= Ho) continue;
            for (int s = 0; s < d.S; ++s) {
                const int tw = iw + d.pad - s;
                if (tw < 0 || tw % d.stride) continue;
                const int ow = tw / d.stride;
                if (ow >= Wo) continue;
                es += (unsigned)__ldg(esum + (nb * Ho + oh) * Wo + ow);
                cnt += (unsigned)d.Cout;
                const int32_t *wp = wsum + (((int64_t)n * d.R + r) * d.S + s) * d.Cin + ci0;
#pragma unroll
                for (int k = 0; k < V; ++k) ws_[k] += (unsigned)__ldg(wp + k);
            }
        }
        const unsigned ze = (unsigned)zE[n], zw = (unsigned)zW[n];
        const unsigned fixed = cnt * ze * zw - zw * es;
        const float sc = dA ? __fmul_rn(sE[n], sW[n]) : 0.f;
        const int64_t oi = pix * d.Cin + ci0;
#pragma unroll
        for (int k = 0; k < V; ++k) {
            const int acc = (int)((unsigned)raw[oi + k] + fixed - ze * ws_[k]);
            if (dAacc) dAacc[oi + k] = acc;
            if (dA) dA[oi + k] = __fmul_rn(__int2float_rn(acc), sc);
        }
    }
}

// Sums of the operands of backward-weight over the output positions whose tap (r, s) lies inside the input image:
//   tabE[n][r][s][co] = sum of E[n][b][oh][ow][co],  tabA[n][r][s][ci] = sum of A[n][b][oh*st+r-pad][ow*st+s-pad][ci].
// Work item = (operand, node, up to `cw` channels, up to `sw` filter columns, image row, share of the batch), a block each.
// The block sums its row over its samples per column (V bytes of consecutive channels per thread), adds a column's sums
// to every filter column that reaches it in shared memory, and the result to every filter row that reaches the row,
// with integer atomics into zeroed tables.  (Batch sums in memory and one serial loop over the positions per tap and
// channel took 141 us at 8 x 32 x 16x16 x 128.)
// (Column sums meet in shared memory with a warp's words on neighbouring banks: stride-4 words, 64-bit divisions of the
// item number and two divisions per entry of the result took 15 us there instead of 9, with the launches around it.)
struct TapSumSide { const uint8_t *src; int32_t *tab; int rows, cols, C, cw, chunks; long long items; };
constexpr int kTapThreads = 512;
template <int V>
__global__ void __launch_bounds__(kTapThreads)
tap_sum_kernel(lpdt_conv_desc d, int Ho, int Wo, TapSumSide sideE, TapSumSide sideA, int sw, int bshares) {
    pdl_enter();
    extern __shared__ unsigned s_acc[];                       // [sw][cw]
    const int tid = threadIdx.x, schunks = (d.S + sw - 1) / sw;
    for (long long item = blockIdx.x; item < sideE.items + sideA.items; item += gridDim.x) {
        const bool in = item >= sideE.items;
        const TapSumSide sd = in ? sideA : sideE;
        long long q = in ? item - sideE.items : item;
        const bool narrow = q <= 0x7fffffff;                  // (a 64-bit division is some hundred instructions in a chain)
        auto take = [&](int by) {
            const long long w = narrow ? (long long)((unsigned)q / (unsigned)by) : q / by;
            const int rest = (int)(q - w * by);
            q = w;
            return rest;
        };
        const int share = take(bshares), row = take(sd.rows), s0 = take(schunks) * sw, c0 = take(sd.chunks) * sd.cw, n = (int)q;
        const int cw = sd.cw, nc = sd.C - c0 < cw ? sd.C - c0 : cw, ns = d.S - s0 < sw ? d.S - s0 : sw;
        for (int i = tid; i < ns * cw; i += kTapThreads) s_acc[i] = 0;
        __syncthreads();
        const int b0 = (int)((int64_t)d.B * share / bshares), b1 = (int)((int64_t)d.B * (share + 1) / bshares);
        const int words = (nc + V - 1) / V;
        const int64_t image = (int64_t)sd.rows * sd.cols * sd.C;
        const uint8_t *src = sd.src + (int64_t)n * d.B * image + (int64_t)row * sd.cols * sd.C + c0;
        // (up to 64 samples, column, word), word fastest
        int plen = 64;                                        // fewer where that leaves threads idle
        while (plen > 16 && (b1 - b0 + plen - 1) / plen * sd.cols * words < kTapThreads) plen /= 2;
        const int parts = (b1 - b0 + plen - 1) / plen, sums = parts * sd.cols * words;
        for (int it = tid; it < sums; it += kTapThreads) {
            const int wd = it % words, r = it / words, col = r % sd.cols, part = r / sd.cols;
            const uint8_t *p = src + (int64_t)col * sd.C + wd * V;
            const int lo = b0 + part * plen, hi = lo + plen < b1 ? lo + plen : b1;
            unsigned sum[V];
            if constexpr (V == 4) {
                unsigned e = 0, o = 0;                        // byte sums in 16-bit halves: at most 64 bytes each
                for (int b = lo; b < hi; b += 16) {
                    unsigned w[16];
#pragma unroll
                    for (int u = 0; u < 16; ++u)              // all in flight at once
                        w[u] = b + u < hi ? __ldg(reinterpret_cast<const unsigned *>(p + (b + u) * image)) : 0u;
#pragma unroll
                    for (int u = 0; u < 16; ++u) { e += w[u] & 0x00ff00ffu; o += (w[u] >> 8) & 0x00ff00ffu; }
                }
                sum[0] = e & 0xffffu; sum[1] = o & 0xffffu; sum[2] = e >> 16; sum[3] = o >> 16;
            } else {
                sum[0] = 0;
                for (int b = lo; b < hi; b += 16) {
                    unsigned w[16];
#pragma unroll
                    for (int u = 0; u < 16; ++u) w[u] = b + u < hi ? __ldg(p + (b + u) * image) : 0u;
#pragma unroll
                    for (int u = 0; u < 16; ++u) sum[0] += w[u];
                }
            }
            for (int k = 0; k < ns; ++k) {
                const int s = s0 + k;
                bool ok;                                      // filter column s reaches this image column
                if (in) { const int t = col + d.pad - s; ok = t >= 0 && (d.stride == 1 || t % d.stride == 0) && t < Wo * d.stride; }
                else { const int iw = col * d.stride + s - d.pad; ok = iw >= 0 && iw < d.W; }
                if (!ok) continue;
#pragma unroll
                for (int v = 0; v < V; ++v) atomicAdd(s_acc + k * cw + v * (cw / V) + wd, sum[v]);      // a warp's words on all banks
            }
        }
        __syncthreads();
        for (int i = tid; i < ns * nc; i += kTapThreads) {
            const int k = i / nc, c = i - k * nc;
            const unsigned v = s_acc[k * cw + c % V * (cw / V) + c / V];
            if (!v) continue;
            int32_t *t = sd.tab + ((int64_t)n * d.R * d.S + s0 + k) * sd.C + c0 + c;
            for (int r = 0; r < d.R; ++r, t += (int64_t)d.S * sd.C) {
                bool ok;
                if (in) { const int u = row + d.pad - r; ok = u >= 0 && (d.stride == 1 || u % d.stride == 0) && u < Ho * d.stride; }
                else { const int ih = row * d.stride + r - d.pad; ok = ih >= 0 && ih < d.H; }
                if (ok) atomicAdd(t, (int)v);
            }
        }
        __syncthreads();
    }
}

// Number of output positions o in [0, No) whose tap r of one axis lies inside an input of length `len`.
__device__ inline int taps_inside(int No, int len, int r, int pad, int st) {
    const int lo = pad > r ? (pad - r + st - 1) / st : 0;
    int hi = len - 1 + pad - r;
    if (hi < 0) return 0;
    hi /= st;
    if (hi > No - 1) hi = No - 1;
    return hi >= lo ? hi - lo + 1 : 0;
}

// A group of G lanes per row (output channel, tap) of a node's filter, V input channels per lane and step: the row's
// tables and counts once per row.  Bound by the sums' traffic: a thread per entry, each
// with its own divisions and counts, took 14.7 us at 8 x 128 x 128 x 9, 6.4 now (9.4 MB), and the whole backward-weight
// call 49.2 us, 34.9 with faster tap sums and one clear for sums and tables.
template <int V>
__global__ void __launch_bounds__(256)
affine_fix_bwd_weight_kernel(lpdt_conv_desc d, int Ho, int Wo, int G, const int32_t *__restrict__ raw,
                             const int32_t *__restrict__ tabE, const int32_t *__restrict__ tabA,
                             const int32_t *__restrict__ zE, const int32_t *__restrict__ zA,
                             const float *__restrict__ sE, const float *__restrict__ sA,
                             float *__restrict__ dW, int64_t dw_stride, int32_t *__restrict__ dWacc) {
    pdl_enter();
    const int taps = d.R * d.S, n = blockIdx.y, lane = threadIdx.x & (G - 1);
    const int64_t rows = (int64_t)d.Cout * taps;
    const unsigned ze = (unsigned)zE[n], za = (unsigned)zA[n];
    const float sc = dW ? __fmul_rn(sE[n], sA[n]) : 0.f;
    for (int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G; row < rows; row += (int64_t)gridDim.x * blockDim.x / G) {
        const int co = rows <= 0x7fffffff ? (int)((uint32_t)row / (uint32_t)taps) : (int)(row / taps), tap = (int)(row - (int64_t)co * taps);
        const int r = tap / d.S, s = tap - r * d.S;
        const unsigned cnt = (unsigned)d.B * (unsigned)taps_inside(Ho, d.H, r, d.pad, d.stride) *
                             (unsigned)taps_inside(Wo, d.W, s, d.pad, d.stride);
        const unsigned te = (unsigned)__ldg(tabE + ((int64_t)n * taps + tap) * d.Cout + co);
        const unsigned fixed = cnt * ze * za - za * te;
        const int64_t o0 = (int64_t)n * rows * d.Cin + row * d.Cin;
        const int32_t *ta = tabA + ((int64_t)n * taps + tap) * d.Cin;
        float *dw = dW ? dW + (int64_t)n * dw_stride + row * d.Cin : nullptr;
#pragma unroll 2
        for (int i = lane * V; i < d.Cin; i += G * V) {
            int rv[V], tv[V], acc[V];
            if constexpr (V == 4) {
                const int4 t = *reinterpret_cast<const int4 *>(raw + o0 + i), u = __ldg(reinterpret_cast<const int4 *>(ta + i));
                rv[0] = t.x; rv[1] = t.y; rv[2] = t.z; rv[3] = t.w;
                tv[0] = u.x; tv[1] = u.y; tv[2] = u.z; tv[3] = u.w;
            } else { rv[0] = raw[o0 + i]; tv[0] = __ldg(ta + i); }
#pragma unroll
            for (int k = 0; k < V; ++k) acc[k] = (int)((unsigned)rv[k] + fixed - ze * (unsigned)tv[k]);
            if constexpr (V == 4) {
                if (dWacc) *reinterpret_cast<int4 *>(dWacc + o0 + i) = make_int4(acc[0], acc[1], acc[2], acc[3]);
                if (dw) *reinterpret_cast<float4 *>(dw + i) = make_float4(__fmul_rn(__int2float_rn(acc[0]), sc), __fmul_rn(__int2float_rn(acc[1]), sc),
                                                                          __fmul_rn(__int2float_rn(acc[2]), sc), __fmul_rn(__int2float_rn(acc[3]), sc));
            } else {
                if (dWacc) dWacc[o0 + i] = acc[0];
                if (dw) dw[i] = __fmul_rn(__int2float_rn(acc[0]), sc);
            }
        }
    }
}

}  // namespace lpdt

static size_t affine_bwd_data_raw_bytes(const lpdt_conv_desc *d) {
    return align_up((size_t)d->nodes * d->B * d->H * d->W * d->Cin * sizeof(int32_t), 256);
}
static size_t affine_esum_bytes(const lpdt_conv_desc *d) {
    const int Ho = conv_out(d->H, d->pad, d->R, d->stride), Wo = conv_out(d->W, d->pad, d->S, d->stride);
    return align_up((size_t)d->nodes * d->B * Ho * Wo * sizeof(int32_t), 256);
}
static size_t affine_wsum_bytes(const lpdt_conv_desc *d) {
    return align_up((size_t)d->nodes * d->R * d->S * d->Cin * sizeof(int32_t), 256);
}

static size_t affine_bwd_data_own(const lpdt_conv_desc *d) {
    return affine_bwd_data_raw_bytes(d) + affine_esum_bytes(d) + affine_wsum_bytes(d);
}

extern "C" size_t lpdt_qconv_bwd_data_affine_workspace_size(const lpdt_conv_desc *d) {
    if (!d || d->nodes <= 0 || check_desc(d) != LPDT_OK) return 256;
    return affine_bwd_data_own(d) + lpdt_qconv_workspace_size(d, 1);
}

extern "C" lpdt_status lpdt_qconv_bwd_data_affine(const lpdt_conv_desc *d, const uint8_t *E, const float *sE,
                                                  const int32_t *zE, const uint8_t *Wq, const float *sW,
                                                  const int32_t *zW, float *dA, int32_t *dAacc, void *ws,
                                                  size_t ws_bytes, int32_t *dev_status, void *stream) {
    lpdt_status s = check_desc(d);
    if (s != LPDT_OK) return s;
    if (d->nodes == 0 || d->B == 0) return LPDT_OK;
    LPDT_CHECK_ARG(E && Wq && zE && zW && (dA || dAacc));
    LPDT_CHECK_ARG(!dA || (sE && sW));
    if (!ws || !aligned(ws, 256) || ws_bytes < affine_bwd_data_own(d) + least_workspace(d, 1)) return LPDT_ERR_WORKSPACE;
    cudaStream_t st = as_stream(stream);
    const int Ho = conv_out(d->H, d->pad, d->R, d->stride), Wo = conv_out(d->W, d->pad, d->S, d->stride);
    int32_t *raw = (int32_t *)ws;
    int32_t *esum = (int32_t *)((char *)ws + affine_bwd_data_raw_bytes(d));
    int32_t *wsum = (int32_t *)((char *)esum + affine_esum_bytes(d));
    void *inner = (char *)wsum + affine_wsum_bytes(d);
    const size_t inner_bytes = ws_bytes - (size_t)((char *)inner - (char *)ws);
    const RowSums sums = row_sums_of(E, (int64_t)d->nodes * d->B * Ho * Wo, d->Cout, esum);
    // Zero-point terms in the contraction's epilogue, as in the forward product; the table takes the place of the raw
    // sums, which do not exist then.  8 x 32 x 16x16 128 -> 128 3x3: 34.8 us, 107.5 us with the raw sums written and
    // corrected in a second pass (80 us of them), which shapes outside the tensor-core path still take.
    const size_t table = (size_t)d->nodes * (d->R + d->stride) * (d->S + d->stride) * d->Cin * sizeof(int32_t);
    if (!affine_separate() && !tiny_bwd_data(*d, reinterpret_cast<const int8_t *>(E)) && table_fits(*d, d->stride) &&
        table <= affine_bwd_data_raw_bytes(d) && use_tc(*d, 1, inner, inner_bytes)) {
        s = weight_table_launch(*d, Wq, 1, d->stride, raw, sums, st);
        if (s != LPDT_OK) return s;
        const tc::AffineArgs aff = {esum, raw, zE, zW};
        s = bwd_data_impl(d, reinterpret_cast<const int8_t *>(E), sE, reinterpret_cast<const int8_t *>(Wq), sW, dA, dAacc,
                          nullptr, inner, inner_bytes, dev_status, st, true, &aff);
        if (s != LPDT_ERR_UNSUPPORTED) return s;
    } else {
        s = row_sum_launch(sums, st);
        if (s != LPDT_OK) return s;
    }
    s = bwd_data_impl(d, reinterpret_cast<const int8_t *>(E), nullptr, reinterpret_cast<const int8_t *>(Wq), nullptr,
                      nullptr, raw, nullptr, inner, inner_bytes, dev_status, st, true);
    if (s != LPDT_OK) return s;
    launch_k(weight_cout_sum_kernel, grid_for((int64_t)d->nodes * d->R * d->S * d->Cin), 256, 0, st, *d, Wq, wsum);
    LPDT_LAUNCH_CHECK();
    const bool v4 = d->Cin % 4 == 0;
    const int64_t work = (int64_t)d->nodes * d->B * d->H * d->W * (d->Cin / (v4 ? 4 : 1));
    if (v4)
        launch_k(affine_fix_bwd_data_kernel<4>, grid_for(work), 256, 0, st, *d, Ho, Wo, raw, esum, wsum, zE, zW, sE, sW, dA, dAacc);
    else
        launch_k(affine_fix_bwd_data_kernel<1>, grid_for(work), 256, 0, st, *d, Ho, Wo, raw, esum, wsum, zE, zW, sE, sW, dA, dAacc);
    LPDT_LAUNCH_CHECK();
    return LPDT_OK;
}

static size_t affine_wg_raw_bytes(const lpdt_conv_desc *d) {
    return align_up((size_t)d->nodes * d->Cout * d->R * d->S * d->Cin * sizeof(int32_t), 256);
}
static size_t affine_tab_bytes(const lpdt_conv_desc *d, int C) {
    return align_up((size_t)d->nodes * d->R * d->S * C * sizeof(int32_t), 256);
}

static size_t affine_bwd_weight_own(const lpdt_conv_desc *d) {
    return affine_wg_raw_bytes(d) + affine_tab_bytes(d, d->Cout) + affine_tab_bytes(d, d->Cin);
}

extern "C" size_t lpdt_qconv_bwd_weight_affine_workspace_size(const lpdt_conv_desc *d) {
    if (!d || d->nodes <= 0 || check_desc(d) != LPDT_OK) return 256;
    return affine_bwd_weight_own(d) + lpdt_qconv_workspace_size(d, 2);
}

extern "C" lpdt_status lpdt_qconv_bwd_weight_affine(const lpdt_conv_desc *d, const uint8_t *E, const float *sE,
                                                    const int32_t *zE, const uint8_t *A, const float *sA,
                                                    const int32_t *zA, float *dW, int64_t dw_node_stride,
                                                    int32_t *dWacc, void *ws, size_t ws_bytes, int32_t *dev_status,
                                                    void *stream) {
    lpdt_status s = check_desc(d);
    if (s != LPDT_OK) return s;
    if (d->nodes == 0) return LPDT_OK;
    LPDT_CHECK_ARG((d->B == 0 || (E && A)) && zE && zA && (dW || dWacc));
    LPDT_CHECK_ARG(!dW || (sE && sA));
    LPDT_CHECK_ARG(!dW || dw_node_stride >= (int64_t)d->Cout * d->R * d->S * d->Cin || d->nodes == 1);
    if (d->nodes > 65535) return LPDT_ERR_UNSUPPORTED;
    if (!ws || !aligned(ws, 256) || ws_bytes < affine_bwd_weight_own(d) + least_workspace(d, 2)) return LPDT_ERR_WORKSPACE;
    cudaStream_t st = as_stream(stream);
    const int Ho = conv_out(d->H, d->pad, d->R, d->stride), Wo = conv_out(d->W, d->pad, d->S, d->stride);
    int32_t *raw = (int32_t *)ws;
    int32_t *tabE = (int32_t *)((char *)ws + affine_wg_raw_bytes(d));
    int32_t *tabA = (int32_t *)((char *)tabE + affine_tab_bytes(d, d->Cout));
    void *inner = (char *)tabA + affine_tab_bytes(d, d->Cin);
    size_t tabs = affine_tab_bytes(d, d->Cout) + affine_tab_bytes(d, d->Cin);      // cleared with the sums where these are
    s = bwd_weight_impl(d, reinterpret_cast<const int8_t *>(E), nullptr, reinterpret_cast<const int8_t *>(A), nullptr,
                        nullptr, 0, raw, inner, ws_bytes - (size_t)((char *)inner - (char *)ws), dev_status, st, true, &tabs);
    if (s != LPDT_OK) return s;
    // both operands' tap sums; samples are shared out until about two waves of blocks exist
    if (tabs) LPDT_CUDA(zero_async(tabE, tabs, st));
    const int sw = d->S < 24 ? d->S : 24, cw = 512;                  // 48 KB of shared memory at most
    const int64_t schunks = ceil_div(d->S, sw);
    TapSumSide sideE = {E, tabE, Ho, Wo, d->Cout, cw, (int)ceil_div(d->Cout, cw), 0};
    TapSumSide sideA = {A, tabA, d->H, d->W, d->Cin, cw, (int)ceil_div(d->Cin, cw), 0};
    sideE.items = d->nodes * sideE.chunks * schunks * Ho; sideA.items = d->nodes * sideA.chunks * schunks * d->H;
    int64_t shares = ceil_div(2 * kNumSMs, sideE.items + sideA.items);
    if (shares > ceil_div(d->B, 64)) shares = ceil_div(d->B, 64);
    if (shares < 1) shares = 1;
    sideE.items *= shares; sideA.items *= shares;
    const int64_t blocks = sideE.items + sideA.items < (int64_t)kNumSMs * 64 ? sideE.items + sideA.items : (int64_t)kNumSMs * 64;
    const bool v4 = d->Cin % 4 == 0 && d->Cout % 4 == 0 && aligned(E, 4) && aligned(A, 4);
    static PerDeviceOnce attr;
    int dev;
    if (attr.pending(&dev)) {
        for (auto fn : {tap_sum_kernel<4>, tap_sum_kernel<1>})
            LPDT_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024));
        attr.mark(dev);
    }
    // Two blocks fit an SM.  Where one operand's blocks have more than twice the other's bytes and are no more than the SMs, each
    // gets one of its own (whole product, 2 x 239 x 21x21, 34 -> 334, 1x1 of stride 2: 84.2 us, 64.4 so; 6 x 38 x 18x18,
    // 249 -> 15, 3x3 of stride 2: 83.8, 68.8).
    const int64_t e_bytes = (int64_t)Wo * (d->Cout < cw ? d->Cout : cw), a_bytes = (int64_t)d->W * (d->Cin < cw ? d->Cin : cw);
    const bool apart = (e_bytes > 2 * a_bytes && sideE.items <= kNumSMs) || (a_bytes > 2 * e_bytes && sideA.items <= kNumSMs);
    launch_k(v4 ? tap_sum_kernel<4> : tap_sum_kernel<1>, (unsigned)blocks, kTapThreads, spread_smem((size_t)sw * cw * 4, apart ? 1 : blocks, 2), st,
             *d, Ho, Wo, sideE, sideA, sw, (int)shares);
    LPDT_LAUNCH_CHECK();
    // four channels a step where every row of the three arrays begins on 16 bytes
    const bool f4 = d->Cin % 4 == 0 && (!dWacc || aligned(dWacc, 16)) && (!dW || (aligned(dW, 16) && (d->nodes == 1 || dw_node_stride % 4 == 0)));
    int G = 1;
    while (G < 32 && G * (f4 ? 4 : 1) < d->Cin) G <<= 1;
    int64_t fblocks = ceil_div((int64_t)d->Cout * d->R * d->S * G, 256);
    const int64_t fcap = ceil_div((int64_t)kNumSMs * 64, d->nodes);
    if (fblocks > fcap) fblocks = fcap;
    launch_k(f4 ? affine_fix_bwd_weight_kernel<4> : affine_fix_bwd_weight_kernel<1>, dim3((unsigned)fblocks, d->nodes), 256, 0, st, *d, Ho, Wo, G,
             raw, tabE, tabA, zE, zA, sE, sA, dW, dw_node_stride, dWacc);
    LPDT_LAUNCH_CHECK();
    return LPDT_OK;
}
