// Internal interface between the convolution front end (argument checks,
// kernel choice) and its back ends.  Not part of the ABI.
#pragma once
#include <cuda.h>
#include "common.cuh"

namespace lpdt {

static inline int conv_out(int H, int pad, int R, int stride) { return (H + 2 * pad - R) / stride + 1; }

lpdt_status generic_fwd(const lpdt_conv_desc &d, const int8_t *A, const float *sA, const int8_t *Wq,
                        const float *sW, const float *bias, int64_t bias_stride, float *Y, int32_t *Yacc,
                        cudaStream_t st, bool uns = false);
lpdt_status generic_bwd_data(const lpdt_conv_desc &d, const int8_t *E, const float *sE, const int8_t *Wq,
                             const float *sW, float *dA, int32_t *dAacc, const float *addend, void *ws, cudaStream_t st,
                             bool uns = false);
lpdt_status generic_bwd_weight(const lpdt_conv_desc &d, const int8_t *E, const float *sE, const int8_t *A,
                               const float *sA, float *dW, int64_t dw_stride, int32_t *dWacc, void *ws,
                               cudaStream_t st, bool uns = false);

lpdt_status dequant_acc_launch(const int32_t *acc, int nodes, int64_t per_node, const float *s1,
                               const float *s2, float *out, int64_t out_stride, cudaStream_t st);

namespace tc {
// Tensor-core engine (tcgen05 kind::i8): convolutions of stride 1 and 2 and GEMMs.
// mode 0 = forward, 1 = backward-data.
// Bytes between the channel rows of the operands in memory (multiples of 16, at least the channel count).
struct Pitches { int in, err, w; };      // activations (Cin), layer gradients (Cout), weights (Cin)
bool tc_supported(const lpdt_conv_desc &d);
bool tc_shape(const lpdt_conv_desc &d);      // the part of it that the shape decides
// Zero-point correction applied in the epilogue (unsigned operands): per-pixel channel sums of operand A (the input, or
// backward-data the layer gradient), the table of the weights' channel sums over the filter taps (see PixParams; up to
// 124 bytes past its end are read), and the per-node zero points of operand A and of the weights.
struct AffineArgs { const int32_t *asum, *wpre, *zA, *zW; };
lpdt_status tc_pix(const lpdt_conv_desc &d, int mode, const int8_t *A, const float *s1, const int8_t *Wq,
                   const float *s2, const float *bias, int64_t bias_stride, float *Y, int32_t *Yacc,
                   int32_t *dev_status, cudaStream_t st, bool uns, const float *addend,
                   const AffineArgs *aff, Pitches pt);
// Halo-tile kernel for 16-channel operands at stride 1 (one TMA request per tile).
bool halo_supported(const lpdt_conv_desc &d, int mode);
lpdt_status tc_pix_halo(const lpdt_conv_desc &d, int mode, const int8_t *A, const float *s1, const int8_t *Wq,
                        const float *s2, const float *bias, int64_t bias_stride, float *Y, int32_t *Yacc,
                        int32_t *dev_status, cudaStream_t st, bool uns = false, const float *addend = nullptr);
// *more_clear bytes behind acc_user (its size rounded up to 256 bytes) are cleared together with it where it is cleared
// at all; *more_clear is 0 then.
lpdt_status tc_wgrad(const lpdt_conv_desc &d, const int8_t *E, const float *sE, const int8_t *A,
                     const float *sA, int32_t *acc_user, int32_t *acc_ws, float *dW, int64_t dw_stride,
                     int32_t *dev_status, cudaStream_t st, bool uns, Pitches pt, size_t *more_clear = nullptr);
// Whether that is one launch that writes dW itself (no split of the pixel loop, no sums in memory).
bool wgrad_direct(const lpdt_conv_desc &d, Pitches pt);
// The same on pairs of SMs (signed codes, stride 1, 128-byte operand rows, 256-channel tiles, fp32 result in rows of 16 bytes): the
// tiling and the operand-A and result maps of tc_pix.  UNSUPPORTED where the one-SM kernel is the better one.
struct PixTile { int TB, TH, TW, tilesB, tilesH, tilesW; };
lpdt_status tc_pix_pair(const lpdt_conv_desc &d, int mode, const PixTile &t, int cpt, const CUtensorMap &mA, const CUtensorMap &mY,
                        const int8_t *Wq, int pitch_w, const float *s1, const float *s2, const float *bias, int64_t bias_stride,
                        int32_t *dev_status, cudaStream_t st, const float *addend);
}  // namespace tc

}  // namespace lpdt
