/*
 * tpfnet — the tensor-core kernels of the warm-start U-Net (training and inference).
 *
 * The paper has no network: this is the learned warm start that predicts steady
 * (phi, u, T) fields of the heated microchannel so that tpflbm_step converges in
 * fewer steps.  Every call is asynchronous on `stream` (cudaStream_t, NULL = legacy
 * default stream), takes device pointers the caller owns, allocates nothing, and
 * returns TPF_OK, TPF_ERR_INVALID_ARG (bad sizes) or TPF_ERR_CUDA (launch failure).
 *
 * Layouts: activations NHWC bfloat16 ("bf16": 2-byte storage); 3x3 weights bf16
 * [9][Cout][Cin] with tap = (dh + 1) * 3 + (dw + 1); biases, the 1x1 head, losses,
 * gradients and Adam state float32.  Convolutions use zero padding 1, stride 1, and
 * accumulate in float32 on the tensor cores.
 */
#ifndef TPFNET_H
#define TPFNET_H

#include <stddef.h>

#ifdef __cplusplus
extern "C" {
#endif

/* y = act(bias + conv3x3(x, wt)); act = ReLU when relu != 0.  Cin % 32 == 0,
 * Cout % 32 == 0; bias may be NULL. */
int tpfnet_conv3x3(const void *x, int N, int H, int W, int Cin, const void *wt, const float *bias, int Cout,
                   int relu, void *y, void *stream);

/* Which kernel tpfnet_conv3x3 (and tpfnet_conv3x3_dgrad, with Cin and Cout swapped)
 * runs for a shape, given 16-byte aligned tensors: the width in output channels of the
 * tcgen05 kernels' tiles (32, 64, 128 or 256), or 0 for the mma.sync kernel.  The
 * tcgen05 kernels take pixel blocks of 128 (8 x 16, or BW x BH with BW = min(W, 128)
 * dividing both 128 and W and BH dividing H); they stage operands with TMA and accumulate
 * in tensor memory.  Images of other extents take them too, from 1,024 pixels up, where the
 * staged blocks of all input channels and the weights fit: with more than 152 tiles two CTAs
 * have to share an SM's memory, and wide layers (from 128 or 192 input channels on, by the
 * tile's width) take the mma.sync kernel then. */
int tpfnet_conv3x3_tcgen05(int N, int H, int W, int Cin, int Cout);

/* 1 when tpfnet_conv3x3_wgrad runs a tcgen05 kernel for a shape (W a multiple of 64, or W of 8
 * and H of 16, or at least 1,024 pixels; 16-byte aligned tensors), 0 for the mma.sync kernel.  The tcgen05 weight gradient
 * reduces over pixels with both operands staged MN-major by TMA (one pixel's channels
 * per 128-byte row) and adds each CTA's FP32 partial sums into dw with atomics. */
int tpfnet_conv3x3_wgrad_tcgen05(int N, int H, int W, int Cin, int Cout);

/* TPF_OK, or TPF_ERR_TIMEOUT once a bounded wait of a tcgen05 kernel has run
 * out in this process (its output is then not to be trusted; the flag stays set);
 * TPF_ERR_CUDA if the flag cannot be read.  Synchronises with the device. */
int tpfnet_status(void);

/* Checks that a warp of the tcgen05 kernels leaves a wait as one: a warp waits on a barrier that
 * completes, first with every lane's polls, then with a lane that has none.  out: lanes that left
 * and error flag, for each (0, 0 and 32, 1). */
int tpfnet_check_bounded_wait(int polls, int out[4]);

/* Data gradient of conv3x3: dx = conv3x3 of dz (the gradient at the convolution's
 * output, ReLU mask already applied) with the flipped, transposed weights, which are
 * written to wflip (9 * Cin * Cout bf16 of caller scratch). */
int tpfnet_conv3x3_dgrad(const void *dz, int N, int H, int W, int Cout, const void *wt, int Cin, void *wflip,
                         void *dx, void *stream);

/* The same pieces in the forms that a whole network's passes join, so that no concatenation,
 * split or ReLU mask is a pass of its own:
 *   conv3x3_into: the output goes to Cout channels of a tensor with ldy channels per pixel
 *     (y points at the first of them, 4-byte aligned; ldy even);
 *   flip_weights: the flipped, transposed weights of up to 16 layers (host arrays of device
 *     pointers and sizes) in one launch;
 *   dgrad_masked: the data gradient from weights flipped before, zero where mask (laid out as
 *     dx; the layer's input, a ReLU output) is not positive; mask may be NULL;
 *   pool_from: pooling of C channels of a tensor with ldx channels per pixel;
 *   pool_back_skip: dx = dy / 4 + skip (lds channels per pixel), zero where mask (ldm) is not
 *     positive;
 *   up_back_masked, head_back_masked: the adjoints, dx zero where the mask (laid out as dx; for
 *     the head its input x) is not positive.
 * Pooling and upsampling in these forms take channel counts and offsets that are multiples of 8
 * and 16-byte aligned tensors. */
int tpfnet_conv3x3_into(const void *x, int N, int H, int W, int Cin, const void *wt, const float *bias, int Cout,
                        int relu, void *y, int ldy, void *stream);
int tpfnet_flip_weights(int layers, const void *const *wt, const int *cin, const int *cout, void *const *wflip,
                        void *stream);
int tpfnet_conv3x3_dgrad_masked(const void *dz, int N, int H, int W, int Cout, const void *wflip, int Cin,
                                const void *mask, void *dx, void *stream);
int tpfnet_pool_from(const void *x, int N, int H, int W, int C, int ldx, void *y, void *stream);
int tpfnet_pool_back_skip(const void *dy, int N, int H, int W, int C, const void *skip, int lds, const void *mask,
                          int ldm, void *dx, void *stream);
int tpfnet_up_back_masked(const void *dy, int N, int H, int W, int Ctot, int cofs, int C, const void *mask, void *dx,
                          void *stream);
int tpfnet_head_back_masked(const void *x, const float *dout, long long pixels, int C, const float *Wt, int Cout,
                            void *dx, float *dW, float *db, void *stream);

/* Weight and bias gradients of conv3x3, ADDED to dw ([9][Cout][Cin] float32) and db
 * (Cout float32, or NULL).  Cin % 32 == 0, Cout % 32 == 0. */
int tpfnet_conv3x3_wgrad(const void *x, const void *dz, int N, int H, int W, int Cin, int Cout, float *dw,
                         float *db, void *stream);

/* Parameter gradients whose float32 sums come out the same on every run: the kernels store what
 * they would have added to dw and db, and one launch adds that up in one order.
 *   wgrad_parts: the number of partial sums of conv3x3_wgrad_part for a shape (0: no such shape);
 *   conv3x3_wgrad_part: partial sum p is stored at part + p (9 Cout Cin + Cout), laid out as dw and
 *     then db; x, dz and part 16-byte aligned;
 *   head_parts, head_back_part: the same for head_back_masked (p (C + 1) Cout; dW and then db; C 8,
 *     16, ... 256, up to 8 outputs, x and dx 16-byte aligned);
 *   sum_parts: for n <= 32 ranges, dst[i][k] += sum over p < parts[i] of part[i][p stride[i] + k],
 *     k < count[i] (host arrays of device pointers and sizes; the ranges of dst do not overlap). */
int tpfnet_wgrad_parts(int N, int H, int W, int Cin, int Cout);
int tpfnet_conv3x3_wgrad_part(const void *x, const void *dz, int N, int H, int W, int Cin, int Cout, float *part,
                              void *stream);
int tpfnet_head_parts(long long pixels, int C, int Cout);
int tpfnet_head_back_part(const void *x, const float *dout, long long pixels, int C, const float *Wt, int Cout,
                          void *dx, float *part, void *stream);
int tpfnet_sum_parts(int n, const float *const *part, const long long *stride, const int *count, const int *parts,
                     float *const *dst, void *stream);

/* d[k] = 0 where y[k] <= 0 (ReLU backward on bf16 tensors of `count` elements). */
int tpfnet_relu_mask(void *d, const void *y, long long count, void *stream);

/* 2 x 2 average pooling (H, W even) and its adjoint (dx = dy / 4 spread over each
 * 2 x 2 block, added to dx when accumulate != 0). */
int tpfnet_pool(const void *x, int N, int H, int W, int C, void *y, void *stream);
int tpfnet_pool_back(const void *dy, int N, int H, int W, int C, void *dx, int accumulate, void *stream);

/* Nearest 2 x 2 upsampling of x (N, H/2, W/2, C) into channels [cofs, cofs + C) of
 * y (N, H, W, Ctot), and its adjoint (sum over each 2 x 2 block into dx (N, H/2, W/2, C)). */
int tpfnet_up_into(const void *x, int N, int H, int W, int C, void *y, int Ctot, int cofs, void *stream);
int tpfnet_up_back(const void *dy, int N, int H, int W, int Ctot, int cofs, int C, void *dx, void *stream);

/* Copy channels [sofs, sofs + C) of src (pixels x Sc) into channels [dofs, dofs + C)
 * of dst (pixels x Dc), adding when accumulate != 0 (concatenation and its adjoint). */
int tpfnet_channels(const void *src, int Sc, int sofs, long long pixels, int C, void *dst, int Dc, int dofs,
                    int accumulate, void *stream);

/* 1 x 1 head: out[p][o] = b[o] + sum_c x[p][c] Wt[c][o] (Wt, b, out float32), and its
 * gradients: dx (bf16) overwritten, dW and db ADDED.  C * Cout + Cout <= 12288. */
int tpfnet_head(const void *x, long long pixels, int C, const float *Wt, const float *b, int Cout, float *out,
                void *stream);
int tpfnet_head_back(const void *x, const float *dout, long long pixels, int C, const float *Wt, int Cout,
                     void *dx, float *dW, float *db, void *stream);

/* The whole forward pass of the 4-level network: the calls above in order, queued by one call.
 * weight and bias: the fourteen 3x3 layers in the order they run (encoder levels 0-3, decoder
 * levels 2-0, two layers each); the activations' buffers are the caller's and keep what a
 * backward pass needs (cat[l]: ch[l + 1] upsampled channels, then the encoder's ch[l]). */
typedef struct tpfnet_unet {
    int cin, cout, ch[4];      /* input channels (padded), outputs, channels per level */
    const void *weight[14];
    const float *bias[14];
    const float *head_w, *head_b;
    void *enc[4];              /* between the two layers of encoder level l */
    void *pool[3];             /* pooled outputs of levels 0-2 */
    void *cat[3];              /* concatenations of levels 0-2 */
    void *deep;                /* output of level 3 */
    void *dec_a[3], *dec[3];   /* between the two layers, and output, of decoder level l */
} tpfnet_unet;
int tpfnet_unet_forward(const tpfnet_unet *u, const void *x, int N, int H, int W, float *out, void *stream);

/* loss += mean_k (pred[k] - target[k])^2 wch[k % C] (FP64, device); grad[k] = d loss /
 * d pred[k] (or NULL to skip); wch may be NULL (all ones). */
int tpfnet_mse(const float *pred, const float *target, const float *wch, long long count, int C, float *grad,
               double *loss, void *stream);

/* One Adam step (bias-corrected, step >= 1) on float32 parameters p with gradient g and
 * moments m, v; writes the bf16 copy pb as well when pb != NULL. */
int tpfnet_adam(float *p, const float *g, float *m, float *v, long long count, float lr, float b1, float b2,
                float eps, int step, void *pb, void *stream);

/* Planar fields to an interleaved tensor and back, with a per-channel affine map
 * (scale, shift: host arrays of C floats, NULL = 1 and 0; 1 <= C <= 8) and optional
 * base planes (device, same layout as the planar side, NULL = 0):
 *   pack:   dst[p * Cd + c] = (src[c * plane + p] - base[c * plane + p]) * scale[c] + shift[c]
 *           for c < C (float32 dst, or bf16 when dst_bf16 != 0; channels C..Cd-1 untouched);
 *   unpack: dst[c * plane + p] = src[p * C + c] * scale[c] + shift[c] + base[c * plane + p]. */
int tpfnet_pack(const float *src, const float *base, long long plane, int C, long long pixels, const float *scale,
                const float *shift, void *dst, int Cd, int dst_bf16, void *stream);
int tpfnet_unpack(const float *src, long long pixels, int C, const float *scale, const float *shift,
                  const float *base, float *dst, long long plane, void *stream);

/* y = bf16(x). */
int tpfnet_to_bf16(const float *x, long long count, void *y, void *stream);

#ifdef __cplusplus
}
#endif

#endif /* TPFNET_H */
