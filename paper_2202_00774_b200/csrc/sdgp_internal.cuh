// Internal declarations shared by the translation units of the SDGP library.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/sdgp.h"

namespace sdgp {

// Multiprocessors of the current device (148 if it cannot be asked).
int sm_count();

// k_pad (0 = none): row pitch, in elements, of the metadata (compressed outputs only, no dense copy): the extra chunks of every
// row name the position pair (0,1), so that a reader can take a row as k_pad channels - those past K of zero value, which it supplies
// itself (TMA reads them as zeros).
cudaError_t launch_prune(const void* dO, int64_t rows, int64_t K, int n, int m, int scheme,
                         uint64_t seed, void* dense, void* values, void* meta, void* mask,
                         cudaStream_t stream, int64_t k_pad = 0, int dtype = SDGP_BF16);

// n > 2 of groups of 8, 16 or 32 (rank.cu): dense pruned copy and / or mask; nvec 8-element vectors, an even number.
cudaError_t launch_rank(const void* dO, int64_t nvec, int n, int m, int scheme, uint64_t seed, void* dense, void* mask,
                        cudaStream_t stream, int dtype);

// The producer of dL/dO below a ReLU fused with its pruning: the gradient above the ReLU (dY) passes where the
// activation `act` is positive; `grad` (optional) receives that unpruned dL/dO, the other outputs are
// launch_prune's. n <= 2, or n == m (nothing pruned: only `grad` and the mask make sense then). skip (optional): a second
// gradient of the same shape, added to dY (fp32 sum, rounded to the 16-bit type) before the gate.
cudaError_t launch_relu_backward_prune(const void* dY, const void* act, int64_t rows, int64_t K, int n, int m, int scheme,
                                       uint64_t seed, void* grad, void* dense, void* values, void* meta, void* mask,
                                       cudaStream_t stream, int dtype = SDGP_BF16, const void* skip = nullptr);

// The same producer below a ReLU that is followed by 2 x 2 max pooling of stride 2: dYp is the pooled gradient
// [B, H/2, W/2, K], act the activation [B, H, W, K]; each pooled gradient goes to the first largest activation of its
// window if that is positive. skip_pooled (optional): a second gradient of the pooled shape, added to dYp first.
// B * H * W * K / 32 must fit 31 bits; H and W even.
cudaError_t launch_maxpool_relu_backward_prune(const void* dYp, const void* act, int B, int H, int W, int64_t K, int n, int m,
                                               int scheme, uint64_t seed, void* grad, void* dense, void* values, void* meta,
                                               void* mask, cudaStream_t stream, int dtype = SDGP_BF16,
                                               const void* skip_pooled = nullptr);

// y [B, H/2, W/2, K] = 2 x 2 max pooling of relu(x), x [B, H, W, K] NHWC (prune.cu); H and W even, K a multiple of 8. A NaN in a window
// gives NaN.
cudaError_t launch_relu_maxpool(const void* x, int64_t B, int64_t H, int64_t W, int64_t K, int dtype, void* y, cudaStream_t stream);

// Per-channel reading of the L1 rescale (channel.cu). sums: 2 * K floats (cleared by the call): the
// column sums of |x| over all rows, then the same over the survivors of the magnitude function.
cudaError_t launch_channel_sums(const void* dO, int64_t rows, int64_t K, int n, int m, int dtype, float* sums,
                                cudaStream_t stream);
// Both at once for n <= 2: launch_channel_sums' sums and launch_prune's compressed form under the magnitude function, in one read of dO.
cudaError_t launch_prune_sums(const void* dO, int64_t rows, int64_t K, int n, int m, int dtype, float* sums, void* values, void* meta,
                              int64_t k_pad, cudaStream_t stream);
// scales[k] = sums[k] / sums[K + k] (1 where the denominator is 0)
cudaError_t launch_channel_scales(const float* sums, int64_t K, float* scales, cudaStream_t stream);
// Wout[k, :] = W[k, :] * scale[k] rounded to the element type (row_elems elements per row, a multiple of 8); also
// writes the K scales.
cudaError_t launch_scale_weights(const void* W, const float* sums, int64_t K, int64_t row_elems, int dtype, void* Wout,
                                 float* scales, cudaStream_t stream);

// Data gradient on the tensor cores (stride 1 or 2). sparse == false: A is dense dL/dO
// [B,P,Q,Cout]; sparse == true: A is the compressed values [B,P,Q,Cout/2] and meta [B,P,Q,Cp/16]
// with Cp = Cout rounded up to a multiple of 128 (see launch_prune's k_pad); values rows are not padded.
// Wt [Cout,R,S,Cin], dD [B,H,W,Cin]. A fully connected layer is B = H = 1, W = rows, R = S = 1.
// fused != nullptr: A is the dense dL/dO and the kernel prunes it on the fly (n <= 2).
struct FusedPrune {
  int n;
  int m;  // group size: 4, 8, 16 (32 in the whole-filter-reuse kernel only)
  int scheme;
  uint64_t seed;
};
// dtype: element type of A, Wt and dD (SDGP_BF16 or SDGP_FP16; accumulation is fp32 either way).
// Fused pruning with the rescaled scheme exists for bf16 only.
// stored != nullptr: Cin and Cout are the channel counts the kernels tile by (multiples of 64; Wt has that
// many rows and columns, the extra ones zero) while the tensors in global memory hold fewer channels per
// pixel: `a` for dL/dO, dense or compressed (0 = Cout), `d` for dD
// (0 = Cin), both multiples of 8. TMA reads the missing channels of A as zeros and clips the stores of dD.
struct StoredChannels {
  int a;
  int d;
};
// conv_groups != nullptr: Wt is block-diagonal - input channels [g * cin_g, (g + 1) * cin_g) are connected to output
// channels [g * cout_g, (g + 1) * cout_g) only, everything else in Wt is zero - so a tile of input channels skips
// the channel blocks of dL/dO that only meet zeros.
struct ConvGroups {
  int cin_g;
  int cout_g;
};
sdgp_status launch_dgrad(bool sparse, const void* A, const void* meta, const void* Wt, void* dD, int B,
                         int H, int W, int Cin, int Cout, int R, int S, int stride, int pad, cudaStream_t stream,
                         const FusedPrune* fused = nullptr, int dtype = SDGP_BF16, const StoredChannels* stored = nullptr,
                         const ConvGroups* conv_groups = nullptr);

// dD [rows, N] = prune(dO [rows, K]) . W [K, N] in one kernel, if that is estimated to be faster than prune kernel + contraction
// (*taken tells; nothing is launched otherwise). K and N multiples of 8, prune.n <= 2.
sdgp_status try_rows_fused(const void* dO, const void* W, void* dD, int64_t rows, int K, int N, const FusedPrune& prune, int dtype,
                           cudaStream_t stream, bool* taken);

// Filters of a grouped convolution, Wg [Cout, R*S, Cin/groups], written as the block-diagonal filters of an
// ordinary one, Wfull [cout_pad, R*S, cin_pad] (zeros outside each group's block and in the padding).
cudaError_t launch_expand_grouped_weights(const void* Wg, int Cout, int taps, int Cin, int groups, int cout_pad, int cin_pad,
                                          void* Wfull, cudaStream_t stream);

// Data gradient of a grouped convolution with C channels on both sides, pruned inside the kernel (n <= 2); Wg [C, R, S, C / groups].
// SDGP_ERR_UNSUPPORTED (nothing launched): groups of other widths than 16 or 32 channels, filters or images that no plan fits or that the
// path over block-diagonal filters is faster on.
sdgp_status launch_grouped_fused(const void* dO, const void* Wg, void* dD, int B, int H, int W, int C, int groups, int R, int S, int stride,
                                 int pad, const FusedPrune& prune, int dtype, cudaStream_t stream);
cudaError_t take_error_grouped(unsigned int* word);
// Estimated time, us, of that other path at stride 1: prune kernel, block-diagonal filters, contraction.
double estimate_block_diagonal(int B, int H, int W, int C, int groups, int R, int S, int pad, const FusedPrune& prune);

// For sdgp_selftest_plan(): whether a call takes the kernel for narrow groups, or the four output parities of a stride-2 layer in one launch, and its
// plan (eight ints). Arguments as launch_grouped_fused's and launch_dgrad's.
bool query_grouped(int B, int H, int W, int C, int groups, int R, int S, int stride, int pad, const FusedPrune& prune, int* plan);
bool query_parities(bool sparse, int B, int H, int W, int Cin, int Cout, int R, int S, int stride, int pad, const StoredChannels* stored,
                    const ConvGroups* conv_groups, int* plan);

// Launches a one-CTA kernel whose only wait can never be satisfied (50 ms limit).
sdgp_status launch_bounded_wait_selftest(cudaStream_t stream);

// Synchronises the device, then reads and clears the kernels' error word.
sdgp_status read_device_error();

}  // namespace sdgp
