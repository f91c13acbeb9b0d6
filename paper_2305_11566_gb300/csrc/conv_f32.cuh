// conv_f32.cuh -- FP32 convolutions and their gradients on the CUDA cores: jobs, packed
// weights and launchers (conv_f32.cu, wgrad_f32.cu).
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <vector>

namespace sv {

// A convolution as window taps over an input grid.  Output grid position (y, x) of a phase
// reads the TY x TX inputs at (S y + dy0 + r, S x + dx0 + c).
//   FK_S2    3x3 stride 2 (encoder)            FK_P1    1x1 (latent heads and their gradient)
//   FK_UP2   nearest x2 + 3x3 (decoder): four output phases of 2x2 taps, the weights that
//            fall on one input pixel summed
//   FK_DS2   input gradient of FK_S2: four phases of 1x1, 1x2, 2x1, 2x2 taps
//   FK_DUP2  input gradient of the nearest-x2 layer: nine taps at each of the four upsampled positions
//   FK_S1_5, FK_S2_5  5x5 stride 1 / 2;  FK_DE5  5x5 stride-2 deconvolution: four phases of
//            3x3, 3x2, 2x3, 2x2 taps
//   FK_Y5    the Table I network's last layer: 5x5 stride-2 deconvolution to one channel, the four
//            output phases taken as four output channels of a 3x3 window
//   FK_UP2X  nearest x2 + 3x3 on the upsampled grid, nine taps (the training forward)
enum F32Kind { FK_S2 = 0, FK_P1, FK_UP2, FK_DS2, FK_DUP2, FK_S1_5, FK_S2_5, FK_DE5, FK_UP2X, FK_Y5, FK_COUNT };

// One pair's operands of a layer.  `in`: the input is the channel concatenation of up to four
// NHWC tensors of Hi x Wi (widths ic, each a whole number of staged channel chunks).
struct F32Job {
  const float* in[4];
  int ic[4];
  const float* mask;  // input gradients: activation whose ReLU masks the result, or null
  float* out;         // [Ho][Wo][N]
  int Hi, Wi, Ho, Wo;
};

// One pair's image, coarse map and the tensors of the first / last layer and the latent.
struct F32Img {
  const uint8_t* L;
  int pitch, W, H, w, h;
  const int16_t* coarse_i;  // integer coarse map, or
  const float* coarse_f;    // real-valued coarse map when non-null
  float* e1;                // [H1][W1][C]
  const float* d3;          // [H][W][C]
  float* Y;                 // [H][W]
  const float* gY;          // gradient of Y
  float* gd3;               // gradient of d3
  const float* ge1;         // gradient of e1
  int W1, H1;
};

// Elementwise latent operands of one pair.
struct F32Lat {
  const float *mu, *lv, *eps, *gz, *gmu_ext, *glv_ext;
  float *z, *gmu, *glv, *mu_copy, *lv_copy, *eps_copy;
  __nv_bfloat16* z16;  // tensor-core forward: z rounded to BF16 (z then holds the rounded value)
  size_t n;
};

// BF16 tensor converted to FP32 (n a multiple of 8, both 16-byte aligned).
struct F32Cvt {
  const __nv_bfloat16* src;
  float* dst;
  size_t n;
};

// Weight gradient operands of one pair: dW += sum over the pixels of g (x) taps of x.
struct F32WJob {
  const float* g;  // [Ho][Wo][Co]
  const float* x;  // [Hi][Wi][Ci]
  int Hi, Wi, Ho, Wo;
  int unit0, units;  // first slot of this pair in its range, its slots
};

// One packed weight block; see f32_pack_kernel.
struct F32PackDesc {
  size_t src;      // offset of W[co][ks][ks][ci] in the flat parameters
  size_t dst;      // offset of the block in the packed buffer
  int kind, phase, border;
  int ks, co, ci;  // of the source layer
  int K, N;        // contraction and output channels of the packed form
  int cic, bn, taps, tx;
  size_t count;
};

// A layer's packed weights and launch constants.
struct F32Layer {
  int kind = 0, K = 0, N = 0, cg = 0;  // cg: groups of 8 output channels per block
  size_t w[4] = {0, 0, 0, 0}, wb = 0;
};

// Adds the pack descriptors of a layer (grad: its input gradient) to `descs` and returns its launch
// constants; `total` is the packed buffer's size so far in floats.
struct F32Src { size_t w_ofs; int ks, co, ci; };
F32Layer f32_plan_layer(int kind, bool grad, const F32Src& src, std::vector<F32PackDesc>& descs, size_t& total);
cudaError_t launch_f32_pack(const F32PackDesc* d_descs, int n, size_t max_count, const float* params, float* packed,
                            cudaStream_t st);

// act: 0 none, 1 ReLU, 2 leaky ReLU 0.1; + 4 (FK_P1): the sums start at the bias; + 8 (FK_P1):
// added to the output.  maxHo / maxWo: largest output of the jobs.
cudaError_t launch_f32_conv(const F32Layer& l, const F32Job* jobs, int n, int maxHo, int maxWo, const float* packed,
                            const float* bias, int act, cudaStream_t st);
cudaError_t launch_f32_enc1(const F32Img* imgs, int n, int maxH1, int maxW1, const float* w, const float* b, int C,
                            cudaStream_t st);
// z = mu + eps exp(lv / 2), with copies of mu, lv and eps where asked for.
cudaError_t launch_f32_reparam(const F32Lat* lat, int n, size_t max_n, cudaStream_t st);
// FK_Y5: out = scale (sum + bias); the jobs' tensors are [Hi][Wi][ic] inputs, [Ho][Wo] outputs.
F32Layer f32_plan_y5(size_t w_ofs, const int* ic, int n_ic, std::vector<F32PackDesc>& descs, size_t& total);
cudaError_t launch_f32_y5(const F32Layer& l, const F32Job* jobs, int n, int maxHo, int maxWo, const float* packed,
                          const float* bias, float scale, cudaStream_t st);
cudaError_t launch_f32_convert(const F32Cvt* jobs, int n, size_t max_n, cudaStream_t st);
// ordered: summed in the training step's order (real-valued coarse maps).
cudaError_t launch_f32_final(const F32Img* imgs, int n, int maxH, int maxW, const float* w, const float* b, int C,
                             bool ordered, cudaStream_t st);

// Weight gradients: plan (fills the jobs' slot ranges), slots (scratch, p.slot_floats) and launch;
// gw / gb are added to.  Every pair needs slots of its own, so the pairs go in ranges of at most
// slot_budget floats of slots (one pair at least), one after the other on the same scratch: the sums are
// added in pair order either way.
struct F32WRange { int i0, n, units; };
struct F32WPlan {
  int kind = 0, co = 0, ci = 0;
  size_t slot = 0, slot_floats = 0;
  std::vector<F32WRange> ranges;
};
F32WPlan f32_wgrad_plan(int kind, int co, int ci, std::vector<F32WJob>& jobs, size_t slot_budget);
cudaError_t launch_f32_wgrad(const F32WPlan& p, const F32WJob* d_jobs, float* gw, float* gb, float* slots,
                             cudaStream_t st);
// Input gradient of the final conv (masked by d3's ReLU).
cudaError_t launch_f32_final_dgrad(const F32Img* imgs, int n, int maxH, int maxW, const float* w, int C,
                                   cudaStream_t st);
// Weight gradients of the final conv (kind FK_WFINAL) and of enc1 (FK_WENC1).
enum { FK_WFINAL = FK_COUNT, FK_WENC1 };
cudaError_t launch_f32_edge_wgrad(const F32WPlan& p, const F32Img* imgs, const F32WJob* d_jobs, float* gw, float* gb,
                                  float* slots, cudaStream_t st);
cudaError_t launch_f32_latent_bwd(const F32Lat* lat, int n, size_t max_n, cudaStream_t st);

}  // namespace sv
