// sv_internal.cuh -- internal declarations shared by the CUDA translation units of
// the StereoVAE library (context, device descriptors, kernel launchers).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <array>
#include <cstdint>
#include <cstring>
#include <cstddef>
#include <string>
#include <vector>

#include "../../include/stereovae.h"

namespace sv {

// ------------------------------------------------------------------ coarse stage
// Device descriptor of one pair for the coarse matcher.
struct ZPair {
  const uint8_t* L;
  const uint8_t* R;
  int W, H, pitch, D;
  int w, h;          // coarse size = (W / 4, H / 4)
  int16_t* disp;     // [h][w]
  float* best;       // [h][w] or nullptr
  float* second;     // [h][w] or nullptr
  float* cost;       // [h][w][D] cost volume 1 - rho (2 where x - d < 0), or nullptr
};

// One CTA job: rows [y0, y0 + ty) and columns [x0, x0 + group width) of a pair.
struct ZJob {
  int pair, y0, x0, pad;
};

constexpr int kZnccTY = 8;      // coarse rows per job
constexpr int kZnccWarps = 8;   // warps per CTA; each owns a column tile of TX(KD) columns
constexpr int kZnccSmallTX = 8, kZnccSmallTY = 4;  // jobs of a call that would leave SMs idle

inline int zncc_kd(int D) { return (D + 31) / 32; }
inline int zncc_tx(int kd) { return kd == 1 ? 32 : kd == 2 ? 20 : kd == 3 ? 16 : 12; }

// Pairs of a small call, passed by value with the launch (no table upload): pair i's jobs start
// at job0[i], tiles_x[i] of them per row of jobs.
constexpr int kZnccInline = 16;
struct ZInline {
  int n, tx, ty;
  int job0[kZnccInline + 1], tiles_x[kZnccInline];
  ZPair p[kZnccInline];
};

// Shared-memory layout of one ZNCC job (window radius r, disparity count D, tile TX).
struct ZLayout {
  int nlc, nrc, gx, nrs;  // staged left / right columns, job width, right-window columns
  size_t off_sl, off_sr, off_suml, off_invl, off_statr, off_cs, off_cs2, total;
};
__host__ __device__ inline size_t align16(size_t v) { return (v + 15) & ~size_t(15); }
__host__ __device__ inline ZLayout zlayout(int r, int D, int tx, int TY) {
  ZLayout z;
  z.gx = kZnccWarps * tx;
  z.nlc = z.gx + 2 * r;
  z.nrc = z.gx + 2 * r + D - 1;
  z.nrs = z.gx + D - 1;
  size_t o = 0;
  z.off_sl = o; o = align16(o + sizeof(uint16_t) * (TY + 2 * r) * z.nlc);
  z.off_sr = o; o = align16(o + sizeof(uint16_t) * (TY + 2 * r) * z.nrc);
  z.off_suml = o; o = align16(o + sizeof(int) * TY * z.gx);
  z.off_invl = o; o = align16(o + sizeof(float) * TY * z.gx);
  z.off_statr = o; o = align16(o + 2 * sizeof(int) * TY * z.nrs);  // {sum, 1/sigma} per right window
  z.off_cs = o; o = align16(o + sizeof(int) * TY * z.nrc);
  z.off_cs2 = o; o = align16(o + sizeof(unsigned) * TY * z.nrc);
  z.total = o;
  return z;
}

// Job shape of a call: the large jobs share their staging and statistics over more pixels; a call
// whose large jobs are fewer than the GPU's SMs takes the small ones, whose chain of dependent work is a fifth
// as long.  One 256 x 128 pair, D = 16: 4 large jobs 38.7 us, 8 small ones 15.0; one 1242 x 375 pair, D = 48: 24
// large jobs 41, 120 small ones 16.7 us.
struct ZShape {
  int tx, ty;
  bool small;
};
inline ZShape zncc_shape(const sv_pair* pairs, int n, int maxD) {
  const int tx = zncc_tx(zncc_kd(maxD)), gx = kZnccWarps * tx;
  long long jobs = 0;
  for (int i = 0; i < n; ++i)
    jobs += (long long)((pairs[i].height / 4 + kZnccTY - 1) / kZnccTY) * ((pairs[i].width / 4 + gx - 1) / gx);
  if (jobs < 152) return {kZnccSmallTX, kZnccSmallTY, true};
  return {tx, kZnccTY, false};
}

// Fused downsample + ZNCC + WTA over the given jobs, one entry per window radius
// r = 1..7 and mode (each compiled in its own translation unit).
// mode 0: disparities only; 1: also the best / second scores of the pairs that ask for them;
// 2: also the cost volume (the pairs' cost pointers are set); 3: the cost volume only (disp unused).
// small: jobs of the small shape; in: the pairs by value (p and j unused), or null.
#define SV_ZNCC_DECL(r, m)                                                                                          \
  cudaError_t launch_zncc_wta_r##r##_m##m(const ZPair* d_pairs, const ZJob* d_jobs, int n_jobs, int maxD, bool small, \
                                          const ZInline* in, cudaStream_t st);
#define SV_ZNCC_EACH(X) X(1) X(2) X(3) X(4) X(5) X(6) X(7)
#define SV_ZNCC_DECLS(r) SV_ZNCC_DECL(r, 0) SV_ZNCC_DECL(r, 1) SV_ZNCC_DECL(r, 2) SV_ZNCC_DECL(r, 3)
SV_ZNCC_EACH(SV_ZNCC_DECLS)
inline cudaError_t launch_zncc_wta(const ZPair* p, const ZJob* j, int n, int r, int maxD, cudaStream_t st,
                                   int mode, bool small, const ZInline* in = nullptr) {
  switch (r * 4 + mode) {
#define SV_ZNCC_CASES(r)                                                          \
  case r * 4: return launch_zncc_wta_r##r##_m0(p, j, n, maxD, small, in, st);     \
  case r * 4 + 1: return launch_zncc_wta_r##r##_m1(p, j, n, maxD, small, in, st); \
  case r * 4 + 2: return launch_zncc_wta_r##r##_m2(p, j, n, maxD, small, in, st); \
  case r * 4 + 3: return launch_zncc_wta_r##r##_m3(p, j, n, maxD, small, in, st);
    SV_ZNCC_EACH(SV_ZNCC_CASES)
  }
  return cudaErrorInvalidValue;
}
#undef SV_ZNCC_CASES
#undef SV_ZNCC_DECLS
#undef SV_ZNCC_DECL
#undef SV_ZNCC_EACH

// ------------------------------------------------------------------ refinement
enum Layer { L_ENC1 = 0, L_ENC2, L_ENC3, L_MU, L_LV, L_DEC1, L_DEC2, L_DEC3, L_FINAL, L_COUNT };

struct NetDims {
  int enc[3], lat, dec[3];
  int cout(int l) const;
  int cin(int l) const;
  int ks(int l) const;
  size_t w_off(int l) const;   // offset of W of layer l in the flat vector
  size_t b_off(int l) const;   // offset of b
  size_t count() const;
};

// Spatial sizes of the four levels of a W x H input.
struct Levels {
  int H[4], W[4];
  explicit Levels(int H0 = 0, int W0 = 0) {
    H[0] = H0; W[0] = W0;
    for (int i = 1; i < 4; ++i) { H[i] = (H[i - 1] + 1) / 2; W[i] = (W[i - 1] + 1) / 2; }
  }
};

// Direct (CUDA-core) convolution arguments, element type T (float or double).
// Activations NHWC; weights canonical [cout][ks][ks][cin].
enum ConvMode { CM_S1 = 0, CM_S2 = 1, CM_UP2 = 2 };
template <typename T>
struct DirectConvArgs {
  const T* in; int Hi, Wi, Ci;
  const T* wt; const T* bias; int Co;
  int Ho, Wo;
  int relu;
  T* out;
};

template <typename T>
cudaError_t launch_conv_direct(const DirectConvArgs<T>& a, int mode, int ks, cudaStream_t st);

// enc1 with the network input built on the fly: x0 = (L / 256, U / 256), U = 4 *
// bilinear(coarse).  CoarseT = int16_t (inference) or T (training).
template <typename T, typename CoarseT>
cudaError_t launch_enc1(const uint8_t* L, int pitch, int W, int H, const CoarseT* coarse, int w, int h,
                        const T* wt, const T* bias, int Co, T* out, cudaStream_t st);

// final 3x3 conv (cin -> 1) + bias + U (recomputed bilinear) -> Y
template <typename T, typename CoarseT, typename OutT>
cudaError_t launch_final(const T* in, int W, int H, int Ci, const T* wt, const T* bias, const CoarseT* coarse,
                         int w, int h, OutT* Y, cudaStream_t st);

// Per-pair descriptors of the batched CUDA-core layers of the tensor-core form.
struct alignas(128) EdgePair {
  const uint8_t* L;
  int pitch, W, H, w, h;
  const int16_t* coarse;    // integer coarse map (inference), or
  const float* coarse_f;    // real-valued coarse map (training) when non-null
  __nv_bfloat16* e1;        // enc1 output [H1][W1][C1]
  const __nv_bfloat16* d3;  // last decoder output [H][W][C]
  float* Y;                 // refined disparity [H][W]
  uint8_t* e1q;             // FP8 form: the tensor-core enc1 writes E4M3 codes of e1 here instead
  CUtensorMap d3_map;       // TMA view of d3 for the final conv (final_staged_by_tma(C))
};
// Row copy between device-accessible buffers (host_io.cu): `height` rows of `width`
// elements of elem_bytes bytes.
struct HostRowCopy {
  const unsigned char* src;
  unsigned char* dst;
  int spitch, dpitch, width, height;  // pitches in bytes
};
cudaError_t launch_copy_rows(const HostRowCopy* jobs, int njobs, int max_rows, int elem_bytes, cudaStream_t st);

// U = 4 x bilinear(coarse) at full-resolution pixel (X, Y), half-pixel centres, source
// clamped to the coarse map (Sec. IV-C "linear scaling", reading N1), FP32.
template <typename CT>
__device__ __forceinline__ float upsample4_f(const CT* __restrict__ c, int w, int h, int X, int Y) {
  float sx = (float)X * 0.25f - 0.375f, sy = (float)Y * 0.25f - 0.375f;
  sx = fminf(fmaxf(sx, 0.f), (float)(w - 1));
  sy = fminf(fmaxf(sy, 0.f), (float)(h - 1));
  const int x0 = (int)sx, y0 = (int)sy;
  const int x1 = min(x0 + 1, w - 1), y1 = min(y0 + 1, h - 1);
  const float fx = sx - (float)x0, fy = sy - (float)y0;
  const float top = (1.f - fx) * (float)c[(size_t)y0 * w + x0] + fx * (float)c[(size_t)y0 * w + x1];
  const float bot = (1.f - fx) * (float)c[(size_t)y1 * w + x0] + fx * (float)c[(size_t)y1 * w + x1];
  return 4.f * ((1.f - fy) * top + fy * bot);
}

// Final conv of the tensor-core form: widths with the register-blocked kernel stage their
// (rows + 2) x 34 x C input tile with one TMA box; its height in output rows per block.
inline bool final_staged_by_tma(int C) { return C == 16 || C == 32 || C == 64 || C == 128; }
inline int final_tile_rows(int C) { return 16 * (C / 8 >= 8 ? 1 : 8 / (C / 8)); }
struct UpFixPair {          // one decoder layer of one pair (input, output, sizes)
  const __nv_bfloat16* in;
  __nv_bfloat16* out;
  int Hi, Wi, Ho, Wo, Hu, Wu;
};
// enc1 for every pair of a call; `tensor`: the tensor-core kernel where C1 allows (16, 32,
// 64), whose bounded wait records code 7 in `err`.
cudaError_t launch_edge_enc1(const EdgePair* pairs, int n, int maxW1, int maxH1, const float* W, const float* B, int C1,
                             int* err, long long spin, bool tensor, cudaStream_t st);
cudaError_t launch_edge_final(const EdgePair* pairs, int n, int maxW, int maxH, const float* W, const float* B, int C,
                              int* err, long long spin, cudaStream_t st);
// Border pixels of a cropped nearest-x2 + 3x3 conv output that the 4-phase form folds
// wrongly: the last row when Ho is odd, the last column (above that row) when Wo is odd.
// The fix kernel takes them in segments of kUpFixSeg pixels, one block per segment.
constexpr int kUpFixSeg = 64;
inline int upfix_segments(int Ho, int Wo) {
  const int nrow = (Ho & 1) ? Wo : 0, ncol = (Wo & 1) ? Ho - (Ho & 1) : 0;
  return (nrow + kUpFixSeg - 1) / kUpFixSeg + (ncol + kUpFixSeg - 1) / kUpFixSeg;
}
cudaError_t launch_edge_up2fix(const UpFixPair* pairs, int n, int max_segments, const __nv_bfloat16* Wb,
                               const float* bias, int cin, int cout, int relu, cudaStream_t st);

// The border recompute of inference on warp MMA: BF16 input and weights, or (f8) E4M3 input codes and
// unfolded weights with their per-output-channel scale (output E4M3 codes, or BF16 when out_f8 = 0).
inline int upfix_pixels(int Ho, int Wo) { return ((Ho & 1) ? Wo : 0) + ((Wo & 1) ? Ho - (Ho & 1) : 0); }
cudaError_t launch_edge_up2fix_mma(const UpFixPair* pairs, int n, int max_pixels, const void* W, const float* wscale,
                                   const float* bias, int cin, int cout, int relu, bool f8, int out_f8,
                                   cudaStream_t st);
// Last two output columns of odd-width pairs after the fused dec3 + final kernel (W: BF16 unfolded dec3
// weights, wf / bf: FP32 final conv).
cudaError_t launch_fused_edge_cols(const UpFixPair* fix, const EdgePair* edges, int n, int maxH, const void* W,
                                   const float* bias, const float* wf, const float* bf, int cin, int NT,
                                   cudaStream_t st);
// E4M3 codes of a BF16 tensor.
cudaError_t launch_bf16_to_e4m3(const __nv_bfloat16* a, uint8_t* b, size_t n, cudaStream_t st);

// Input gradient of enc1 in FP32 (Ci = 2): d loss / d (L / 256, U / 256).
cudaError_t launch_enc1_dgrad(const float* gout, int Ho, int Wo, int Co, const float* w, int Hi, int Wi, float* gin,
                              cudaStream_t st);

// One pair of the loss: smooth-L1 of Y against gt, KL of (mu, lv); gradients where not null.
template <typename T>
struct LossJob {
  const T* Y;
  const float* gt;
  T* gY;
  size_t P;
  const T *mu, *lv;
  T *gmu, *glv;
  size_t n;
};

// latent heads on the H3 x W3 grid: mu = 1x1(e3) + b; optionally logvar and z = mu + eps * exp(lv / 2).
template <typename T>
cudaError_t launch_latent(const T* e3, int H3, int W3, int Ci, const T* wmu, const T* bmu, const T* wlv, const T* blv,
                          int lat, const T* eps, T* mu, T* lv, T* z, cudaStream_t st);

}  // namespace sv
