// enc1_dgrad.cu -- input gradient of the first encoder layer in FP32, for the gradient of the
// coarse map: dX(i, ci) = sum over the taps k with o = (i + 1 - k) / 2 an output pixel of
// dY(o, co) W[co][k][ci], two channels.  A block owns 8 x 16 input pixels and stages dY of the output
// region they reach (zero outside) and the weights, eight output channels at a time.
#include "sv_internal.cuh"

namespace sv {

namespace {

constexpr int kTH = 8, kTW = 16;               // input pixels per block
constexpr int kGR = (kTH - 1 + 2) / 2 + 2, kGC = (kTW - 1 + 2) / 2 + 2;  // output rows / columns they reach
constexpr int kCoc = 8;

__device__ __forceinline__ int floor_half(int a) { return a >= 0 ? a / 2 : -((-a + 1) / 2); }

__global__ void __launch_bounds__(kTH * kTW)
enc1_dgrad_kernel(const float* __restrict__ gout, int Ho, int Wo, int Co, const float* __restrict__ w, int Hi, int Wi,
                  float* __restrict__ gin) {
  __shared__ float gp[kGR][kGC][kCoc];
  __shared__ __align__(8) float wsm[9][kCoc][2];
  const int tid = threadIdx.x, ty = tid / kTW, tx = tid % kTW;
  const int I0 = blockIdx.y * kTH, J0 = blockIdx.x * kTW;
  const int iy = I0 + ty, ix = J0 + tx;
  const int oy0 = floor_half(I0 - 1), ox0 = floor_half(J0 - 1);
  float acc[2] = {0.f, 0.f};
  for (int c0 = 0; c0 < Co; c0 += kCoc) {
    __syncthreads();
    for (int e = tid; e < kGR * kGC * kCoc; e += kTH * kTW) {
      const int c = e % kCoc, q = e / kCoc;
      const int oy = oy0 + q / kGC, ox = ox0 + q % kGC;
      gp[q / kGC][q % kGC][c] =
          (oy >= 0 && ox >= 0 && oy < Ho && ox < Wo && c0 + c < Co) ? gout[((size_t)oy * Wo + ox) * Co + c0 + c] : 0.f;
    }
    for (int e = tid; e < 9 * kCoc * 2; e += kTH * kTW) {
      const int ci = e % 2, co = e / 2 % kCoc, tap = e / (2 * kCoc);
      wsm[tap][co][ci] = c0 + co < Co ? w[((size_t)(c0 + co) * 9 + tap) * 2 + ci] : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int ky = 0; ky < 3; ++ky) {
      const int ny = iy + 1 - ky;
      if (ny & 1) continue;
      const int ry = floor_half(ny) - oy0;
#pragma unroll
      for (int kx = 0; kx < 3; ++kx) {
        const int nx = ix + 1 - kx;
        if (nx & 1) continue;
        const int rx = floor_half(nx) - ox0;
#pragma unroll
        for (int co = 0; co < kCoc; ++co) {
          const float g = gp[ry][rx][co];
          acc[0] = fmaf(g, wsm[ky * 3 + kx][co][0], acc[0]);
          acc[1] = fmaf(g, wsm[ky * 3 + kx][co][1], acc[1]);
        }
      }
    }
  }
  if (iy >= Hi || ix >= Wi) return;
  *reinterpret_cast<float2*>(gin + ((size_t)iy * Wi + ix) * 2) = make_float2(acc[0], acc[1]);
}

}  // namespace

cudaError_t launch_enc1_dgrad(const float* gout, int Ho, int Wo, int Co, const float* w, int Hi, int Wi, float* gin,
                              cudaStream_t st) {
  enc1_dgrad_kernel<<<dim3((Wi + kTW - 1) / kTW, (Hi + kTH - 1) / kTH), kTH * kTW, 0, st>>>(gout, Ho, Wo, Co, w, Hi,
                                                                                            Wi, gin);
  return cudaGetLastError();
}

}  // namespace sv
