// wgrad_f32.cu -- weight gradients of the FP32 refinement layers on the CUDA cores, all pairs of
// a call per launch.
//
// dW[co][ky][kx][ci] = sum over output pixels p of g(p, co) V(p S + k - pad, ci), V the layer's input
// view.  The summation order is fixed and does not depend on the block shape (conv_f32.cu says
// why the training step keeps one order): a pair's 8 x 16 output tiles go to `units` chains, tile t to
// chain t mod units; a chain adds its tiles' pixels in row order, each weight in one accumulator; the
// chains' sums are added in chain order, the pairs' in pair order.  No atomics.
//
// A block runs one chain for a block of output x input channels.  A warp owns one kernel row: a lane
// holds COL output x 4 input channels x 3 kernel columns in registers and slides the three input
// columns along the row, so a pixel costs it 2 loads of g and 0.5 (nearest x2), 1 or 2 (stride 2) of x
// for 96 multiply-adds (one thread holding 4 x 2 channels x 9 taps loaded 10 vectors for 72).  g and
// x of a few rows (a whole tile where the input is low-resolution) are staged by cp.async in two
// buffers, the next step's once the step's one barrier has shown everyone done with the last; one
// warp adds the bias gradient from the g it holds anyway (lanes of their own, reading g once more
// behind the others, cost 5 %).  16 pairs of 1242 x 375, 16/32/64 net: dec3 and dec2 3.23 ms (6.8
// before, one pair a launch) at 43 TFLOP/s; the whole training step with the input gradients of
// conv_f32.cu 31.1 -> 10.6 ms.  The FMA pipes are 60 % busy: 96-168 registers a thread leave 12-18
// warps an SM, in blocks of 3 or 6 that meet at the barrier.  Summing the folded phase-taps instead
// ran dec3 and dec2 in 1.6 ms but moves the gradient's bits (see conv_f32.cu).
#include "conv_f32.cuh"

#include <algorithm>
#include <type_traits>

#include "sv_internal.cuh"

namespace sv {

namespace {

typedef unsigned long long u64;
__device__ __forceinline__ u64 dup2(float a) {
  u64 r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a));
  return r;
}
__device__ __forceinline__ void fma2(u64& d, u64 a, u64 b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b)); }
__device__ __forceinline__ float2 unpack2(u64 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ void cp16z(float* dst, const float* src, bool ok) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(dst);
  const int n = ok ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(s), "l"(src), "r"(n));
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N)); }

constexpr int kTR = 8, kTC = 16;  // pixels of a tile

// Kernel rows (= warps per channel block) and columns, tile rows staged per step, staged x.
template <int KIND> struct WK;
template <> struct WK<FK_S2> { static constexpr int KR = 3, KC = 3, ROWS = 2, XR = 5, XC = 33; };
template <> struct WK<FK_P1> { static constexpr int KR = 1, KC = 1, ROWS = 4, XR = 4, XC = 16; };
template <> struct WK<FK_UP2> { static constexpr int KR = 3, KC = 3, ROWS = 8, XR = 6, XC = 10; };

// COL output channels per lane, CGN x IGN lanes of a warp, NB input-channel blocks (warps) per kernel row.
template <int KIND, int COL_, int CGN_, int IGN_, int NB_>
struct WG {
  using K = WK<KIND>;
  static constexpr int COL = COL_, CGN = CGN_, IGN = IGN_, NB = NB_;
  static constexpr int BCO = COL * CGN, WCI = 4 * IGN, BCI = WCI * NB, NT = 32 * K::KR * NB;
  static constexpr int NG = K::ROWS * kTC;
  static constexpr int GF = NG * BCO, XF = K::XR * K::XC * BCI, BUF = GF + XF;
  static constexpr size_t SMEM = 2 * sizeof(float) * BUF;
  static constexpr int WARPS = K::KR * NB, MINB = COL == 8 ? (WARPS > 6 ? 1 : WARPS > 3 ? 2 : 4) : (WARPS > 6 ? 2 : WARPS > 3 ? 3 : 6);
};

template <int KIND, int COL, int CGN, int IGN, int NB>
__global__ void __launch_bounds__(WG<KIND, COL, CGN, IGN, NB>::NT, WG<KIND, COL, CGN, IGN, NB>::MINB)
wgrad_f32_kernel(const F32WJob* __restrict__ jobs, int n, int Co, int Ci, size_t slot, float* __restrict__ slots) {
  using G = WG<KIND, COL, CGN, IGN, NB>;
  using K = WK<KIND>;
  constexpr int BCO = G::BCO, BCI = G::BCI, KC = K::KC;
  extern __shared__ __align__(16) float wf_sm[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int ky = warp % K::KR, cib = warp / K::KR;
  const int cg = lane % CGN, ig = lane / CGN % IGN;  // (fewer than 32 lanes: the others repeat)
  const int nci = (Ci + BCI - 1) / BCI, co0 = ((int)blockIdx.y / nci) * BCO, ci0 = ((int)blockIdx.y % nci) * BCI;
  int job = 0;
  while (job + 1 < n && (int)blockIdx.x >= jobs[job + 1].unit0) ++job;
  const F32WJob& J = jobs[job];
  const int Ho = J.Ho, Wo = J.Wo, Hi = J.Hi, Wi = J.Wi;
  const int tiles_x = (Wo + kTC - 1) / kTC, ntiles = tiles_x * ((Ho + kTR - 1) / kTR);
  const int t0 = blockIdx.x - J.unit0;
  constexpr int STEPS = kTR / K::ROWS;
  const int nsteps = (ntiles - t0 + J.units - 1) / J.units * STEPS;
  u64 acc[KC][COL][2];
#pragma unroll
  for (int k = 0; k < KC; ++k)
#pragma unroll
    for (int j = 0; j < COL; ++j) acc[k][j][0] = acc[k][j][1] = 0ull;
  u64 bacc[COL / 2];  // bias gradient: one warp adds the g it reads anyway
#pragma unroll
  for (int j = 0; j < COL / 2; ++j) bacc[j] = 0ull;
  const bool bias_warp = ci0 == 0 && cib == 0 && ky == K::KR / 2;

  auto stage = [&](int step) {
    const int t = t0 + step / STEPS * J.units;
    const int Y0 = t / tiles_x * kTR + step % STEPS * K::ROWS, X0 = t % tiles_x * kTC;
    float* gs = wf_sm + (step & 1) * G::BUF;
    float* xs = gs + G::GF;
#pragma unroll 4
    for (int e = threadIdx.x; e < G::NG * (BCO / 4); e += G::NT) {
      const int c = e % (BCO / 4), p = e / (BCO / 4);
      const int oy = Y0 + p / kTC, ox = X0 + p % kTC;
      const bool ok = oy < Ho && ox < Wo;
      cp16z(gs + p * BCO + 4 * c, ok ? J.g + ((size_t)oy * Wo + ox) * Co + co0 + 4 * c : J.g, ok);
    }
    const int iy0 = KIND == FK_S2 ? 2 * Y0 - 1 : KIND == FK_UP2 ? Y0 / 2 - 1 : Y0;
    const int ix0 = KIND == FK_S2 ? 2 * X0 - 1 : KIND == FK_UP2 ? X0 / 2 - 1 : X0;
#pragma unroll 4
    for (int e = threadIdx.x; e < K::XR * K::XC * (BCI / 4); e += G::NT) {
      const int c = e % (BCI / 4), p = e / (BCI / 4), r = p / K::XC, q = p - r * K::XC;
      const int iy = iy0 + r, ix = ix0 + q;
      const bool ok = iy >= 0 && ix >= 0 && iy < Hi && ix < Wi && ci0 + 4 * c < Ci;
      cp16z(xs + p * BCI + 4 * c, ok ? J.x + ((size_t)iy * Wi + ix) * Ci + ci0 + 4 * c : J.x, ok);
    }
    cp_commit();
  };
  auto add2 = [](u64& d, u64 a) { asm("add.rn.f32x2 %0, %0, %1;" : "+l"(d) : "l"(a)); };
  auto loadg = [&](auto bias, const float* g, u64 (&gv)[COL]) {
#pragma unroll
    for (int h = 0; h < COL / 4; ++h) {
      const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(g + h * (BCO / 2) + cg * 4);
      const float2 u = unpack2(q.x), v = unpack2(q.y);
      gv[4 * h] = dup2(u.x); gv[4 * h + 1] = dup2(u.y); gv[4 * h + 2] = dup2(v.x); gv[4 * h + 3] = dup2(v.y);
      if constexpr (decltype(bias)::value) {
        add2(bacc[2 * h], q.x);
        add2(bacc[2 * h + 1], q.y);
      }
    }
  };
  auto madd = [&](u64 (&a)[COL][2], const u64 (&gv)[COL], const ulonglong2& x) {
#pragma unroll
    for (int j = 0; j < COL; ++j) {
      fma2(a[j][0], gv[j], x.x);
      fma2(a[j][1], gv[j], x.y);
    }
  };

  if (nsteps > 0) stage(0);
  for (int step = 0; step < nsteps; ++step) {
    cp_wait<0>();
    __syncthreads();  // this step's rows are there, and everyone is done with the last step's buffer
    if (step + 1 < nsteps) stage(step + 1);
    const int t = t0 + step / STEPS * J.units;
    const int Y0 = t / tiles_x * kTR + step % STEPS * K::ROWS, X0 = t % tiles_x * kTC;
    const float* gs = wf_sm + (step & 1) * G::BUF;
    const float* xs = gs + G::GF + cib * G::WCI + ig * 4;
    auto X = [&](int r, int c) { return *reinterpret_cast<const ulonglong2*>(xs + (r * K::XC + c) * BCI); };
    auto rows = [&](auto bias) {
#pragma unroll 1
      for (int r = 0; r < K::ROWS; ++r) {
        const float* gr = gs + r * kTC * BCO;
        if constexpr (KIND == FK_UP2) {
          if (Y0 + r + ky - 1 >= Ho) continue;  // the cropped upsampled row adds nothing
          const int xr = ((r + ky - 1) >> 1) + 1;
          ulonglong2 xm = X(xr, 0), x0 = X(xr, 1);
#pragma unroll 2
          for (int c = 0; c < kTC / 2; ++c) {
            const ulonglong2 xp = X(xr, c + 2);
            u64 gv[COL];
            loadg(bias, gr + 2 * c * BCO, gv);
            madd(acc[0], gv, xm);
            madd(acc[1], gv, x0);
            if (X0 + 2 * c + 1 < Wo) madd(acc[2], gv, x0);  // (else cropped)
            loadg(bias, gr + (2 * c + 1) * BCO, gv);
            madd(acc[0], gv, x0);
            madd(acc[1], gv, x0);
            madd(acc[2], gv, xp);
            xm = x0;
            x0 = xp;
          }
        } else if constexpr (KIND == FK_S2) {
          const int xr = 2 * r + ky;
          ulonglong2 xa = X(xr, 0);
#pragma unroll 2
          for (int c = 0; c < kTC; ++c) {
            const ulonglong2 xb = X(xr, 2 * c + 1), xc = X(xr, 2 * c + 2);
            u64 gv[COL];
            loadg(bias, gr + c * BCO, gv);
            madd(acc[0], gv, xa);
            madd(acc[1], gv, xb);
            madd(acc[2], gv, xc);
            xa = xc;
          }
        } else {
#pragma unroll 4
          for (int c = 0; c < kTC; ++c) {
            u64 gv[COL];
            loadg(bias, gr + c * BCO, gv);
            madd(acc[0], gv, X(r, c));
          }
        }
      }
    };
    if (bias_warp)
      rows(std::true_type());
    else
      rows(std::false_type());
  }
  float* out = slots + (size_t)blockIdx.x * slot;
  constexpr int TAPS = K::KR * KC;
  const int ci = ci0 + cib * G::WCI + ig * 4;
  if (lane < CGN * IGN && ci < Ci) {
#pragma unroll
    for (int k = 0; k < KC; ++k)
#pragma unroll
      for (int j = 0; j < COL; ++j) {
        const int co = co0 + (j >> 2) * (BCO / 2) + cg * 4 + (j & 3);
        const float2 u = unpack2(acc[k][j][0]), v = unpack2(acc[k][j][1]);
        *reinterpret_cast<float4*>(out + ((size_t)co * TAPS + ky * KC + k) * Ci + ci) = make_float4(u.x, u.y, v.x, v.y);
      }
  }
  if (bias_warp && ig == 0)
#pragma unroll
    for (int h = 0; h < COL / 4; ++h)
      *reinterpret_cast<ulonglong2*>(out + (size_t)TAPS * Co * Ci + co0 + h * (BCO / 2) + cg * 4) =
          make_ulonglong2(bacc[2 * h], bacc[2 * h + 1]);
}

// gw[e] += the pairs' sums (e < nWw), gb[e - nWw] likewise: a pair's chains in chain order, the pairs in
// pair order.  A block takes 32 elements, its 8 rows one pair each.
__global__ void __launch_bounds__(256)
wgrad_f32_reduce(const float* __restrict__ slots, const F32WJob* __restrict__ jobs, int n, size_t slot, int nW, int nWw,
                 float* __restrict__ gw, float* __restrict__ gb) {
  __shared__ float part[8][32];
  const int e = blockIdx.x * 32 + threadIdx.x, y = threadIdx.y;
  float tot = 0.f;
  if (y == 0 && e < nW) tot = e < nWw ? gw[e] : gb[e - nWw];
  for (int i0 = 0; i0 < n; i0 += 8) {
    float s = 0.f;
    if (i0 + y < n && e < nW) {
      const float* p = slots + (size_t)jobs[i0 + y].unit0 * slot + e;
      const int u = jobs[i0 + y].units;
      int b = 0;
      for (; b + 8 <= u; b += 8) {
        float v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = p[(size_t)(b + j) * slot];
#pragma unroll
        for (int j = 0; j < 8; ++j) s += v[j];
      }
      for (; b < u; ++b) s += p[(size_t)b * slot];
    }
    part[y][threadIdx.x] = s;
    __syncthreads();
    if (y == 0)
      for (int j = 0; j < 8 && i0 + j < n; ++j) tot += part[j][threadIdx.x];
    __syncthreads();
  }
  if (y == 0 && e < nW) {
    if (e < nWw)
      gw[e] = tot;
    else
      gb[e - nWw] = tot;
  }
}

// Input gradient of the final conv (C channels -> 1), masked by d3's ReLU.  C / 4 lanes hold a
// pixel's channels; a thread walks down the rows of one column with the nine neighbouring output
// gradients from shared memory.  Bound by reading d3 and writing its gradient once.
constexpr int kFbRows = 16, kFbThreads = 256;
__global__ void __launch_bounds__(kFbThreads)
f32_final_dgrad_kernel(const F32Img* __restrict__ imgs, const float* __restrict__ w, int C, int tiles_x) {
  extern __shared__ __align__(16) float fb_sm[];
  const int L = C / 4, NC = kFbThreads / L;  // lanes of a pixel, columns of a tile
  const int l = threadIdx.x % L, col = threadIdx.x / L, P = NC + 2;
  const F32Img& I = imgs[blockIdx.z];
  const int Y0 = (blockIdx.x / tiles_x) * kFbRows, X0 = (blockIdx.x % tiles_x) * NC;
  if (Y0 >= I.H || X0 >= I.W) return;
  float4 k[9];
#pragma unroll
  for (int t = 0; t < 9; ++t) k[t] = *reinterpret_cast<const float4*>(w + t * C + 4 * l);
  for (int e = threadIdx.x; e < (kFbRows + 2) * P; e += kFbThreads) {
    const int r = e / P, c = e - r * P, y = Y0 - 1 + r, x = X0 - 1 + c;
    fb_sm[e] = y >= 0 && x >= 0 && y < I.H && x < I.W ? I.gY[(size_t)y * I.W + x] : 0.f;
  }
  __syncthreads();
  const int x = X0 + col;
  if (col >= NC || x >= I.W) return;
  const int rows = min(kFbRows, I.H - Y0);
  const size_t base = ((size_t)Y0 * I.W + x) * C + 4 * l, step = (size_t)I.W * C;
#pragma unroll 1
  for (int r0 = 0; r0 < rows; r0 += 4) {
    float4 v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (r0 + j < rows) v[j] = *reinterpret_cast<const float4*>(I.d3 + base + (r0 + j) * step);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (r0 + j >= rows) break;
      const int r = r0 + j;
      float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int q = 0; q < 9; ++q) {
        // output (y + 1 - ky, x + 1 - kx) read this pixel through tap (ky, kx)
        const float g = fb_sm[(r + 2 - q / 3) * P + col + 2 - q % 3];
        d.x = fmaf(g, k[q].x, d.x);
        d.y = fmaf(g, k[q].y, d.y);
        d.z = fmaf(g, k[q].z, d.z);
        d.w = fmaf(g, k[q].w, d.w);
      }
      d.x = v[j].x > 0.f ? d.x : 0.f;
      d.y = v[j].y > 0.f ? d.y : 0.f;
      d.z = v[j].z > 0.f ? d.z : 0.f;
      d.w = v[j].w > 0.f ? d.w : 0.f;
      *reinterpret_cast<float4*>(I.gd3 + base + r * step) = d;
    }
  }
}

// Weight gradient of the final conv: a lane owns one kernel row, 4 input channels and their three
// kernel columns, and reads d3 and the output gradient of its chain's rows straight from memory (the
// lanes of a pixel read whole sectors; the three kernel rows and neighbouring tiles meet in the
// caches).  3 C / 4 lanes run a chain; a lane of the middle kernel row, which sees every output, adds the
// bias (a lane of its own walked the tile one dependent load at a time while its warp waited: 16 pairs
// of 1242 x 375, 16 channels, 317 -> 263 us with its reduction).  Bound by the loads' latency.
__global__ void __launch_bounds__(256)
f32_final_wgrad_kernel(const F32Img* __restrict__ imgs, const F32WJob* __restrict__ jobs, int n, int units, int C,
                       int lanes, size_t slot, float* __restrict__ slots) {
  const int per = blockDim.x / lanes;  // chains of a block
  const int u = blockIdx.x * per + threadIdx.x / lanes, l = threadIdx.x % lanes;
  if (threadIdx.x / lanes >= per || u >= units) return;
  int job = 0;
  while (job + 1 < n && u >= jobs[job + 1].unit0) ++job;
  const F32WJob& J = jobs[job];
  const int H = J.Ho, W = J.Wo;
  const int tiles_x = (W + kTC - 1) / kTC, ntiles = tiles_x * ((H + kTR - 1) / kTR);
  const float* g = imgs[job].gY;
  float* out = slots + (size_t)u * slot;
  const int ky = l / (C / 4), c4 = 4 * (l % (C / 4));
  const bool bias = l == C / 4;  // (ky 1, channel 0)
  float bacc = 0.f;
  float4 acc[3] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
  for (int t = u - J.unit0; t < ntiles; t += J.units) {
    const int Y0 = t / tiles_x * kTR, X0 = t % tiles_x * kTC, ye = min(Y0 + kTR, H);
    for (int y = Y0; y < ye; ++y) {
      const int vy = y + ky - 1;
      if (vy < 0 || vy >= H) continue;
      const float* x = J.x + ((size_t)vy * W + X0) * C + c4;
      const float* gr = g + (size_t)y * W + X0;
      const int m = W - X0;  // columns of the row that exist
      float4 v[kTC + 2];
      float gv[kTC];
#pragma unroll
      for (int j = 0; j < kTC + 2; ++j)
        v[j] = (j > 0 || X0 > 0) && j - 1 < m ? *reinterpret_cast<const float4*>(x + (j - 1) * C)
                                              : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int j = 0; j < kTC; ++j) gv[j] = j < m ? gr[j] : 0.f;
      if (bias)
#pragma unroll
        for (int j = 0; j < kTC; ++j) bacc += gv[j];
#pragma unroll
      for (int j = 0; j < kTC; ++j)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          acc[k].x = fmaf(gv[j], v[j + k].x, acc[k].x);
          acc[k].y = fmaf(gv[j], v[j + k].y, acc[k].y);
          acc[k].z = fmaf(gv[j], v[j + k].z, acc[k].z);
          acc[k].w = fmaf(gv[j], v[j + k].w, acc[k].w);
        }
    }
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) *reinterpret_cast<float4*>(out + (ky * 3 + k) * C + c4) = acc[k];
  if (bias) out[9 * C] = bacc;
}

// Weight and bias gradient of enc1 (2 channels -> C, stride 2): a warp builds the network input
// (L / 256, U / 256) under its chain's tile in shared memory; a lane owns one kernel row and 4 output
// channels: 4 x 3 columns x 2 channels.  Up to 20 channels a chain fills half a warp at most: two
// chains share it (CW = 2; 16 channels, 16 pairs of 1242 x 375: 324 -> 264 us with its
// reduction).
constexpr int kEwWarps = 4, kEwR = 2 * kTR + 1, kEwC = 2 * kTC + 1;
template <int CW>
__global__ void __launch_bounds__(32 * kEwWarps)
f32_enc1_wgrad_kernel(const F32Img* __restrict__ imgs, const F32WJob* __restrict__ jobs, int n, int units, int C,
                      size_t slot, float* __restrict__ slots) {
  constexpr int LW = 32 / CW;  // lanes of a chain
  __shared__ float2 sm[kEwWarps * CW][kEwR][kEwC];
  const int chain = threadIdx.x / LW, lane = threadIdx.x % LW, u = blockIdx.x * kEwWarps * CW + chain;
  int job = 0;
  while (job + 1 < n && u >= jobs[job + 1].unit0) ++job;
  const F32WJob& J = jobs[job];
  const F32Img& I = imgs[job];
  const int tiles_x = (I.W1 + kTC - 1) / kTC, ntiles = u < units ? tiles_x * ((I.H1 + kTR - 1) / kTR) : 0;
  float* out = slots + (size_t)u * slot;
  const int q0 = C / 4;
  // 3 q0 (kernel row, 4 channels) tasks, LW at a time
  for (int base = 0; base < 3 * q0; base += LW) {
    const int task = base + lane;
    const bool on = task < 3 * q0;
    const int ky = on ? task / q0 : 0, c4 = on ? 4 * (task % q0) : 0;
    float4 acc[6], bacc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int k = 0; k < 6; ++k) acc[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int t = u - J.unit0; __any_sync(0xffffffffu, t < ntiles); t += J.units) {
      const bool live = t < ntiles;  // (the warp's other chain may have a tile more)
      const int Y0 = t / tiles_x * kTR, X0 = t % tiles_x * kTC;
      __syncwarp();
      for (int e = lane; live && e < kEwR * kEwC; e += LW) {
        const int r = e / kEwC, c = e - r * kEwC, vy = 2 * Y0 - 1 + r, vx = 2 * X0 - 1 + c;
        float2 v = make_float2(0.f, 0.f);
        if (vy >= 0 && vx >= 0 && vy < I.H && vx < I.W) {
          v.x = (float)I.L[(size_t)vy * I.pitch + vx] * (1.0f / 256.0f);
          v.y = upsample4_f(I.coarse_f, I.w, I.h, vx, vy) * (1.0f / 256.0f);
        }
        sm[chain][r][c] = v;
      }
      __syncwarp();
      const int ye = live && on ? min(kTR, I.H1 - Y0) : 0, xe = min(kTC, I.W1 - X0);
      for (int y = 0; y < ye; ++y) {
        const float* g = I.ge1 + ((size_t)(Y0 + y) * I.W1 + X0) * C + c4;
        const float2* xr = sm[chain][2 * y + ky];
        float2 xa = xr[0];
#pragma unroll 8
        for (int x = 0; x < xe; ++x) {
          const float4 gv = *reinterpret_cast<const float4*>(g + (size_t)x * C);
          const float2 xb = xr[2 * x + 1], xc = xr[2 * x + 2];
          auto madd = [&](float4& a, float v) {
            a.x = fmaf(gv.x, v, a.x);
            a.y = fmaf(gv.y, v, a.y);
            a.z = fmaf(gv.z, v, a.z);
            a.w = fmaf(gv.w, v, a.w);
          };
          madd(acc[0], xa.x); madd(acc[1], xa.y);
          madd(acc[2], xb.x); madd(acc[3], xb.y);
          madd(acc[4], xc.x); madd(acc[5], xc.y);
          bacc.x += gv.x; bacc.y += gv.y; bacc.z += gv.z; bacc.w += gv.w;
          xa = xc;
        }
      }
    }
    if (on && u < units) {
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        const float v[4] = {acc[k].x, acc[k].y, acc[k].z, acc[k].w};
#pragma unroll
        for (int j = 0; j < 4; ++j) out[(size_t)(c4 + j) * 18 + ky * 6 + k] = v[j];
      }
      if (ky == 0) {
        out[18 * C + c4] = bacc.x; out[18 * C + c4 + 1] = bacc.y; out[18 * C + c4 + 2] = bacc.z; out[18 * C + c4 + 3] = bacc.w;
      }
    }
  }
}

// gmu = gz + the loss's own term; glv = gz eps exp(lv / 2) / 2 + the loss's own term.
__global__ void f32_latent_bwd_kernel(const F32Lat* __restrict__ lat) {
  const F32Lat& q = lat[blockIdx.y];
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < q.n; i += (size_t)gridDim.x * blockDim.x) {
    const float gz = q.gz[i];
    q.gmu[i] = gz + (q.gmu_ext ? q.gmu_ext[i] : 0.f);
    q.glv[i] = gz * q.eps[i] * 0.5f * expf(0.5f * q.lv[i]) + (q.glv_ext ? q.glv_ext[i] : 0.f);
  }
}

cudaError_t reduce(const F32WPlan& p, const F32WJob* d_jobs, int n, int taps, float* gw, float* gb, const float* slots,
                   cudaStream_t st) {
  const int nWw = p.co * taps * p.ci, nW = nWw + p.co;
  wgrad_f32_reduce<<<(nW + 31) / 32, dim3(32, 8), 0, st>>>(slots, d_jobs, n, p.slot, nW, nWw, gw, gb);
  return cudaGetLastError();
}

template <int KIND, int COL, int CGN, int IGN, int NB>
cudaError_t run_wgrad(const F32WJob* d_jobs, const F32WPlan& p, const F32WRange& r, float* gw, float* gb,
                      float* slots, cudaStream_t st) {
  using G = WG<KIND, COL, CGN, IGN, NB>;
  auto kern = wgrad_f32_kernel<KIND, COL, CGN, IGN, NB>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::SMEM);
  if (e != cudaSuccess) return e;
  kern<<<dim3(r.units, (p.co / G::BCO) * ((p.ci + G::BCI - 1) / G::BCI)), G::NT, G::SMEM, st>>>(d_jobs, r.n, p.co, p.ci,
                                                                                             p.slot, slots);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  return reduce(p, d_jobs, r.n, WK<KIND>::KR * WK<KIND>::KC, gw, gb, slots, st);
}

// Channel blocks by the layer's widths: as many output channels as fit a warp's lanes, then input
// channels up to 12 warps a block.
template <int KIND>
cudaError_t wgrad_by_width(const F32WJob* d_jobs, const F32WPlan& p, const F32WRange& r, float* gw, float* gb,
                           float* slots, cudaStream_t st) {
  if (p.co % 64 == 0) {
    if (p.ci > 32) return run_wgrad<KIND, 8, 8, 4, 4>(d_jobs, p, r, gw, gb, slots, st);
    return run_wgrad<KIND, 8, 8, 4, 2>(d_jobs, p, r, gw, gb, slots, st);
  }
  if (p.co % 32 == 0) {
    if (p.ci > 32) return run_wgrad<KIND, 8, 4, 8, 2>(d_jobs, p, r, gw, gb, slots, st);
    if (p.ci > 16) return run_wgrad<KIND, 8, 4, 8, 1>(d_jobs, p, r, gw, gb, slots, st);
    return run_wgrad<KIND, 4, 8, 4, 1>(d_jobs, p, r, gw, gb, slots, st);
  }
  if (p.ci > 32) return run_wgrad<KIND, 4, 4, 8, 2>(d_jobs, p, r, gw, gb, slots, st);
  return run_wgrad<KIND, 4, 4, 8, 1>(d_jobs, p, r, gw, gb, slots, st);
}

}  // namespace

F32WPlan f32_wgrad_plan(int kind, int co, int ci, std::vector<F32WJob>& jobs, size_t slot_budget) {
  F32WPlan p;
  p.kind = kind;
  p.co = co;
  p.ci = ci;
  const int taps = kind == FK_P1 ? 1 : 9;
  // chains of a pair (part of the summation order: a change moves the gradient's last bits)
  const bool few = co * taps * ci + co <= 512 && (co < 16 || ci < 16);
  const int most = few ? 608 : 304;
  p.slot = ((size_t)taps * co * ci + co + 31) / 32 * 32;
  size_t total = 0;
  for (F32WJob& j : jobs) {
    const int tiles = ((j.Wo + kTC - 1) / kTC) * ((j.Ho + kTR - 1) / kTR);
    j.units = std::min(tiles, most);
    total += j.units;
  }
  // ranges of about equal work, so that no small one is left over
  const size_t cap = std::max<size_t>(1, slot_budget / p.slot), parts = (total + cap - 1) / cap,
               share = (total + parts - 1) / std::max<size_t>(1, parts);
  for (int i = 0; i < (int)jobs.size(); ++i) {
    const size_t u = p.ranges.empty() ? 0 : p.ranges.back().units;
    if (p.ranges.empty() || u >= share || u + jobs[i].units > cap) p.ranges.push_back({i, 0, 0});
    F32WRange& r = p.ranges.back();
    jobs[i].unit0 = r.units;
    r.units += jobs[i].units;
    ++r.n;
    p.slot_floats = std::max(p.slot_floats, p.slot * r.units);
  }
  return p;
}

cudaError_t launch_f32_wgrad(const F32WPlan& p, const F32WJob* d_jobs, float* gw, float* gb, float* slots,
                             cudaStream_t st) {
  for (const F32WRange& r : p.ranges) {
    cudaError_t e = cudaErrorInvalidValue;
    switch (p.kind) {
      case FK_S2: e = wgrad_by_width<FK_S2>(d_jobs + r.i0, p, r, gw, gb, slots, st); break;
      case FK_P1: e = wgrad_by_width<FK_P1>(d_jobs + r.i0, p, r, gw, gb, slots, st); break;
      case FK_UP2: e = wgrad_by_width<FK_UP2>(d_jobs + r.i0, p, r, gw, gb, slots, st); break;
    }
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_f32_final_dgrad(const F32Img* imgs, int n, int maxH, int maxW, const float* w, int C,
                                   cudaStream_t st) {
  const int NC = kFbThreads / (C / 4);
  const int tx = (maxW + NC - 1) / NC, ty = (maxH + kFbRows - 1) / kFbRows;
  f32_final_dgrad_kernel<<<dim3(tx * ty, 1, n), kFbThreads, sizeof(float) * (kFbRows + 2) * (NC + 2), st>>>(imgs, w, C,
                                                                                                          tx);
  return cudaGetLastError();
}

cudaError_t launch_f32_edge_wgrad(const F32WPlan& p, const F32Img* imgs, const F32WJob* d_jobs, float* gw, float* gb,
                                  float* slots, cudaStream_t st) {
  for (const F32WRange& r : p.ranges) {
    const F32Img* im = imgs + r.i0;
    const F32WJob* j = d_jobs + r.i0;
    if (p.kind == FK_WENC1) {
      const bool two = 3 * p.co / 4 <= 16;
      const int per = kEwWarps * (two ? 2 : 1);
      (two ? f32_enc1_wgrad_kernel<2> : f32_enc1_wgrad_kernel<1>)<<<(r.units + per - 1) / per, 32 * kEwWarps, 0, st>>>(
          im, j, r.n, r.units, p.co, p.slot, slots);
    } else {
      const int lanes = 3 * p.ci / 4,  // of a chain (C <= 256: at most 192)
                threads = std::max(lanes, 128), per = threads / lanes;
      f32_final_wgrad_kernel<<<(r.units + per - 1) / per, threads, 0, st>>>(im, j, r.n, r.units, p.ci, lanes, p.slot,
                                                                            slots);
    }
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = reduce(p, j, r.n, 9, gw, gb, slots, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_f32_latent_bwd(const F32Lat* lat, int n, size_t max_n, cudaStream_t st) {
  if (n == 0 || max_n == 0) return cudaSuccess;
  const unsigned gx = (unsigned)std::min<size_t>(256, (max_n + 255) / 256);
  f32_latent_bwd_kernel<<<dim3(gx, n), 256, 0, st>>>(lat);
  return cudaGetLastError();
}

}  // namespace sv
