// wgrad_f32.cu -- weight gradients of the FP32 refinement layers on the CUDA cores, all pairs of
// a call per launch, and the fused backward of the one- and two-channel layers.
//
// dW[co][tap][ci] = sum over output pixels p of g(p, co) x(p S + tap, ci): one GEMM per tap whose
// reduction runs over the pixels.  A warp owns one tap of a block of BCO output x BCI input
// channels (8 x 8 in registers per lane; lanes left over split the pixels), so each staged pixel
// costs a lane 4 vector loads for 64 multiply-adds; the block's warps share the staged g and x of
// 64 pixels (cp.async, two buffers).  (One lane holding every tap of 4 x 2 channels needed
// 10 loads for 72 multiply-adds.)  Nearest-x2 layers run on the folded form: output phase (py, px)
// reads 2x2 input pixels, 16 phase-taps instead of 4 x 9, and the reduction adds each kernel
// element's four phase-taps; the last row / column of an odd output, whose cropped neighbour the
// folded taps would count, goes to extra blocks that take the nine taps one by one.
// Every block writes its sums to its own slot; wgrad_f32_reduce adds the slots in a fixed order
// (no atomics: the same call gives the same bits).  Backward of 16 pairs of 1242 x 375, 16/32/64 net:
// dec3 + dec2 weight gradients 6.8 -> 1.6 ms, final conv's two gradients 2.5 -> 0.27 ms; the whole
// training step (with the input gradients of conv_f32.cu) 31.0 -> 6.7 ms.
#include "conv_f32.cuh"

#include <algorithm>

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

constexpr int kTR = 4, kTC = 16;  // pixels of a tile (input pixels for FK_UP2)

// Warps (= taps, or pixel groups of the 1x1 form), staged pixels of g and x per tile.
template <int KIND> struct WK;
template <> struct WK<FK_S2> { static constexpr int NW = 9, NG = 64, XR = 9, XC = 33; };
template <> struct WK<FK_P1> { static constexpr int NW = 8, NG = 64, XR = 4, XC = 16; };
template <> struct WK<FK_UP2> { static constexpr int NW = 16, NG = 256, XR = 6, XC = 18; };

template <int KIND, int CGN, int IGN>
struct WG {
  using K = WK<KIND>;
  static constexpr int BCO = 8 * CGN, BCI = 8 * IGN, KSP = 32 / (CGN * IGN), NT = 32 * K::NW;
  // FK_UP2's edge tiles stage 64 pixels of g and their nine taps of x
  static constexpr int GF = K::NG * BCO, XF = (KIND == FK_UP2 ? 64 * 9 : K::XR * K::XC) * BCI;
  static constexpr int MAINF = GF + K::XR * K::XC * BCI, EDGEF = 64 * BCO + 64 * 9 * BCI;
  static constexpr int BUF = KIND == FK_UP2 && EDGEF > MAINF ? EDGEF : MAINF;
  static constexpr size_t SMEM = 2 * sizeof(float) * BUF;
};

struct WArgs {
  int n, Co, Ci, n_tiles, n_main, n_btiles, n_edge;  // tiles and blocks of the main and edge parts
  size_t slot, bslot, edge_ofs;  // floats of a main / edge slot; first edge slot
  float* slots;
};

__device__ __forceinline__ int tiles_of(int h, int w) { return ((h + kTR - 1) / kTR) * ((w + kTC - 1) / kTC); }

template <int KIND, int CGN, int IGN>
__global__ void __launch_bounds__(WG<KIND, CGN, IGN>::NT, KIND == FK_UP2 ? 1 : 2)
wgrad_f32_kernel(const F32WJob* __restrict__ jobs, const WArgs A) {
  using G = WG<KIND, CGN, IGN>;
  using K = WK<KIND>;
  constexpr int BCO = G::BCO, BCI = G::BCI, KSP = G::KSP;
  extern __shared__ __align__(16) float wf_sm[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cg = lane % CGN, ig = lane / CGN % IGN, ks = lane / (CGN * IGN);
  const int nci = A.Ci / BCI, co0 = ((int)blockIdx.y / nci) * BCO, ci0 = ((int)blockIdx.y % nci) * BCI;
  const bool edge = KIND == FK_UP2 && (int)blockIdx.x >= A.n_main;
  const int b = edge ? blockIdx.x - A.n_main : blockIdx.x, nb = edge ? A.n_edge : A.n_main;
  const int nt = edge ? A.n_btiles : A.n_tiles;
  const int t0 = (int)((long long)nt * b / nb), t1 = (int)((long long)nt * (b + 1) / nb);
  u64 acc[8][4];
#pragma unroll
  for (int j = 0; j < 8; ++j)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[j][q] = 0ull;
  float4 bacc = make_float4(0.f, 0.f, 0.f, 0.f);  // bias gradient: lane l the channels 4 l .. of g
  const bool want_bias = ci0 == 0;

  int job = 0;  // pair of the tile being staged
  auto stage = [&](int t, int buf) {
    while (job + 1 < A.n && t >= (edge ? jobs[job + 1].btile0 : jobs[job + 1].tile0)) ++job;
    const F32WJob& J = jobs[job];
    float* gs = wf_sm + buf * G::BUF;
    if (!edge) {
      float* xs = gs + G::GF;
      const int Hp = KIND == FK_UP2 ? J.Ho / 2 : J.Ho, Wp = KIND == FK_UP2 ? J.Wo / 2 : J.Wo;  // tiled grid
      const int tx = (Wp + kTC - 1) / kTC, tl = t - J.tile0;
      const int Y0 = tl / tx * kTR, X0 = tl % tx * kTC;
#pragma unroll 4
      for (int e = threadIdx.x; e < K::NG * (BCO / 4); e += G::NT) {
        const int c = e % (BCO / 4), p = e / (BCO / 4);
        int oy, ox;
        bool ok;
        if (KIND == FK_UP2) {  // p = row of 8, column of 32 output pixels
          oy = 2 * Y0 + p / 32;
          ox = 2 * X0 + p % 32;
          ok = oy < 2 * Hp && ox < 2 * Wp;
        } else {
          oy = Y0 + p / kTC;
          ox = X0 + p % kTC;
          ok = oy < Hp && ox < Wp;
        }
        cp16z(gs + p * BCO + 4 * c, ok ? J.g + ((size_t)oy * J.Wo + ox) * A.Co + co0 + 4 * c : J.g, ok);
      }
      const int iy0 = KIND == FK_S2 ? 2 * Y0 - 1 : KIND == FK_UP2 ? Y0 - 1 : Y0;
      const int ix0 = KIND == FK_S2 ? 2 * X0 - 1 : KIND == FK_UP2 ? X0 - 1 : X0;
#pragma unroll 4
      for (int e = threadIdx.x; e < K::XR * K::XC * (BCI / 4); e += G::NT) {
        const int c = e % (BCI / 4), p = e / (BCI / 4), r = p / K::XC, q = p - r * K::XC;
        const int iy = iy0 + r, ix = ix0 + q;
        const bool ok = iy >= 0 && ix >= 0 && iy < J.Hi && ix < J.Wi;
        cp16z(xs + p * BCI + 4 * c, ok ? J.x + ((size_t)iy * J.Wi + ix) * A.Ci + ci0 + 4 * c : J.x, ok);
      }
    } else if constexpr (KIND == FK_UP2) {
      // edge pixels in order: the last row when Ho is odd, then the last column above it
      float* xs = gs + 64 * BCO;
      const int nrow = J.Ho & 1 ? J.Wo : 0, ncol = J.Wo & 1 ? J.Ho - (J.Ho & 1) : 0;
      const int p0 = (t - J.btile0) * 64;
      for (int e = threadIdx.x; e < 64 * (BCO / 4); e += G::NT) {
        const int c = e % (BCO / 4), q = e / (BCO / 4), p = p0 + q;
        const bool ok = p < nrow + ncol;
        const int oy = p < nrow ? J.Ho - 1 : p - nrow, ox = p < nrow ? p : J.Wo - 1;
        cp16z(gs + q * BCO + 4 * c, ok ? J.g + ((size_t)oy * J.Wo + ox) * A.Co + co0 + 4 * c : J.g, ok);
      }
      for (int e = threadIdx.x; e < 64 * 9 * (BCI / 4); e += G::NT) {
        const int c = e % (BCI / 4), m = e / (BCI / 4), q = m / 9, tp = m - 9 * q, p = p0 + q;
        const int oy = p < nrow ? J.Ho - 1 : p - nrow, ox = p < nrow ? p : J.Wo - 1;
        const int vy = oy + tp / 3 - 1, vx = ox + tp % 3 - 1;
        const bool ok = p < nrow + ncol && vy >= 0 && vx >= 0 && vy < J.Ho && vx < J.Wo;
        cp16z(xs + m * BCI + 4 * c, ok ? J.x + ((size_t)(vy >> 1) * J.Wi + (vx >> 1)) * A.Ci + ci0 + 4 * c : J.x, ok);
      }
    }
    cp_commit();
  };
  auto madd = [&](const float* g, const float* x) {
    const float4 g0 = *reinterpret_cast<const float4*>(g + cg * 4);
    const float4 g1 = *reinterpret_cast<const float4*>(g + BCO / 2 + cg * 4);
    const ulonglong2 x0 = *reinterpret_cast<const ulonglong2*>(x + ig * 4);
    const ulonglong2 x1 = *reinterpret_cast<const ulonglong2*>(x + BCI / 2 + ig * 4);
    const float gv[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const u64 v = dup2(gv[j]);
      fma2(acc[j][0], v, x0.x);
      fma2(acc[j][1], v, x0.y);
      fma2(acc[j][2], v, x1.x);
      fma2(acc[j][3], v, x1.y);
    }
  };

  if (t0 < t1) stage(t0, 0);
  for (int t = t0; t < t1; ++t) {
    const int buf = (t - t0) & 1;
    if (t + 1 < t1) {
      stage(t + 1, buf ^ 1);
      cp_wait<1>();
    } else {
      cp_wait<0>();
    }
    __syncthreads();
    const float* gs = wf_sm + buf * G::BUF;
    if (!edge) {
      const float* xs = gs + G::GF;
      if constexpr (KIND == FK_S2) {
        const int ky = warp / 3, kx = warp % 3;
        for (int r = 0; r < kTR; ++r) {
          const float* gp = gs + r * kTC * BCO;
          const float* xp = xs + ((2 * r + ky) * K::XC + kx) * BCI;
#pragma unroll 2
          for (int c = ks; c < kTC; c += KSP) madd(gp + c * BCO, xp + 2 * c * BCI);
        }
      } else if constexpr (KIND == FK_P1) {
#pragma unroll 2
        for (int p = warp * 8 + ks; p < warp * 8 + 8; p += KSP) madd(gs + p * BCO, xs + p * BCI);
      } else {
        const int ph = warp >> 2, py = ph >> 1, px = ph & 1, dr = (warp >> 1 & 1) + py, dc = (warp & 1) + px;
        for (int r = 0; r < kTR; ++r) {
          const float* gp = gs + ((2 * r + py) * 32 + px) * BCO;
          const float* xp = xs + ((r + dr) * K::XC + dc) * BCI;
#pragma unroll 2
          for (int c = ks; c < kTC; c += KSP) madd(gp + 2 * c * BCO, xp + c * BCI);
        }
      }
    } else if constexpr (KIND == FK_UP2) {
      if (warp < 9) {
        const float* xs = gs + 64 * BCO;
#pragma unroll 2
        for (int p = ks; p < 64; p += KSP) madd(gs + p * BCO, xs + (p * 9 + warp) * BCI);
      }
    }
    if (want_bias && lane < BCO / 4) {
      const int np = edge ? 64 : K::NG;
      for (int p = warp; p < np; p += K::NW) {
        const float4 g = *reinterpret_cast<const float4*>(gs + p * BCO + 4 * lane);
        bacc.x += g.x;
        bacc.y += g.y;
        bacc.z += g.z;
        bacc.w += g.w;
      }
    }
    __syncthreads();
  }
  // lanes that split the pixels add up
#pragma unroll
  for (int o = CGN * IGN; o < 32; o <<= 1)
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const u64 v = __shfl_xor_sync(0xffffffffu, acc[j][q], o);
        asm("add.rn.f32x2 %0, %0, %1;" : "+l"(acc[j][q]) : "l"(v));
      }
  float* out = A.slots + (edge ? A.edge_ofs + (size_t)b * A.bslot : (size_t)b * A.slot);
  // main FK_UP2 slots: [phase-tap][co][ci]; every other slot in the parameters' order
  const int taps = KIND == FK_P1 ? 1 : KIND == FK_UP2 && !edge ? 16 : 9;
  auto put = [&](int co, int ci, int t, float4 v) {
    const size_t o = KIND == FK_UP2 && !edge ? ((size_t)t * A.Co + co) * A.Ci + ci : ((size_t)co * taps + t) * A.Ci + ci;
    *reinterpret_cast<float4*>(out + o) = v;
  };
  if constexpr (KIND == FK_P1) {  // the warps split the pixels too: add them up in warp order
    for (int w = 1; w < K::NW; ++w) {
      if (warp == w && ks == 0)
#pragma unroll
        for (int j = 0; j < 8; ++j)
#pragma unroll
          for (int q = 0; q < 4; ++q) reinterpret_cast<u64*>(wf_sm)[(j * 4 + q) * (CGN * IGN) + cg + CGN * ig] = acc[j][q];
      __syncthreads();
      if (warp == 0 && ks == 0)
#pragma unroll
        for (int j = 0; j < 8; ++j)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const u64 v = reinterpret_cast<u64*>(wf_sm)[(j * 4 + q) * (CGN * IGN) + cg + CGN * ig];
            asm("add.rn.f32x2 %0, %0, %1;" : "+l"(acc[j][q]) : "l"(v));
          }
      __syncthreads();
    }
  }
  if (ks == 0 && (KIND == FK_P1 ? warp == 0 : !edge || warp < 9)) {
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float2 u = unpack2(acc[j][2 * h]), v = unpack2(acc[j][2 * h + 1]);
        put(co0 + (j >> 2) * (BCO / 2) + cg * 4 + (j & 3), ci0 + h * (BCI / 2) + ig * 4, KIND == FK_P1 ? 0 : warp,
            make_float4(u.x, u.y, v.x, v.y));
      }
  }
  if (want_bias) {
    float4* bs = reinterpret_cast<float4*>(wf_sm);
    __syncthreads();
    if (lane < BCO / 4) bs[warp * (BCO / 4) + lane] = bacc;
    __syncthreads();
    if (threadIdx.x < BCO) {
      float s = 0.f;
      for (int w = 0; w < K::NW; ++w) s += wf_sm[w * BCO + threadIdx.x];
      out[(size_t)taps * A.Co * A.Ci + co0 + threadIdx.x] = s;
    }
  }
}

// gw[e] += the slots' sums (e < nWw), gb[e - nWw] likewise.  A block takes 32 elements; its 8
// rows add every 8th slot, then each other, in a fixed order.  folded: main slots hold the 16
// phase-taps of a nearest-x2 layer.
__global__ void __launch_bounds__(256)
wgrad_f32_reduce(const float* __restrict__ slots, int n_main, size_t slot, int n_edge, size_t bslot, size_t edge_ofs,
                 int nWw, int Co, int Ci, int taps, int folded, float* __restrict__ gw, float* __restrict__ gb) {
  __shared__ float part[8][32];
  const int e = blockIdx.x * 32 + threadIdx.x, y = threadIdx.y;
  const int nW = nWw + Co;
  float s = 0.f;
  if (e < nW) {
    if (folded) {
      size_t o[4];
      int no = 1;
      if (e < nWw) {
        const int ci = e % Ci, t = e / Ci % 9, co = e / (9 * Ci), ky = t / 3, kx = t % 3;
        no = 4;
        for (int ph = 0; ph < 4; ++ph) {
          const int py = ph >> 1, px = ph & 1, r = (ky + 1 - py) >> 1, c = (kx + 1 - px) >> 1;
          o[ph] = ((size_t)(ph * 4 + r * 2 + c) * Co + co) * Ci + ci;
        }
      } else {
        o[0] = (size_t)16 * Co * Ci + (e - nWw);
        o[1] = o[2] = o[3] = o[0];
      }
      for (int b = y; b < n_main; b += 8) {
        const float* p = slots + (size_t)b * slot;
        s += no == 4 ? (p[o[0]] + p[o[1]]) + (p[o[2]] + p[o[3]]) : p[o[0]];
      }
    } else {
#pragma unroll 4
      for (int b = y; b < n_main; b += 8) s += slots[(size_t)b * slot + e];
    }
    for (int b = y; b < n_edge; b += 8) s += slots[edge_ofs + (size_t)b * bslot + e];
  }
  part[y][threadIdx.x] = s;
  __syncthreads();
  if (y == 0 && e < nW) {
    float t = part[0][threadIdx.x];
#pragma unroll
    for (int j = 1; j < 8; ++j) t += part[j][threadIdx.x];
    if (e < nWw)
      gw[e] += t;
    else
      gb[e - nWw] += t;
  }
}

// Backward of the final conv (C channels -> 1): input gradient masked by d3's ReLU, and weight and bias
// gradient, in one pass over d3.  C / 4 lanes hold a pixel's channels; a thread walks down the
// rows of one column with the nine neighbouring output gradients from shared memory.  Bound by
// reading d3 and writing its gradient once.
constexpr int kFbRows = 16, kFbThreads = 256;
__global__ void __launch_bounds__(kFbThreads, 2)
f32_final_bwd_kernel(const F32Img* __restrict__ imgs, int n, const float* __restrict__ w, int C, int tiles_x,
                     int tiles_y, float* __restrict__ slots) {
  extern __shared__ __align__(16) float fb_sm[];
  const int L = C / 4, NC = kFbThreads / L;  // lanes of a pixel, columns of a tile
  const int l = threadIdx.x % L, col = threadIdx.x / L, P = NC + 2;
  const bool on = col < NC;
  float* gs = fb_sm;  // [kFbRows + 2][P]
  float4 k[9], acc[9];
#pragma unroll
  for (int t = 0; t < 9; ++t) {
    k[t] = *reinterpret_cast<const float4*>(w + t * C + 4 * l);
    acc[t] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  float bacc = 0.f;
  const int nt = n * tiles_x * tiles_y;
  for (int t = blockIdx.x; t < nt; t += gridDim.x) {
    const F32Img& I = imgs[t / (tiles_x * tiles_y)];
    const int tl = t % (tiles_x * tiles_y), Y0 = tl / tiles_x * kFbRows, X0 = tl % tiles_x * NC;
    if (Y0 >= I.H || X0 >= I.W) continue;
    __syncthreads();
    for (int e = threadIdx.x; e < (kFbRows + 2) * P; e += kFbThreads) {
      const int r = e / P, c = e - r * P, y = Y0 - 1 + r, x = X0 - 1 + c;
      gs[e] = y >= 0 && x >= 0 && y < I.H && x < I.W ? I.gY[(size_t)y * I.W + x] : 0.f;
    }
    __syncthreads();
    const int x = X0 + col;
    if (!on || x >= I.W) continue;
    const int rows = min(kFbRows, I.H - Y0);
    const size_t base = ((size_t)Y0 * I.W + x) * C + 4 * l, step = (size_t)I.W * C;
#pragma unroll 1
    for (int r0 = 0; r0 < rows; r0 += 4) {
      float4 v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (r0 + j < rows) v[j] = __ldcs(reinterpret_cast<const float4*>(I.d3 + base + (r0 + j) * step));
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (r0 + j >= rows) break;
        const int r = r0 + j;
        float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int ky = 0; ky < 3; ++ky)
#pragma unroll
          for (int kx = 0; kx < 3; ++kx) {
            // output (y + 1 - ky, x + 1 - kx) read this pixel through tap (ky, kx)
            const float g = gs[(r + 2 - ky) * P + col + 2 - kx];
            const int q = ky * 3 + kx;
            d.x = fmaf(g, k[q].x, d.x);
            d.y = fmaf(g, k[q].y, d.y);
            d.z = fmaf(g, k[q].z, d.z);
            d.w = fmaf(g, k[q].w, d.w);
            acc[q].x = fmaf(g, v[j].x, acc[q].x);
            acc[q].y = fmaf(g, v[j].y, acc[q].y);
            acc[q].z = fmaf(g, v[j].z, acc[q].z);
            acc[q].w = fmaf(g, v[j].w, acc[q].w);
            if (q == 4 && l == 0) bacc += g;
          }
        d.x = v[j].x > 0.f ? d.x : 0.f;
        d.y = v[j].y > 0.f ? d.y : 0.f;
        d.z = v[j].z > 0.f ? d.z : 0.f;
        d.w = v[j].w > 0.f ? d.w : 0.f;
        *reinterpret_cast<float4*>(I.gd3 + base + r * step) = d;
      }
    }
  }
  // the columns of a block add up in column order, tap by tap
  float* slot = slots + (size_t)blockIdx.x * (9 * C + 1);
  float4* red = reinterpret_cast<float4*>(fb_sm);
#pragma unroll
  for (int t = 0; t < 9; ++t) {
    __syncthreads();
    if (on) red[threadIdx.x] = acc[t];
    __syncthreads();
    if (threadIdx.x < C) {
      float s = 0.f;
      for (int c = 0; c < NC; ++c) s += fb_sm[c * C + threadIdx.x];
      slot[t * C + threadIdx.x] = s;
    }
  }
  __syncthreads();
  if (on && l == 0) fb_sm[col] = bacc;
  __syncthreads();
  if (threadIdx.x == 0) {
    float s = 0.f;
    for (int c = 0; c < NC; ++c) s += fb_sm[c];
    slot[9 * C] = s;
  }
}

// Weight and bias gradient of enc1 (2 channels -> C, stride 2): the input patch (L / 256,
// U / 256) of a tile is built in shared memory, C / 4 lanes hold a pixel's output gradient and every
// lane sums its 4 output channels x 18 taps.
constexpr int kEwRows = 8, kEwThreads = 256;
__global__ void __launch_bounds__(kEwThreads, 2)
f32_enc1_wgrad_kernel(const F32Img* __restrict__ imgs, int n, int C, int tiles_x, int tiles_y,
                      float* __restrict__ slots) {
  extern __shared__ __align__(16) float ew_sm[];
  const int L = C / 4, NC = kEwThreads / L;
  const int l = threadIdx.x % L, col = threadIdx.x / L, P = 2 * NC + 1;
  const bool on = col < NC;
  float2* xs = reinterpret_cast<float2*>(ew_sm);  // [2 kEwRows + 1][P]
  float4 acc[18], bacc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int t = 0; t < 18; ++t) acc[t] = make_float4(0.f, 0.f, 0.f, 0.f);
  const int nt = n * tiles_x * tiles_y;
  for (int t = blockIdx.x; t < nt; t += gridDim.x) {
    const F32Img& I = imgs[t / (tiles_x * tiles_y)];
    const int tl = t % (tiles_x * tiles_y), Y0 = tl / tiles_x * kEwRows, X0 = tl % tiles_x * NC;
    if (Y0 >= I.H1 || X0 >= I.W1) continue;
    __syncthreads();
    for (int e = threadIdx.x; e < (2 * kEwRows + 1) * P; e += kEwThreads) {
      const int r = e / P, c = e - r * P, vy = 2 * Y0 - 1 + r, vx = 2 * X0 - 1 + c;
      float2 v = make_float2(0.f, 0.f);
      if (vy >= 0 && vx >= 0 && vy < I.H && vx < I.W) {
        v.x = (float)I.L[(size_t)vy * I.pitch + vx] * (1.0f / 256.0f);
        v.y = upsample4_f(I.coarse_f, I.w, I.h, vx, vy) * (1.0f / 256.0f);
      }
      xs[e] = v;
    }
    __syncthreads();
    const int x = X0 + col;
    if (!on || x >= I.W1) continue;
    const int rows = min(kEwRows, I.H1 - Y0);
    const float* g0 = I.ge1 + ((size_t)Y0 * I.W1 + x) * C + 4 * l;
#pragma unroll 2
    for (int r = 0; r < rows; ++r) {
      const float4 g = *reinterpret_cast<const float4*>(g0 + (size_t)r * I.W1 * C);
      bacc.x += g.x;
      bacc.y += g.y;
      bacc.z += g.z;
      bacc.w += g.w;
#pragma unroll
      for (int t9 = 0; t9 < 9; ++t9) {
        const float2 v = xs[(2 * r + t9 / 3) * P + 2 * col + t9 % 3];
        float4 &a = acc[2 * t9], &c = acc[2 * t9 + 1];
        a.x = fmaf(g.x, v.x, a.x);
        a.y = fmaf(g.y, v.x, a.y);
        a.z = fmaf(g.z, v.x, a.z);
        a.w = fmaf(g.w, v.x, a.w);
        c.x = fmaf(g.x, v.y, c.x);
        c.y = fmaf(g.y, v.y, c.y);
        c.z = fmaf(g.z, v.y, c.z);
        c.w = fmaf(g.w, v.y, c.w);
      }
    }
  }
  float* slot = slots + (size_t)blockIdx.x * (19 * C);
  float4* red = reinterpret_cast<float4*>(ew_sm);
#pragma unroll
  for (int t = 0; t < 19; ++t) {
    __syncthreads();
    if (on) red[threadIdx.x] = t < 18 ? acc[t < 18 ? t : 0] : bacc;
    __syncthreads();
    if (threadIdx.x < C) {
      float s = 0.f;
      for (int c = 0; c < NC; ++c) s += ew_sm[c * C + threadIdx.x];
      if (t < 18)
        slot[(size_t)threadIdx.x * 18 + t] = s;
      else
        slot[(size_t)18 * C + threadIdx.x] = s;
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

template <int KIND, int CGN, int IGN>
cudaError_t run_wgrad(const F32WJob* d_jobs, const F32WPlan& p, int n, float* gw, float* gb, float* slots,
                      cudaStream_t st) {
  using G = WG<KIND, CGN, IGN>;
  WArgs a{n, p.co, p.ci, p.n_tiles, p.n_main, p.n_btiles, p.n_edge, p.slot, p.bslot, p.edge_ofs, slots};
  auto kern = wgrad_f32_kernel<KIND, CGN, IGN>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::SMEM);
  if (e != cudaSuccess) return e;
  kern<<<dim3(p.n_main + p.n_edge, (p.co / G::BCO) * (p.ci / G::BCI)), G::NT, G::SMEM, st>>>(d_jobs, a);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const int taps = KIND == FK_P1 ? 1 : 9, nWw = p.co * taps * p.ci;
  wgrad_f32_reduce<<<(nWw + p.co + 31) / 32, dim3(32, 8), 0, st>>>(slots, p.n_main, p.slot, p.n_edge, p.bslot,
                                                                   p.edge_ofs, nWw, p.co, p.ci, taps,
                                                                   KIND == FK_UP2 ? 1 : 0, gw, gb);
  return cudaGetLastError();
}

template <int KIND>
cudaError_t wgrad_by_width(const F32WJob* d_jobs, const F32WPlan& p, int n, float* gw, float* gb, float* slots,
                           cudaStream_t st) {
  const int cgn = p.cgn, ign = p.ign;
  if (cgn == 8 && ign == 4) return run_wgrad<KIND, 8, 4>(d_jobs, p, n, gw, gb, slots, st);
  if (cgn == 8 && ign == 2) return run_wgrad<KIND, 8, 2>(d_jobs, p, n, gw, gb, slots, st);
  if (cgn == 4 && ign == 4) return run_wgrad<KIND, 4, 4>(d_jobs, p, n, gw, gb, slots, st);
  if (cgn == 4 && ign == 2) return run_wgrad<KIND, 4, 2>(d_jobs, p, n, gw, gb, slots, st);
  if (cgn == 2 && ign == 4) return run_wgrad<KIND, 2, 4>(d_jobs, p, n, gw, gb, slots, st);
  return run_wgrad<KIND, 2, 2>(d_jobs, p, n, gw, gb, slots, st);
}

}  // namespace

// Blocks: about one wave of the GPU over all channel blocks (each block walks its share of the
// tiles, so more blocks only add slots to write and read); the edge tiles, which cost what a main
// tile costs, get their share of them.
F32WPlan f32_wgrad_plan(int kind, int co, int ci, std::vector<F32WJob>& jobs) {
  F32WPlan p;
  p.kind = kind;
  p.co = co;
  p.ci = ci;
  p.cgn = co % 64 == 0 ? 8 : co % 32 == 0 ? 4 : 2;
  p.ign = ci % 32 == 0 ? 4 : 2;
  long long tiles = 0, btiles = 0;
  for (F32WJob& j : jobs) {
    j.tile0 = (int)tiles;
    j.btile0 = (int)btiles;
    const int h = kind == FK_UP2 ? j.Ho / 2 : j.Ho, w = kind == FK_UP2 ? j.Wo / 2 : j.Wo;
    tiles += (long long)((h + kTR - 1) / kTR) * ((w + kTC - 1) / kTC);
    if (kind == FK_UP2) btiles += ((j.Ho & 1 ? j.Wo : 0) + (j.Wo & 1 ? j.Ho - (j.Ho & 1) : 0) + 63) / 64;
  }
  p.n_tiles = (int)tiles;
  p.n_btiles = (int)btiles;
  const int blocks = (co / (8 * p.cgn)) * (ci / (8 * p.ign)), per_sm = kind == FK_UP2 ? 1 : 2;
  const int want = std::max(1, 152 * per_sm / blocks);
  if (btiles > 0)
    p.n_edge = (int)std::min<long long>(btiles, std::max<long long>(1, (want * btiles + tiles) / (tiles + btiles)));
  p.n_main = (int)std::max<long long>(1, std::min<long long>(tiles, std::max(1, want - p.n_edge)));
  const int taps = kind == FK_P1 ? 1 : 9;
  p.slot = ((size_t)(kind == FK_UP2 ? 16 : taps) * co * ci + co + 31) / 32 * 32;
  p.bslot = ((size_t)9 * co * ci + co + 31) / 32 * 32;
  p.edge_ofs = p.slot * p.n_main;
  p.slot_floats = p.edge_ofs + (p.n_edge ? p.bslot * p.n_edge : 0);
  return p;
}

cudaError_t launch_f32_wgrad(const F32WPlan& p, const F32WJob* d_jobs, int n, float* gw, float* gb, float* slots,
                             cudaStream_t st) {
  switch (p.kind) {
    case FK_S2: return wgrad_by_width<FK_S2>(d_jobs, p, n, gw, gb, slots, st);
    case FK_P1: return wgrad_by_width<FK_P1>(d_jobs, p, n, gw, gb, slots, st);
    case FK_UP2: return wgrad_by_width<FK_UP2>(d_jobs, p, n, gw, gb, slots, st);
  }
  return cudaErrorInvalidValue;
}

size_t f32_edge_slot_floats(int C) { return (size_t)2 * 152 * std::max(9 * C + 1, 19 * C); }

cudaError_t launch_f32_final_bwd(const F32Img* imgs, int n, int maxH, int maxW, const float* w, int C, float* gw,
                                 float* gb, float* slots, cudaStream_t st) {
  const int NC = kFbThreads / (C / 4);
  const int tx = (maxW + NC - 1) / NC, ty = (maxH + kFbRows - 1) / kFbRows;
  const int grid = (int)std::min<long long>((long long)tx * ty * n, 2 * 152);
  const size_t smem = std::max(sizeof(float) * (kFbRows + 2) * (NC + 2), sizeof(float4) * kFbThreads);
  f32_final_bwd_kernel<<<grid, kFbThreads, smem, st>>>(imgs, n, w, C, tx, ty, slots);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  wgrad_f32_reduce<<<(9 * C + 1 + 31) / 32, dim3(32, 8), 0, st>>>(slots, grid, 9 * C + 1, 0, 0, 0, 9 * C, 1, C, 9, 0, gw,
                                                                  gb);
  return cudaGetLastError();
}

cudaError_t launch_f32_enc1_wgrad(const F32Img* imgs, int n, int maxH1, int maxW1, int C, float* gw, float* gb,
                                  float* slots, cudaStream_t st) {
  const int NC = kEwThreads / (C / 4);
  const int tx = (maxW1 + NC - 1) / NC, ty = (maxH1 + kEwRows - 1) / kEwRows;
  const int grid = (int)std::min<long long>((long long)tx * ty * n, 2 * 152);
  const size_t smem = std::max(sizeof(float2) * (2 * kEwRows + 1) * (2 * NC + 1), sizeof(float4) * kEwThreads);
  f32_enc1_wgrad_kernel<<<grid, kEwThreads, smem, st>>>(imgs, n, C, tx, ty, slots);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  wgrad_f32_reduce<<<(19 * C + 31) / 32, dim3(32, 8), 0, st>>>(slots, grid, 19 * C, 0, 0, 0, 18 * C, C, 2, 9, 0, gw, gb);
  return cudaGetLastError();
}

cudaError_t launch_f32_latent_bwd(const F32Lat* lat, int n, size_t max_n, cudaStream_t st) {
  if (n == 0 || max_n == 0) return cudaSuccess;
  const unsigned gx = (unsigned)std::min<size_t>(256, (max_n + 255) / 256);
  f32_latent_bwd_kernel<<<dim3(gx, n), 256, 0, st>>>(lat);
  return cudaGetLastError();
}

}  // namespace sv
