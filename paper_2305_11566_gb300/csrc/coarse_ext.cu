// coarse_ext.cu -- variants of the coarse stage (Sec. III-A and the robustness study of
// Sec. IV-C): a matching cost, an aggregation, winner-take-all and post-processing, for
// every pair of a call.
//
//   cost volume C [h][w][D]
//     ZNCC     1 - rho of Eq. 1-3, written by the coarse matcher itself (zncc_wta.cu): the cost
//              alone where an aggregation follows, beside its own winner-take-all where not;
//     census   box4 (4 x 4 box sums of L and R), census_codes (kc x kc census bit strings of
//              the box sums, clamped windows), census_cost (Hamming distance of the codes of
//              (x, y) and (x - d, y); kc^2 - 1 where x - d < 0)
//   aggregation A [h][w][D]
//     SGM      sgm_axis: Eq. 4 along both directions of one axis per launch, 8 or 16 lanes per
//              path line, each holding V consecutive disparities, so that the d - 1 and d + 1 terms are
//              registers but for one shuffle each way; the directions add into A in order
//              (Eq. 5, deterministic); the last one also takes the winner-take-all of the sum
//              (Eq. 6).  The pairs of a call go through cost and paths in parts of bounded
//              volume
//     DT       dt_weights (the edge weights of an iteration), dt_rows / dt_cols: the recursive
//              domain-transform filter on every disparity slice, guided by the left box sums, one
//              thread per (row, d) or (column, d)
//   wta        Eq. 6 on a volume: 8 or 16 lanes per pixel, argmin over d, lowest d on ties
//   smp        single-matching-phase check (Eq. 7, read as uniqueness of the target column),
//              one block per row; median3: 3 x 3 median filter, one thread per pixel
#include "sv_ctx.cuh"

namespace sv {

namespace {

struct XPair {
  const uint8_t* L;
  const uint8_t* R;
  int pitch, w, h, D;
  int32_t* SL;      // [h][w] box sums of L
  int32_t* SR;      // [h][w] box sums of R
  uint64_t* CL;     // [h][w] census codes of L
  uint64_t* CR;     // [h][w] census codes of R
  float* C;         // [h][w][D] cost
  float* A;         // [h][w][D] aggregated cost
  float* WX;        // [h][w] DT weight between (x - 1, y) and (x, y)
  float* WY;        // [h][w] DT weight between (x, y - 1) and (x, y)
  int16_t* wta;     // [h][w] winner-take-all map
  int16_t* mid;     // [h][w] after the occlusion check, when the median filter follows
  int16_t* disp;    // [h][w] result
};

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

// Order-preserving float -> int key (finite values): smaller float, smaller key.
__device__ __forceinline__ int fkey(float f) {
  int i = __float_as_int(f + 0.0f);
  return i >= 0 ? i : (i ^ 0x7FFFFFFF);
}

__global__ void box4_kernel(const XPair* __restrict__ P) {
  const XPair& p = P[blockIdx.z];
  const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
  if (y >= p.h || x >= p.w) return;
  int32_t sl = 0, sr = 0;
  for (int j = 0; j < 4; ++j) {
    const unsigned a = *reinterpret_cast<const unsigned*>(p.L + (size_t)(4 * y + j) * p.pitch + 4 * x);
    const unsigned b = *reinterpret_cast<const unsigned*>(p.R + (size_t)(4 * y + j) * p.pitch + 4 * x);
    sl += (a & 0xFF) + ((a >> 8) & 0xFF) + ((a >> 16) & 0xFF) + (a >> 24);
    sr += (b & 0xFF) + ((b >> 8) & 0xFF) + ((b >> 16) & 0xFF) + (b >> 24);
  }
  p.SL[(size_t)y * p.w + x] = sl;
  p.SR[(size_t)y * p.w + x] = sr;
}

// Census bit strings: bit b (window offsets in raster order, the centre skipped) is set
// where the neighbour's box sum is below the centre's.
template <int RC>
__global__ void census_codes_kernel(const XPair* __restrict__ P) {
  const XPair& p = P[blockIdx.z];
  const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
  if (y >= p.h || x >= p.w) return;
  const int w = p.w, h = p.h;
  const int32_t cl = p.SL[(size_t)y * w + x], cr = p.SR[(size_t)y * w + x];
  uint64_t ml = 0, mr = 0;
  int bit = 0;
#pragma unroll
  for (int j = -RC; j <= RC; ++j) {
    const size_t row = (size_t)clampi(y + j, 0, h - 1) * w;
#pragma unroll
    for (int i = -RC; i <= RC; ++i) {
      if (i == 0 && j == 0) continue;
      const int xx = clampi(x + i, 0, w - 1);
      if (p.SL[row + xx] < cl) ml |= 1ull << bit;
      if (p.SR[row + xx] < cr) mr |= 1ull << bit;
      ++bit;
    }
  }
  p.CL[(size_t)y * w + x] = ml;
  p.CR[(size_t)y * w + x] = mr;
}

// One block per row or piece of `piece` pixels of one: its left codes and the right ones it reaches in shared
// memory, 8, 16 or 32 lanes (as D asks for) per pixel with the lanes over d, so that neighbouring stores are
// contiguous.  Bound by writing the volume.  Calls of few rows cut them into pieces, and no pixel waits for
// a load of its own: with whole rows, a warp a pixel and its left code from memory, a call on one 640 x 128
// pair, D = 64, waited for, took 51 us instead of 42, four of 1242 x 375, D = 8, 72 instead of 59.
__global__ void __launch_bounds__(256) census_cost_kernel(const XPair* __restrict__ P, int kc2m1, int piece) {
  extern __shared__ uint64_t code_sm[];  // [piece] left, then right from x0 - (D - 1) on
  const XPair& p = P[blockIdx.y];
  const int y = blockIdx.x, w = p.w, D = p.D, x0 = blockIdx.z * piece, x1 = min(w, x0 + piece);
  if (y >= p.h || x0 >= w) return;
  const int base = max(0, x0 - (D - 1));
  uint64_t* cr = code_sm + piece;
  for (int x = base + threadIdx.x; x < x1; x += blockDim.x) {
    cr[x - base] = p.CR[(size_t)y * w + x];
    if (x >= x0) code_sm[x - x0] = p.CL[(size_t)y * w + x];
  }
  __syncthreads();
  const int shift = D <= 8 ? 3 : D <= 16 ? 4 : 5, lane = threadIdx.x & ((1 << shift) - 1);
  for (int x = x0 + (threadIdx.x >> shift); x < x1; x += blockDim.x >> shift) {
    const uint64_t cl = code_sm[x - x0];
    float* c = p.C + ((size_t)y * w + x) * D;
    for (int d = lane; d < D; d += 1 << shift)
      c[d] = x - d >= 0 ? (float)__popcll(cl ^ cr[x - d - base]) : (float)kc2m1;
  }
}

// V consecutive values of a line's pixel from d0 on, INF beyond D (or 0: PAD0).  VEC: pairs of floats
// (D even and 8-byte aligned volumes).
template <int V, bool VEC, bool PAD0>
__device__ __forceinline__ void load_d(const float* p, int d0, int D, float (&v)[V]) {
  const float pad = PAD0 ? 0.f : __int_as_float(0x7f800000);
  if constexpr (VEC) {
#pragma unroll
    for (int k = 0; k < V; k += 2) {
      float2 f = make_float2(pad, pad);
      if (d0 + k < D) f = *reinterpret_cast<const float2*>(p + d0 + k);
      v[k] = f.x;
      v[k + 1] = f.y;
    }
  } else {
#pragma unroll
    for (int k = 0; k < V; ++k) v[k] = d0 + k < D ? p[d0 + k] : pad;
  }
}

// Lowest d among the smallest values over the LG lanes of a group, in every lane.
template <int V, int LG>
__device__ __forceinline__ int group_argmin(const float (&v)[V], int d0, int D) {
  int key = INT_MAX, bd = 0x7FFFFFFF;
#pragma unroll
  for (int k = 0; k < V; ++k) {
    const int kk = d0 + k < D ? fkey(v[k]) : INT_MAX;
    if (kk < key) { key = kk; bd = d0 + k; }
  }
#pragma unroll
  for (int o = 1; o < LG; o <<= 1) {
    const int ok = __shfl_xor_sync(0xffffffffu, key, o), od = __shfl_xor_sync(0xffffffffu, bd, o);
    if (ok < key || (ok == key && od < bd)) { key = ok; bd = od; }
  }
  return bd;
}

// One direction of Eq. 4 along a line of `len` pixels, `step` floats (and qstep pixels) apart, from pixel
// q0 on.  FIRST: A = L, else A += L.  The costs and sums of the next PF pixels are loaded ahead.
template <int V, int LG, bool VEC, bool FIRST>
__device__ __forceinline__ void sgm_line(const XPair& p, int q0, int qstep, int len, int l, bool active, bool last,
                                         bool keep, float P1, float P2) {
  constexpr int PF = 8;
  const unsigned FULL = 0xffffffffu;
  const float INF = __int_as_float(0x7f800000);
  const int D = p.D, d0 = l * V;
  const float* C = p.C;
  float* A = p.A;
  const ptrdiff_t step = (ptrdiff_t)qstep * D;
  ptrdiff_t o = (ptrdiff_t)q0 * D;
  float c[PF][V], a[PF][V];
  auto fetch = [&](int slot, int s) {
    if (s >= len) return;
    load_d<V, VEC, false>(C + o + slot * step, d0, D, c[slot]);
    if constexpr (!FIRST) load_d<V, VEC, true>(A + o + slot * step, d0, D, a[slot]);
  };
#pragma unroll
  for (int j = 0; j < PF; ++j) fetch(j, j);
  float prev[V], m = 0.f;
#pragma unroll 1
  for (int s0 = 0; s0 < len; s0 += PF) {
#pragma unroll
    for (int j = 0; j < PF; ++j) {
      const int s = s0 + j;
      if (s >= len) break;
      float cur[V];
      if (s == 0) {
#pragma unroll
        for (int k = 0; k < V; ++k) cur[k] = c[j][k];
      } else {
        float lo = __shfl_up_sync(FULL, prev[V - 1], 1, LG), hi = __shfl_down_sync(FULL, prev[0], 1, LG);
        if (l == 0) lo = INF;
        if (l == LG - 1) hi = INF;
        const float mp = m + P2;
#pragma unroll
        for (int k = 0; k < V; ++k) {
          float best = fminf(prev[k], fminf(k > 0 ? prev[k - 1] : lo, k + 1 < V ? prev[k + 1] : hi) + P1);
          best = fminf(best, mp);
          cur[k] = c[j][k] + (best - m);
        }
      }
      float mn = cur[0];
#pragma unroll
      for (int k = 1; k < V; ++k) mn = fminf(mn, cur[k]);
#pragma unroll
      for (int x = 1; x < LG; x <<= 1) mn = fminf(mn, __shfl_xor_sync(FULL, mn, x));
      m = mn;
      float tot[V];
#pragma unroll
      for (int k = 0; k < V; ++k) {
        prev[k] = cur[k];
        tot[k] = FIRST ? cur[k] : a[j][k] + cur[k];
      }
      float* out = A + o + j * step;
      if (active && (keep || !last)) {
        if constexpr (VEC) {
#pragma unroll
          for (int k = 0; k < V; k += 2)
            if (d0 + k < D) *reinterpret_cast<float2*>(out + d0 + k) = make_float2(tot[k], tot[k + 1]);
        } else {
#pragma unroll
          for (int k = 0; k < V; ++k)
            if (d0 + k < D) out[d0 + k] = tot[k];
        }
      }
      if (last) {
        const int bd = group_argmin<V, LG>(tot, d0, D);
        if (active && l == 0) p.wta[q0 + s * qstep] = (int16_t)bd;
      }
      // the slot's next pixel, PF ahead
      if (s + PF < len) {
        load_d<V, VEC, false>(C + o + (j + PF) * step, d0, D, c[j]);
        if constexpr (!FIRST) load_d<V, VEC, true>(A + o + (j + PF) * step, d0, D, a[j]);
      }
    }
    o += PF * step;
  }
}

// Eq. 4 along rows (axis 0: left to right, then right to left) or columns (axis 1: top to bottom, then
// bottom to top), LG lanes per line and 32 / LG lines per warp; ndir: 1 or both directions.  first: the
// axis's first direction writes A, every other adds; last: the axis's last direction also takes the
// winner-take-all into wta; keep: it stores A too (else only the map).  A lane's values of the
// second direction are the ones it stored in the first.  (One warp per line with the lanes over d
// spent 10 shuffles on a line's minimum and used 48 of 64 lane slots at D = 48.)  Four paths of 64
// pairs of 1242 x 375, D = 48: 1294 -> 577 us; reading and writing the volumes once per direction takes
// 470 us at the measured 6.8 TB/s.
template <int V, int LG, bool VEC>
__global__ void __launch_bounds__(128) sgm_axis_kernel(const XPair* __restrict__ P, int axis, int ndir, int first,
                                                       int last, int keep, float P1, float P2) {
  const XPair& p = P[blockIdx.y];
  const int w = p.w, h = p.h, nlines = axis == 0 ? h : w, len = axis == 0 ? w : h;
  constexpr int NL = 32 / LG;
  const int base = (blockIdx.x * 4 + (threadIdx.x >> 5)) * NL;
  if (base >= nlines) return;  // whole warp
  const int l = threadIdx.x % LG, line0 = base + threadIdx.x / LG % NL;
  const bool active = line0 < nlines;
  const int line = min(line0, nlines - 1);
  const int qstep = axis == 0 ? 1 : w, q0 = axis == 0 ? line * w : line;
  const bool one = ndir == 1;
  if (first)
    sgm_line<V, LG, VEC, true>(p, q0, qstep, len, l, active, last && one, keep, P1, P2);
  else
    sgm_line<V, LG, VEC, false>(p, q0, qstep, len, l, active, last && one, keep, P1, P2);
  if (!one) sgm_line<V, LG, VEC, false>(p, q0 + (len - 1) * qstep, -qstep, len, l, active, last, keep, P1, P2);
}

// The weights of one DT iteration, once for all disparities: a^t between a pixel and its left / upper
// neighbour.
__global__ void dt_weights_kernel(const XPair* __restrict__ P, float lna, float ratio) {
  const XPair& p = P[blockIdx.z];
  const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
  if (y >= p.h || x >= p.w) return;
  const size_t q = (size_t)y * p.w + x;
  const int32_t g = p.SL[q];
  if (x > 0) p.WX[q] = expf(lna * (1.0f + ratio * fabsf((float)(g - p.SL[q - 1]) * 0.0625f)));
  if (y > 0) p.WY[q] = expf(lna * (1.0f + ratio * fabsf((float)(g - p.SL[q - p.w]) * 0.0625f)));
}

// (Two iterations on 16 pairs of 1242 x 375, D = 48, census: rows and columns 430 -> 223 us with the weights
// computed once instead of per disparity and the loads running ahead.)
// J[n] = c[n] + wt[n] (J[n - 1] - c[n]) for n = 1 .. len - 1, written to dst; src, dst and wt advance by
// `step`, `step` and `wstep` per n (wt points at the weight of n = 1).  The loads of the next U
// elements are out while the current U go through the recurrence.
__device__ __forceinline__ void dt_line(const float* src, float* dst, ptrdiff_t step, const float* wt, ptrdiff_t wstep,
                                        int len, float J) {
  constexpr int U = 8;
  float c[2][U], k[2][U];
  auto fetch = [&](int b, int n0) {
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (n0 + u < len) {
        c[b][u] = src[(n0 + u) * step];
        k[b][u] = wt[(n0 + u - 1) * wstep];
      }
  };
  fetch(0, 1);
#pragma unroll 1
  for (int n0 = 1; n0 < len; n0 += 2 * U) {
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int n1 = n0 + b * U;
      fetch(b ^ 1, n1 + U);
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (n1 + u < len) {
          J = c[b][u] + k[b][u] * (J - c[b][u]);
          dst[(n1 + u) * step] = J;
        }
    }
  }
}

// One domain-transform pass along rows (both ways) for every (row, d) of a pair; src is
// read once (the first pass reads C), dst written (the aggregated volume).
__global__ void dt_rows_kernel(const XPair* __restrict__ P, int from_cost) {
  const XPair& p = P[blockIdx.y];
  const int w = p.w, h = p.h, D = p.D;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= h * D) return;
  const int y = t / D, d = t - y * D;
  const size_t base = (size_t)y * w * D + d;
  const float* src = (from_cost ? p.C : p.A) + base;
  float* dst = p.A + base;
  const float* wx = p.WX + (size_t)y * w;
  const float J = src[0];
  dst[0] = J;
  dt_line(src, dst, D, wx + 1, 1, w, J);
  float* end = dst + (size_t)(w - 1) * D;
  dt_line(end, end, -(ptrdiff_t)D, wx + w - 1, -1, w, end[0]);
}

// The same along columns, in place on A, one thread per (column, d): consecutive threads
// touch consecutive addresses of a row.
__global__ void dt_cols_kernel(const XPair* __restrict__ P) {
  const XPair& p = P[blockIdx.y];
  const int w = p.w, h = p.h, D = p.D;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= w * D) return;
  const int x = t / D;
  float* A = p.A + t;
  const ptrdiff_t row = (ptrdiff_t)w * D;
  dt_line(A, A, row, p.WY + x + w, w, h, A[0]);
  float* end = A + (size_t)(h - 1) * row;
  dt_line(end, end, -row, p.WY + x + (size_t)(h - 1) * w, -(ptrdiff_t)w, h, end[0]);
}

// Eq. 6 on a volume (vol_sel 0: C, 1: A): LG lanes per pixel, lowest d among the minima.
template <int V, int LG, bool VEC>
__global__ void __launch_bounds__(256) vol_wta_kernel(const XPair* __restrict__ P, int vol_sel) {
  const XPair& p = P[blockIdx.y];
  constexpr int NP = 32 / LG;  // pixels of a warp
  const int D = p.D, npix = p.w * p.h, l = threadIdx.x % LG;
  const float* A = vol_sel ? p.A : p.C;
  const int stride = gridDim.x * 8 * NP;
  for (int q0 = (blockIdx.x * 8 + (threadIdx.x >> 5)) * NP; q0 < npix; q0 += stride) {  // whole warps
    const int q = q0 + threadIdx.x / LG % NP;
    float v[V];
    load_d<V, VEC, false>(A + (size_t)min(q, npix - 1) * D, l * V, D, v);
    const int bd = group_argmin<V, LG>(v, l * V, D);
    if (l == 0 && q < npix) p.wta[q] = (int16_t)bd;
  }
}

// Single-matching-phase check of one row: pixel x keeps its disparity unless a pixel x - k
// (0 < k < D) of the row has the same target column x - disp; the others take the
// disparity of the nearest kept pixel of the row (left first at equal distance).  A row
// without a kept pixel is copied.  in / out: the pair's maps selected by sel_in / sel_out
// (0: wta, 1: mid, 2: disp).
// Disparities in [0, D) put every pixel of one target within D of the others, so the keeper of a target
// is its leftmost pixel: one shared-memory minimum per pixel.  A row with values outside that
// range (maps the caller brings) looks back over its D - 1 neighbours instead.
__global__ void smp_kernel(const XPair* __restrict__ P, int sel_in, int sel_out) {
  extern __shared__ int smp_sm[];
  const XPair& p = P[blockIdx.y];
  const int y = blockIdx.x, w = p.w, D = p.D;
  if (y >= p.h) return;
  const int16_t* in = (sel_in == 0 ? p.wta : sel_in == 1 ? p.mid : p.disp) + (size_t)y * w;
  int16_t* out = (sel_out == 0 ? p.wta : sel_out == 1 ? p.mid : p.disp) + (size_t)y * w;
  int* val = smp_sm;                                               // [w] disparities
  int* own = smp_sm + w;                                           // [w + D] leftmost pixel of target t - D
  unsigned char* ok = reinterpret_cast<unsigned char*>(own + w + D);  // [w] kept
  int odd = 0;
  for (int x = threadIdx.x; x < w + D; x += blockDim.x) own[x] = INT_MAX;
  for (int x = threadIdx.x; x < w; x += blockDim.x) {
    val[x] = in[x];
    odd |= val[x] < 0 || val[x] >= D;
  }
  odd = __syncthreads_or(odd);
  if (!odd) {
    for (int x = threadIdx.x; x < w; x += blockDim.x) atomicMin(&own[x - val[x] + D], x);
    __syncthreads();
  }
  int any = 0;
  for (int x = threadIdx.x; x < w; x += blockDim.x) {
    int keep = 1;
    if (!odd) {
      keep = own[x - val[x] + D] == x;
    } else {
      const int lo = max(0, x - D + 1);
      for (int u = x - 1; u >= lo; --u)
        if (u - val[u] == x - val[x]) { keep = 0; break; }
    }
    ok[x] = (unsigned char)keep;
    any |= keep;
  }
  any = __syncthreads_or(any);
  for (int x = threadIdx.x; x < w; x += blockDim.x) {
    int v = val[x];
    if (!ok[x] && any) {
      for (int dist = 1; dist < w; ++dist) {
        if (x - dist >= 0 && ok[x - dist]) { v = val[x - dist]; break; }
        if (x + dist < w && ok[x + dist]) { v = val[x + dist]; break; }
      }
    }
    out[x] = (int16_t)v;
  }
}

// 3 x 3 median with clamped edges: the 5th smallest of the 9 values (partial selection).
__global__ void median3_kernel(const XPair* __restrict__ P, int sel_in) {
  const XPair& p = P[blockIdx.z];
  const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
  if (y >= p.h || x >= p.w) return;
  const int w = p.w, h = p.h;
  const int16_t* in = sel_in == 0 ? p.wta : p.mid;
  int v[9];
  int n = 0;
#pragma unroll
  for (int j = -1; j <= 1; ++j)
#pragma unroll
    for (int i = -1; i <= 1; ++i) v[n++] = in[(size_t)clampi(y + j, 0, h - 1) * w + clampi(x + i, 0, w - 1)];
#pragma unroll
  for (int a = 0; a < 5; ++a)
#pragma unroll
    for (int b = a + 1; b < 9; ++b) {
      const int lo = min(v[a], v[b]), hi = max(v[a], v[b]);
      v[a] = lo;
      v[b] = hi;
    }
  p.disp[(size_t)y * w + x] = (int16_t)v[4];
}

cudaError_t launch_census_codes(const XPair* T, int kc, int maxw, int maxh, int n, cudaStream_t st) {
  const dim3 g((maxw + 127) / 128, maxh, n);
  switch (kc / 2) {
    case 1: census_codes_kernel<1><<<g, 128, 0, st>>>(T); break;
    case 2: census_codes_kernel<2><<<g, 128, 0, st>>>(T); break;
    case 3: census_codes_kernel<3><<<g, 128, 0, st>>>(T); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// Disparities per lane and lanes per line (or pixel) for the largest range of the call; vec: every pair's
// volumes can be read in pairs of floats.  Ranges above 64 take 16 lanes: 12 or 16 disparities in one of 8
// lanes hold so many registers that too few lines are in flight (four paths, D = 128: one 640 x 128 pair
// 331 us with 8 lanes, 165 with 16; 16 census pairs of 1242 x 375 1038, 669).
template <int V_, int LG_, bool VEC_>
struct Range {
  static constexpr int V = V_, LG = LG_;
  static constexpr bool VEC = VEC_;
};
template <typename F>
cudaError_t by_range(int maxD, bool vec, F&& f) {
#define SV_RANGE(v, lg)               \
  if (maxD <= lg * v) {               \
    if (vec)                          \
      f(Range<v, lg, true>());        \
    else                              \
      f(Range<v, lg, false>());       \
    return cudaGetLastError();        \
  }
  SV_RANGE(2, 8) SV_RANGE(4, 8) SV_RANGE(6, 8) SV_RANGE(8, 8) SV_RANGE(6, 16) SV_RANGE(8, 16)
#undef SV_RANGE
  return cudaErrorInvalidValue;
}

cudaError_t launch_sgm_axis(const XPair* T, int maxD, bool vec, int nlines, int n, int axis, int ndir, int first,
                            int last, int keep, float P1, float P2, cudaStream_t st) {
  return by_range(maxD, vec, [&](auto r) {
    using R = decltype(r);
    constexpr int lines = 4 * 32 / R::LG;  // of a block
    sgm_axis_kernel<R::V, R::LG, R::VEC><<<dim3((nlines + lines - 1) / lines, n), 128, 0, st>>>(
        T, axis, ndir, first, last, keep, P1, P2);
  });
}

cudaError_t launch_vol_wta(const XPair* T, int maxD, bool vec, int n, int maxpix, int vol_sel, cudaStream_t st) {
  return by_range(maxD, vec, [&](auto r) {
    using R = decltype(r);
    constexpr int pixels = 8 * 32 / R::LG;  // of a block
    vol_wta_kernel<R::V, R::LG, R::VEC><<<dim3(std::min(8 * 152, (maxpix + pixels - 1) / pixels), n), 256, 0, st>>>(
        T, vol_sel);
  });
}

// Volume bytes (cost and aggregated) the pairs of one part may hold, which bounds the workspace.  The path
// kernels need the lines of many pairs to cover a step's latency more than they need a part to fit the L2:
// 64 pairs of 1242 x 375 (11 MB each) take 577 us in one part, 733 in two, 932 in four.
constexpr size_t kPartBytes = size_t(1) << 30;

}  // namespace

// Post-processing launches on a prepared table: SMP (wta -> mid or disp), median (wta or
// mid -> disp).  With neither flag nothing runs (the caller wrote disp directly).
sv_status Ctx::post_launch(const void* table, int n, int maxw, int maxh, int post, cudaStream_t st) {
  const XPair* T = (const XPair*)table;
  sv_status s;
  const bool smp = post & SV_POST_SMP, med = post & SV_POST_MEDIAN;
  if (smp) {
    LaunchScope ls(*this, "smp", st);
    const size_t sm = ((size_t)maxw * 2 + kMaxDisp) * sizeof(int) + (maxw + 3) / 4 * sizeof(int);
    if (sm > 48 * 1024 &&
        (s = cuda(cudaFuncSetAttribute(smp_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm),
                  "occlusion check shared memory")))
      return s;
    smp_kernel<<<dim3(maxh, n), 256, sm, st>>>(T, 0, med ? 1 : 2);
    if ((s = cuda(cudaGetLastError(), "occlusion check"))) return s;
  }
  if (med) {
    LaunchScope ls(*this, "median3", st);
    median3_kernel<<<dim3((maxw + 127) / 128, maxh, n), 128, 0, st>>>(T, smp ? 1 : 0);
    if ((s = cuda(cudaGetLastError(), "median filter"))) return s;
  }
  return SV_OK;
}

sv_status Ctx::coarse_ext(const sv_pair* pairs, int n, const sv_coarse_opts& o, int16_t* const* disp,
                          float* const* cost_out, cudaStream_t st) {
  if (n == 0) return SV_OK;
  const bool want_cost = cost_out != nullptr;
  const bool zncc = o.cost == SV_COST_ZNCC;
  const int post = o.post & (SV_POST_SMP | SV_POST_MEDIAN);
  // the plain matcher: its own exact winner-take-all straight into the output (or into the
  // map the post-processing reads)
  const bool plain = zncc && o.aggregation == SV_AGG_NONE;
  int maxw = 0, maxh = 0, maxD = 1;
  size_t nS = 0;
  // parts: the volumes of a part's pairs share the workspace with every other part's
  std::vector<int> part(1, 0);
  size_t nV = 0, nA = 0, pV = 0, pA = 0;
  const bool agg = o.aggregation != SV_AGG_NONE;
  auto own_c = [&](int i) { return !(want_cost && cost_out[i] && !agg); };
  auto own_a = [&](int i) { return agg && !(want_cost && cost_out[i]); };
  for (int i = 0; i < n; ++i) {
    const int w = pairs[i].width / 4, h = pairs[i].height / 4, D = pairs[i].max_disp;
    const size_t vol = plain && !want_cost ? 0 : (size_t)w * h * D;
    maxw = std::max(maxw, w);
    maxh = std::max(maxh, h);
    maxD = std::max(maxD, D);
    nS += (size_t)w * h;
    if (i > part.back() && (pV + pA + 2 * vol) * sizeof(float) > kPartBytes) {
      part.push_back(i);
      pV = pA = 0;
    }
    if (own_c(i)) pV += vol;
    if (own_a(i)) pA += vol;
    nV = std::max(nV, pV);
    nA = std::max(nA, pA);
  }
  part.push_back(n);
  if (plain && !want_cost) nV = 0;
  const bool dt = o.aggregation == SV_AGG_DT;
  const bool need_box = !zncc || dt;
  sv_status s;
  if (need_box && (s = cuda(sgm_s.ensure(2 * nS * sizeof(int32_t)), "alloc box sums"))) return s;
  if (!zncc && (s = cuda(x_codes.ensure(2 * nS * sizeof(uint64_t)), "alloc census codes"))) return s;
  if (dt && (s = cuda(dt_w.ensure(2 * nS * sizeof(float)), "alloc DT weights"))) return s;
  if (nV && (s = cuda(sgm_c.ensure(nV * sizeof(float)), "alloc cost volume"))) return s;
  if (nA && (s = cuda(sgm_a.ensure(nA * sizeof(float)), "alloc aggregated volume"))) return s;
  if ((s = cuda(x_maps.ensure(2 * nS * sizeof(int16_t)), "alloc coarse maps"))) return s;
  if ((s = cuda(sgm_tab.ensure(sizeof(XPair) * n), "alloc pair table"))) return s;
  std::vector<XPair> tab(n);
  size_t oS = 0, oV = 0, oA = 0;
  bool vec = true;
  for (int i = 0, k = 0; i < n; ++i) {
    const int w = pairs[i].width / 4, h = pairs[i].height / 4, D = pairs[i].max_disp;
    if (i == part[k + 1]) {
      ++k;
      oV = oA = 0;
    }
    XPair& q = tab[i];
    q = XPair{};
    q.L = (const uint8_t*)pairs[i].left;
    q.R = (const uint8_t*)pairs[i].right;
    q.pitch = pairs[i].pitch;
    q.w = w;
    q.h = h;
    q.D = D;
    q.SL = need_box ? (int32_t*)sgm_s.p + oS : nullptr;
    q.SR = need_box ? (int32_t*)sgm_s.p + nS + oS : nullptr;
    q.CL = !zncc ? (uint64_t*)x_codes.p + oS : nullptr;
    q.CR = !zncc ? (uint64_t*)x_codes.p + nS + oS : nullptr;
    q.WX = dt ? (float*)dt_w.p + oS : nullptr;
    q.WY = dt ? (float*)dt_w.p + nS + oS : nullptr;
    if (own_c(i)) {
      q.C = nV ? (float*)sgm_c.p + oV : nullptr;
      oV += (size_t)w * h * D;
    } else {
      q.C = cost_out[i];
    }
    if (own_a(i)) {
      q.A = (float*)sgm_a.p + oA;
      oA += (size_t)w * h * D;
    } else {
      q.A = agg ? cost_out[i] : nullptr;
    }
    vec = vec && D % 2 == 0 && (((uintptr_t)q.C | (uintptr_t)q.A) & 7) == 0;
    q.disp = disp[i];
    q.wta = post ? (int16_t*)x_maps.p + oS : disp[i];
    q.mid = (int16_t*)x_maps.p + nS + oS;
    oS += (size_t)w * h;
  }
  if ((s = cuda(cudaMemcpyAsync(sgm_tab.p, tab.data(), sizeof(XPair) * n, cudaMemcpyHostToDevice, st),
                "upload pair table")))
    return s;
  const XPair* T = (const XPair*)sgm_tab.p;

  const bool with_cost = !plain || want_cost;
  ZRun z;
  std::vector<int> job0;  // first job of every pair
  if (zncc) {
    std::vector<int16_t*> wta(n);
    for (int i = 0; i < n; ++i) wta[i] = tab[i].wta;
    coarse_prepare(pairs, n, wta.data(), nullptr, nullptr, z);
    if (with_cost)
      for (int i = 0; i < n; ++i) z.pairs[i].cost = tab[i].C;
    job0.assign(n + 1, (int)z.jobs.size());
    for (int j = (int)z.jobs.size() - 1; j >= 0; --j) job0[z.jobs[j].pair] = j;
    if ((s = cuda(zpairs.ensure(sizeof(ZPair) * n), "alloc pair table"))) return s;
    if ((s = cuda(zjobs.ensure(sizeof(ZJob) * z.jobs.size()), "alloc job table"))) return s;
    if ((s = cuda(cudaMemcpyAsync(zpairs.p, z.pairs.data(), sizeof(ZPair) * n, cudaMemcpyHostToDevice, st),
                  "upload pairs")))
      return s;
    if ((s = cuda(cudaMemcpyAsync(zjobs.p, z.jobs.data(), sizeof(ZJob) * z.jobs.size(), cudaMemcpyHostToDevice, st),
                  "upload jobs")))
      return s;
  }
  if (need_box) {
    LaunchScope ls(*this, "box4", st);
    box4_kernel<<<dim3((maxw + 127) / 128, maxh, n), 128, 0, st>>>(T);
    if ((s = cuda(cudaGetLastError(), "box sums"))) return s;
  }
  if (!zncc) {
    LaunchScope ls(*this, "census_codes", st);
    if ((s = cuda(launch_census_codes(T, o.census_window, maxw, maxh, n, st), "census codes"))) return s;
  }
  for (size_t k = 0; k + 1 < part.size(); ++k) {
    const int i0 = part[k], m = part[k + 1] - i0;
    // ---- cost volume (and, for the plain matcher, its winner-take-all)
    if (zncc) {
      LaunchScope ls(*this, with_cost ? "zncc_cost" : "zncc_wta", st);
      if ((s = cuda(launch_zncc_wta((const ZPair*)zpairs.p, (const ZJob*)zjobs.p + job0[i0], job0[i0 + m] - job0[i0],
                                    cfg.window / 2, z.maxD, st, !with_cost ? 0 : agg ? 3 : 2, z.shape.small),
                    "zncc cost")))
        return s;
    } else {
      LaunchScope ls(*this, "census_cost", st);
      // pieces of 32 to 2048 pixels (34 KB of codes), as many as four blocks for every SM ask for
      const int want = std::max(1, 4 * 152 / (maxh * m)),
                piece = std::min(2048, std::max(32, (maxw + want - 1) / want));
      const size_t sm = (size_t)(piece + std::min(maxw, piece + maxD - 1)) * sizeof(uint64_t);
      census_cost_kernel<<<dim3(maxh, m, (maxw + piece - 1) / piece), 256, sm, st>>>(
          T + i0, o.census_window * o.census_window - 1, piece);
      if ((s = cuda(cudaGetLastError(), "census cost"))) return s;
    }

    // ---- aggregation and winner-take-all
    if (o.aggregation == SV_AGG_SGM) {
      for (int axis = 0; 2 * axis < o.npaths; ++axis) {
        LaunchScope ls(*this, "sgm_path", st);
        const int ndir = std::min(2, o.npaths - 2 * axis);
        if ((s = cuda(launch_sgm_axis(T + i0, maxD, vec, axis == 0 ? maxh : maxw, m, axis, ndir, axis == 0,
                                      2 * axis + ndir == o.npaths, want_cost ? 1 : 0, o.P1, o.P2, st),
                      "SGM path")))
          return s;
      }
    } else if (dt) {
      const double N = o.dt_iters;
      const float ratio = (float)((double)o.dt_sigma_s / (double)o.dt_sigma_r);
      for (int it = 1; it <= o.dt_iters; ++it) {
        const double sig = o.dt_sigma_s * std::sqrt(3.0) * std::pow(2.0, N - it) / std::sqrt(std::pow(4.0, N) - 1.0);
        const float lna = (float)(-std::sqrt(2.0) / sig);
        {
          LaunchScope ls(*this, "dt_weights", st);
          dt_weights_kernel<<<dim3((maxw + 127) / 128, maxh, m), 128, 0, st>>>(T + i0, lna, ratio);
          if ((s = cuda(cudaGetLastError(), "DT weights"))) return s;
        }
        {
          LaunchScope ls(*this, "dt_rows", st);
          dt_rows_kernel<<<dim3((maxh * maxD + 127) / 128, m), 128, 0, st>>>(T + i0, it == 1);
          if ((s = cuda(cudaGetLastError(), "DT rows"))) return s;
        }
        LaunchScope ls(*this, "dt_cols", st);
        dt_cols_kernel<<<dim3((maxw * maxD + 127) / 128, m), 128, 0, st>>>(T + i0);
        if ((s = cuda(cudaGetLastError(), "DT columns"))) return s;
      }
      LaunchScope ls(*this, "vol_wta", st);
      if ((s = cuda(launch_vol_wta(T + i0, maxD, vec, m, maxw * maxh, 1, st), "winner-take-all"))) return s;
    } else if (!zncc) {
      LaunchScope ls(*this, "vol_wta", st);
      if ((s = cuda(launch_vol_wta(T + i0, maxD, vec, m, maxw * maxh, 0, st), "winner-take-all"))) return s;
    }
  }

  // ---- post-processing
  return post_launch(T, n, maxw, maxh, post, st);
}

sv_status Ctx::postprocess(const sv_pair* pairs, int n, const int16_t* const* in, int post, int16_t* const* out,
                           cudaStream_t st) {
  if (n == 0) return SV_OK;
  int maxw = 0, maxh = 0;
  size_t nS = 0;
  for (int i = 0; i < n; ++i) {
    maxw = std::max(maxw, pairs[i].width / 4);
    maxh = std::max(maxh, pairs[i].height / 4);
    nS += (size_t)(pairs[i].width / 4) * (pairs[i].height / 4);
  }
  sv_status s;
  if (!(post & (SV_POST_SMP | SV_POST_MEDIAN))) {
    for (int i = 0; i < n; ++i)
      if ((s = cuda(cudaMemcpyAsync(out[i], in[i], sizeof(int16_t) * (pairs[i].width / 4) * (pairs[i].height / 4),
                                    cudaMemcpyDeviceToDevice, st),
                    "copy map")))
        return s;
    return SV_OK;
  }
  if ((s = cuda(x_maps.ensure(2 * nS * sizeof(int16_t)), "alloc coarse maps"))) return s;
  if ((s = cuda(sgm_tab.ensure(sizeof(XPair) * n), "alloc pair table"))) return s;
  std::vector<XPair> tab(n);
  size_t oS = 0;
  for (int i = 0; i < n; ++i) {
    XPair& q = tab[i];
    q = XPair{};
    q.w = pairs[i].width / 4;
    q.h = pairs[i].height / 4;
    q.D = pairs[i].max_disp;
    q.wta = const_cast<int16_t*>(in[i]);  // only read
    q.mid = (int16_t*)x_maps.p + nS + oS;
    q.disp = out[i];
    oS += (size_t)q.w * q.h;
  }
  if ((s = cuda(cudaMemcpyAsync(sgm_tab.p, tab.data(), sizeof(XPair) * n, cudaMemcpyHostToDevice, st),
                "upload pair table")))
    return s;
  return post_launch(sgm_tab.p, n, maxw, maxh, post, st);
}

sv_status Ctx::pipeline_ex(const sv_pair* pairs, int n, const sv_coarse_opts& o, float* const* out, cudaStream_t st) {
  std::vector<size_t> off(n + 1, 0);
  for (int i = 0; i < n; ++i) off[i + 1] = off[i] + (size_t)(pairs[i].width / 4) * (pairs[i].height / 4);
  sv_status s = cuda(coarse_maps.ensure(std::max<size_t>(1, off[n]) * sizeof(int16_t)), "alloc coarse maps");
  if (s) return s;
  std::vector<int16_t*> maps(n);
  for (int i = 0; i < n; ++i) maps[i] = (int16_t*)coarse_maps.p + off[i];
  if ((s = coarse_ext(pairs, n, o, maps.data(), nullptr, st))) return s;
  std::vector<const int16_t*> cm(maps.begin(), maps.end());
  return refine_infer(pairs, cm.data(), n, out, st);
}

}  // namespace sv

namespace {

sv_status check_opts(sv::Ctx* c, const sv_coarse_opts* o) {
  if (!o) return c->fail(SV_ERR_INVALID_ARG, "opts is NULL");
  if (o->cost != SV_COST_ZNCC && o->cost != SV_COST_CENSUS) return c->fail(SV_ERR_INVALID_ARG, "unknown cost %d", o->cost);
  if (o->cost == SV_COST_CENSUS && o->census_window != 3 && o->census_window != 5 && o->census_window != 7)
    return c->fail(SV_ERR_INVALID_ARG, "census_window must be 3, 5 or 7");
  if (o->aggregation == SV_AGG_SGM) {
    if (!(o->P1 >= 0.f) || !(o->P2 >= 0.f)) return c->fail(SV_ERR_INVALID_ARG, "penalties must be >= 0");
    if (o->npaths < 1 || o->npaths > 4) return c->fail(SV_ERR_INVALID_ARG, "npaths must be 1..4");
  } else if (o->aggregation == SV_AGG_DT) {
    if (!(o->dt_sigma_s > 0.f) || !(o->dt_sigma_r > 0.f)) return c->fail(SV_ERR_INVALID_ARG, "DT scales must be > 0");
    if (o->dt_iters < 1 || o->dt_iters > 8) return c->fail(SV_ERR_INVALID_ARG, "dt_iters must be 1..8");
  } else if (o->aggregation != SV_AGG_NONE) {
    return c->fail(SV_ERR_INVALID_ARG, "unknown aggregation %d", o->aggregation);
  }
  if (o->post & ~(SV_POST_SMP | SV_POST_MEDIAN)) return c->fail(SV_ERR_INVALID_ARG, "unknown post-processing flag");
  return SV_OK;
}

sv_status check_outputs(sv::Ctx* c, int n, void* const* out, const char* what) {
  if (n == 0) return SV_OK;
  if (!out) return c->fail(SV_ERR_INVALID_ARG, "%s is NULL", what);
  for (int i = 0; i < n; ++i)
    if (!out[i]) return c->fail(SV_ERR_INVALID_ARG, "%s[%d] is NULL", what, i);
  return SV_OK;
}

}  // namespace

extern "C" sv_status sv_coarse_match_ex(sv_ctx* ctx, const sv_pair* pairs, int n_pairs, const sv_coarse_opts* opts,
                                        int16_t* const* disp_out, float* const* cost_out, sv_stream stream) {
  if (!ctx) return SV_ERR_INVALID_ARG;
  sv::Ctx* c = reinterpret_cast<sv::Ctx*>(ctx);
  c->err.clear();
  sv_status s = c->check_pairs(pairs, n_pairs);
  if (s) return s;
  if ((s = check_opts(c, opts))) return s;
  if ((s = check_outputs(c, n_pairs, (void* const*)disp_out, "disp_out"))) return s;
  if (n_pairs == 0) return SV_OK;
  sv::DeviceGuardInt g(c->device);
  return c->coarse_ext(pairs, n_pairs, *opts, disp_out, cost_out, (cudaStream_t)stream);
}

extern "C" sv_status sv_coarse_match_sgm(sv_ctx* ctx, const sv_pair* pairs, int n_pairs, float P1, float P2, int npaths,
                                         int16_t* const* disp_out, float* const* cost_out, sv_stream stream) {
  sv_coarse_opts o{};
  o.cost = SV_COST_ZNCC;
  o.aggregation = SV_AGG_SGM;
  o.P1 = P1;
  o.P2 = P2;
  o.npaths = npaths;
  return sv_coarse_match_ex(ctx, pairs, n_pairs, &o, disp_out, cost_out, stream);
}

extern "C" sv_status sv_postprocess(sv_ctx* ctx, const sv_pair* pairs, int n_pairs, const int16_t* const* disp_in,
                                    int post, int16_t* const* disp_out, sv_stream stream) {
  if (!ctx) return SV_ERR_INVALID_ARG;
  sv::Ctx* c = reinterpret_cast<sv::Ctx*>(ctx);
  c->err.clear();
  if (n_pairs < 0 || (n_pairs > 0 && !pairs)) return c->fail(SV_ERR_INVALID_ARG, "invalid pair list");
  if (post & ~(SV_POST_SMP | SV_POST_MEDIAN)) return c->fail(SV_ERR_INVALID_ARG, "unknown post-processing flag");
  sv_status s;
  if ((s = check_outputs(c, n_pairs, (void* const*)disp_in, "disp_in"))) return s;
  if ((s = check_outputs(c, n_pairs, (void* const*)disp_out, "disp_out"))) return s;
  for (int i = 0; i < n_pairs; ++i) {
    const sv_pair& p = pairs[i];
    if (p.width < 4 || p.height < 4 || p.width > sv::kMaxSide || p.height > sv::kMaxSide)
      return c->fail(SV_ERR_INVALID_ARG, "pair %d: size %dx%d", i, p.width, p.height);
    if (p.max_disp < 1 || p.max_disp > sv::kMaxDisp || p.max_disp > p.width / 4)
      return c->fail(SV_ERR_INVALID_ARG, "pair %d: max_disp %d", i, p.max_disp);
    const size_t bytes = sizeof(int16_t) * (p.width / 4) * (p.height / 4);
    const char* a = (const char*)disp_in[i];
    const char* b = (const char*)disp_out[i];
    if (a < b + bytes && b < a + bytes) return c->fail(SV_ERR_INVALID_ARG, "pair %d: disp_out overlaps disp_in", i);
  }
  if (n_pairs == 0) return SV_OK;
  sv::DeviceGuardInt g(c->device);
  return c->postprocess(pairs, n_pairs, disp_in, post, disp_out, (cudaStream_t)stream);
}

extern "C" sv_status sv_pipeline_ex(sv_ctx* ctx, const sv_pair* pairs, int n_pairs, const sv_coarse_opts* opts,
                                    float* const* disp_out, sv_stream stream) {
  if (!ctx) return SV_ERR_INVALID_ARG;
  sv::Ctx* c = reinterpret_cast<sv::Ctx*>(ctx);
  c->err.clear();
  sv_status s = c->check_pairs(pairs, n_pairs);
  if (s) return s;
  if ((s = check_opts(c, opts))) return s;
  if ((s = check_outputs(c, n_pairs, (void* const*)disp_out, "disp_out"))) return s;
  if (n_pairs == 0) return SV_OK;
  sv::DeviceGuardInt g(c->device);
  return c->pipeline_ex(pairs, n_pairs, *opts, disp_out, (cudaStream_t)stream);
}
