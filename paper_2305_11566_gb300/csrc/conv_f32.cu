// conv_f32.cu -- FP32 convolutions of the refinement networks on the CUDA cores, all pairs of a
// call per launch: the plain form's layers, their input gradients and the Table I network's
// 5x5 layers (kinds in conv_f32.cuh).
//
// A block of 128 threads computes TH x TW positions of one output phase x 8 CG output channels;
// a thread holds 8 consecutive positions x 8 channels in registers.  The input patch is staged
// channel-planar (CIC channels a step) and the packed weights as [tap][channel][output], both by
// cp.async into two buffers, with one barrier a step (two cost the Table I net 1.3 %).  Per channel and window row a thread reads its row segment once
// and reuses it for the TX taps: 64 TX multiply-adds for 2 TX + 3 vector loads, so the FMA pipe and
// not shared memory bounds the kernel (one output channel group per thread and one position
// needed 9 loads for 32 multiply-adds).  The multiply-adds are issued as packed pairs.  8 pairs of
// 1242 x 375, 32/64/128 net: 22.1 -> 3.8 ms (dec2 at 51, dec1 at 45 TFLOP/s of 80 on the FP32 pipes).
//
// Nearest-x2 layers run as four output phases of 2x2 taps (2.25x fewer multiply-adds than the
// 3x3 window on the upsampled grid).  Where an odd size crops the last upsampled row or column, the
// summed weights hold one kernel row or column too many there: tiles that touch that edge run the
// unsummed 3x3 taps with the cropped taps left out.
#include "conv_f32.cuh"

#include <algorithm>
#include <type_traits>

#include "sv_internal.cuh"

namespace sv {

namespace {

constexpr int kThreads = 128;
constexpr int PX = 8;  // positions per thread, along x (FK_DUP2 launches that leave SMs idle take 4)

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
__device__ __forceinline__ void cp4(float* dst, const float* src, bool ok) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(dst);
  const int n = ok ? 4 : 0;
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(s), "l"(src), "r"(n));
}
__device__ __forceinline__ void cp16z(float* dst, const float* src, bool ok) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(dst);
  const int n = ok ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(s), "l"(src), "r"(n));
}
__device__ __forceinline__ void cp16(float* dst, const float* src) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(src));
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N)); }

// Window and stepping of a kind: largest window, input stride, phases, taps of the edge form.
template <int KIND> struct Kind;
template <> struct Kind<FK_S2> { static constexpr int TY = 3, TX = 3, S = 2, PH = 1, BT = 0; };
template <> struct Kind<FK_P1> { static constexpr int TY = 1, TX = 1, S = 1, PH = 1, BT = 0; };
template <> struct Kind<FK_UP2> { static constexpr int TY = 2, TX = 2, S = 1, PH = 4, BT = 9; };
template <> struct Kind<FK_DS2> { static constexpr int TY = 2, TX = 2, S = 1, PH = 4, BT = 0; };
template <> struct Kind<FK_DUP2> { static constexpr int TY = 3, TX = 3, S = 2, PH = 1, BT = 0; };
template <> struct Kind<FK_S1_5> { static constexpr int TY = 5, TX = 5, S = 1, PH = 1, BT = 0; };
template <> struct Kind<FK_S2_5> { static constexpr int TY = 5, TX = 5, S = 2, PH = 1, BT = 0; };
template <> struct Kind<FK_DE5> { static constexpr int TY = 3, TX = 3, S = 1, PH = 4, BT = 0; };
template <> struct Kind<FK_UP2X> { static constexpr int TY = 3, TX = 3, S = 1, PH = 1, BT = 0; };

// Channels staged per step: kinds with a large stride-2 patch stage fewer.
constexpr int kind_cic(int kind) { return kind == FK_P1 ? 16 : kind == FK_S1_5 || kind == FK_S2_5 ? 4 : 8; }

constexpr int imax(int a, int b) { return a > b ? a : b; }

template <int KIND, int CG_, int CIC_, int PX_ = 8>
struct Geo {
  using K = Kind<KIND>;
  static constexpr int CG = CG_, CIC = CIC_, BN = 8 * CG, S = K::S, PX = PX_;
  static constexpr int TW = CG >= 4 ? 16 : 32, GX = TW / PX, TH = kThreads / CG / GX;
  static constexpr int PR = (TH - 1) * S + K::TY, PC = (TW - 1) * S + K::TX;
  static constexpr int NV = ((PX - 1) * S + K::TX + 3) / 4;  // float4 loads of a thread's row segment
  static constexpr int PITCH = imax((PC + 3) / 4 * 4, (TW - PX) * S + 4 * NV);
  // planes 4 banks apart (mod 32): the transposing copies of a pixel's channels do not collide
  static constexpr int PLANE = (PR * PITCH + 31 - 4) / 32 * 32 + 4;
  static constexpr int WT = imax(K::TY * K::TX, K::BT) * CIC * BN;
  static constexpr int BUF = CIC * PLANE + WT, NBUF = 2;
  static constexpr size_t SMEM = NBUF * sizeof(float) * BUF;
  static constexpr bool SPLIT = false;  // columns split by parity
  static constexpr int EVEN = 0;
};

// FK_S2: the patch's even and odd columns are staged apart (a tap's stride-2 reads of 8 positions
// are then consecutive), in one buffer: the 8 channels of a step and their weights take 38 KB, and
// four blocks share an SM.
template <int CG_, int CIC_, int PX_>
struct Geo<FK_S2, CG_, CIC_, PX_> {
  static constexpr int CG = CG_, CIC = CIC_, BN = 8 * CG, S = 2, PX = PX_;
  static constexpr int TW = CG >= 4 ? 16 : 32, GX = TW / PX, TH = kThreads / CG / GX;
  static constexpr int PR = 2 * TH + 1, PC = 2 * TW + 1;
  // row: odd columns 2x - 1 (TW + 1 of them, to a multiple of 4, + 4 read past the last), then even
  static constexpr int EVEN = TW + 4, PITCH = EVEN + TW;
  static constexpr int PLANE = (PR * PITCH + 31 - 4) / 32 * 32 + 4;
  static constexpr int BUF = CIC * PLANE + 9 * CIC * BN, NBUF = 1;
  static constexpr size_t SMEM = sizeof(float) * BUF;
  static constexpr bool SPLIT = true;
};

// FK_DUP2: columns 2x - 1 .. 2x + 2 of the upsampled grid, split by parity, in one buffer.
template <int CG_, int CIC_, int PX_>
struct Geo<FK_DUP2, CG_, CIC_, PX_> {
  static constexpr int CG = CG_, CIC = CIC_, BN = 8 * CG, S = 2, PX = PX_;
  static constexpr int TW = CG >= 4 ? 16 : 32, GX = TW / PX, TH = kThreads / CG / GX;
  static constexpr int PR = 2 * TH + 2, PC = 2 * TW + 2;
  static constexpr int EVEN = TW + 4, PITCH = 2 * EVEN;
  static constexpr int PLANE = (PR * PITCH + 31 - 4) / 32 * 32 + 4;
  static constexpr int BUF = CIC * PLANE + 9 * CIC * BN, NBUF = 1;
  static constexpr size_t SMEM = sizeof(float) * BUF;
  static constexpr bool SPLIT = true;
};

// FK_UP2X: the patch holds the input pixels under the tile, (TH / 2 + 2) x (TW / 2 + 2); column 0 sits
// at offset 3, so that a thread's four input pixels are one aligned vector.
template <int CG_, int CIC_, int PX_>
struct Geo<FK_UP2X, CG_, CIC_, PX_> {
  static constexpr int CG = CG_, CIC = CIC_, BN = 8 * CG, S = 1, PX = PX_;
  static constexpr int TW = CG >= 4 ? 16 : 32, GX = TW / PX, TH = kThreads / CG / GX;
  static constexpr int PR = TH / 2 + 2, PC = TW / 2 + 2, PITCH = TW / 2 + 8;
  static constexpr int PLANE = (PR * PITCH + 31 - 4) / 32 * 32 + 4;
  static constexpr int BUF = CIC * PLANE + 9 * CIC * BN, NBUF = 2;
  static constexpr size_t SMEM = NBUF * sizeof(float) * BUF;
  static constexpr bool SPLIT = false;
  static constexpr int EVEN = 0;
};

struct F32Args {
  const float* packed;
  size_t w[4], wb;
  const float* bias;
  int K, N, nb, tiles_x, act;
  int accumulate;  // 1: added to the output
  int bias_first;  // 1: the sum starts at the bias (else the bias is added to it)
};

// The patch rows iy0 .. of one channel chunk, channel-planar; zero outside the input.
template <class G, int PR, int PC>
__device__ __forceinline__ void load_patch(float* dst, const float* src, int C, int iy0, int ix0, int Hi, int Wi) {
  constexpr int SL = kThreads / G::CIC, CW = SL < 32 ? SL : 32, RG = SL / CW;
  const int t = threadIdx.x, ci = t % G::CIC, cc = (t / G::CIC) % CW, rg = t / (G::CIC * CW);
  const ptrdiff_t step = (ptrdiff_t)RG * Wi * C;
  for (int c = cc; c < PC; c += CW) {
    const int ix = ix0 + c;
    const bool cok = (unsigned)ix < (unsigned)Wi;
    ptrdiff_t o = ((ptrdiff_t)(iy0 + rg) * Wi + ix) * C + ci;
    const int cd = G::SPLIT ? (c & 1 ? G::EVEN : 0) + (c >> 1) : c;  // (patch column 0 is odd)
    float* d = dst + ci * G::PLANE + rg * G::PITCH + cd;
#pragma unroll 4
    for (int r = rg; r < PR; r += RG) {
      const bool ok = cok && (unsigned)(iy0 + r) < (unsigned)Hi;
      cp4(d, ok ? src + o : src, ok);
      o += step;
      d += RG * G::PITCH;
    }
  }
}

template <class G, int NV>
__device__ __forceinline__ void load_row(const float* p, float* a) {
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const float4 f = *reinterpret_cast<const float4*>(p + 4 * v);
    a[4 * v] = f.x;
    a[4 * v + 1] = f.y;
    a[4 * v + 2] = f.z;
    a[4 * v + 3] = f.w;
  }
}

// acc[p][..] += a[p S + c] * w: weights of one tap and channel, 4 + 4 outputs of this thread.
template <class G, int OFS>
__device__ __forceinline__ void tap(u64 (&acc)[G::PX][4], const float* a, const float* w) {
  const ulonglong2 w0 = *reinterpret_cast<const ulonglong2*>(w);
  const ulonglong2 w1 = *reinterpret_cast<const ulonglong2*>(w + G::BN / 2);
#pragma unroll
  for (int p = 0; p < G::PX; ++p) {
    const u64 v = dup2(a[p * G::S + OFS]);
    fma2(acc[p][0], v, w0.x);
    fma2(acc[p][1], v, w0.y);
    fma2(acc[p][2], v, w1.x);
    fma2(acc[p][3], v, w1.y);
  }
}
// The same with position `drop` left out (-1: none).
template <class G, int OFS>
__device__ __forceinline__ void tap_but(u64 (&acc)[G::PX][4], const float* a, const float* w, int drop) {
  const ulonglong2 w0 = *reinterpret_cast<const ulonglong2*>(w);
  const ulonglong2 w1 = *reinterpret_cast<const ulonglong2*>(w + G::BN / 2);
#pragma unroll
  for (int p = 0; p < G::PX; ++p) {
    const u64 v = dup2(p == drop ? 0.f : a[p * G::S + OFS]);
    fma2(acc[p][0], v, w0.x);
    fma2(acc[p][1], v, w0.y);
    fma2(acc[p][2], v, w1.x);
    fma2(acc[p][3], v, w1.y);
  }
}

template <class G, int TY, int TX, int C = 0>
__device__ __forceinline__ void taps_of_row(u64 (&acc)[G::PX][4], const float* a, const float* w) {
  if constexpr (C < TX) {
    tap<G, C>(acc, a, w + C * G::CIC * G::BN);
    taps_of_row<G, TY, TX, C + 1>(acc, a, w);
  }
}

// Main form: TY x TX window.
template <class G, int TY, int TX>
struct Window {
  static constexpr int PR = (G::TH - 1) * G::S + TY, PC = (G::TW - 1) * G::S + TX, TAPS = TY * TX;
  __device__ __forceinline__ void operator()(u64 (&acc)[G::PX][4], const float* pa, const float* pw) const {
    constexpr int NV = ((G::PX - 1) * G::S + TX + 3) / 4;
#pragma unroll 1
    for (int ci = 0; ci < G::CIC; ++ci, pa += G::PLANE, pw += G::BN)
#pragma unroll
      for (int r = 0; r < TY; ++r) {
        float a[4 * NV];
        load_row<G, NV>(pa + r * G::PITCH, a);
        taps_of_row<G, TY, TX>(acc, a, pw + r * TX * G::CIC * G::BN);
      }
  }
};

// Edge form of FK_UP2: 3x3 taps of phase (py, px) on the 2x2 patch; kernel row / column 2 of
// an even phase falls on the cropped row / column at the edge.
template <class G>
struct UpEdge {
  static constexpr int PR = G::PR, PC = G::PC, TAPS = 9;
  int py, px, drop;
  bool last_row;
  __device__ __forceinline__ void operator()(u64 (&acc)[G::PX][4], const float* pa, const float* pw) const {
    constexpr int NV = (G::PX + 1 + 3) / 4, WS = G::CIC * G::BN;
#pragma unroll 1
    for (int ci = 0; ci < G::CIC; ++ci, pa += G::PLANE, pw += G::BN)
#pragma unroll 1
      for (int ky = 0; ky < 3; ++ky) {
        if (ky == 2 && last_row) continue;
        float a[4 * NV];
        load_row<G, NV>(pa + ((ky + 1 - py) >> 1) * G::PITCH, a);
        const float* w = pw + ky * 3 * WS;
        tap<G, 0>(acc, a, w);
        if (px == 0)
          tap<G, 1>(acc, a, w + WS);
        else
          tap<G, 0>(acc, a, w + WS);
        tap_but<G, 1>(acc, a, w + 2 * WS, drop);
      }
  }
};

// The training step keeps one summation order, whatever tile computes it: FK_S2 and FK_UP2X kernel
// row, kernel column, channel within a step of 8 channels; FK_DUP2 the four upsampled positions of an
// input pixel, then the same; FK_DS2 the same over the taps a phase has.  A reordered sum flips a few
// ReLUs, after one Adam step (whose update is +-lr for every weight) also through the weights, and
// moves an FP32 gradient by up to 1e-4 of its norm on small batches; in this order the step gives the
// same bits as one thread per pixel does.  So these kinds run the unsummed nine taps (dec2 of 8 pairs of
// 256 x 128: 229 us against 105 us for the summed 2x2 form, which inference uses).
template <class G, int OFS>
__device__ __forceinline__ void tap_unit(u64 (&acc)[G::PX][4], const float* a, const float* w) {
  const ulonglong2 w0 = *reinterpret_cast<const ulonglong2*>(w);
  const ulonglong2 w1 = *reinterpret_cast<const ulonglong2*>(w + G::BN / 2);
#pragma unroll
  for (int p = 0; p < G::PX; ++p) {
    const u64 v = dup2(a[p + OFS]);
    fma2(acc[p][0], v, w0.x);
    fma2(acc[p][1], v, w0.y);
    fma2(acc[p][2], v, w1.x);
    fma2(acc[p][3], v, w1.y);
  }
}
// All channels of a step for one tap; drop: position left out (EDGE tiles).
template <class G, int OFS, bool EDGE = false>
__device__ __forceinline__ void columns(u64 (&acc)[G::PX][4], const float* pa, const float* w, int drop = -1) {
  constexpr int NV = (G::PX + OFS + 3) / 4;
#pragma unroll 2
  for (int ci = 0; ci < G::CIC; ++ci) {
    float a[4 * NV];
    load_row<G, NV>(pa + ci * G::PLANE, a);
    if constexpr (EDGE) {
#pragma unroll
      for (int p = 0; p < G::PX; ++p) a[p + OFS] = p == drop ? 0.f : a[p + OFS];
    }
    tap_unit<G, OFS>(acc, a, w + ci * G::BN);
  }
}

template <class G>
struct OrderedS2 {
  static constexpr int PR = G::PR, PC = G::PC, TAPS = 9;
  __device__ __forceinline__ void operator()(u64 (&acc)[G::PX][4], const float* pa, const float* pw) const {
    constexpr int WS = G::CIC * G::BN;
#pragma unroll 1
    for (int ky = 0; ky < 3; ++ky, pa += G::PITCH, pw += 3 * WS) {
      columns<G, 0>(acc, pa, pw);
      columns<G, 0>(acc, pa + G::EVEN, pw + WS);
      columns<G, 1>(acc, pa, pw + 2 * WS);
    }
  }
};

// FK_DUP2: input pixel (y, x) gathers the upsampled positions (2y + a, 2x + b) through the taps: row
// 2y + a + 1 - ky, column 2x + b + 1 - kx.  The last row's a = 1 and the last column's b = 1 are cropped
// away when the grid is odd.
template <class G, bool EDGE>
struct OrderedDup {
  static constexpr int PR = G::PR, PC = G::PC, TAPS = 9;
  int na, drop;  // na: 1 where a = 1 is cropped
  __device__ __forceinline__ void operator()(u64 (&acc)[G::PX][4], const float* pa, const float* pw) const {
    constexpr int WS = G::CIC * G::BN;
#pragma unroll 1
    for (int a = 0; a < (EDGE ? na : 2); ++a) {
      const float* p = pa + (a + 2) * G::PITCH;
#pragma unroll 1
      for (int ky = 0; ky < 3; ++ky) {
        const float *q = p - ky * G::PITCH, *w = pw + ky * 3 * WS;
        columns<G, 1>(acc, q, w);
        columns<G, 0>(acc, q + G::EVEN, w + WS);
        columns<G, 0>(acc, q, w + 2 * WS);
      }
#pragma unroll 1
      for (int ky = 0; ky < 3; ++ky) {
        const float *q = p - ky * G::PITCH, *w = pw + ky * 3 * WS;
        columns<G, 1, EDGE>(acc, q + G::EVEN, w, drop);
        columns<G, 1, EDGE>(acc, q, w + WS, drop);
        columns<G, 0, EDGE>(acc, q + G::EVEN, w + 2 * WS, drop);
      }
    }
  }
};

// FK_DS2: window taps from the last to the first (kernel rows and columns ascending).
template <class G, int TY, int TX>
struct OrderedDs {
  static constexpr int PR = G::TH - 1 + TY, PC = G::TW - 1 + TX, TAPS = TY * TX;
  __device__ __forceinline__ void operator()(u64 (&acc)[G::PX][4], const float* pa, const float* pw) const {
    constexpr int WS = G::CIC * G::BN;
#pragma unroll
    for (int r = TY - 1; r >= 0; --r) {
      if (TX == 2) columns<G, 1>(acc, pa + r * G::PITCH, pw + (r * TX + 1) * WS);
      columns<G, 0>(acc, pa + r * G::PITCH, pw + r * TX * WS);
    }
  }
};

// FK_UP2X: position p of a thread reads the input pixels (p + kx - 1) >> 1 of its four (and one to
// either side).  vy0: the upsampled row of ky = 0 relative to the patch, rows: kernel rows above
// the crop; drop: position whose kx = 2 falls on the cropped column (-1: none).
template <class G>
struct OrderedUp {
  static constexpr int PR = G::PR, PC = G::PC, TAPS = 9;
  int vy0, rows, drop;
  __device__ __forceinline__ void operator()(u64 (&acc)[G::PX][4], const float* pa, const float* pw) const {
    constexpr int WS = G::CIC * G::BN;
#pragma unroll 1
    for (int ky = 0; ky < rows; ++ky) {
      const float* p = pa + ((vy0 + ky) >> 1) * G::PITCH;
      const float* w = pw + ky * 3 * WS;
#pragma unroll 2
      for (int ci = 0; ci < G::CIC; ++ci) column<0>(acc, p + ci * G::PLANE, w + ci * G::BN);
#pragma unroll 2
      for (int ci = 0; ci < G::CIC; ++ci) column<1>(acc, p + ci * G::PLANE, w + WS + ci * G::BN);
#pragma unroll 2
      for (int ci = 0; ci < G::CIC; ++ci) column<2>(acc, p + ci * G::PLANE, w + 2 * WS + ci * G::BN);
    }
  }
  template <int KX>
  __device__ __forceinline__ void column(u64 (&acc)[G::PX][4], const float* p, const float* w) const {
    const float4 f = *reinterpret_cast<const float4*>(p);
    const ulonglong2 w0 = *reinterpret_cast<const ulonglong2*>(w);
    const ulonglong2 w1 = *reinterpret_cast<const ulonglong2*>(w + G::BN / 2);
    u64 v[5];
    const int o = KX == 0 ? 1 : 0;
    if (KX == 0) v[0] = dup2(p[-1]);
    v[o] = dup2(f.x);
    v[o + 1] = dup2(f.y);
    v[o + 2] = dup2(f.z);
    v[o + 3] = dup2(f.w);
    if (KX == 2) v[4] = dup2(p[4]);
#pragma unroll
    for (int q = 0; q < G::PX; ++q) {
      u64 x = v[KX == 1 ? q >> 1 : (q + 1) >> 1];
      if (KX == 2 && q == drop) x = 0ull;
      fma2(acc[q][0], x, w0.x);
      fma2(acc[q][1], x, w0.y);
      fma2(acc[q][2], x, w1.x);
      fma2(acc[q][3], x, w1.y);
    }
  }
};

// Runs the channel chunks through the staging buffers; pa0: the thread's place in a patch.
template <class G, class Form>
__device__ __forceinline__ void contract(const Form& form, u64 (&acc)[G::PX][4], float* sm, const F32Job& J,
                                         const float* w, int K, int iy0, int ix0, int pa0, int cg) {
  const int nch = K / G::CIC;
  constexpr int WF = Form::TAPS * G::CIC * G::BN;
  constexpr int COL0 = std::is_same<Form, OrderedUp<G>>::value ? 3 : 0;
  int s = 0, c0 = 0;  // source tensor of the chunk being staged, its first channel
  auto stage = [&](int ch) {
    float* b = sm + (ch % G::NBUF) * G::BUF;
    while (ch * G::CIC - c0 >= J.ic[s]) c0 += J.ic[s++];
    load_patch<G, Form::PR, Form::PC>(b + COL0, J.in[s] + (ch * G::CIC - c0), J.ic[s], iy0, ix0, J.Hi, J.Wi);
    const float* ws = w + (size_t)ch * WF;
    float* wd = b + G::CIC * G::PLANE;
#pragma unroll 4
    for (int e = threadIdx.x; e < WF / 4; e += kThreads) cp16(wd + 4 * e, ws + 4 * e);
    cp_commit();
  };
  stage(0);
  for (int ch = 0; ch < nch; ++ch) {
    cp_wait<0>();
    __syncthreads();  // chunk ch is there, and everyone is done with chunk ch - 1: its buffer may be refilled
    if (G::NBUF == 2 && ch + 1 < nch) stage(ch + 1);
    const float* b = sm + (ch % G::NBUF) * G::BUF;
    form(acc, b + pa0, b + G::CIC * G::PLANE + cg * 4);
    if (G::NBUF == 1 && ch + 1 < nch) {
      __syncthreads();
      stage(ch + 1);
    }
  }
}

__device__ __forceinline__ float activate(float v, int act) {
  if (act == 1) return v < 0.f ? 0.f : v;
  if (act == 2) return v < 0.f ? v * 0.1f : v;
  return v;
}

template <int KIND, int CG, int CIC, int PXV>
__global__ void __launch_bounds__(kThreads, 4) f32_conv_kernel(const F32Job* __restrict__ jobs, const F32Args A) {
  using G = Geo<KIND, CG, CIC, PXV>;
  extern __shared__ __align__(16) float f32_sm[];
  constexpr int PH = Kind<KIND>::PH, OS = PH == 4 ? 2 : 1;
  const F32Job& J = jobs[blockIdx.z];
  const int phase = PH == 4 ? blockIdx.y / A.nb : 0, nblk = blockIdx.y - phase * A.nb;
  const int py = phase >> 1, px = phase & 1;
  const int Ho = J.Ho, Wo = J.Wo;
  const int GH = (Ho - py + OS - 1) / OS, GW = (Wo - px + OS - 1) / OS;
  const int Y0 = (blockIdx.x / A.tiles_x) * G::TH, X0 = (blockIdx.x % A.tiles_x) * G::TW;
  if (Y0 >= GH || X0 >= GW) return;
  const int cg = threadIdx.x % CG, pg = threadIdx.x / CG, gx = pg % G::GX, row = pg / G::GX;
  const int y = Y0 + row, xb = X0 + gx * G::PX, n0 = nblk * G::BN + cg * 4;
  u64 acc[G::PX][4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const u64 b = KIND == FK_P1 && A.bias_first
                      ? *reinterpret_cast<const u64*>(A.bias + n0 + (q >> 1) * (G::BN / 2) + 2 * (q & 1))
                      : 0ull;
#pragma unroll
    for (int p = 0; p < G::PX; ++p) acc[p][q] = b;
  }
  const float* wm = A.packed + A.w[phase];
  auto run = [&](auto form, const float* base, int dy, int dx) {
    using Form = decltype(form);
    contract<G>(form, acc, f32_sm, J, base + (size_t)nblk * Form::TAPS * A.K * G::BN, A.K, Y0 * G::S + dy,
                X0 * G::S + dx, row * G::S * G::PITCH + gx * G::PX * (G::SPLIT ? 1 : G::S), cg);
  };
  if constexpr (KIND == FK_S2) {
    run(OrderedS2<G>{}, wm, -1, -1);
  } else if constexpr (KIND == FK_UP2X) {
    const int rows = min(3, Ho - (y - 1));
    const int drop = (Wo & 1) && X0 + G::TW >= GW ? GW - 1 - xb : -1;
    contract<G>(OrderedUp<G>{row + 1, rows, drop}, acc, f32_sm, J, wm + (size_t)nblk * 9 * A.K * G::BN, A.K, Y0 / 2 - 1,
                X0 / 2 - 1, gx * (G::PX / 2) + 4, cg);
  } else if constexpr (KIND == FK_P1) {
    run(Window<G, 1, 1>{}, wm, 0, 0);
  } else if constexpr (KIND == FK_S1_5 || KIND == FK_S2_5) {
    run(Window<G, 5, 5>{}, wm, -2, -2);
  } else if constexpr (KIND == FK_UP2) {
    const bool er = py == 0 && (Ho & 1) && Y0 + G::TH >= GH, ec = px == 0 && (Wo & 1) && X0 + G::TW >= GW;
    if (er || ec)
      run(UpEdge<G>{py, px, ec ? GW - 1 - xb : -1, er && y == GH - 1}, A.packed + A.wb, py - 1, px - 1);
    else
      run(Window<G, 2, 2>{}, wm, py - 1, px - 1);
  } else if constexpr (KIND == FK_DUP2) {
    const bool er = (J.Hi & 1) && Y0 + G::TH >= GH, ec = (J.Wi & 1) && X0 + G::TW >= GW;
    if (er || ec)
      run(OrderedDup<G, true>{er && y == GH - 1 ? 1 : 2, ec ? GW - 1 - xb : -1}, wm, -1, -1);
    else
      run(OrderedDup<G, false>{2, -1}, wm, -1, -1);
  } else if constexpr (KIND == FK_DS2) {
    if (phase == 0) run(OrderedDs<G, 1, 1>{}, wm, 0, 0);
    else if (phase == 1) run(OrderedDs<G, 1, 2>{}, wm, 0, 0);
    else if (phase == 2) run(OrderedDs<G, 2, 1>{}, wm, 0, 0);
    else run(OrderedDs<G, 2, 2>{}, wm, 0, 0);
  } else if constexpr (KIND == FK_DE5) {
    if (phase == 0) run(Window<G, 3, 3>{}, wm, -1, -1);
    else if (phase == 1) run(Window<G, 3, 2>{}, wm, -1, 0);
    else if (phase == 2) run(Window<G, 2, 3>{}, wm, 0, -1);
    else run(Window<G, 2, 2>{}, wm, 0, 0);
  }
  if (y >= GH) return;
  float bs[8];
#pragma unroll
  for (int q = 0; q < 8; ++q)
    bs[q] = A.bias && !(KIND == FK_P1 && A.bias_first) ? A.bias[n0 + (q >> 2) * (G::BN / 2) + (q & 3)] : 0.f;
#pragma unroll
  for (int p = 0; p < G::PX; ++p) {
    const int x = xb + p;
    if (x >= GW) break;
    const size_t o = ((size_t)(y * OS + py) * Wo + x * OS + px) * A.N + n0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float2 u = unpack2(acc[p][2 * h]), v = unpack2(acc[p][2 * h + 1]);
      float4 f = make_float4(activate(u.x + bs[4 * h], A.act), activate(u.y + bs[4 * h + 1], A.act),
                             activate(v.x + bs[4 * h + 2], A.act), activate(v.y + bs[4 * h + 3], A.act));
      const size_t oo = o + h * (G::BN / 2);
      if (J.mask) {
        const float4 m = *reinterpret_cast<const float4*>(J.mask + oo);
        f.x = m.x > 0.f ? f.x : 0.f;
        f.y = m.y > 0.f ? f.y : 0.f;
        f.z = m.z > 0.f ? f.z : 0.f;
        f.w = m.w > 0.f ? f.w : 0.f;
      }
      if (KIND == FK_P1 && A.accumulate) {
        const float4 g = *reinterpret_cast<const float4*>(J.out + oo);
        f = make_float4(g.x + f.x, g.y + f.y, g.z + f.z, g.w + f.w);
      }
      *reinterpret_cast<float4*>(J.out + oo) = f;
    }
  }
}

template <int KIND, int CG, int CIC, int PXV = PX>
cudaError_t run_conv(const F32Layer& l, const F32Job* jobs, int n, int maxHo, int maxWo, const float* packed,
                     const float* bias, int act, cudaStream_t st) {
  using G = Geo<KIND, CG, CIC, PXV>;
  constexpr int PH = Kind<KIND>::PH, OS = PH == 4 ? 2 : 1;
  F32Args a{packed, {l.w[0], l.w[1], l.w[2], l.w[3]}, l.wb, bias, l.K, l.N, l.N / G::BN, 0, act & 3, act & 8 ? 1 : 0, act & 4 ? 1 : 0};
  a.tiles_x = ((maxWo + OS - 1) / OS + G::TW - 1) / G::TW;
  const int tiles_y = ((maxHo + OS - 1) / OS + G::TH - 1) / G::TH;
  const dim3 grid(a.tiles_x * tiles_y, PH * a.nb, n);
  // FK_DUP2 launches of blocks for half the SMs at most: half the positions per thread.  A thread's chain
  // (36 taps x K channels, one after the other) is then all the time there is, and half as long with half
  // the independent sums; larger launches need the 8 positions' reuse of loads.  One pair: 36 x 36,
  // 32/64/128 net, dec1 289 -> 207 us, dec2 141 -> 99; 256 x 128, 16/32/64 net, 138 -> 97 and 78 -> 55.
  if constexpr (KIND == FK_DUP2 && PXV == PX) {
    if (2LL * grid.x * grid.y * grid.z <= 152)
      return run_conv<KIND, CG, CIC, 4>(l, jobs, n, maxHo, maxWo, packed, bias, act, st);
  }
  auto kern = f32_conv_kernel<KIND, CG, CIC, PXV>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::SMEM);
  if (e != cudaSuccess) return e;
  kern<<<grid, kThreads, G::SMEM, st>>>(jobs, a);
  return cudaGetLastError();
}

template <int KIND>
cudaError_t by_width(const F32Layer& l, const F32Job* jobs, int n, int maxHo, int maxWo, const float* packed,
                     const float* bias, int act, cudaStream_t st) {
  constexpr int C = kind_cic(KIND);
  if (l.cg == 8) return run_conv<KIND, 8, C>(l, jobs, n, maxHo, maxWo, packed, bias, act, st);
  if (l.cg == 4) return run_conv<KIND, 4, C>(l, jobs, n, maxHo, maxWo, packed, bias, act, st);
  if (l.cg == 2) return run_conv<KIND, 2, C>(l, jobs, n, maxHo, maxWo, packed, bias, act, st);
  return cudaErrorInvalidValue;
}

// Packed weights: a block per (output channel block, staged channel chunk), each
// [tap][channel][output channel], so that a step's weights are one contiguous copy.
__global__ void f32_pack_kernel(const F32PackDesc* __restrict__ descs, const float* __restrict__ params,
                                float* __restrict__ packed) {
  const F32PackDesc& D = descs[blockIdx.y];
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < D.count; i += (size_t)gridDim.x * blockDim.x) {
    const int n = (int)(i % D.bn), ci = (int)(i / D.bn % D.cic), t = (int)(i / (D.bn * D.cic) % D.taps);
    const int rest = (int)(i / ((size_t)D.bn * D.cic * D.taps)), kc = D.K / D.cic;
    const int chunk = rest % kc, nblk = rest / kc;
    const int k = chunk * D.cic + ci, nn = nblk * D.bn + n;
    const int r = t / D.tx, c = t % D.tx, py = D.phase >> 1, px = D.phase & 1;
    auto W = [&](int o, int ky, int kx, int ii) {
      return params[D.src + (((size_t)o * D.ks + ky) * D.ks + kx) * D.ci + ii];
    };
    float v = 0.f;
    if (D.kind == FK_Y5) {
      // one source of the last layer: output "channel" n is phase (n >> 1, n & 1)
      const int ky = ((n >> 1) ? 3 : 4) - 2 * (r - (n >> 1)), kx = ((n & 1) ? 3 : 4) - 2 * (c - (n & 1));
      if (k < D.co && ky >= 0 && ky <= 4 && kx >= 0 && kx <= 4) v = params[D.src + (ky * 5 + kx) * D.ci + D.N + k];
    } else if (D.kind == FK_UP2 && !D.border) {
      for (int ky = 0; ky < 3; ++ky)
        for (int kx = 0; kx < 3; ++kx)
          if (((ky + 1 - py) >> 1) == r && ((kx + 1 - px) >> 1) == c) v += W(nn, ky, kx, k);
    } else if (D.kind == FK_DUP2) {
      v = W(k, r, c, nn);
    } else if (D.kind == FK_DS2) {
      v = W(k, py ? 2 - 2 * r : 1, px ? 2 - 2 * c : 1, nn);
    } else if (D.kind == FK_DE5) {
      v = W(nn, (py ? 3 : 4) - 2 * r, (px ? 3 : 4) - 2 * c, k);
    } else if (D.kind == FK_P1 && D.phase == 1) {  // gradient of a 1x1: transposed
      v = W(k, 0, 0, nn);
    } else {
      v = W(nn, r, c, k);
    }
    packed[D.dst + i] = v;
  }
}

template <int CG_>
struct Enc1Geo {
  static constexpr int CG = CG_, CIC = 2, BN = 8 * CG, S = 2, PX = 8;
  static constexpr int TW = CG >= 4 ? 16 : 32, GX = TW / PX, TH = kThreads / CG / GX;
  static constexpr int PR = 2 * TH + 1, PC = 2 * TW + 1, PITCH = (TW - PX) * 2 + 20, PLANE = PR * PITCH;
  static constexpr int BUF = 2 * PLANE + 18 * BN;
};

// enc1: the input patch (L / 256, U / 256) is built while staging, U = 4 x bilinear(coarse).
template <int CG>
__global__ void __launch_bounds__(kThreads, 4)
f32_enc1_kernel(const F32Img* __restrict__ imgs, const float* __restrict__ w, const float* __restrict__ b, int C,
                int tiles_x) {
  using G = Enc1Geo<CG>;
  __shared__ __align__(16) float sm[G::BUF];
  const F32Img& I = imgs[blockIdx.z];
  const int Y0 = (blockIdx.x / tiles_x) * G::TH, X0 = (blockIdx.x % tiles_x) * G::TW;
  if (Y0 >= I.H1 || X0 >= I.W1) return;
  for (int e = threadIdx.x; e < G::PR * G::PC; e += kThreads) {
    const int r = e / G::PC, c = e - r * G::PC;
    const int vy = 2 * Y0 - 1 + r, vx = 2 * X0 - 1 + c;
    float l = 0.f, u = 0.f;
    if (vy >= 0 && vx >= 0 && vy < I.H && vx < I.W) {
      l = (float)I.L[(size_t)vy * I.pitch + vx] * (1.0f / 256.0f);
      u = (I.coarse_f ? upsample4_f(I.coarse_f, I.w, I.h, vx, vy) : upsample4_f(I.coarse_i, I.w, I.h, vx, vy)) *
          (1.0f / 256.0f);
    }
    sm[r * G::PITCH + c] = l;
    sm[G::PLANE + r * G::PITCH + c] = u;
  }
  float* ws = sm + 2 * G::PLANE;
  for (int e = threadIdx.x; e < 18 * G::BN; e += kThreads) {
    const int n = e % G::BN, tc = e / G::BN;  // tc = tap * 2 + channel: the source order
    ws[e] = w[(size_t)(blockIdx.y * G::BN + n) * 18 + tc];
  }
  __syncthreads();
  const int cg = threadIdx.x % CG, pg = threadIdx.x / CG, gx = pg % G::GX, row = pg / G::GX;
  u64 acc[PX][4];
#pragma unroll
  for (int p = 0; p < PX; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[p][q] = 0ull;
#pragma unroll
  for (int r = 0; r < 3; ++r) {  // kernel row, column, channel
    float a0[20], a1[20];
    const float* pa = sm + (row * 2 + r) * G::PITCH + gx * PX * 2;
    load_row<G, 5>(pa, a0);
    load_row<G, 5>(pa + G::PLANE, a1);
    const float* wr = ws + cg * 4 + r * 6 * G::BN;
    tap<G, 0>(acc, a0, wr);
    tap<G, 0>(acc, a1, wr + G::BN);
    tap<G, 1>(acc, a0, wr + 2 * G::BN);
    tap<G, 1>(acc, a1, wr + 3 * G::BN);
    tap<G, 2>(acc, a0, wr + 4 * G::BN);
    tap<G, 2>(acc, a1, wr + 5 * G::BN);
  }
  const int y = Y0 + row, n0 = blockIdx.y * G::BN + cg * 4;
  if (y >= I.H1) return;
#pragma unroll
  for (int p = 0; p < PX; ++p) {
    const int x = X0 + gx * PX + p;
    if (x >= I.W1) break;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int nn = n0 + h * (G::BN / 2);
      const float2 u = unpack2(acc[p][2 * h]), v = unpack2(acc[p][2 * h + 1]);
      *reinterpret_cast<float4*>(I.e1 + ((size_t)y * I.W1 + x) * C + nn) =
          make_float4(activate(u.x + b[nn], 1), activate(u.y + b[nn + 1], 1), activate(v.x + b[nn + 2], 1),
                      activate(v.y + b[nn + 3], 1));
    }
  }
}

// final 3x3 conv to one channel + bias + the residual U.  The layer is bound by reading d3 once
// (60 MB a 1242 x 375 pair at 32 channels), so d3 goes straight to registers: LPP lanes hold
// one pixel's channels (4 each, 4 LPP a pass), walk down the rows of a column and keep the three
// kernel rows' sums running; the finished row's three kernel-column sums are added over the lanes
// and left in shared memory, where each output adds its three columns.  44 -> 18 us a 1242 x 375
// pair of 32 channels against a block that staged d3 channel-planar.
constexpr int kFinRows = 16;  // output rows of a block
template <int LPP>
__global__ void __launch_bounds__(256)
f32_final_kernel(const F32Img* __restrict__ imgs, const float* __restrict__ w, const float* __restrict__ b, int C,
                 int tiles_x) {
  constexpr int NC = 256 / LPP, NO = NC - 2;  // staged columns, output columns
  __shared__ float P[kFinRows][NC][3];
  const F32Img& I = imgs[blockIdx.z];
  const int Y0 = (blockIdx.x / tiles_x) * kFinRows, X0 = (blockIdx.x % tiles_x) * NO;
  if (Y0 >= I.H || X0 >= I.W) return;
  const int l = threadIdx.x % LPP, col = threadIdx.x / LPP, x = X0 - 1 + col;
  const bool xok = x >= 0 && x < I.W;
  for (int c0 = 0; c0 < C; c0 += 4 * LPP) {
    float4 k[9];
#pragma unroll
    for (int t = 0; t < 9; ++t) k[t] = *reinterpret_cast<const float4*>(w + t * C + c0 + 4 * l);
    float fin[3] = {0.f, 0.f, 0.f}, mid[3] = {0.f, 0.f, 0.f};
    const float* src = I.d3 + ((ptrdiff_t)(Y0 - 1) * I.W + x) * C + c0 + 4 * l;
    const ptrdiff_t step = (ptrdiff_t)I.W * C;
    constexpr int AHEAD = 6;  // rows loaded before they are used
    static_assert((kFinRows + 2) % AHEAD == 0, "whole groups of rows");
#pragma unroll 1
    for (int r0 = 0; r0 < kFinRows + 2; r0 += AHEAD) {
      float4 v[AHEAD];
#pragma unroll
      for (int j = 0; j < AHEAD; ++j) {
        const int y = Y0 - 1 + r0 + j;
        v[j] = xok && y >= 0 && y < I.H ? __ldcs(reinterpret_cast<const float4*>(src + (r0 + j) * step))
                                        : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int j = 0; j < AHEAD; ++j) {
        const int r = r0 + j;  // input row Y0 - 1 + r completes output row Y0 + r - 2
        float f[3];
#pragma unroll
        for (int kx = 0; kx < 3; ++kx) {
          auto dot = [&](const float4& q, float s) {
            return fmaf(q.w, v[j].w, fmaf(q.z, v[j].z, fmaf(q.y, v[j].y, fmaf(q.x, v[j].x, s))));
          };
          f[kx] = dot(k[6 + kx], fin[kx]);
          fin[kx] = dot(k[3 + kx], mid[kx]);
          mid[kx] = dot(k[kx], 0.f);
        }
        if (r >= 2) {
#pragma unroll
          for (int kx = 0; kx < 3; ++kx) {
#pragma unroll
            for (int o = LPP / 2; o > 0; o >>= 1) f[kx] += __shfl_xor_sync(0xffffffffu, f[kx], o);
            if (l == 0) P[r - 2][col][kx] = c0 == 0 ? f[kx] : P[r - 2][col][kx] + f[kx];
          }
        }
      }
    }
  }
  __syncthreads();
  for (int e = threadIdx.x; e < kFinRows * NO; e += 256) {
    const int r = e / NO, c = e - r * NO, y = Y0 + r, X = X0 + c;
    if (y >= I.H || X >= I.W) continue;
    const float acc = P[r][c][0] + P[r][c + 1][1] + P[r][c + 2][2];
    const float u = I.coarse_f ? upsample4_f(I.coarse_f, I.w, I.h, X, y) : upsample4_f(I.coarse_i, I.w, I.h, X, y);
    I.Y[(size_t)y * I.W + X] = u + (b[0] + acc);
  }
}

// The final conv of the training forward: the same layer summed in the training step's order
// (8 channels a step; kernel row, kernel column, channel).  A thread owns 8 consecutive pixels and holds
// a kernel row's 8 channels of them in registers; 32 x 32 pixels a block.
struct FinalGeo {
  static constexpr int CIC = 8, TW = 32, TH = 32, S = 1, PR = 34, PC = 34, PITCH = 36;
  static constexpr int PLANE = (PR * PITCH + 31 - 4) / 32 * 32 + 4;
  static constexpr bool SPLIT = false;
  static constexpr int EVEN = 0;
};
__global__ void __launch_bounds__(kThreads, 4)
f32_final_ordered_kernel(const F32Img* __restrict__ imgs, const float* __restrict__ w, const float* __restrict__ b,
                         int C, int tiles_x) {
  using G = FinalGeo;
  __shared__ __align__(16) float sm[G::CIC * G::PLANE];
  __shared__ float ws[9 * G::CIC];  // [tap][channel]
  const F32Img& I = imgs[blockIdx.z];
  const int Y0 = (blockIdx.x / tiles_x) * G::TH, X0 = (blockIdx.x % tiles_x) * G::TW;
  if (Y0 >= I.H || X0 >= I.W) return;
  const int gx = threadIdx.x % 4, row = threadIdx.x / 4;
  float acc[PX];
#pragma unroll
  for (int p = 0; p < PX; ++p) acc[p] = 0.f;
  for (int c0 = 0; c0 < C; c0 += G::CIC) {
    __syncthreads();
    load_patch<G, G::PR, G::PC>(sm, I.d3 + c0, C, Y0 - 1, X0 - 1, I.H, I.W);
    cp_commit();
    if (threadIdx.x < 9 * G::CIC) ws[threadIdx.x] = w[(threadIdx.x / G::CIC) * C + c0 + threadIdx.x % G::CIC];
    cp_wait<0>();
    __syncthreads();
#pragma unroll 1
    for (int ky = 0; ky < 3; ++ky) {
      float a[G::CIC][12];
#pragma unroll
      for (int ci = 0; ci < G::CIC; ++ci) load_row<G, 3>(sm + ci * G::PLANE + (row + ky) * G::PITCH + gx * PX, a[ci]);
#pragma unroll
      for (int kx = 0; kx < 3; ++kx)
#pragma unroll
        for (int ci = 0; ci < G::CIC; ++ci) {
          const float k = ws[(ky * 3 + kx) * G::CIC + ci];
#pragma unroll
          for (int p = 0; p < PX; ++p) acc[p] = fmaf(k, a[ci][p + kx], acc[p]);
        }
    }
  }
  const int y = Y0 + row;
  if (y >= I.H) return;
#pragma unroll
  for (int p = 0; p < PX; ++p) {
    const int x = X0 + gx * PX + p;
    if (x >= I.W) break;
    I.Y[(size_t)y * I.W + x] = upsample4_f(I.coarse_f, I.w, I.h, x, y) + (b[0] + acc[p]);
  }
}

// FK_Y5: a thread owns 8 input positions along x and their four output phases; the phase pair
// py = 1 has no tap in window row 0.  Channels go 4 a step (a one-channel source fills its step
// with zeros); the packed weights are [step][tap][channel][phase].
// A position's four channels are one 16-byte word, staged by one copy: the wide kinds' channel planes
// take four 4-byte copies, whose issue slots a kernel of 15 multiply-add pairs per word cannot hide (16
// pairs of 1242 x 375: 457 -> 300 us).  A gap after every eighth word and rows 4 words apart modulo 8
// keep a quarter-warp's reads on different banks.  Sources that are no multiple of 4 channels wide or not
// 16-byte aligned are copied by channels, zeros in the missing ones.
struct Y5Geo {
  static constexpr int CIC = 4, TW = 32, TH = 32, PR = 34, PC = 34, PITCH = 44;  // (in words)
  static constexpr int PATCH = PR * PITCH * 4, WF = 9 * CIC * 4, BUF = PATCH + WF;
  __device__ static constexpr int word(int c) { return c + (c >> 3); }
};
__global__ void __launch_bounds__(kThreads, 4)
f32_y5_kernel(const F32Job* __restrict__ jobs, const float* __restrict__ w, const float* __restrict__ bias, int steps,
              float scale, int tiles_x) {
  using G = Y5Geo;
  __shared__ __align__(16) float sm[2 * G::BUF];
  const F32Job& J = jobs[blockIdx.z];
  const int Y0 = (blockIdx.x / tiles_x) * G::TH, X0 = (blockIdx.x % tiles_x) * G::TW;
  if (Y0 >= J.Hi || X0 >= J.Wi) return;
  const int gx = threadIdx.x % 4, row = threadIdx.x / 4;
  int s = 0, c0 = 0;
  auto stage = [&](int ch) {
    float* b = sm + (ch & 1) * G::BUF;
    if (c0 >= J.ic[s]) { c0 = 0; ++s; }
    const int ic = J.ic[s], avail = ic - c0;
    const float* src = J.in[s] + c0;
    const bool vec = ic % 4 == 0 && reinterpret_cast<size_t>(src) % 16 == 0;
    for (int e = threadIdx.x; e < G::PR * G::PC; e += kThreads) {
      const int r = e / G::PC, c = e - r * G::PC, iy = Y0 - 1 + r, ix = X0 - 1 + c;
      const bool ok = iy >= 0 && ix >= 0 && iy < J.Hi && ix < J.Wi;
      const float* p = ok ? src + ((size_t)iy * J.Wi + ix) * ic : src;
      float* d = b + (r * G::PITCH + G::word(c)) * 4;
      if (vec) {
        cp16z(d, p, ok);
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) cp4(d + q, q < avail ? p + q : p, ok && q < avail);
      }
    }
    c0 += G::CIC;
    if (threadIdx.x < G::WF / 4) cp16(b + G::PATCH + 4 * threadIdx.x, w + (size_t)ch * G::WF + 4 * threadIdx.x);
    cp_commit();
  };
  u64 acc[PX][2];
#pragma unroll
  for (int p = 0; p < PX; ++p) acc[p][0] = acc[p][1] = 0ull;
  stage(0);
  for (int ch = 0; ch < steps; ++ch) {
    cp_wait<0>();
    __syncthreads();  // (as in contract)
    if (ch + 1 < steps) stage(ch + 1);
    const float* pa = sm + (ch & 1) * G::BUF + (row * G::PITCH + G::word(gx * PX)) * 4;
    const float* pw = sm + (ch & 1) * G::BUF + G::PATCH;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      float4 a[PX + 2];
#pragma unroll
      for (int q = 0; q < PX + 2; ++q)
        a[q] = *reinterpret_cast<const float4*>(pa + (r * G::PITCH + G::word(q)) * 4);
#pragma unroll
      for (int ci = 0; ci < G::CIC; ++ci) {
        u64 v[PX + 2];
#pragma unroll
        for (int q = 0; q < PX + 2; ++q) v[q] = dup2(ci == 0 ? a[q].x : ci == 1 ? a[q].y : ci == 2 ? a[q].z : a[q].w);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const ulonglong2 k = *reinterpret_cast<const ulonglong2*>(pw + ((r * 3 + c) * G::CIC + ci) * 4);
#pragma unroll
          for (int p = 0; p < PX; ++p) {
            fma2(acc[p][0], v[p + c], k.x);
            if (r > 0) fma2(acc[p][1], v[p + c], k.y);
          }
        }
      }
    }
  }
  const float b0 = bias[0];
#pragma unroll
  for (int py = 0; py < 2; ++py) {
    const int oy = 2 * (Y0 + row) + py;
    if (oy >= J.Ho) break;
#pragma unroll
    for (int p = 0; p < PX; ++p) {
      const int ox = 2 * (X0 + gx * PX + p);
      const float2 f = unpack2(acc[p][py]);
      if (ox < J.Wo) J.out[(size_t)oy * J.Wo + ox] = (f.x + b0) * scale;
      if (ox + 1 < J.Wo) J.out[(size_t)oy * J.Wo + ox + 1] = (f.y + b0) * scale;
    }
  }
}

__global__ void f32_reparam_kernel(const F32Lat* __restrict__ lat) {
  const F32Lat& q = lat[blockIdx.y];
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < q.n; i += (size_t)gridDim.x * blockDim.x) {
    const float m = q.mu[i], l = q.lv[i], e = q.eps[i];
    const float z = m + e * expf(0.5f * l);
    if (q.z16) {
      const __nv_bfloat16 r = __float2bfloat16_rn(z);
      q.z16[i] = r;
      q.z[i] = __bfloat162float(r);
    } else {
      q.z[i] = z;
    }
    if (q.mu_copy) q.mu_copy[i] = m;
    if (q.lv_copy) q.lv_copy[i] = l;
    if (q.eps_copy) q.eps_copy[i] = e;
  }
}

__global__ void f32_convert_kernel(const F32Cvt* __restrict__ jobs) {
  const F32Cvt& q = jobs[blockIdx.y];
  const size_t n8 = q.n / 8;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n8; i += (size_t)gridDim.x * blockDim.x) {
    const uint4 v = *reinterpret_cast<const uint4*>(q.src + 8 * i);
    float4* d = reinterpret_cast<float4*>(q.dst + 8 * i);
    auto lo = [](unsigned u) { return __uint_as_float(u << 16); };
    auto hi = [](unsigned u) { return __uint_as_float(u & 0xFFFF0000u); };
    d[0] = make_float4(lo(v.x), hi(v.x), lo(v.y), hi(v.y));
    d[1] = make_float4(lo(v.z), hi(v.z), lo(v.w), hi(v.w));
  }
}

}  // namespace

cudaError_t launch_f32_convert(const F32Cvt* jobs, int n, size_t max_n, cudaStream_t st) {
  if (n == 0 || max_n == 0) return cudaSuccess;
  const unsigned gx = (unsigned)std::min<size_t>(1024, (max_n / 8 + 255) / 256);
  constexpr int kMost = 65535;  // jobs of a launch (the grid's y extent)
  for (int i = 0; i < n; i += kMost) {
    f32_convert_kernel<<<dim3(std::max(1u, gx), std::min(kMost, n - i)), 256, 0, st>>>(jobs + i);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_f32_reparam(const F32Lat* lat, int n, size_t max_n, cudaStream_t st) {
  if (n == 0 || max_n == 0) return cudaSuccess;
  const unsigned gx = (unsigned)std::min<size_t>(256, (max_n + 255) / 256);
  f32_reparam_kernel<<<dim3(gx, n), 256, 0, st>>>(lat);
  return cudaGetLastError();
}

F32Layer f32_plan_layer(int kind, bool grad, const F32Src& src, std::vector<F32PackDesc>& descs, size_t& total) {
  F32Layer l;
  l.kind = kind;
  l.N = grad ? src.ci : src.co;
  l.K = grad ? src.co : src.ci;
  l.cg = l.N % 64 == 0 ? 8 : l.N % 32 == 0 ? 4 : l.N % 16 == 0 ? 2 : 1;
  const int cic = std::min(kind_cic(kind), l.K), bn = 8 * l.cg;
  const int phases = kind == FK_UP2 || kind == FK_DS2 || kind == FK_DE5 ? 4 : 1;
  static const int ty0[FK_COUNT] = {3, 1, 2, 1, 3, 5, 5, 3, 3};
  const bool edge = kind == FK_UP2;
  for (int ph = 0; ph < phases + (edge ? 1 : 0); ++ph) {
    const bool border = ph == phases;
    const int py = ph >> 1, px = ph & 1;
    int ty = ty0[kind], tx = ty0[kind];
    if (kind == FK_DS2) { ty = 1 + py; tx = 1 + px; }
    if (kind == FK_DE5) { ty = 3 - py; tx = 3 - px; }
    if (border) ty = tx = 3;
    (border ? l.wb : l.w[ph]) = total;
    F32PackDesc d{};
    d.src = src.w_ofs;
    d.dst = total;
    d.kind = kind;
    d.phase = kind == FK_P1 ? (grad ? 1 : 0) : (border ? 0 : ph);
    d.border = border;
    d.ks = src.ks;
    d.co = src.co;
    d.ci = src.ci;
    d.K = l.K;
    d.N = l.N;
    d.cic = cic;
    d.bn = bn;
    d.taps = ty * tx;
    d.tx = tx;
    d.count = (size_t)l.K * l.N * d.taps;
    descs.push_back(d);
    total += (size_t)l.K * l.N * ty * tx;
  }
  return l;
}

F32Layer f32_plan_y5(size_t w_ofs, const int* ic, int n_ic, std::vector<F32PackDesc>& descs, size_t& total) {
  F32Layer l;
  l.kind = FK_Y5;
  l.w[0] = total;
  int channels = 0;
  for (int i = 0; i < n_ic; ++i) channels += ic[i];
  int c0 = 0;
  for (int i = 0; i < n_ic; ++i) {
    F32PackDesc d{};
    d.src = w_ofs;
    d.dst = total;
    d.kind = FK_Y5;
    d.ks = 5;
    d.co = ic[i];     // channels of this source
    d.ci = channels;  // channels of the layer
    d.N = c0;         // first channel of this source
    d.cic = Y5Geo::CIC;
    d.K = (ic[i] + d.cic - 1) / d.cic * d.cic;
    d.bn = 4;
    d.taps = 9;
    d.tx = 3;
    d.count = (size_t)d.K * 9 * 4;
    descs.push_back(d);
    total += d.count;
    l.K += d.K;
    c0 += ic[i];
  }
  return l;
}

cudaError_t launch_f32_y5(const F32Layer& l, const F32Job* jobs, int n, int maxHo, int maxWo, const float* packed,
                          const float* bias, float scale, cudaStream_t st) {
  const int tx = ((maxWo + 1) / 2 + Y5Geo::TW - 1) / Y5Geo::TW, ty = ((maxHo + 1) / 2 + Y5Geo::TH - 1) / Y5Geo::TH;
  f32_y5_kernel<<<dim3(tx * ty, 1, n), kThreads, 0, st>>>(jobs, packed + l.w[0], bias, l.K / Y5Geo::CIC, scale, tx);
  return cudaGetLastError();
}

cudaError_t launch_f32_pack(const F32PackDesc* d, int n, size_t max_count, const float* params, float* packed,
                            cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  const unsigned gx = (unsigned)std::min<size_t>(64, (max_count + 255) / 256);
  f32_pack_kernel<<<dim3(gx, n), 256, 0, st>>>(d, params, packed);
  return cudaGetLastError();
}

cudaError_t launch_f32_conv(const F32Layer& l, const F32Job* jobs, int n, int maxHo, int maxWo, const float* packed,
                            const float* bias, int act, cudaStream_t st) {
  switch (l.kind) {
    case FK_S2: return by_width<FK_S2>(l, jobs, n, maxHo, maxWo, packed, bias, act, st);
    case FK_P1: return by_width<FK_P1>(l, jobs, n, maxHo, maxWo, packed, bias, act, st);
    case FK_UP2: return by_width<FK_UP2>(l, jobs, n, maxHo, maxWo, packed, bias, act, st);
    case FK_DS2: return by_width<FK_DS2>(l, jobs, n, maxHo, maxWo, packed, bias, act, st);
    case FK_DUP2: return by_width<FK_DUP2>(l, jobs, n, maxHo, maxWo, packed, bias, act, st);
    case FK_S1_5:
      if (l.K == 1) return run_conv<FK_S1_5, 4, 1>(l, jobs, n, maxHo, maxWo, packed, bias, act, st);
      if (l.cg == 2) return run_conv<FK_S1_5, 2, 4>(l, jobs, n, maxHo, maxWo, packed, bias, act, st);
      return run_conv<FK_S1_5, 1, 4>(l, jobs, n, maxHo, maxWo, packed, bias, act, st);
    case FK_S2_5:
      if (l.cg == 4) return run_conv<FK_S2_5, 4, 4>(l, jobs, n, maxHo, maxWo, packed, bias, act, st);
      return run_conv<FK_S2_5, 2, 4>(l, jobs, n, maxHo, maxWo, packed, bias, act, st);
    case FK_UP2X: return by_width<FK_UP2X>(l, jobs, n, maxHo, maxWo, packed, bias, act, st);
    case FK_DE5: return run_conv<FK_DE5, 2, 8>(l, jobs, n, maxHo, maxWo, packed, bias, act, st);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_f32_enc1(const F32Img* imgs, int n, int maxH1, int maxW1, const float* w, const float* b, int C,
                            cudaStream_t st) {
  auto go = [&](auto kern, int bn, int th, int tw) {
    const int tx = (maxW1 + tw - 1) / tw, ty = (maxH1 + th - 1) / th;
    kern<<<dim3(tx * ty, C / bn, n), kThreads, 0, st>>>(imgs, w, b, C, tx);
    return cudaGetLastError();
  };
  if (C % 64 == 0) return go(f32_enc1_kernel<8>, 64, Enc1Geo<8>::TH, Enc1Geo<8>::TW);
  if (C % 32 == 0) return go(f32_enc1_kernel<4>, 32, Enc1Geo<4>::TH, Enc1Geo<4>::TW);
  return go(f32_enc1_kernel<2>, 16, Enc1Geo<2>::TH, Enc1Geo<2>::TW);
}

cudaError_t launch_f32_final(const F32Img* imgs, int n, int maxH, int maxW, const float* w, const float* b, int C,
                             bool ordered, cudaStream_t st) {
  if (ordered) {
    const int tx = (maxW + FinalGeo::TW - 1) / FinalGeo::TW, ty = (maxH + FinalGeo::TH - 1) / FinalGeo::TH;
    f32_final_ordered_kernel<<<dim3(tx * ty, 1, n), kThreads, 0, st>>>(imgs, w, b, C, tx);
    return cudaGetLastError();
  }
  auto go = [&](auto kern, int no) {
    const int tx = (maxW + no - 1) / no, ty = (maxH + kFinRows - 1) / kFinRows;
    kern<<<dim3(tx * ty, 1, n), 256, 0, st>>>(imgs, w, b, C, tx);
    return cudaGetLastError();
  };
  if (C % 32 == 0) return go(f32_final_kernel<8>, 256 / 8 - 2);
  return go(f32_final_kernel<4>, 256 / 4 - 2);
}

}  // namespace sv
