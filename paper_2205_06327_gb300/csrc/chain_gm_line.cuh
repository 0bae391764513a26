// Line passes of the generic-window slice chain (any window M = 2^a 3^b other
// than the register-resident 64 and 128): what one launch does, and its kernels.
//
// The Fresnel factor is separable, so a propagation is a 1-D propagation P_d
// (FFT, h_1(k)/M, inverse) along each axis d, in either order.  Slice s is
// transmitted between two propagations, so with the axes taken alternately
// (x first after slice 0, y first after slice 1, ...) the second half of one
// propagation, the transmission and the first half of the next all act on the
// same lines:
//   pass 0        load the probe,     x O_0,                     P_x
//   pass s        P_d,                keep psi_s, x O_s,         P_d     d = s mod 2 (0: rows, 1: columns)
//   pass S-1      P_d,                keep, x O_{S-1},           F_d
//   residual      F_d',               residual of Eq. 1,         F_d'^-1
//   adjoint S-1   F_d^-1,             keep g_phi, x conj O_{S-1}, P_d^*
//   adjoint s     P_d^*,              keep g_phi_s, x conj O_s,  P_d^*
//   adjoint 0     P_x^*,              keep g_phi_0, x conj O_0   -> probe gradient
// One evaluation is 2S + 1 passes over the chunk's waves, each reading and
// writing them once (the waves of a chunk stay in L2).
#pragma once

#include "../../include/ptycho.h"
#include "bounds.h"
#include "fft2d.cuh"
#include "internal.h"

namespace ptycho {

enum GmOp : int { GM_NONE = 0, GM_PROP = 1, GM_FFT = 2, GM_IFFT = 3 };
enum GmKind : int { GM_FWD = 0, GM_ADJ = 1, GM_RES = 2 };

struct GmPass {
  const float2* src;  // waves read [n][M][M], or the probe [M][M]
  float2* dst;        // waves written [n][M][M] (null: only `save` is written)
  float2* save;       // psi_s (forward) or g_phi_s (adjoint) of every position, or null
  int cols;           // 0: the lines are rows, 1: columns
  int s;              // slice transmitted
  int from_probe;
  int op1, op2;       // GmOp before and after the transmission (conjugated in the adjoint)
  int mode;           // residual pass: the ChainMode
};

// Launches of one window's instance.
struct GmInstance {
  int M;
  int r1, r2, r3;
  int parts;  // loss parts per position (blocks of the residual pass)
  cudaError_t (*prepare)();
  int (*blocks_per_sm)();  // resident blocks of a pass (0 if unknown)
  cudaError_t (*launch)(GmKind kind, const ChainArgs& a, const GmPass& g, cudaStream_t st);
};

// Constants of the composite radices: w_R^e = exp(-2 pi i e / R) (the inverse
// uses the conjugate).
namespace gmr {

template <int R>
struct Wr;
template <>
struct Wr<16> {
  static constexpr float c[16] = {1.f, 0.92387953251128674f, 0.70710678118654752f, 0.38268343236508977f,
                                  0.f, -0.38268343236508977f, -0.70710678118654752f, -0.92387953251128674f,
                                  -1.f, -0.92387953251128674f, -0.70710678118654752f, -0.38268343236508977f,
                                  0.f, 0.38268343236508977f, 0.70710678118654752f, 0.92387953251128674f};
  static constexpr float s[16] = {0.f, -0.38268343236508977f, -0.70710678118654752f, -0.92387953251128674f,
                                  -1.f, -0.92387953251128674f, -0.70710678118654752f, -0.38268343236508977f,
                                  0.f, 0.38268343236508977f, 0.70710678118654752f, 0.92387953251128674f,
                                  1.f, 0.92387953251128674f, 0.70710678118654752f, 0.38268343236508977f};
};
template <>
struct Wr<12> {
  static constexpr float c[12] = {1.f, 0.86602540378443865f, 0.5f, 0.f, -0.5f, -0.86602540378443865f,
                                  -1.f, -0.86602540378443865f, -0.5f, 0.f, 0.5f, 0.86602540378443865f};
  static constexpr float s[12] = {0.f, -0.5f, -0.86602540378443865f, -1.f, -0.86602540378443865f, -0.5f,
                                  0.f, 0.5f, 0.86602540378443865f, 1.f, 0.86602540378443865f, 0.5f};
};
template <>
struct Wr<9> {
  static constexpr float c[9] = {1.f, 0.76604444311897804f, 0.17364817766693035f, -0.5f, -0.93969262078590838f,
                                 -0.93969262078590838f, -0.5f, 0.17364817766693035f, 0.76604444311897804f};
  static constexpr float s[9] = {0.f, -0.64278760968653933f, -0.98480775301220806f, -0.86602540378443865f,
                                 -0.34202014332566873f, 0.34202014332566873f, 0.86602540378443865f,
                                 0.98480775301220806f, 0.64278760968653933f};
};
template <>
struct Wr<6> {
  static constexpr float c[6] = {1.f, 0.5f, -0.5f, -1.f, -0.5f, 0.5f};
  static constexpr float s[6] = {0.f, -0.86602540378443865f, -0.86602540378443865f, 0.f,
                                 0.86602540378443865f, 0.86602540378443865f};
};

// R = R1 R2 for the composite radices.
template <int R>
struct Split;
template <>
struct Split<16> {
  static constexpr int R1 = 4, R2 = 4;
};
template <>
struct Split<12> {
  static constexpr int R1 = 4, R2 = 3;
};
template <>
struct Split<9> {
  static constexpr int R1 = 3, R2 = 3;
};
template <>
struct Split<6> {
  static constexpr int R1 = 2, R2 = 3;
};

}  // namespace gmr

namespace {

// v w_R^e (forward) or v conj(w_R^e) (inverse), with the trivial factors
// (1, -i, -1, +i) as sign and swap operations.
template <int R, int E, bool INV>
__device__ __forceinline__ float2 mul_wr(float2 v) {
  constexpr int e = E % R;
  if constexpr (e == 0) {
    return v;
  } else if constexpr (4 * e == R) {
    return mul_mi<INV>(v);
  } else if constexpr (2 * e == R) {
    return make_float2(-v.x, -v.y);
  } else if constexpr (4 * e == 3 * R) {
    return mul_mi<!INV>(v);
  } else {
    const float c = gmr::Wr<R>::c[e], sn = INV ? -gmr::Wr<R>::s[e] : gmr::Wr<R>::s[e];
    return make_float2(fmaf(v.x, c, -v.y * sn), fmaf(v.x, sn, v.y * c));
  }
}

template <int R, bool INV>
__device__ __forceinline__ void dft_r(float2 (&x)[R]);

// Composite small DFT (one Cooley-Tukey step in registers): with n = R2 n1 + n2
// and k = k1 + R1 k2, X[k] = sum_n2 w_R2^(n2 k2) w_R^(n2 k1) sum_n1 w_R1^(n1 k1) x[n].
template <int R, bool INV>
__device__ __forceinline__ void dft_composite(float2 (&x)[R]) {
  constexpr int R1 = gmr::Split<R>::R1, R2 = gmr::Split<R>::R2;
  float2 y[R];  // y[n2 R1 + k1]
  static_for<0, R2>([&](auto n2c) {
    constexpr int n2 = decltype(n2c)::value;
    float2 u[R1];
#pragma unroll
    for (int n1 = 0; n1 < R1; ++n1) u[n1] = x[R2 * n1 + n2];
    dft_r<R1, INV>(u);
    static_for<0, R1>([&](auto k1c) {
      constexpr int k1 = decltype(k1c)::value;
      y[n2 * R1 + k1] = mul_wr<R, n2 * k1, INV>(u[k1]);
    });
  });
#pragma unroll
  for (int k1 = 0; k1 < R1; ++k1) {
    float2 u[R2];
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) u[n2] = y[n2 * R1 + k1];
    dft_r<R2, INV>(u);
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) x[k1 + R1 * k2] = u[k2];
  }
}

// Small DFT of a register array in natural order, forward kernel
// exp(-2 pi i n k / R), inverse its conjugate, unnormalised.
template <int R, bool INV>
__device__ __forceinline__ void dft_r(float2 (&x)[R]) {
  if constexpr (R == 2) {
    dft2(x[0], x[1]);
  } else if constexpr (R == 3) {
    // X1 = t2 -+ i s3 (b - c), X2 = t2 +- i s3 (b - c), t2 = a - (b + c)/2
    const float s3 = 0.86602540378443864676f;
    const float2 a = x[0], b = x[1], c = x[2];
    const float2 t1 = cadd(b, c);
    const float2 t2 = make_float2(fmaf(-0.5f, t1.x, a.x), fmaf(-0.5f, t1.y, a.y));
    const float2 d = make_float2(s3 * (b.x - c.x), s3 * (b.y - c.y));
    const float2 mid = mul_mi<INV>(d);
    x[0] = cadd(a, t1);
    x[1] = cadd(t2, mid);
    x[2] = csub(t2, mid);
  } else if constexpr (R == 4) {
    dft4<INV>(x[0], x[1], x[2], x[3]);
  } else if constexpr (R == 8) {
    dft8<INV>(x[0], x[1], x[2], x[3], x[4], x[5], x[6], x[7]);
  } else {
    static_assert(R == 6 || R == 9 || R == 12 || R == 16, "radix 2, 3, 4, 6, 8, 9, 12 or 16");
    dft_composite<R, INV>(x);
  }
}

__device__ __forceinline__ bool window_ok(int2 r, int M, int H, int W) {
  return r.x >= 0 && r.y >= 0 && r.x <= H - M && r.y <= W - M;
}

// A block's lines and where its elements sit in the waves and the object.
struct GmBlock {
  const ChainArgs& a;
  const GmPass& g;
  int M, l0, il;     // window, first line, position in the chunk
  int2 r;            // window corner (y, x)
  bool cols;

  __device__ __forceinline__ int at(int li, int i) const { return cols ? i * M + (l0 + li) : (l0 + li) * M + i; }
  __device__ __forceinline__ int64_t obj_at(int li, int i) const {
    return cols ? window_at(i, l0 + li, a.W) : window_at(l0 + li, i, a.W);
  }
  __device__ __forceinline__ const float2* obj_window(const float2* o) const {
    return o + (size_t)g.s * a.H * a.W + (size_t)r.x * a.W + r.y;
  }

  // The slice's transmission on R elements i0 + q di of line li: forward
  // keeps psi_s and multiplies by O_s (at the line search's trial point when
  // the call has one), the adjoint keeps g_phi_s and multiplies by conj(O_s).
  template <int KIND, int R>
  __device__ __forceinline__ void transmit(float2 (&x)[R], int li, int i0, int di) const {
    const int64_t step = cols ? window_at(di, 0, a.W) : di;  // from one of the elements to the next
    const float2* ow = obj_window(a.obj) + obj_at(li, i0);
    float2 o[R];
#pragma unroll
    for (int q = 0; q < R; ++q, ow += step) o[q] = __ldg(ow);
    if constexpr (KIND == GM_FWD) {
      if (g.from_probe && a.probe_dir) {
#pragma unroll
        for (int q = 0; q < R; ++q) {
          const float2 d = a.probe_dir[at(li, i0 + q * di)];
          x[q].x = fmaf(a.probe_step, d.x, x[q].x);
          x[q].y = fmaf(a.probe_step, d.y, x[q].y);
        }
      }
      if (a.obj_dir) {
        const float2* dw = obj_window(a.obj_dir) + obj_at(li, i0);
#pragma unroll
        for (int q = 0; q < R; ++q, dw += step) {
          const float2 d = __ldg(dw);
          o[q].x = fmaf(a.obj_step, d.x, o[q].x);
          o[q].y = fmaf(a.obj_step, d.y, o[q].y);
        }
      }
    }
    if (g.save) {
      float2* sv = g.save + (size_t)il * M * M;
#pragma unroll
      for (int q = 0; q < R; ++q) __stcs(sv + at(li, i0 + q * di), x[q]);
    }
#pragma unroll
    for (int q = 0; q < R; ++q) x[q] = KIND == GM_FWD ? cmul(x[q], o[q]) : cmulc(x[q], o[q]);
  }
};

// Far field z (unnormalised along both axes: M Psi) of element e -> outputs
// (forward mode).
__device__ __forceinline__ void gm_output(const GmBlock& b, float2 z, size_t e) {
  const float inv_m = 1.0f / (float)b.M;
  const float2 p = make_float2(z.x * inv_m, z.y * inv_m);
  if (b.a.psi_out) b.a.psi_out[e] = p;
  if (b.a.int_out) b.a.int_out[e] = fmaf(p.x, p.x, p.y * p.y);
}

// The residual of Eq. 1 against the measured intensity: adds the loss term to
// lsum and returns the adjoint seed 2 d Psi/|Psi| / M, pre-scaled for the
// unnormalised inverse.
__device__ __forceinline__ float2 gm_residual(int M, float2 z, float intensity, double& lsum) {
  const float A = sqrtf(intensity);
  const float mag = sqrtf(fmaf(z.x, z.x, z.y * z.y));
  const float d = mag * (1.0f / (float)M) - A;
  lsum += (double)d * (double)d;
  const float sc = mag > 0.0f ? (2.0f * d) / (mag * (float)M) : 0.0f;
  return make_float2(z.x * sc, z.y * sc);
}

// Fixed-order FP64 sum over the block, written by thread 0.
template <int T>
__device__ __forceinline__ void gm_store_loss(double lsum, double* red, double* out, int t) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) lsum += __shfl_down_sync(0xffffffffu, lsum, off);
  if ((t & 31) == 0) red[t >> 5] = lsum;
  __syncthreads();
  if (t == 0) {
    double tot = 0.0;
    for (int k = 0; k < T / 32; ++k) tot += red[k];
    *out = tot;
  }
}

// A window outside the object contributes nothing: flag it, no loss, no
// gradient (the object-gradient accumulation skips such windows).
template <int KIND>
__device__ __forceinline__ void gm_skip(const GmBlock& b, int L, int parts, int part, int t, int T) {
  if (KIND == GM_FWD && t == 0) *b.a.pos_status = PTYCHO_ERR_POSITION;
  if (KIND == GM_RES && t == 0 && b.g.mode != MODE_FORWARD) b.a.loss_part[(size_t)b.il * parts + part] = 0.0;
  if (KIND == GM_ADJ && b.g.s == 0)
    for (int k = t; k < L * b.M; k += T) b.g.dst[(size_t)b.il * b.M * b.M + b.at(k % L, k / L)] = make_float2(0.f, 0.f);
}

// ---------------------------------------------------------------------------
// Compile-time instances.  M = R1 R2 R3 (R2 = 1: two factors), L lines per
// block.  Decimation in frequency forward, exactly reversed inverse, so a 1-D
// propagation needs no reordering: a thread of phase A holds the R1 elements
// j + (M/R1) q of a line, transforms over q and writes them to the line's
// slots (k1, j); phase B (three factors) transforms the R2 digit of j, phase C
// the R3 digit, multiplies by the factor and goes straight back; phase A'
// inverts the R1 digit into the same registers phase A loaded.  A two-factor
// propagation so costs two shared-memory round trips per element (Stockham
// stages of radix 8/8/3 cost five) and the last phase of one propagation, the
// transmission and the first phase of the next run in registers.  ncu on 225
// positions at M = 192 (4 blocks of 256 threads, 64 registers): the shared
// pipe 60-67 %, FP32 37-39 %, issue 45 %, the largest stall the block barrier,
// then global loads.  So the shapes below take small blocks (96-128 threads,
// several items each, many blocks per SM to cover the barriers) and registers
// enough not to spill.
//
// Slots: rows keep line li's element (k1, k2, j2) at li LS + k1 PK + k2 PJ + j2
// with PJ odd and PK = 16/R1 modulo 16 for R1 | 16, so that the 16 lanes of a
// half-warp fall on different 8-byte banks in every phase; columns
// interleave the block's lines ((k1 PK + k2 PJ + j2) L + li), so consecutive
// lanes take consecutive columns, in shared and in global memory; with fewer
// than 16 lines PJ and PK are odd, for the same reason.
// ---------------------------------------------------------------------------
constexpr int gm_pk(int R1, int R2, int PJ) {
  int p = R2 * PJ;
  if (R2 == 1) return p;
  if (16 % R1 == 0)
    while (p % 16 != (16 / R1) % 16) ++p;
  else
    while (p % 2 == 0) ++p;
  return p;
}

template <int R1_, int R2_, int R3_, int L_, int T_, int MINB_>
struct GmShape {
  static constexpr int R1 = R1_, R2 = R2_, R3 = R3_, L = L_, T = T_, MINB = MINB_;
  static constexpr int M = R1 * R2 * R3, MI = R2 * R3;
  static constexpr int PT = R3 | 1;  // pitch of the phase-C twiddle rows
  static constexpr int TA = R2 == 1 ? R1 * PT : M, TB = R2 == 1 ? 0 : R2 * PT;
  static_assert(M % L == 0 && T % 32 == 0, "whole lines per block, whole warps");
  static constexpr int pj(bool cols) { return cols && L % 16 == 0 ? R3 : R3 | 1; }
  static constexpr int pk(bool cols) {
    return !cols ? gm_pk(R1, R2, pj(false)) : R2 == 1 ? pj(true) : L % 16 == 0 ? R2 * R3 : (R2 * pj(true)) | 1;
  }
  static constexpr int line_slots(bool cols) { return R1 * pk(cols); }
  static constexpr size_t smem(bool cols) {
    return ((size_t)L * line_slots(cols) + TA + TB + M) * sizeof(float2) + (T / 32) * sizeof(double);
  }
};

template <class P, bool COLS>
struct GmLines {
  static constexpr int R1 = P::R1, R2 = P::R2, R3 = P::R3, L = P::L, T = P::T, MI = P::MI;
  static constexpr int PJ = P::pj(COLS), PK = P::pk(COLS), LS = R1 * PK;
  // Rows, when the warps share the lines evenly and fill their lanes (or have
  // three factors): each warp keeps its lines to itself, so its phases need no
  // block barrier.  Measured, block / warp: 1024 positions, M = 256 8033 / 7925
  // us, 42 at 384 1050 / 1033, 20 at 512 912 / 883, 4 at 1024 x 100 slices 14143
  // / 13741; 506 at 192, where a quarter of the lanes would idle, 3308 / 3345.
  static constexpr bool WARP =
      !COLS && L % (T / 32) == 0 && (R2 > 1 || L / (T / 32) * R1 * R2 % 32 == 0);
  static constexpr int LW = WARP ? L / (T / 32) : L, TW = WARP ? 32 : T;
  float2* D;         // the block's lines
  const float2* TA;  // w_M^(k1 j): [R1][PT] (two factors) or [R1][M/R1]
  const float2* TB;  // w_(M/R1)^(k2 j2): [R2][PT] (three factors)
  const float2* H;   // h_1(k) / M
  int t;

  __device__ __forceinline__ float2& slot(int li, int k1, int k2, int j2) const {
    return COLS ? D[(k1 * PK + k2 * PJ + j2) * L + li] : D[li * LS + k1 * PK + k2 * PJ + j2];
  }
  // f(li, r) for every item (line li, r < N) of this thread.
  template <int N, class F>
  __device__ __forceinline__ void items(F&& f) const {
    const int first = WARP ? t % 32 : t, line0 = WARP ? t / 32 * LW : 0;
#pragma unroll 1
    for (int idx = first; idx < LW * N; idx += TW) {
      const int r = COLS ? idx / L : idx % N, li = COLS ? idx % L : idx / N;
      f(line0 + li, r);
    }
  }
  // Between phases: the lines' slots are written.
  __device__ __forceinline__ void sync() const {
    if constexpr (WARP) __syncwarp(); else __syncthreads();
  }
  __device__ __forceinline__ void put_a(const float2 (&x)[R1], int li, int j) const {
#pragma unroll
    for (int q = 0; q < R1; ++q) slot(li, q, j / R3, j % R3) = x[q];
  }
  __device__ __forceinline__ void get_a(float2 (&x)[R1], int li, int j) const {
#pragma unroll
    for (int q = 0; q < R1; ++q) x[q] = slot(li, q, j / R3, j % R3);
  }
  template <bool INV>
  __device__ __forceinline__ void phase_b() const {
    if constexpr (R2 > 1) {
      items<R1 * R3>([&](int li, int r) {
        const int j2 = r % R3, k1 = r / R3;
        float2 x[R2];
#pragma unroll
        for (int q = 0; q < R2; ++q) x[q] = slot(li, k1, q, j2);
        if constexpr (INV) dft_r<R2, true>(x);
#pragma unroll
        for (int q = 0; q < R2; ++q) x[q] = cmul_opt<INV>(x[q], TA[k1 * MI + j2 + R3 * q]);
        if constexpr (!INV) dft_r<R2, false>(x);
#pragma unroll
        for (int q = 0; q < R2; ++q) slot(li, k1, q, j2) = x[q];
      });
      sync();
    }
  }
  __device__ __forceinline__ const float2* twc(int k1, int k2) const {
    return R2 > 1 ? TB + k2 * P::PT : TA + k1 * P::PT;
  }
  __device__ __forceinline__ void get_c(float2 (&x)[R3], int li, int k1, int k2) const {
    const float2* w = twc(k1, k2);
#pragma unroll
    for (int q = 0; q < R3; ++q) x[q] = slot(li, k1, k2, q);
#pragma unroll
    for (int q = 1; q < R3; ++q) x[q] = cmul(x[q], w[q]);
    dft_r<R3, false>(x);
  }
  __device__ __forceinline__ void put_c(float2 (&x)[R3], int li, int k1, int k2) const {
    const float2* w = twc(k1, k2);
    dft_r<R3, true>(x);
#pragma unroll
    for (int q = 1; q < R3; ++q) x[q] = cmulc(x[q], w[q]);
#pragma unroll
    for (int q = 0; q < R3; ++q) slot(li, k1, k2, q) = x[q];
  }
  // 1-D propagation between put_a and get_a.
  template <bool CONJ>
  __device__ __forceinline__ void propagate() const {
    sync();
    phase_b<false>();
    items<R1 * R2>([&](int li, int r) {
      const int k1 = r % R1, k2 = r / R1;
      float2 x[R3];
      get_c(x, li, k1, k2);
#pragma unroll
      for (int q = 0; q < R3; ++q) x[q] = cmul_opt<CONJ>(x[q], H[r + R1 * R2 * q]);
      put_c(x, li, k1, k2);
    });
    sync();
    phase_b<true>();
  }
};

// Twiddle and factor tables of the block.
template <class P>
__device__ __forceinline__ void gm_tables(const ChainArgs& a, float2* TA, float2* TB, float2* H, int t) {
  constexpr int MI = P::MI, PA = P::R2 == 1 ? P::PT : MI;
  for (int e = t; e < P::R1 * MI; e += P::T) {
    const int k1 = e / MI, j = e % MI;
    TA[k1 * PA + j] = a.tw[k1 * j];
  }
  if constexpr (P::R2 > 1)
    for (int e = t; e < MI; e += P::T) {
      const int k2 = e / P::R3, j = e % P::R3;
      TB[k2 * P::PT + j] = a.tw[P::R1 * k2 * j];
    }
  for (int e = t; e < P::M; e += P::T) H[e] = a.hs[e];
}

template <class P, int KIND, bool COLS>
__global__ void __launch_bounds__(P::T, P::MINB) k_gm_pass(const ChainArgs a, const GmPass g) {
  constexpr int M = P::M, L = P::L, T = P::T, R1 = P::R1, R2 = P::R2, R3 = P::R3, MI = P::MI, PARTS = M / L;
  extern __shared__ float2 gsm[];
  float2* D = gsm;
  float2* TA = D + (size_t)L * P::line_slots(COLS);
  float2* TB = TA + P::TA;
  float2* H = TB + P::TB;
  [[maybe_unused]] double* red = reinterpret_cast<double*>(H + M);
  const int t = threadIdx.x;
  gm_tables<P>(a, TA, TB, H, t);
  dependency_wait();
  const GmLines<P, COLS> ln{D, TA, TB, H, t};
  const int il = blockIdx.x / PARTS, part = blockIdx.x % PARTS;
  const GmBlock b{a, g, M, part * L, il, a.pos[a.pos_begin + il], COLS};
  if (!window_ok(b.r, M, a.H, a.W)) {
    gm_skip<KIND>(b, L, PARTS, part, t, T);
    return;
  }
  const float2* src = g.src + (g.from_probe ? 0 : (size_t)il * M * M);
  float2* dst = g.dst + (size_t)il * M * M;
  auto load_a = [&](float2(&x)[R1], int li, int j) {
#pragma unroll
    for (int q = 0; q < R1; ++q) x[q] = src[b.at(li, j + MI * q)];
  };
  auto store_a = [&](const float2(&x)[R1], int li, int j) {
#pragma unroll
    for (int q = 0; q < R1; ++q) dst[b.at(li, j + MI * q)] = x[q];
  };

  if constexpr (KIND == GM_RES) {
    ln.template items<MI>([&](int li, int j) {
      float2 x[R1];
      load_a(x, li, j);
      dft_r<R1, false>(x);
      ln.put_a(x, li, j);
    });
    __syncthreads();  // (and the tables are filled)
    ln.template phase_b<false>();
    double lsum = 0.0;
    const size_t e0 = (size_t)(a.pos_begin + il) * M * M;
    if (g.mode == MODE_FORWARD) {
      ln.template items<R1 * R2>([&](int li, int r) {
        float2 x[R3];
        ln.get_c(x, li, r % R1, r / R1);
#pragma unroll
        for (int q = 0; q < R3; ++q) gm_output(b, x[q], e0 + b.at(li, r + R1 * R2 * q));
      });
      return;
    }
    ln.template items<R1 * R2>([&](int li, int r) {
      const int k1 = r % R1, k2 = r / R1;
      float I[R3];  // from DRAM: fetched before the transform
#pragma unroll
      for (int q = 0; q < R3; ++q) I[q] = __ldcs(a.meas + e0 + b.at(li, r + R1 * R2 * q));
      float2 x[R3];
      ln.get_c(x, li, k1, k2);
#pragma unroll
      for (int q = 0; q < R3; ++q) x[q] = gm_residual(M, x[q], I[q], lsum);
      if (g.dst) ln.put_c(x, li, k1, k2);
    });
    gm_store_loss<T>(lsum, red, a.loss_part + (size_t)il * PARTS + part, t);
    if (!g.dst) return;
    ln.sync();
    ln.template phase_b<true>();
    launch_dependents();
    ln.template items<MI>([&](int li, int j) {
      float2 x[R1];
      ln.get_a(x, li, j);
      dft_r<R1, true>(x);
      store_a(x, li, j);
    });
  } else {
    constexpr bool ADJ = KIND == GM_ADJ;
    __syncthreads();
    bool staged = false;  // the lines sit in the slots, one inverse R1 digit short of the elements
    if (ADJ && g.op1 == GM_IFFT) {
      ln.template items<R1 * R2>([&](int li, int r) {
        float2 x[R3];
#pragma unroll
        for (int q = 0; q < R3; ++q) x[q] = src[b.at(li, r + R1 * R2 * q)];
        ln.put_c(x, li, r % R1, r / R1);
      });
      ln.sync();
      ln.template phase_b<true>();
      staged = true;
    }
    const int mid = g.op1 == GM_PROP ? 1 : 0;
    const int last = g.op2 == GM_PROP ? mid + 1 : mid;
#pragma unroll 1
    for (int step = 0;; ++step) {
      if (step == last) launch_dependents();
      ln.template items<MI>([&](int li, int j) {
        float2 x[R1];
        if (staged) {
          ln.get_a(x, li, j);
          dft_r<R1, true>(x);
        } else {
          load_a(x, li, j);
        }
        if (step == mid) b.template transmit<KIND, R1>(x, li, j, MI);
        if (step == last && g.op2 != GM_FFT) {
          if (g.dst) store_a(x, li, j);
        } else {
          dft_r<R1, false>(x);
          ln.put_a(x, li, j);
        }
      });
      if (step == last) break;
      ln.template propagate<ADJ>();
      staged = true;
    }
    if (!ADJ && g.op2 == GM_FFT) {
      ln.sync();
      ln.template phase_b<false>();
      ln.template items<R1 * R2>([&](int li, int r) {
        float2 x[R3];
        ln.get_c(x, li, r % R1, r / R1);
#pragma unroll
        for (int q = 0; q < R3; ++q) dst[b.at(li, r + R1 * R2 * q)] = x[q];
      });
    }
  }
}

template <class P, int KIND>
cudaError_t gm_set_smem() {
  cudaError_t e = cudaFuncSetAttribute(k_gm_pass<P, KIND, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)P::smem(false));
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_gm_pass<P, KIND, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)P::smem(true));
}

template <class P>
cudaError_t gm_prepare_ct() {
  cudaError_t e;
  if ((e = gm_set_smem<P, GM_FWD>()) != cudaSuccess) return e;
  if ((e = gm_set_smem<P, GM_ADJ>()) != cudaSuccess) return e;
  return gm_set_smem<P, GM_RES>();
}

template <class P>
cudaError_t gm_launch_ct(GmKind kind, const ChainArgs& a, const GmPass& g, cudaStream_t st) {
  const unsigned grid = (unsigned)a.n_pos * (P::M / P::L);
  const size_t smem = P::smem(g.cols != 0);
  void (*k)(ChainArgs, GmPass) =
      g.cols ? (kind == GM_FWD ? k_gm_pass<P, GM_FWD, true>
                               : kind == GM_ADJ ? k_gm_pass<P, GM_ADJ, true> : k_gm_pass<P, GM_RES, true>)
             : (kind == GM_FWD ? k_gm_pass<P, GM_FWD, false>
                               : kind == GM_ADJ ? k_gm_pass<P, GM_ADJ, false> : k_gm_pass<P, GM_RES, false>);
  return launch_after(k, grid, P::T, smem, st, a, g);
}

template <class P>
int gm_blocks_ct() {
  int n = 0;
  const cudaError_t e =
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_gm_pass<P, GM_ADJ, false>, P::T, P::smem(false));
  return e == cudaSuccess ? n : 0;
}

template <class P>
constexpr GmInstance gm_instance() {
  return GmInstance{P::M, P::R1, P::R2, P::R3, P::M / P::L, gm_prepare_ct<P>, gm_blocks_ct<P>, gm_launch_ct<P>};
}

}  // namespace

// The compile-time instances, grouped by translation unit.
extern const GmInstance kGmSmall[], kGmMiddle[], kGmLarge[];
extern const int kGmSmallCount, kGmMiddleCount, kGmLargeCount;

}  // namespace ptycho
