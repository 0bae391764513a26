// Generic-window slice chain: any probe window M = 2^a 3^b (8 <= M <= 4096)
// that the register-resident kernels do not cover (they take M = 64, 128).
//
// The chunk's positions advance through the multislice model (Sec. II-B)
// together, slice by slice: their waves live in a global buffer wv[n][M][M],
// and every launch is one pass over their rows or columns (chain_gm_line.cuh
// says what a pass does).  The workspace it fills (entering waves, exit-wave
// gradients, probe-gradient parts, loss parts) has the layout of the
// register-resident kernels, so the tiled reductions are shared.
//
// This file holds the passes with a runtime radix schedule (windows without a
// compile-time instance) and the launch sequence.
#include "chain_gm_line.cuh"
#include "gm_gain.h"

#include <algorithm>
#include <cmath>

namespace ptycho {

namespace {

struct GmPlan {
  int n;      // radix stages
  int r[16];  // radices (8, 4, 2, 3)
};

// Shared-memory slot of element i of a line: one padding slot every 16
// elements, which spreads the radix-8 first stage (outputs 8 apart across
// threads) over the banks; the odd line stride does the same for the column
// transposes.
__host__ __device__ constexpr int gm_pad(int i) { return i + (i >> 4); }
__host__ __device__ constexpr int gm_line_stride(int M) { return M + M / 16 + 1; }
// Block shape: threads and the most elements (lines x M) a block takes.
constexpr int kGmThreads = 256, kGmElems = 4096;

bool gm_plan(int M, GmPlan* plan) {
  if (M < 8 || M > 4096) return false;
  GmPlan p{};
  int m = M;
  for (int r : {8, 4, 2, 3})
    while (m % r == 0 && p.n < 16) {
      p.r[p.n++] = r;
      m /= r;
    }
  if (m != 1) return false;
  if (plan) *plan = p;
  return true;
}

// Lines per block: the largest divisor of M with L M <= kGmElems.
__host__ __device__ int gm_lines(int M) {
  int best = 1;
  for (int L = 1; L <= M && L * M <= kGmElems; ++L)
    if (M % L == 0) best = L;
  return best;
}

size_t gm_rt_smem(int M) {
  return (2 * (size_t)gm_lines(M) * gm_line_stride(M) + 2 * (size_t)M) * sizeof(float2) +
         (kGmThreads / 32) * sizeof(double);
}

// One Stockham autosort stage of radix R over the block's L lines of length
// M, after spans of Ns: butterfly j takes x[j + q M/R], twiddles it by
// w_{Ns R}^{q (j mod Ns)} (per-stage table at toff, contiguous in j mod Ns),
// and writes y[(j - k) R + k + q Ns].
template <int R, bool INV>
__device__ __forceinline__ void gm_stage(const float2* __restrict__ src, float2* __restrict__ dst, int M, int L,
                                         int Ns, const float2* __restrict__ tw, int t) {
  const int nb = M / R, LS = gm_line_stride(M);
  for (int idx = t; idx < L * nb; idx += kGmThreads) {
    const int li = idx / nb, j = idx - li * nb;
    const int k = j % Ns;
    float2 x[R];
#pragma unroll
    for (int q = 0; q < R; ++q) x[q] = src[li * LS + gm_pad(j + q * nb)];
    if (Ns > 1) {
#pragma unroll
      for (int q = 1; q < R; ++q) x[q] = cmul_opt<INV>(x[q], tw[(q - 1) * Ns + k]);
    }
    dft_r<R, INV>(x);
    const int d0 = (j - k) * R + k;
#pragma unroll
    for (int q = 0; q < R; ++q) dst[li * LS + gm_pad(d0 + q * Ns)] = x[q];
  }
}

// All stages of one transform from buffer A; returns the buffer that holds
// the result (A or B).  Every stage ends in a block barrier.
template <bool INV>
__device__ __forceinline__ float2* gm_transform(const GmPlan& plan, float2* A, float2* B, int M, int L,
                                                const float2* Tst, int t) {
  int Ns = 1;
  for (int i = 0; i < plan.n; ++i) {
    const int R = plan.r[i];
    if (R == 8)
      gm_stage<8, INV>(A, B, M, L, Ns, Tst, t);
    else if (R == 4)
      gm_stage<4, INV>(A, B, M, L, Ns, Tst, t);
    else if (R == 2)
      gm_stage<2, INV>(A, B, M, L, Ns, Tst, t);
    else
      gm_stage<3, INV>(A, B, M, L, Ns, Tst, t);
    if (Ns > 1) Tst += (R - 1) * Ns;
    Ns *= R;
    float2* s = A;
    A = B;
    B = s;
    __syncthreads();
  }
  return A;
}

// For n stages 4n + 4 shared-memory round trips an element and propagation,
// against 4n - 2 when each propagation was two passes of its own (rows, then
// columns) whose first and last stages worked on global memory; but half as many
// passes read and write the waves.  us of an evaluation, those two passes / these (8
// slices): 36, 930 positions 1323 / 849; 243, 135 5468 / 5065; 324, 76 5273 /
// 4936; 576, 24 4560 / 4061; 4 slices: 768, 13 2520 / 1917; 1152, 6 4063 / 2901;
// 3 slices: 2048, 2 4749 / 1976; 4096, 2 34707 / 13538.  The 31 windows without an
// instance gain 1.07 to 3.3 times, single positions 1.4 to 4.7.
template <int KIND>
__global__ void __launch_bounds__(kGmThreads, 4)
    k_gm_pass_rt(const ChainArgs a, const GmPass g, const int M, const int L, const GmPlan plan) {
  constexpr bool ADJ = KIND == GM_ADJ;
  const int LS = gm_line_stride(M), parts = M / L;
  extern __shared__ float2 gsm[];
  float2* A = gsm;
  float2* B = A + (size_t)L * LS;
  float2* Tst = B + (size_t)L * LS;  // sum over stages of (R - 1) Ns < M entries
  float2* H = Tst + M;
  [[maybe_unused]] double* red = reinterpret_cast<double*>(H + M);
  const int t = threadIdx.x;
  {
    int Ns = 1, toff = 0;
    for (int i = 0; i < plan.n; ++i) {
      const int R = plan.r[i];
      if (Ns > 1) {
        const int tstep = M / (Ns * R);
        for (int e = t; e < (R - 1) * Ns; e += kGmThreads) {
          const int q = 1 + e / Ns, k = e - (q - 1) * Ns;
          Tst[toff + e] = a.tw[tstep * q * k];
        }
        toff += (R - 1) * Ns;
      }
      Ns *= R;
    }
    for (int k = t; k < M; k += kGmThreads) H[k] = a.hs[k];
  }
  dependency_wait();
  const int il = blockIdx.x / parts, part = blockIdx.x % parts;
  const GmBlock b{a, g, M, part * L, il, a.pos[a.pos_begin + il], g.cols != 0};
  if (!window_ok(b.r, M, a.H, a.W)) {
    gm_skip<KIND>(b, L, parts, part, t, kGmThreads);
    return;
  }
  const float2* src = g.src + (g.from_probe ? 0 : (size_t)il * M * M);
  // f(li, i) for every element of the block's lines, consecutive threads on
  // consecutive addresses of the waves
  auto each = [&](auto&& f) {
    for (int e = t; e < L * M; e += kGmThreads)
      if (b.cols) f(e % L, e / L); else f(e / M, e % M);
  };
  auto other = [&](float2* x) { return x == A ? B : A; };
  each([&](int li, int i) { A[li * LS + gm_pad(i)] = src[b.at(li, i)]; });
  __syncthreads();
  float2* x = A;
  auto transform = [&](auto inv) {
    x = gm_transform<decltype(inv)::value>(plan, x, other(x), M, L, Tst, t);
  };
  auto propagate = [&]() {
    transform(std::false_type{});
    each([&](int li, int i) {
      float2& v = x[li * LS + gm_pad(i)];
      v = cmul_opt<ADJ>(v, H[i]);
    });
    __syncthreads();
    transform(std::true_type{});
  };
  if constexpr (KIND == GM_RES) {
    transform(std::false_type{});
    double lsum = 0.0;
    const size_t e0 = (size_t)(a.pos_begin + il) * M * M;
    if (g.mode == MODE_FORWARD) {
      each([&](int li, int i) { gm_output(b, x[li * LS + gm_pad(i)], e0 + b.at(li, i)); });
      return;
    }
    each([&](int li, int i) {
      float2& v = x[li * LS + gm_pad(i)];
      v = gm_residual(M, v, __ldcs(a.meas + e0 + b.at(li, i)), lsum);
    });
    gm_store_loss<kGmThreads>(lsum, red, a.loss_part + (size_t)il * parts + part, t);
    if (!g.dst) return;
    __syncthreads();
    transform(std::true_type{});
  } else {
    if (g.op1 == GM_PROP) propagate();
    if (g.op1 == GM_IFFT) transform(std::true_type{});
    each([&](int li, int i) {
      float2 v[1] = {x[li * LS + gm_pad(i)]};
      b.template transmit<KIND, 1>(v, li, i, 0);
      x[li * LS + gm_pad(i)] = v[0];
    });
    if (!g.dst) return;
    __syncthreads();
    if (g.op2 == GM_PROP) propagate();
    if (g.op2 == GM_FFT) transform(std::false_type{});
  }
  launch_dependents();
  float2* dst = g.dst + (size_t)il * M * M;
  each([&](int li, int i) { dst[b.at(li, i)] = x[li * LS + gm_pad(i)]; });
}

// The compile-time instance of a window, or null.
const GmInstance* gm_find(int M) {
  for (int i = 0; i < kGmSmallCount; ++i)
    if (kGmSmall[i].M == M) return &kGmSmall[i];
  for (int i = 0; i < kGmMiddleCount; ++i)
    if (kGmMiddle[i].M == M) return &kGmMiddle[i];
  for (int i = 0; i < kGmLargeCount; ++i)
    if (kGmLarge[i].M == M) return &kGmLarge[i];
  return nullptr;
}

}  // namespace

void gm_factor_gain(int M, double* gain) {
  if (const GmInstance* in = gm_find(M))
    gm_transform_gain(in->r1, in->r2, in->r3, gain);
  else
    std::fill(gain, gain + M, 1.0);
}

bool gm_supported(int M) { return gm_plan(M, nullptr); }

int gm_loss_parts(int M) {
  const GmInstance* in = gm_find(M);
  return in ? in->parts : M / gm_lines(M);
}

// The shared-memory limit is an attribute of the kernel, shared by every plan
// in the process: the runtime kernels' is raised to what the largest window
// they serve needs.
cudaError_t gm_prepare(int M) {
  if (const GmInstance* in = gm_find(M)) return in->prepare();
  size_t most = 0;
  for (int m = 8; m <= 4096; ++m)
    if (gm_supported(m) && gm_rt_smem(m) > most) most = gm_rt_smem(m);
  cudaError_t e;
  const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
  if ((e = cudaFuncSetAttribute(k_gm_pass_rt<GM_FWD>, attr, (int)most)) != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(k_gm_pass_rt<GM_ADJ>, attr, (int)most)) != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_gm_pass_rt<GM_RES>, attr, (int)most);
}

// Positions per chunk for n positions, at most cap.  A pass runs in waves of
// resident blocks; a chunk that ends in a nearly empty wave, or a small last
// chunk, wastes them in each of its 2S + 1 passes.  Takes the chunk with the
// fewest waves in all, a fifth of a wave counted per chunk for its launches.
// us of an evaluation, largest chunk / this rule: 506 positions, M = 192 3107 /
// 3068; 306 simulated at 256 791 / 777; 400, M = 81 420 / 413; 1024, M = 256
// 7445 / 7483.
int gm_chunk(int M, int n, int cap, int sm_count) {
  if (n <= cap) return n;
  const GmInstance* in = gm_find(M);
  int per_sm = 0;
  if (in)
    per_sm = in->blocks_per_sm();
  else if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_gm_pass_rt<GM_ADJ>, kGmThreads, gm_rt_smem(M)) !=
           cudaSuccess)
    per_sm = 0;
  const double resident = (double)per_sm * sm_count;
  if (resident <= 0) return cap;
  const int parts = gm_loss_parts(M);
  auto waves = [&](int positions) { return std::ceil(positions * (double)parts / resident) + 0.2; };
  int best = cap;
  double least = 0;
  for (int c = cap; c >= 1 && 2 * c >= cap; --c) {
    const double w = n / c * waves(c) + (n % c ? waves(n % c) : 0);
    if (c == cap || w < least) {
      best = c;
      least = w;
    }
  }
  return best;
}

namespace {

struct GmLauncher {
  const ChainArgs& a;
  int M;
  cudaStream_t st;
  GmPlan plan{};
  const GmInstance* in = nullptr;
  int launches = 0;

  cudaError_t pass(GmKind kind, const GmPass& g) {
    ++launches;
    if (in) return in->launch(kind, a, g, st);
    const int L = gm_lines(M);
    const unsigned grid = (unsigned)((size_t)a.n_pos * (M / L));
    const size_t smem = gm_rt_smem(M);
    void (*k)(ChainArgs, GmPass, int, int, GmPlan) =
        kind == GM_FWD ? k_gm_pass_rt<GM_FWD> : kind == GM_ADJ ? k_gm_pass_rt<GM_ADJ> : k_gm_pass_rt<GM_RES>;
    return launch_after(k, grid, kGmThreads, smem, st, a, g, M, L, plan);
  }
};

}  // namespace

// Recompute mode (ckpt_L = L, K = ceil(S / L) segments) follows the
// register-resident kernels' schedule with the chunk's waves in wv:
// MODE_GRAD_RC runs the forward keeping the waves entering segments 1..K-2
// (ws_psi slots 0..K-3) and the last segment's waves (slots K-2 ..), the
// residual, the adjoint through the last segment (g_phi in ws_gphi slots
// s - s0), whose last pass writes the adjoint state to slot K-2+L;
// MODE_RC_SEG rebuilds segment a.seg's waves from its checkpoint (or the
// probe) and runs the adjoint through the segment from and to that slot.  The
// caller sums each segment's (psi, g_phi) pairs into the object gradient in
// between.
cudaError_t launch_chain_gm(ChainMode mode, const ChainArgs& a, float2* wv, int M, int* n_launches,
                            cudaStream_t st) {
  if (a.n_pos <= 0) return cudaSuccess;
  GmLauncher g{a, M, st};
  if (!gm_plan(M, &g.plan)) return cudaErrorInvalidValue;
  g.in = gm_find(M);
  const size_t MM = (size_t)M * M;
  const int S = a.S, L = a.ckpt_L > 0 ? a.ckpt_L : 1, K = (S + L - 1) / L;
  const int seg_slot = K - 2, park_slot = K - 2 + L;
  auto psi_slot = [&](int k) { return a.ws_psi + (size_t)k * a.ws_n * MM; };
  // slice s forward: from the probe (s = 0), `from` (no propagation before
  // it) or wv; `stop` keeps psi_s only
  auto forward = [&](int s, float2* save, const float2* from, bool stop) {
    GmPass p{};
    p.from_probe = s == 0;
    p.src = s == 0 ? a.probe : from ? from : wv;
    p.dst = stop ? nullptr : wv;
    p.save = save;
    p.cols = s % 2;
    p.s = s;
    p.op1 = s == 0 || from ? GM_NONE : GM_PROP;
    p.op2 = stop ? GM_NONE : s == S - 1 ? GM_FFT : GM_PROP;
    return g.pass(GM_FWD, p);
  };
  // adjoint through slices s_hi .. s_lo, g_phi_s into slot s - base, from
  // `from` (or wv); the state after s_lo > 0 goes to `to` (or wv)
  auto adjoint = [&](int s_hi, int s_lo, int base, const float2* from, float2* to) -> cudaError_t {
    for (int s = s_hi; s >= s_lo; --s) {
      GmPass p{};
      p.src = s == s_hi && from ? from : wv;
      p.dst = s == 0 ? a.ws_gp : s == s_lo && to ? to : wv;
      p.save = a.ws_gphi + (size_t)(s - base) * a.ws_n * MM;
      p.cols = s % 2;
      p.s = s;
      p.op1 = s == S - 1 ? GM_IFFT : GM_PROP;
      p.op2 = s == 0 ? GM_NONE : GM_PROP;
      const cudaError_t r = g.pass(GM_ADJ, p);
      if (r != cudaSuccess) return r;
    }
    return cudaSuccess;
  };
  cudaError_t e;
  if (mode == MODE_RC_SEG) {
    const int j = a.seg, s0 = j * L, s1 = s0 + L;
    for (int s = s0; s < s1; ++s) {
      if (s == 0 && s1 == 1) break;  // psi_0 is the probe
      if ((e = forward(s, s > 0 ? psi_slot(seg_slot + (s - s0)) : nullptr,
                       s == s0 && j > 0 ? psi_slot(j - 1) : nullptr, s == s1 - 1)) != cudaSuccess)
        return e;
    }
    if ((e = adjoint(s1 - 1, s0, s0, psi_slot(park_slot), psi_slot(park_slot))) != cudaSuccess) return e;
    if (n_launches) *n_launches = g.launches;
    return cudaSuccess;
  }
  const bool grad = mode == MODE_GRAD, rc = mode == MODE_GRAD_RC;
  const int s_last = (K - 1) * L;  // first slice of the last segment (recompute mode)
  for (int s = 0; s < S; ++s) {
    float2* save = nullptr;
    if (grad && s > 0)
      save = psi_slot(s - 1);
    else if (rc && s > 0 && s % L == 0 && s / L <= K - 2)
      save = psi_slot(s / L - 1);
    else if (rc && s >= s_last)
      save = psi_slot(seg_slot + (s - s_last));
    if ((e = forward(s, save, nullptr, false)) != cudaSuccess) return e;
  }
  GmPass p{};
  p.src = wv;
  p.dst = grad || rc ? wv : nullptr;
  p.cols = S % 2;
  p.mode = mode;
  if ((e = g.pass(GM_RES, p)) != cudaSuccess) return e;
  if (grad && (e = adjoint(S - 1, 0, 0, nullptr, nullptr)) != cudaSuccess) return e;
  if (rc && (e = adjoint(S - 1, s_last, s_last, nullptr, psi_slot(park_slot))) != cudaSuccess) return e;
  if (n_launches) *n_launches = g.launches;
  return cudaSuccess;
}

}  // namespace ptycho
