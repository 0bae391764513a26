// Register-resident 2-D FFT of one M x M complex64 tile per thread block.
//
// The multislice model (Sec. II-B) Fourier transforms each slice's wave,
// multiplies by the propagator and inverse transforms it; the exit wave is
// transformed once more to the detector.  Here one thread block owns one
// probe position's M x M wave for the whole slice chain: each thread keeps
// V = M*M/T complex values in registers and the transform is three radix
// passes, each a 2-D pass that applies one mixed-radix digit of y and one of
// x at once (decimation in frequency).  Between passes the wave is exchanged
// through shared memory in a swizzled row-major layout that is free of bank
// conflicts for all three access patterns.
//
// Forward passes leave the spectrum in digit-reversed storage order; the
// inverse passes undo the forward ones exactly in reverse order on the same
// storage.  So propagate = fwd, pointwise multiply, inv needs no reordering,
// and the register grouping before pass 1 equals the grouping after inverse
// pass 1: consecutive slices chain without any extra exchange.
//
// Transforms here are unnormalised; callers fold the orthonormal 1/M factors
// into the propagator table or the residual.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "tc_bf16.cuh"

namespace ptycho {

template <int I, int N, class F>
__device__ __forceinline__ void static_for(F&& f) {
  if constexpr (I < N) {
    f(std::integral_constant<int, I>{});
    static_for<I + 1, N>(f);
  }
}

// Complex sums as packed pairs of FP32 operations: one instruction for both
// components, each rounded as the scalar operation, so results are unchanged.
// A packed instruction takes two slots of the FP32 pipe (probe: 0.46 packed
// against 0.90 scalar per clock and scheduler), so it buys issue slots, not
// arithmetic: the chain issued 1.84 M instructions per position against an
// FP32 pipe 40 % busy.  Measured (scalar -> packed sums): 576 positions,
// M = 128, 16 slices 2.28 -> 2.20 ms; 960 positions, M = 64 1.17 -> 1.06 ms;
// 506 positions, M = 192 7.16 -> 6.80 ms.
__device__ __forceinline__ unsigned long long pack2(float2 a) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
  return r;
}
__device__ __forceinline__ float2 unpack2(unsigned long long a) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
  return r;
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)));
  return unpack2(r);
}
__device__ __forceinline__ float2 csub(float2 a, float2 b) {
  unsigned long long r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)));
  return unpack2(r);
}
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
// a * conj(b)
__device__ __forceinline__ float2 cmulc(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, a.y * b.y), fmaf(a.y, b.x, -a.x * b.y));
}
// conj(a) * b
__device__ __forceinline__ float2 cconjmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, a.y * b.y), fmaf(a.x, b.y, -a.y * b.x));
}
// The same products with packed instructions (identical rounding): fewer issue
// slots, but their operands need aligned register pairs.  They pay in the
// register-resident chain (below) and cost spills in the line passes of
// chain_gm_line.cuh.
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)));
  return unpack2(r);
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)), "l"(pack2(c)));
  return unpack2(r);
}
__device__ __forceinline__ float2 pmul(float2 a, float2 b) {
  return fma2(make_float2(a.x, a.x), b, mul2(make_float2(a.y, a.y), make_float2(-b.y, b.x)));
}
__device__ __forceinline__ float2 pmulc(float2 a, float2 b) {
  return fma2(a, make_float2(b.x, b.x), mul2(make_float2(a.y, -a.x), make_float2(b.y, b.y)));
}
template <bool CONJ>
__device__ __forceinline__ float2 pmul_opt(float2 a, float2 b) { return CONJ ? pmulc(a, b) : pmul(a, b); }
template <bool CONJ>
__device__ __forceinline__ float2 cmul_opt(float2 a, float2 b) { return CONJ ? cmulc(a, b) : cmul(a, b); }

// multiply by -i (forward kernel) or +i (inverse kernel)
template <bool INV>
__device__ __forceinline__ float2 mul_mi(float2 a) {
  return INV ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}

// Small DFTs in natural order, forward kernel exp(-2 pi i n k / R), inverse
// kernel its conjugate, both unnormalised.
__device__ __forceinline__ void dft2(float2& x0, float2& x1) {
  const float2 t = x0;
  x0 = cadd(t, x1);
  x1 = csub(t, x1);
}

template <bool INV>
__device__ __forceinline__ void dft4(float2& x0, float2& x1, float2& x2, float2& x3) {
  const float2 t0 = cadd(x0, x2), t1 = csub(x0, x2);
  const float2 t2 = cadd(x1, x3), t3 = mul_mi<INV>(csub(x1, x3));
  x0 = cadd(t0, t2);
  x2 = csub(t0, t2);
  x1 = cadd(t1, t3);
  x3 = csub(t1, t3);
}

template <bool INV>
__device__ __forceinline__ void dft8(float2& x0, float2& x1, float2& x2, float2& x3,
                                     float2& x4, float2& x5, float2& x6, float2& x7) {
  dft4<INV>(x0, x2, x4, x6);  // even samples -> E0..E3
  dft4<INV>(x1, x3, x5, x7);  // odd samples  -> O0..O3
  const float r = 0.70710678118654752440f;
  // O_k *= w8^k, w8 = exp(-+ 2 pi i / 8)
  const float2 o1 = INV ? make_float2((x3.x - x3.y) * r, (x3.x + x3.y) * r)
                        : make_float2((x3.x + x3.y) * r, (x3.y - x3.x) * r);
  const float2 o2 = mul_mi<INV>(x5);
  const float2 o3 = INV ? make_float2((-x7.x - x7.y) * r, (x7.x - x7.y) * r)
                        : make_float2((x7.y - x7.x) * r, (-x7.x - x7.y) * r);
  const float2 e0 = x0, e1 = x2, e2 = x4, e3 = x6, o0 = x1;
  x0 = cadd(e0, o0); x4 = csub(e0, o0);
  x1 = cadd(e1, o1); x5 = csub(e1, o1);
  x2 = cadd(e2, o2); x6 = csub(e2, o2);
  x3 = cadd(e3, o3); x7 = csub(e3, o3);
}

template <int R, bool INV, int OFF, int ST, int N>
__device__ __forceinline__ void dft_at(float2 (&v)[N]) {
  if constexpr (R == 1) {
  } else if constexpr (R == 2) {
    dft2(v[OFF], v[OFF + ST]);
  } else if constexpr (R == 4) {
    dft4<INV>(v[OFF], v[OFF + ST], v[OFF + 2 * ST], v[OFF + 3 * ST]);
  } else if constexpr (R == 8) {
    dft8<INV>(v[OFF], v[OFF + ST], v[OFF + 2 * ST], v[OFF + 3 * ST],
              v[OFF + 4 * ST], v[OFF + 5 * ST], v[OFF + 6 * ST], v[OFF + 7 * ST]);
  } else {
    static_assert(R == 1 || R == 2 || R == 4 || R == 8, "unsupported radix");
  }
}

// ---------------------------------------------------------------------------
// Tile configurations.  Storage index of y: py = d0*SY0 + d1*SY1 + d2 with
// digit j in [0, RY(j)); likewise px for x.  Pass j transforms digit j of y
// and of x.  base<J>(t, q) returns the storage coordinates of the (a=0, b=0)
// element of the q-th group that thread t owns in pass J; element (a, b) of
// that group sits at (py + a*SY(J), px + b*SX(J)).  swz() permutes columns
// inside each 16-element block of a row (bank-conflict-free exchanges).
// ---------------------------------------------------------------------------
// Where a thread finds its per-pass factors (filled once per block by
// fill_factors, every entry rounded once from FP64).  Read from shared and
// global memory, each with its own index arithmetic, the twiddles and the
// propagator were a third of the chain's shared-memory wavefronts and a fifth
// of its instructions, and spilled registers.  A thread needs the same 2 V
// pass-0 and spectrum factors for the whole chain, and tensor memory (unused
// otherwise by this kernel) holds exactly 4 V = 128 words per thread and has a
// data path of its own.  With the packed products below: one wave of 152
// positions, M = 128, 16 slices 445 -> 380 us; 576 positions 2.20 -> 2.04 ms;
// 960 positions, M = 64 1.06 -> 0.98 ms.  The adjoint now reads the exact
// twiddles too (it multiplied two table entries per element before).
//   tmem  this warp's 128 tensor-memory columns: words [0, 2V) hold the pass-0
//         twiddles of the thread's V elements, words [2V, 4V) the propagator
//         at its V spectrum elements (pass-2 grouping);
//   tw1   shared table of the pass-1 twiddles, one row of G entries per
//         (ey, ex) class (16 classes).
struct Factors {
  uint32_t tmem;
  const float2* tw1;
  // cluster only: the mbarriers of the two row buffers, the parity of their
  // next completion, the device error word, and whether this thread still takes
  // part in the exchanges
  uint64_t* mbar = nullptr;
  uint32_t phase = 0;
  int* status = nullptr;
  int state = 0;
};
// Factors::state.  Muted (self-test): no exchange stores, a short wait, which
// therefore expires.  Gave up: a wait expired.
constexpr int kMuted = 1, kGaveUp = 2;
constexpr int kWaitExpired = -5;  // PTYCHO_ERR_TIMEOUT

template <int M>
struct Cfg;

template <>
struct Cfg<128> {
  static constexpr int M = 128, T = 512, V = 32, MIN_BLOCKS = 1;
  static constexpr int CL = 1, TB = T, kSmemWave = M * M;  // blocks per position, threads per block
  static constexpr int TWB = 16;  // complex factors fetched from tensor memory at a time
  __device__ static __forceinline__ void sync() { __syncthreads(); }
  __device__ static __forceinline__ void arrived(const Factors&, int) { __syncthreads(); }
  __device__ static __forceinline__ void put_loss(double* red, int w, double v) { red[w] = v; }
  static constexpr int ry(int j) { return j == 0 ? 8 : 4; }
  static constexpr int rx(int j) { return j == 1 ? 8 : 4; }
  static constexpr int sy(int j) { return j == 0 ? 16 : (j == 1 ? 4 : 1); }
  static constexpr int sx(int j) { return j == 0 ? 32 : (j == 1 ? 4 : 1); }
  __device__ static __forceinline__ int swz(int px) { return px ^ (5 * ((px >> 5) & 3)); }
  // The pass-1 <-> pass-2 exchange stays inside warp pairs {2k, 2k+1}: a
  // 64-thread named barrier (ids 1..8) orders it.
  __device__ static __forceinline__ void sync12(int t) {
    asm volatile("bar.sync %0, 64;" ::"r"(1 + (t >> 6)) : "memory");
  }
  // After a block barrier the 16 warps would load their next pass together
  // and then compute together, so the shared-memory pipe and the FP32 pipe
  // would take turns (ncu on one wave of positions: 54 % and 45 % of 380 us,
  // which add up).  Instead the block starts in kTurns groups of warps, each
  // loading once the group before it has issued its loads: one group computes
  // while the next loads, and the offset persists to the next block barrier.
  // Measured with 1 / 2 / 4 / 8 groups: 576 positions, 16 slices 2.04 / 1.93 /
  // 1.86 / 1.85 ms; forward model alone 0.615 / 0.555 / 0.537 / 0.532 ms;
  // 16632 positions in recompute mode - / - / 119.5 / 121.1 ms.
  static constexpr int kTurns = 4;
  __device__ static __forceinline__ void turn_wait(int t) {
    constexpr int GT = T / kTurns;
    if (t / GT > 0) asm volatile("bar.sync %0, %1;" ::"r"(8 + t / GT), "n"(2 * GT) : "memory");
  }
  __device__ static __forceinline__ void turn_pass(int t) {
    constexpr int GT = T / kTurns;
    if (t / GT < kTurns - 1) asm volatile("bar.arrive %0, %1;" ::"r"(9 + t / GT), "n"(2 * GT) : "memory");
  }
  template <int J>
  __device__ static __forceinline__ void base(int t, int q, int& py, int& px) {
    const int w = t >> 5, l = t & 31;
    if constexpr (J == 0) {
      py = w; px = l;
    } else if constexpr (J == 1) {
      const int e3 = l & 3, e1 = (l >> 2) & 3;
      const int d3 = ((l >> 4) & 1) | ((w & 1) << 1), d1 = w >> 1;
      py = 16 * d1 + d3; px = 32 * e1 + e3;
    } else {
      const int e1 = l & 3, e2 = l >> 2, g = 2 * w + q;
      py = 16 * (g >> 2) + 4 * (g & 3); px = 32 * e1 + 4 * e2;
    }
  }
};

// The same wave over a cluster of 8 thread blocks of 64 threads (thread t of
// the 512 is thread t % 64 of block t / 64), each on its own SM when few
// positions run.  Block k owns the pass-1 and pass-2 groups of rows
// 16 k .. 16 k + 15, so only the exchange between passes 0 and 1 crosses
// blocks: forward, every element is stored into its pass-1 owner's row buffer;
// inverse, into its pass-0 owner's.  The arithmetic of every element is that
// of Cfg<128>, so results are bit-identical.
struct ClusterCfg128 : Cfg<128> {
  static constexpr int CL = 8, TB = T / CL, ROWS = M / CL;
  static constexpr int kSmemWave = 2 * ROWS * M;  // float2: the two row buffers
  __device__ static __forceinline__ void sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
  __device__ static __forceinline__ void sync12(int) { __syncthreads(); }
  __device__ static __forceinline__ void turn_wait(int) {}
  __device__ static __forceinline__ void turn_pass(int) {}
  // The exchanges need no cluster barrier: every store counts its bytes on the
  // receiving buffer's mbarrier, and a block waits for its 16 KB.  A buffer may
  // be written again once the exchange through the other one is complete: by
  // then every block has sent, so has read what the first one held.
  static constexpr uint32_t kBytes = ROWS * M * sizeof(float2);
  static constexpr long long kWaitCycles = 2000000000LL;  // about 1 s
  static constexpr long long kShortWaitCycles = 2000000LL;  // about 1 ms
  // address of p in block `rank` of the cluster
  __device__ static __forceinline__ uint32_t peer(const void* p, int rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(tc::smem_u32(p)), "r"(rank));
    return r;
  }
  __device__ static __forceinline__ void put(uint32_t addr, uint32_t mbar, float2 v) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(addr),
                 "f"(v.x), "f"(v.y), "r"(mbar)
                 : "memory");
  }
  // Buffer `which`'s exchange number `phase` has arrived.  A thread whose wait
  // expires reports it and gives up: it neither waits nor arms an mbarrier nor
  // stores into another block from then on (what it computes is meaningless), so
  // the other blocks' next wait expires too and the kernel ends within two
  // limits.  An mbarrier is only armed again by a thread that saw its last phase
  // complete.
  __device__ static __forceinline__ void arrived(Factors& f, int which) {
    if (!(f.state & kGaveUp)) {
      uint64_t* mbar = f.mbar + which;
      if (threadIdx.x == 0)
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(tc::smem_u32(mbar)), "r"(kBytes)
                     : "memory");
      const long long limit = f.state & kMuted ? kShortWaitCycles : kWaitCycles;
      if (tc::mbar_wait_bounded(mbar, f.phase >> which & 1u, limit)) {
        f.phase ^= 1u << which;
      } else {
        *f.status = kWaitExpired;
        f.state |= kGaveUp;
      }
    }
    __syncwarp();  // tensor memory is read by whole warps
  }
  // Before a block gives its memory back: no block leaves while another may
  // still store into it.  A block whose exchanges all arrived has nothing in
  // flight towards it; one that gave up lets late stores of the exchange it left
  // land first (its peers have issued theirs by the barrier).
  __device__ static __forceinline__ void leave(const Factors& f) {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
    if (f.state & kGaveUp)
      for (int which = 0; which < 2; ++which)
        tc::mbar_wait_bounded(f.mbar + which, f.phase >> which & 1u, kShortWaitCycles);
  }
  __device__ static __forceinline__ void put_loss(double* red, int w, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(peer(red + w, 0)), "d"(v) : "memory");
  }
};

template <>
struct Cfg<64> {
  static constexpr int M = 64, T = 128, V = 32, MIN_BLOCKS = 4;
  static constexpr int CL = 1, TB = T, kSmemWave = M * M, TWB = 16;
  __device__ static __forceinline__ void sync() { __syncthreads(); }
  __device__ static __forceinline__ void arrived(const Factors&, int) { __syncthreads(); }
  __device__ static __forceinline__ void put_loss(double* red, int w, double v) { red[w] = v; }
  static constexpr int ry(int) { return 4; }
  static constexpr int rx(int) { return 4; }
  static constexpr int sy(int j) { return j == 0 ? 16 : (j == 1 ? 4 : 1); }
  static constexpr int sx(int j) { return j == 0 ? 16 : (j == 1 ? 4 : 1); }
  __device__ static __forceinline__ int swz(int px) { return px ^ (5 * ((px >> 4) & 3)); }
  // (four independent blocks per SM overlap by themselves)
  __device__ static __forceinline__ void turn_wait(int) {}
  __device__ static __forceinline__ void turn_pass(int) {}
  // The pass-1 <-> pass-2 exchange stays inside each warp.
  __device__ static __forceinline__ void sync12(int) { __syncwarp(); }
  template <int J>
  __device__ static __forceinline__ void base(int t, int q, int& py, int& px) {
    const int w = t >> 5, l = t & 31;
    if constexpr (J == 0) {
      py = (l >> 4) | (w << 1) | (q << 3); px = l & 15;
    } else if constexpr (J == 1) {
      const int e3 = l & 3, e1 = (l >> 2) & 3, d3 = ((l >> 4) & 1) | (q << 1);
      py = 16 * w + d3; px = 16 * e1 + e3;
    } else {
      const int e1 = l & 3, e2 = (l >> 2) & 3, d2 = ((l >> 4) & 1) | (q << 1);
      py = 16 * w + 4 * d2; px = 16 * e1 + 4 * e2;
    }
  }
};

// Tensor-memory columns a block takes: 128 per 4 warps.
template <class C>
constexpr int kTmemTake = C::TB < 128 ? 128 : C::TB;

// The same with half the factors fetched at a time.  Fewer, wider fetches wait
// less but hold more registers: 576 positions, M = 128, 16 slices, gradient
// 1606 us with 8 at a time, 1587 with 16 (4560 positions in recompute mode 27.3
// and 26.9 ms); forward model alone 538 and 554 us.
template <class B>
struct HalfFetch : B {
  static constexpr int TWB = 8;
};

// Frequency index of storage row/column after the three forward passes:
// k = d0 + R0*d1 + R0*R1*d2 (digit reversal of the storage index).
template <class C>
__device__ __forceinline__ int freq_y(int py) {
  return py / C::sy(0) + C::ry(0) * ((py / C::sy(1)) % C::ry(1)) + C::ry(0) * C::ry(1) * (py % C::ry(2));
}
template <class C>
__device__ __forceinline__ int freq_x(int px) {
  return px / C::sx(0) + C::rx(0) * ((px / C::sx(1)) % C::rx(1)) + C::rx(0) * C::rx(1) * (px % C::rx(2));
}

template <class C, int J>
struct PassShape {
  static constexpr int RY = C::ry(J), RX = C::rx(J), G = RY * RX, Q = C::V / G;
  static constexpr int SY = C::sy(J), SX = C::sx(J);
  static_assert(Q * G == C::V, "group size must divide the per-thread count");
};

// Launder a value through an empty asm so index arithmetic derived from it
// is recomputed where it is used instead of being hoisted out of the slice
// loop and pinned in registers.
__device__ __forceinline__ int opaque(int x) {
  asm volatile("" : "+r"(x));
  return x;
}

// FAR: the exchange between passes 0 and 1 (the one that crosses the blocks of
// a cluster; stored by pass 0 going forward and by pass 1 going back).
template <class C, int J, bool FAR>
__device__ __forceinline__ void xch_store(const float2 (&v)[C::V], float2* sm, const Factors& f, int t) {
  using P = PassShape<C, J>;
  if constexpr (C::CL > 1 && FAR) {
    if (f.state) return;  // muted, or gave up
  }
  t = opaque(t);
  static_for<0, P::Q>([&](auto qq) {
    constexpr int q = decltype(qq)::value;
    int py, px;
    C::template base<J>(t, q, py, px);
    static_for<0, P::RY>([&](auto aa) {
      constexpr int a = decltype(aa)::value;
      const int y = py + a * P::SY;
      [[maybe_unused]] uint32_t row = 0, mbar = 0;
      if constexpr (C::CL > 1 && FAR) {  // into row buffer 0 by rows, or row buffer 1 by pass-0 owner
        const int rank = J == 0 ? y / C::ROWS : y % 16 / 2;
        row = C::peer(sm + (J == 0 ? y % C::ROWS : C::ROWS + y % 2 * 8 + y / 16) * C::M, rank);
        mbar = C::peer(f.mbar + (J == 0 ? 0 : 1), rank);
      }
      static_for<0, P::RX>([&](auto bb) {
        constexpr int b = decltype(bb)::value;
        const int x = C::swz(px + b * P::SX);
        const float2 e = v[q * P::G + a * P::RX + b];
        if constexpr (C::CL == 1)
          sm[y * C::M + x] = e;
        else if constexpr (FAR)
          C::put(row + 8 * x, mbar, e);
        else
          sm[(y % C::ROWS) * C::M + x] = e;
      });
    });
  });
}

template <class C, int J>
__device__ __forceinline__ void xch_load(float2 (&v)[C::V], const float2* sm, int t) {
  using P = PassShape<C, J>;
  t = opaque(t);
  static_for<0, P::Q>([&](auto qq) {
    constexpr int q = decltype(qq)::value;
    int py, px;
    C::template base<J>(t, q, py, px);
    static_for<0, P::RY>([&](auto aa) {
      constexpr int a = decltype(aa)::value;
      int y = py + a * P::SY;
      if constexpr (C::CL > 1) y = J == 0 ? C::ROWS + y % 2 * 8 + y / 16 : y % C::ROWS;
      static_for<0, P::RX>([&](auto bb) {
        constexpr int b = decltype(bb)::value;
        v[q * P::G + a * P::RX + b] = sm[y * C::M + C::swz(px + b * P::SX)];
      });
    });
  });
}

template <class C>
__host__ __device__ constexpr int tw1_stride() {  // float2; odd in 16-byte units: the classes fall on different banks
  return C::ry(1) * C::rx(1) + 2;
}

// 8 complex values of the thread's tensor-memory row from word `word` on.
__device__ __forceinline__ void tmem_factors8(uint32_t taddr, float2 (&w)[8]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
#pragma unroll
  for (int i = 0; i < 8; ++i) w[i] = make_float2(__uint_as_float(r[2 * i]), __uint_as_float(r[2 * i + 1]));
}

// 16 of them.
__device__ __forceinline__ void tmem_factors16(uint32_t taddr, float2 (&w)[16]) {
  float2* p = w;
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n\ttcgen05.wait::ld.sync.aligned;"
      : "=f"(p[0].x), "=f"(p[0].y), "=f"(p[1].x), "=f"(p[1].y), "=f"(p[2].x), "=f"(p[2].y), "=f"(p[3].x),
        "=f"(p[3].y), "=f"(p[4].x), "=f"(p[4].y), "=f"(p[5].x), "=f"(p[5].y), "=f"(p[6].x), "=f"(p[6].y),
        "=f"(p[7].x), "=f"(p[7].y), "=f"(p[8].x), "=f"(p[8].y), "=f"(p[9].x), "=f"(p[9].y), "=f"(p[10].x),
        "=f"(p[10].y), "=f"(p[11].x), "=f"(p[11].y), "=f"(p[12].x), "=f"(p[12].y), "=f"(p[13].x), "=f"(p[13].y),
        "=f"(p[14].x), "=f"(p[14].y), "=f"(p[15].x), "=f"(p[15].y)
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_factors(uint32_t a, float2 (&w)[8]) { tmem_factors8(a, w); }
__device__ __forceinline__ void tmem_factors(uint32_t a, float2 (&w)[16]) { tmem_factors16(a, w); }

// All V complex values of the thread's tensor-memory words [word, word + 2V):
// issued here, usable after tmem_factors_wait.
__device__ __forceinline__ void tmem_factors_issue(uint32_t taddr, float2 (&w)[32]) {
  static_for<0, 2>([&](auto hh) {
    constexpr int h = decltype(hh)::value;
    float2* p = w + 16 * h;
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=f"(p[0].x), "=f"(p[0].y), "=f"(p[1].x), "=f"(p[1].y), "=f"(p[2].x), "=f"(p[2].y), "=f"(p[3].x),
          "=f"(p[3].y), "=f"(p[4].x), "=f"(p[4].y), "=f"(p[5].x), "=f"(p[5].y), "=f"(p[6].x), "=f"(p[6].y),
          "=f"(p[7].x), "=f"(p[7].y), "=f"(p[8].x), "=f"(p[8].y), "=f"(p[9].x), "=f"(p[9].y), "=f"(p[10].x),
          "=f"(p[10].y), "=f"(p[11].x), "=f"(p[11].y), "=f"(p[12].x), "=f"(p[12].y), "=f"(p[13].x), "=f"(p[13].y),
          "=f"(p[14].x), "=f"(p[14].y), "=f"(p[15].x), "=f"(p[15].y)
        : "r"(taddr + 32 * h));
  });
}
__device__ __forceinline__ void tmem_factors_wait(float2 (&w)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+f"(w[0].x), "+f"(w[0].y), "+f"(w[1].x), "+f"(w[1].y), "+f"(w[2].x), "+f"(w[2].y), "+f"(w[3].x),
                 "+f"(w[3].y), "+f"(w[4].x), "+f"(w[4].y), "+f"(w[5].x), "+f"(w[5].y), "+f"(w[6].x), "+f"(w[6].y),
                 "+f"(w[7].x), "+f"(w[7].y), "+f"(w[8].x), "+f"(w[8].y), "+f"(w[9].x), "+f"(w[9].y), "+f"(w[10].x),
                 "+f"(w[10].y), "+f"(w[11].x), "+f"(w[11].y), "+f"(w[12].x), "+f"(w[12].y), "+f"(w[13].x),
                 "+f"(w[13].y), "+f"(w[14].x), "+f"(w[14].y), "+f"(w[15].x), "+f"(w[15].y));
  asm volatile("" : "+f"(w[16].x), "+f"(w[16].y), "+f"(w[17].x), "+f"(w[17].y), "+f"(w[18].x), "+f"(w[18].y),
                    "+f"(w[19].x), "+f"(w[19].y), "+f"(w[20].x), "+f"(w[20].y), "+f"(w[21].x), "+f"(w[21].y),
                    "+f"(w[22].x), "+f"(w[22].y), "+f"(w[23].x), "+f"(w[23].y), "+f"(w[24].x), "+f"(w[24].y),
                    "+f"(w[25].x), "+f"(w[25].y), "+f"(w[26].x), "+f"(w[26].y), "+f"(w[27].x), "+f"(w[27].y),
                    "+f"(w[28].x), "+f"(w[28].y), "+f"(w[29].x), "+f"(w[29].y), "+f"(w[30].x), "+f"(w[30].y),
                    "+f"(w[31].x), "+f"(w[31].y));
}
template <bool CONJ, int FIRST_STEP>
__device__ __forceinline__ void mul_factors(float2 (&v)[32], const float2 (&w)[32]) {
  static_for<0, 32>([&](auto ee) {
    constexpr int e = decltype(ee)::value;
    if constexpr (e % FIRST_STEP != 0 || FIRST_STEP == 1) v[e] = pmul_opt<CONJ>(v[e], w[e]);
  });
}

// One radix pass on the registers.  Forward: DFT over digit J of y (for every
// x element), DFT over digit J of x (for every y element), then the twiddle
// w_M^(ey*a' + ex*b') that couples digit J to the lower digits.  Inverse: the
// conjugate twiddle, then the inverse DFTs (exact inverse up to the factor RY*RX).
template <class C, int J, bool INV>
__device__ __forceinline__ void pass_dft(float2 (&v)[C::V]) {
  using P = PassShape<C, J>;
  static_for<0, P::Q>([&](auto qq) {
    constexpr int o = decltype(qq)::value * P::G;
    static_for<0, P::RX>([&](auto bb) {
      constexpr int b = decltype(bb)::value;
      dft_at<P::RY, INV, o + b, P::RX>(v);
    });
    static_for<0, P::RY>([&](auto aa) {
      constexpr int a = decltype(aa)::value;
      dft_at<P::RX, INV, o + a * P::RX, 1>(v);
    });
  });
}

template <class C, int J, bool INV>
__device__ __forceinline__ void pass_compute(float2 (&v)[C::V], const Factors& f, int t) {
  using P = PassShape<C, J>;
  t = opaque(t);
  auto twiddle = [&]() {
    if constexpr (J == 0) {
      static_for<0, C::V / C::TWB>([&](auto cc) {
        constexpr int c = decltype(cc)::value;
        float2 w[C::TWB];
        tmem_factors(f.tmem + 2 * C::TWB * c, w);
        static_for<0, C::TWB>([&](auto ii) {
          constexpr int e = C::TWB * c + decltype(ii)::value;
          if constexpr (e % P::G != 0) v[e] = pmul_opt<INV>(v[e], w[e % C::TWB]);
        });
      });
    } else if constexpr (J == 1) {
      static_for<0, P::Q>([&](auto qq) {
        constexpr int q = decltype(qq)::value;
        int py, px;
        C::template base<1>(t, q, py, px);
        const float4* row =
            reinterpret_cast<const float4*>(f.tw1 + ((py & (P::SY - 1)) * P::SX + (px & (P::SX - 1))) * tw1_stride<C>());
        static_for<0, P::G / 2>([&](auto ee) {
          constexpr int e = 2 * decltype(ee)::value;
          const float4 w = row[e / 2];
          if constexpr (e != 0) v[q * P::G + e] = pmul_opt<INV>(v[q * P::G + e], make_float2(w.x, w.y));
          v[q * P::G + e + 1] = pmul_opt<INV>(v[q * P::G + e + 1], make_float2(w.z, w.w));
        });
      });
    }
  };
  if constexpr (INV) twiddle();
  pass_dft<C, J, INV>(v);
  if constexpr (!INV) twiddle();
}

// registers in pass-0 grouping (natural storage) -> unnormalised forward DFT,
// registers in pass-2 grouping (digit-reversed storage).  The cluster's blocks
// have registers to spare and only one warp per scheduler to hide latency, so
// there the pass-0 twiddles are fetched whole while the wave is transformed.
template <class C>
__device__ __forceinline__ void fft_fwd(float2 (&v)[C::V], float2* sm, Factors& f, int t) {
  if constexpr (C::CL > 1) {
    float2 w[C::V];
    tmem_factors_issue(f.tmem, w);
    pass_dft<C, 0, false>(v);
    tmem_factors_wait(w);
    mul_factors<false, PassShape<C, 0>::G>(v, w);
  } else {
    pass_compute<C, 0, false>(v, f, t);
  }
  xch_store<C, 0, true>(v, sm, f, t);
  C::arrived(f, 0);
  C::turn_wait(t);
  xch_load<C, 1>(v, sm, t);
  C::turn_pass(t);
  pass_compute<C, 1, false>(v, f, t);
  xch_store<C, 1, false>(v, sm, f, t);
  C::sync12(t);
  xch_load<C, 2>(v, sm, t);
  pass_compute<C, 2, false>(v, f, t);
}

// exact reverse of fft_fwd: unnormalised inverse DFT (times M*M relative to
// the true inverse), registers back in pass-0 grouping
template <class C>
__device__ __forceinline__ void fft_inv(float2 (&v)[C::V], float2* sm, Factors& f, int t) {
  pass_compute<C, 2, true>(v, f, t);
  xch_store<C, 2, false>(v, sm, f, t);
  C::sync12(t);
  xch_load<C, 1>(v, sm, t);
  pass_compute<C, 1, true>(v, f, t);
  xch_store<C, 1, true>(v, sm, f, t);
  if constexpr (C::CL > 1) {
    float2 w[C::V];
    tmem_factors_issue(f.tmem, w);
    C::arrived(f, 1);
    xch_load<C, 0>(v, sm, t);
    tmem_factors_wait(w);
    mul_factors<true, PassShape<C, 0>::G>(v, w);
    pass_dft<C, 0, true>(v);
  } else {
    C::arrived(f, 1);
    C::turn_wait(t);
    xch_load<C, 0>(v, sm, t);
    C::turn_pass(t);
    pass_compute<C, 0, true>(v, f, t);
  }
}

// Multiply the spectrum (pass-2 grouping) by the propagator h(ky, kx) / M^2 or
// its conjugate.
template <class C, bool CONJ>
__device__ __forceinline__ void mul_prop(float2 (&v)[C::V], const Factors& f) {
  if constexpr (C::CL > 1) {
    float2 w[C::V];
    tmem_factors_issue(f.tmem + 2 * C::V, w);
    tmem_factors_wait(w);
    mul_factors<CONJ, 1>(v, w);
    return;
  }
  static_for<0, C::V / C::TWB>([&](auto cc) {
    constexpr int c = decltype(cc)::value;
    float2 w[C::TWB];
    tmem_factors(f.tmem + 2 * C::V + 2 * C::TWB * c, w);
    static_for<0, C::TWB>([&](auto ii) {
      constexpr int e = C::TWB * c + decltype(ii)::value;
      v[e] = pmul_opt<CONJ>(v[e], w[e % C::TWB]);
    });
  });
}

// Fill the block's factors from the twiddle table tw[M] and the propagator
// table h2[M][M] (global memory; with_h = false leaves the propagator out).
// The caller synchronises the block before tw1 is read; the tensor-memory
// words are read back only by the thread's own warp.
template <class C>
__device__ __forceinline__ void fill_factors(uint32_t taddr, float2* tw1, const float2* __restrict__ tw,
                                             const float2* __restrict__ h2, bool with_h, int t) {
  {  // (each block of a cluster keeps the whole table)
    using P = PassShape<C, 1>;
    constexpr int EY = C::M / (P::RY * P::SY), EX = C::M / (P::RX * P::SX);
    for (int k = t % C::TB; k < P::SY * P::SX * P::G; k += C::TB) {
      const int cls = k / P::G, e = k % P::G;
      const int ex = EY * (cls / P::SX) * (e / P::RX) + EX * (cls % P::SX) * (e % P::RX);
      tw1[cls * tw1_stride<C>() + e] = __ldg(tw + (ex & (C::M - 1)));
    }
  }
  auto put = [&](uint32_t addr, const float2 (&w)[8]) {
    uint32_t r[16];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      r[2 * i] = __float_as_uint(w[i].x);
      r[2 * i + 1] = __float_as_uint(w[i].y);
    }
    tc::tmem_st16(addr, r);
  };
  static_for<0, C::V / 8>([&](auto cc) {
    constexpr int c = decltype(cc)::value;
    using P = PassShape<C, 0>;
    float2 w[8];
    static_for<0, 8>([&](auto ii) {
      constexpr int i = decltype(ii)::value, e = 8 * c + i, q = e / P::G, a = e % P::G / P::RX, b = e % P::RX;
      int py, px;
      C::template base<0>(t, q, py, px);
      constexpr int EY = C::M / (P::RY * P::SY), EX = C::M / (P::RX * P::SX);
      w[i] = __ldg(tw + ((EY * (py & (P::SY - 1)) * a + EX * (px & (P::SX - 1)) * b) & (C::M - 1)));
    });
    put(taddr + 16 * c, w);
  });
  if (with_h)
    static_for<0, C::V / 8>([&](auto cc) {
      constexpr int c = decltype(cc)::value;
      using P = PassShape<C, 2>;
      float2 w[8];
      static_for<0, 8>([&](auto ii) {
        constexpr int i = decltype(ii)::value, e = 8 * c + i, q = e / P::G, a = e % P::G / P::RX, b = e % P::RX;
        int py, px;
        C::template base<2>(t, q, py, px);
        const int ky = freq_y<C>(py) + C::ry(0) * C::ry(1) * a, kx = freq_x<C>(px) + C::rx(0) * C::rx(1) * b;
        w[i] = __ldg(h2 + ky * C::M + kx);
      });
      put(taddr + 2 * C::V + 16 * c, w);
    });
  tc::tmem_wait_st();
}

}  // namespace ptycho
