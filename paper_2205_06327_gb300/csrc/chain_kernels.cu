// Per-position multislice chain: forward model G (Sec. II-B), amplitude
// residual of Eq. 1 and the exact adjoint back to the slices and the probe
// (the per-position term of Eq. 2, Sec. III).
//
// One thread block owns one probe position for its whole slice chain; the
// wave never leaves the SM between slices.  Per slice s the forward pass
// multiplies by the object window O_s[y_i:y_i+M, x_i:x_i+M] (read straight
// from global memory, L2-resident) and, if s < S-1, propagates by
// FFT -> x h -> IFFT.  The exit wave is transformed to the detector; the
// residual gives the loss term and the seed of the adjoint, which runs the
// chain backwards with conjugated factors.
//
// Gradient mode writes, per position, the wave entering every slice s >= 1
// and the gradient w.r.t. every slice's exit wave (streaming stores); the
// object gradient conj(psi_s) * g_phi_s is formed and summed per object tile
// by the deterministic owner-computes reduction in reduce_kernels.cu.
//
// Recompute mode (checkpoint every L slices, K = ceil(S / L) segments) runs
// as K launches so that the workspace does not hold a patch per slice: the
// first (MODE_GRAD_RC) runs the forward model keeping only the checkpoints
// entering segments 1..K-2 and the waves of the last segment, then the
// residual and the adjoint through the last segment, writing its finished
// gradient patches conj(psi_s) g_phi_s over those waves and parking the
// adjoint state.  Each later launch (MODE_RC_SEG, segment j = K-2 .. 0)
// rebuilds segment j's waves from its checkpoint (or the probe) with the
// forward model's exact operations, runs the adjoint through the segment from
// the parked state and parks the state again (segment 0: the probe gradient).
// The host accumulates each segment's patches into the object gradient
// before the next launch overwrites them.
#include "bounds.h"
#include "fft2d.cuh"
#include "internal.h"
#include "../../include/ptycho.h"

namespace ptycho {

static_assert(kWaitExpired == PTYCHO_ERR_TIMEOUT, "the cluster's expired wait reports the library's code");

namespace {

// Elementwise over the pass-0 grouping (natural order), element (py, px).
template <class C, class F>
__device__ __forceinline__ void for_p0(int t, F&& f) {
  using P = PassShape<C, 0>;
  t = opaque(t);
  static_for<0, P::Q>([&](auto qq) {
    constexpr int q = decltype(qq)::value;
    int py0, px0;
    C::template base<0>(t, q, py0, px0);
    static_for<0, P::RY>([&](auto aa) {
      constexpr int a = decltype(aa)::value;
      static_for<0, P::RX>([&](auto bb) {
        constexpr int b = decltype(bb)::value;
        f(q * P::G + a * P::RX + b, py0 + a * P::SY, px0 + b * P::SX);
      });
    });
  });
}

// Elementwise over the pass-2 grouping (spectrum), frequency (ky, kx).
template <class C, class F>
__device__ __forceinline__ void for_p2(int t, F&& f) {
  using P = PassShape<C, 2>;
  t = opaque(t);
  static_for<0, P::Q>([&](auto qq) {
    constexpr int q = decltype(qq)::value;
    int py, px;
    C::template base<2>(t, q, py, px);
    const int ky0 = freq_y<C>(py), kx0 = freq_x<C>(px);
    static_for<0, P::RY>([&](auto aa) {
      constexpr int a = decltype(aa)::value;
      static_for<0, P::RX>([&](auto bb) {
        constexpr int b = decltype(bb)::value;
        f(q * P::G + a * P::RX + b, ky0 + C::ry(0) * C::ry(1) * a, kx0 + C::rx(0) * C::rx(1) * b);
      });
    });
  });
}

__device__ __forceinline__ float2 ldg2(const float2* p) { return __ldg(p); }

// Recompute mode's finished patches are read once, by the accumulation that
// follows each launch: streaming stores.
__device__ __forceinline__ void store_patch(float2* p, float2 v) { __stcs(p, v); }

}  // namespace


template <int M, int MODE>
__global__ void __launch_bounds__(Cfg<M>::T, Cfg<M>::MIN_BLOCKS) k_chain(const ChainArgs a) {
  using C = std::conditional_t<MODE == MODE_FORWARD || MODE == MODE_LOSS, HalfFetch<Cfg<M>>, Cfg<M>>;
  const int il = blockIdx.x, t = threadIdx.x;
#include "chain_body.inc"
}

// Few positions (Algorithm 1's per-location update, small batches, the last
// partial wave of a chunk): one position per cluster of 8 blocks.  On one SM
// its 16 warps take turns, 4 per scheduler, while most SMs idle; on 8 SMs each
// warp has a scheduler to itself and what is left is the latency of a transform
// (about 2.3 us, 4700 clocks).  Exchanges by cluster barriers and plain remote
// stores took 184 us for one position of 16 slices, stores counted on the
// receiver's mbarrier 168 us.
template <int MODE>
__global__ void __cluster_dims__(ClusterCfg128::CL, 1, 1) __launch_bounds__(ClusterCfg128::TB, 4)
    k_chain_cluster(const ChainArgs a) {
  using C = ClusterCfg128;
  constexpr int M = C::M;
  const int il = blockIdx.x / C::CL, t = (blockIdx.x % C::CL) * C::TB + threadIdx.x;
#include "chain_body.inc"
}

// Several problems' chunks in one launch (the batched workload): block b runs
// position b - start[p] of problem p's chunk, start[p] <= b < start[p + 1].
template <int M>
__global__ void __launch_bounds__(Cfg<M>::T, Cfg<M>::MIN_BLOCKS)
    k_chain_multi(const __grid_constant__ MultiChainArgs m) {
  constexpr int MODE = MODE_GRAD;
  __shared__ ChainArgs sa;
  const int b = blockIdx.x;
  int p = 0;
  while (p + 1 < m.n && b >= m.start[p + 1]) ++p;
  if (threadIdx.x == 0) sa = m.a[p];
  __syncthreads();
  const ChainArgs& a = sa;
  using C = Cfg<M>;
  const int il = b - m.start[p], t = threadIdx.x;
#include "chain_body.inc"
}

int chain_threads(int M) { return M == 128 ? Cfg<128>::T : Cfg<64>::T; }

// The exchange buffer, the pass-1 twiddle table, the loss partials of the
// position's warps and the tensor-memory address.
//
// A cluster's block holds tensor memory while it waits for the other blocks of
// its cluster, and the allocation waits without limit.  If more of them were
// resident on an SM than its tensor memory serves, two clusters could each hold
// columns that the other one's blocks wait for, for ever.  Registers (218 to
// 241 a thread) happen to allow four blocks; shared memory makes it certain,
// also for launches of several streams together.
template <class C>
static constexpr size_t chain_smem() {
  const size_t need = (C::kSmemWave + 16 * (size_t)tw1_stride<C>()) * sizeof(float2) +
                      (C::T / 32 + 1) * sizeof(double) + (C::CL > 1 ? 2 * sizeof(uint64_t) : 0);
  return C::CL > 1 ? smem_for_at_most(kTmemColumns / kTmemTake<C>, need) : need;
}
static_assert(chain_smem<ClusterCfg128>() <= 48 << 10, "a launch may ask for it without raising the kernel's limit");

size_t chain_smem_bytes(int M) { return M == 128 ? chain_smem<Cfg<128>>() : chain_smem<Cfg<64>>(); }

template <int M>
static cudaError_t prepare_m() {
  const int bytes = (int)chain_smem_bytes(M);
  cudaError_t e;
  if ((e = cudaFuncSetAttribute(k_chain<M, MODE_FORWARD>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes)) != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(k_chain<M, MODE_LOSS>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes)) != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(k_chain<M, MODE_GRAD_RC>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes)) != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(k_chain<M, MODE_RC_SEG>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes)) != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(k_chain_multi<M>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes)) != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_chain<M, MODE_GRAD>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

cudaError_t chain_prepare(int M) { return M == 128 ? prepare_m<128>() : prepare_m<64>(); }

int chain_blocks_per_sm(int M) {
  int n = 0;
  const cudaError_t e =
      M == 128 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_chain<128, MODE_GRAD>, Cfg<128>::T,
                                                               chain_smem_bytes(128))
               : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_chain<64, MODE_GRAD>, Cfg<64>::T,
                                                               chain_smem_bytes(64));
  return e == cudaSuccess ? n : 0;
}

template <int M>
static cudaError_t launch_m(ChainMode mode, const ChainArgs& a, cudaStream_t st) {
  const dim3 grid(a.n_pos), block(Cfg<M>::T);
  const size_t smem = chain_smem_bytes(M);
  switch (mode) {
    case MODE_FORWARD: return launch_after(k_chain<M, MODE_FORWARD>, grid, block, smem, st, a);
    case MODE_LOSS: return launch_after(k_chain<M, MODE_LOSS>, grid, block, smem, st, a);
    case MODE_GRAD_RC: return launch_after(k_chain<M, MODE_GRAD_RC>, grid, block, smem, st, a);
    case MODE_RC_SEG: return launch_after(k_chain<M, MODE_RC_SEG>, grid, block, smem, st, a);
    default: return launch_after(k_chain<M, MODE_GRAD>, grid, block, smem, st, a);
  }
}

static cudaError_t launch_cluster(ChainMode mode, const ChainArgs& a, cudaStream_t st) {
  using C = ClusterCfg128;
  const dim3 grid(a.n_pos * C::CL), block(C::TB);
  const size_t smem = chain_smem<C>();
  switch (mode) {
    case MODE_FORWARD: return launch_after(k_chain_cluster<MODE_FORWARD>, grid, block, smem, st, a);
    case MODE_LOSS: return launch_after(k_chain_cluster<MODE_LOSS>, grid, block, smem, st, a);
    case MODE_GRAD_RC: return launch_after(k_chain_cluster<MODE_GRAD_RC>, grid, block, smem, st, a);
    case MODE_RC_SEG: return launch_after(k_chain_cluster<MODE_RC_SEG>, grid, block, smem, st, a);
    default: return launch_after(k_chain_cluster<MODE_GRAD>, grid, block, smem, st, a);
  }
}

// Does a launch take the cluster kernel?  Results are the same bit for bit, so
// this is where it is the faster one.  us of an evaluation, one block / one
// cluster per position: 16 slices, 1 position 332 / 198, 24 352 / 248, 40 358 /
// 297, 48 362 / 332 (76: the chain alone 312 / 520, as the blocks of different
// positions compete); 48 positions of 4 slices 128 / 123, of 3 109 / 109; forward
// model of 16 slices, 48 positions 137 / 134.  Gradients of one or two slices
// have few exchanges to win by: 2 slices, 16 positions 77 / 74, 32 91 / 92, 48 90
// / 94; one slice, 48 positions 65 / 68.
// As a chunk's tail it takes SMs from the accumulation of the chunk's `beside`
// full waves, which runs at the same time, the more the longer that lasts: 16
// slices, 152 + 48 positions 693 / 660, 304 + 32 1022 / 982, 304 + 48 1029 /
// 1063, 456 + 16 1386 / 1348, 456 + 48 1362 / 1477, 608 + 16 1708 / 1740; 8
// slices, 152 + 32 380 / 360, 152 + 48 385 / 401; 4 slices, 152 + 16 219 / 209,
// 304 + 16 317 / 323; 2 slices, 152 + 8 142 / 148.
bool cluster_faster(ChainMode mode, const ChainArgs& a, int beside) {
  int most = 48;
  if (beside > 0)
    most = a.S < 4 ? 0 : (a.S < 12 ? 4 * a.S : 48) - 16 * (beside - 1);
  else if (mode != MODE_FORWARD && mode != MODE_LOSS && a.S < 3)
    most = a.S == 2 ? 16 : 0;
  return a.n_pos <= most;
}

cudaError_t launch_chain(int M, ChainMode mode, const ChainArgs& a, cudaStream_t st, int beside) {
  if (a.n_pos <= 0) return cudaSuccess;
  if (M == 128 && cluster_faster(mode, a, beside)) return launch_cluster(mode, a, st);
  return M == 128 ? launch_m<128>(mode, a, st) : launch_m<64>(mode, a, st);
}

cudaError_t launch_chain_multi(int M, const MultiChainArgs& m, cudaStream_t st) {
  if (m.n < 0 || m.n > kMultiChainMax) return cudaErrorInvalidValue;
  if (m.n == 0 || m.start[m.n] <= 0) return cudaSuccess;
  const dim3 grid(m.start[m.n]), block(chain_threads(M));
  const size_t smem = chain_smem_bytes(M);
  return M == 128 ? launch_after(k_chain_multi<128>, grid, block, smem, st, m)
                  : launch_after(k_chain_multi<64>, grid, block, smem, st, m);
}

}  // namespace ptycho
