// Deterministic reductions: the object gradient as an owner-computes tiled
// accumulation (the one-GPU form of the image-gradient decomposition of
// Sec. III), the probe gradient, the FP64 loss, and the small vector kernels
// of the gradient-descent step.
//
// Object gradient (Eq. 2 with the locality of Sec. III): slice s of dF/dO is
// sum_i conj(psi_{i,s}) * g_phi_{i,s} placed at window i.  The object is
// tessellated into tiles; one block owns one (tile, slice), walks the
// positions whose window meets its tile in ascending order and sums their
// contributions on chip.  Every output pixel therefore has exactly one
// writer and a fixed summation order: no atomics, bit-reproducible.
#include "internal.h"
#include "../../include/ptycho.h"

namespace ptycho {

namespace {

constexpr int kAccThreads = 256;
constexpr int kAccWarps = kAccThreads / 32;
constexpr int kAccDefaultCols = 512;
constexpr int kAccMaxCols = 1024;
constexpr int kAccBatch = 4 * kAccThreads;  // positions listed at a time
constexpr int kSmCount = 152;               // of the GPU this is built for

// float2 a warp's row takes per column parity
__host__ __device__ constexpr int acc_half(int tile_w) { return tile_w / 2 + 1; }

template <int VEC>
struct AccVec;
template <>
struct AccVec<2> {
  using type = float4;
  static __device__ __forceinline__ float4 zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }
  static __device__ __forceinline__ float2 get(const float4& v, int i) {
    return i ? make_float2(v.z, v.w) : make_float2(v.x, v.y);
  }
};
template <>
struct AccVec<1> {
  using type = float2;
  static __device__ __forceinline__ float2 zero() { return make_float2(0.f, 0.f); }
  static __device__ __forceinline__ float2 get(const float2& v, int) { return v; }
};

// The probe need not be 16-byte aligned (8 bytes are asked of the caller).
template <int VEC>
__device__ __forceinline__ typename AccVec<VEC>::type probe_load(const float2* p) {
  if constexpr (VEC == 2) {
    const float2 u = __ldg(p), v = __ldg(p + 1);
    return make_float4(u.x, u.y, v.x, v.y);
  } else {
    return __ldg(p);
  }
}

// One block owns one (tile, slice) and each of its 8 warps one row of the
// tile: the row's sums live in shared memory and only that warp touches them.
// The warp walks the positions whose window covers its row in ascending order
// and streams that window row of psi and g_phi, VEC pixels per lane and step
// (16-byte loads for even windows), K steps per position, with the loads of
// groups of U positions in flight before they are added.
//
// The kernel is bound by HBM: it reads the two workspace arrays once.  With
// threads tied to the pixels of a 32 x 32 tile, a third of the loads fell
// outside the window and the rest came in 256-byte pieces of rows 1 KB apart.
// Here lanes follow the window, so a full row keeps every lane busy, and
// neighbouring warps read neighbouring rows of the same windows.  Measured
// (tile 32 x 32 -> bands): 576 positions, M = 128, 16 slices 876 -> 620 us (both
// parts, one beside the chain's last wave); 225 positions, M = 192, 12 slices
// 362 -> 238 us (6.7 TB/s); 930 positions, M = 96 499 -> 338 us; finished
// patches of 3600 positions, M = 128, 30 slices 4.72 -> 3.43 ms.  Fewer loads
// in flight with more blocks per SM (half of them, 4 blocks) gave 721 / 276 /
// 451 us; 8 steps instead of 16 for finished patches 4.02 ms.
template <int K, int VEC, bool PATCH>
__global__ void __launch_bounds__(kAccThreads, 2) k_accum_obj_grad(const AccumArgs a) {
  using V = AccVec<VEC>;
  using vec = typename V::type;
  // Two groups of loads in turn, one in flight while the other is added, or one
  // twice as large.  ncu on the latter (patches, M = 128): waiting for loads is
  // half of all stalls at 4 TB/s.  One group / two: 4560 patches of 30 slices,
  // M = 128 (K = 2) 4.49 / 3.20 ms, M = 64 (K = 1) 0.93 / 1.06 ms; waves of 930
  // positions, M = 96 (K = 2) 311 / 274 us, 576 at 128 606 / 593, 225 at 192 (K =
  // 3) 235 / 234, 4 at 1024 (K = 8) 81 / 111.
  constexpr bool PIPE = PATCH ? K >= 2 : K <= 3;
  constexpr int STEPS = PIPE ? (PATCH ? 8 : 4) : (PATCH ? 16 : 8), U = STEPS / K > 0 ? STEPS / K : 1;
  struct Group {  // positions whose loads are in flight together
    vec g[U][K];
    vec p[PATCH ? 1 : U][PATCH ? 1 : K];
    int cx[U], lo[U], hi[U];  // tile column of window column 0; window columns [lo, hi) of the segment
  };
  __shared__ int2 lpos[kAccBatch];
  __shared__ int lidx[kAccBatch];
  __shared__ int wcount[kAccWarps];
  extern __shared__ float2 acc[];  // [8][2 acc_half(tile_w)]: a row's even columns, then its odd ones
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  dependency_wait();
  const int z = blockIdx.x % a.n_slices, b = blockIdx.x / a.n_slices;  // slice s_begin + z
  const int s = a.s_begin + z;
  const int M = a.M;
  // Blocks in launch order: slices, then tile columns, then tile rows from
  // the middle outwards (the middle rows, which most windows cover, first).
  const int nc = (a.W + a.tile_w - 1) / a.tile_w, nr = (a.H + kAccWarps - 1) / kAccWarps;
  const int rank = b / nc;
  const int ty0 = kAccWarps * (nr / 2 + (rank % 2 ? -(rank + 1) / 2 : rank / 2));
  const int tx0 = a.tile_w * (b % nc);
  const int th = min(kAccWarps, a.H - ty0), tw = min(a.tile_w, a.W - tx0);
  const int y = ty0 + w;                  // this warp's object row (if w < th)
  // Lanes that hold pairs of pixels touch every other column at a time: with
  // the columns apart by parity no bank idles (finished patches of 16632
  // positions, 30 slices: 18.8 -> 17.7 ms).
  const int half = acc_half(a.tile_w);
  float2* arow = acc + w * 2 * half;
  auto at = [&](int x) { return VEC == 2 ? (x & 1) * half + (x >> 1) : x; };
  const size_t MM = (size_t)M * M;
  const float2* gphi_s = a.ws_gphi + (size_t)(a.seg_slots ? z : s) * a.ws_n * MM;
  const float2* psi_s = s > 0 && !PATCH ? a.ws_psi + (size_t)(a.seg_slots ? z : s - 1) * a.ws_n * MM : nullptr;
  for (int x = lane; x < 2 * half; x += 32) arow[x] = make_float2(0.f, 0.f);

  for (int base = 0; base < a.n_pos; base += kAccBatch) {
    // Positions of this batch whose window meets the tile, in ascending order
    // (four consecutive positions per thread, block prefix sum).
    int2 r[4];
    unsigned hit = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int il = base + 4 * t + k;
      r[k] = il < a.n_pos ? a.pos[a.pos_begin + il] : make_int2(-1, -1);
      const bool ok = r[k].x >= 0 && r[k].y >= 0 && r[k].x <= a.H - M && r[k].y <= a.W - M;
      if (ok && r[k].x < ty0 + th && r[k].x + M > ty0 && r[k].y < tx0 + tw && r[k].y + M > tx0) hit |= 1u << k;
    }
    const int n = __popc(hit);
    int off = n;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, off, d);
      if (lane >= d) off += v;
    }
    __syncthreads();  // the previous batch's list is read
    if (lane == 31) wcount[w] = off;
    __syncthreads();
    int slot = off - n, total = 0;
#pragma unroll
    for (int k = 0; k < kAccWarps; ++k) {
      slot += k < w ? wcount[k] : 0;
      total += wcount[k];
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (hit >> k & 1) {
        lpos[slot] = r[k];
        lidx[slot++] = base + 4 * t + k;
      }
    __syncthreads();

    if (w >= th) continue;
    for (int sx0 = 0; sx0 < tw; sx0 += a.seg_w) {
      const int sx1 = min(tw, sx0 + a.seg_w);
      for (int j0 = 0; j0 < total; j0 += 32) {
        int2 rj = make_int2(0, 0);
        int ij = 0;
        bool in = false;
        if (j0 + lane < total) {
          rj = lpos[j0 + lane];
          ij = lidx[j0 + lane];
          in = rj.x <= y && y < rj.x + M && rj.y - tx0 < sx1 && rj.y - tx0 + M > sx0;
        }
        unsigned todo = __ballot_sync(0xffffffffu, in);
        // The next up to U of them: issue their loads.
        auto fetch = [&](Group& f) {
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const bool live = todo != 0;
            const int src = live ? __ffs(todo) - 1 : 0;
            todo &= todo - 1;
            const int ry = __shfl_sync(0xffffffffu, rj.x, src), rx = __shfl_sync(0xffffffffu, rj.y, src);
            const int i = __shfl_sync(0xffffffffu, ij, src);
            f.cx[u] = rx - tx0;
            f.lo[u] = max(0, sx0 - f.cx[u]);
            f.hi[u] = live ? min(M, sx1 - f.cx[u]) : 0;
            const size_t row_off = (size_t)i * MM + (size_t)(y - ry) * M;
            const float2* gp = gphi_s + row_off;
            const float2* pp = PATCH ? nullptr : s > 0 ? psi_s + row_off : a.probe + (size_t)(y - ry) * M;
            const int x0 = (f.lo[u] & ~(VEC - 1)) + VEC * lane;
#pragma unroll
            for (int k = 0; k < K; ++k) {
              const int x = x0 + 32 * VEC * k;
              const bool ld = x < f.hi[u];
              f.g[u][k] = ld ? __ldcs(reinterpret_cast<const vec*>(gp + x)) : V::zero();
              if constexpr (!PATCH)
                f.p[u][k] = !ld ? V::zero()
                                : s > 0 ? __ldcs(reinterpret_cast<const vec*>(pp + x)) : probe_load<VEC>(pp + x);
            }
          }
        };
        // Add them in order.
        auto add = [&](const Group& f) {
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int x0 = (f.lo[u] & ~(VEC - 1)) + VEC * lane;
#pragma unroll
            for (int e = 0; e < VEC; ++e) {
              // pixel (step k, e) is tile column cx + x0 + 32 VEC k + e (it may start at -1)
              float2* oe = arow + (VEC == 2 ? ((f.cx[u] + e) & 1) * half + ((f.cx[u] + x0 + e) >> 1) : f.cx[u] + x0);
#pragma unroll
              for (int k = 0; k < K; ++k) {
                const int x = x0 + 32 * VEC * k + e;
                if (x >= f.lo[u] && x < f.hi[u]) {
                  float2* o = oe + 32 * k;
                  float2 v = *o;
                  const float2 g = V::get(f.g[u][k], e);
                  if constexpr (PATCH) {  // finished patches conj(psi) g_phi
                    v.x += g.x;
                    v.y += g.y;
                  } else {
                    const float2 p = V::get(f.p[u][k], e);
                    v.x = fmaf(p.x, g.x, fmaf(p.y, g.y, v.x));
                    v.y = fmaf(p.x, g.y, fmaf(-p.y, g.x, v.y));
                  }
                  *o = v;
                }
              }
            }
            __syncwarp();  // the next position's lanes fall on other columns
          }
        };
        if constexpr (PIPE) {
          if (!todo) continue;
          Group f0, f1;
          fetch(f0);
          for (;;) {
            const bool more1 = todo != 0;
            if (more1) fetch(f1);
            add(f0);
            if (!more1) break;
            const bool more0 = todo != 0;
            if (more0) fetch(f0);
            add(f1);
            if (!more0) break;
          }
        } else {
          while (todo) {
            Group f;
            fetch(f);
            add(f);
          }
        }
      }
    }
  }
  __syncwarp();
  if (w >= th) return;
  float2* out = a.grad_obj + (size_t)s * a.H * a.W + (size_t)y * a.W + tx0;
  for (int x = lane; x < tw; x += 32) {
    float2 val = arow[at(x)];
    if (a.accumulate) {
      const float2 prev = out[x];
      val.x += prev.x;
      val.y += prev.y;
    }
    out[x] = val;
  }
}

// part[sp][pix] = sum over positions of split sp (ascending) of ws_gp[i][pix]
__global__ void k_probe_grad_part(const float2* __restrict__ ws_gp, int n_pos, int MM, int n_split,
                                  float2* __restrict__ part) {
  launch_dependents();
  dependency_wait();
  const int pix = blockIdx.x * blockDim.x + threadIdx.x;
  const int sp = blockIdx.y;
  if (pix >= MM) return;
  const int per = (n_pos + n_split - 1) / n_split;
  const int i0 = sp * per, i1 = min(n_pos, i0 + per);
  float2 acc = make_float2(0.f, 0.f);
  for (int i = i0; i < i1; ++i) {
    const float2 g = __ldcs(ws_gp + (size_t)i * MM + pix);
    acc.x += g.x;
    acc.y += g.y;
  }
  part[(size_t)sp * MM + pix] = acc;
}

// Fixed-order FP64 sum of n values into acc[0] (one block of 256 threads).
__device__ __forceinline__ void loss_sum(const double* __restrict__ part, int n, double* acc, int accumulate) {
  __shared__ double sh[256];
  const int t = threadIdx.x;
  double s = 0.0;
  for (int i = t; i < n; i += 256) s += part[i];
  sh[t] = s;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if (t < h) sh[t] += sh[t + h];
    __syncthreads();
  }
  if (t == 0) acc[0] = (accumulate ? acc[0] : 0.0) + sh[0];
}

__global__ void k_loss_accum(const double* __restrict__ part, int n, double* acc, int accumulate) {
  launch_dependents();
  dependency_wait();
  loss_sum(part, n, acc, accumulate);
}

// The end of an evaluation in one launch: the probe gradient's splits and, in
// one more block, the loss.  PER > 0 (splits of at most PER positions, few
// positions): sums the positions of each split here, in the order of
// k_probe_grad_part, so that its launch falls away too.
template <int PER>
__global__ void __launch_bounds__(256) k_probe_loss(const float2* __restrict__ src, int n, int MM,
                                                    float2* __restrict__ gp, const double* __restrict__ loss_part,
                                                    int n_loss, double* loss, int accumulate) {
  launch_dependents();
  dependency_wait();
  if (blockIdx.x == gridDim.x - 1) {
    loss_sum(loss_part, n_loss, loss, accumulate);
    return;
  }
  const int pix = blockIdx.x * 256 + threadIdx.x;
  if (pix >= MM) return;
  constexpr int U = 8, P = PER > 0 ? PER : 1;
  float2 acc = accumulate ? gp[pix] : make_float2(0.f, 0.f);
  for (int i0 = 0; i0 < n; i0 += U) {
    float2 g[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
      g[u] = i0 + u < n ? __ldcs(src + (size_t)(i0 + u) * MM + pix) : make_float2(0.f, 0.f);
#pragma unroll
    for (int u = 0; u < U; u += P) {
      float2 part = g[u];
#pragma unroll
      for (int k = 1; k < P; ++k) {
        part.x += g[u + k].x;
        part.y += g[u + k].y;
      }
      acc.x += part.x;
      acc.y += part.y;
    }
  }
  gp[pix] = acc;
}

// The update of a step in one launch: O += a_o dF/dO, P += a_p dF/dP, and for
// the delayed accumulation (ACC) acc += dF/dO and, with `flush`, the second
// update O += a_o acc, acc = 0.  No launch_dependents here: the next chain reads O
// and P through the read-only path (__ldg), so it must not start before they are
// written (8 per-location updates 1446 us with it, 1437 without; plain loads
// instead of read-only ones cost the chain 3 %).
template <bool ACC>
__global__ void __launch_bounds__(256) k_update(const UpdateArgs u) {
  dependency_wait();
  const size_t stride = (size_t)gridDim.x * 256;
  for (size_t i = blockIdx.x * (size_t)256 + threadIdx.x; i < u.n_obj; i += stride) {
    const float2 d = u.g_obj[i];
    float2 o = u.obj[i];
    o = make_float2(fmaf(u.a_obj, d.x, o.x), fmaf(u.a_obj, d.y, o.y));
    if constexpr (ACC) {
      float2 c = u.acc[i];
      c = make_float2(c.x + d.x, c.y + d.y);
      if (u.flush) {
        o = make_float2(fmaf(u.a_obj, c.x, o.x), fmaf(u.a_obj, c.y, o.y));
        c = make_float2(0.f, 0.f);
      }
      u.acc[i] = c;
    }
    u.obj[i] = o;
  }
  for (size_t i = blockIdx.x * (size_t)256 + threadIdx.x; i < u.n_probe; i += stride) {
    const float2 d = u.g_probe[i], p = u.probe[i];
    u.probe[i] = make_float2(fmaf(u.a_probe, d.x, p.x), fmaf(u.a_probe, d.y, p.y));
  }
}

// Sum of |x|^2 in FP64: per-block partials over a fixed index assignment.
__global__ void k_norm2_part(const float2* __restrict__ x, size_t n, double* part) {
  __shared__ double sh[256];
  const int t = threadIdx.x;
  double s = 0.0;
  for (size_t i = blockIdx.x * (size_t)256 + t; i < n; i += (size_t)gridDim.x * 256) {
    const float2 v = x[i];
    s += (double)v.x * v.x + (double)v.y * v.y;
  }
  sh[t] = s;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if (t < h) sh[t] += sh[t + h];
    __syncthreads();
  }
  if (t == 0) part[blockIdx.x] = sh[0];
}

// O = exp(i sigma V) for a real potential V (Sec. II-B's unknown).
__global__ void k_potential_to_transmission(const float* __restrict__ V, float2* __restrict__ O, float sigma,
                                            size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    float sn, cs;
    sincosf(sigma * V[i], &sn, &cs);
    O[i] = make_float2(cs, sn);
  }
}

// dF/dV = sigma * Im(conj(O) dF/dO) for O = exp(i sigma V), V real.
__global__ void k_potential_grad(const float2* __restrict__ O, const float2* __restrict__ g, float* __restrict__ gV,
                                 float sigma, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const float2 o = O[i], d = g[i];
    gV[i] = sigma * fmaf(o.x, d.y, -o.y * d.x);
  }
}

__global__ void k_check_positions(const int2* __restrict__ pos, int n, int M, int H, int W, int* status) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int2 r = pos[i];
  if (r.x < 0 || r.y < 0 || r.x > H - M || r.y > W - M) *status = PTYCHO_ERR_POSITION;
}

}  // namespace

namespace {

template <int K, int VEC>
cudaError_t accum_launch(const AccumArgs& a, dim3 grid, cudaStream_t st) {
  const size_t smem = (size_t)kAccWarps * 2 * acc_half(a.tile_w) * sizeof(float2);
  void (*const k)(AccumArgs) = a.patch_mode ? k_accum_obj_grad<K, VEC, true> : k_accum_obj_grad<K, VEC, false>;
  if (smem > 2 * acc_half(kAccDefaultCols) * kAccWarps * sizeof(float2)) {  // beyond the 48 KB every kernel may use
    const cudaError_t e =
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * acc_half(kAccMaxCols) * kAccWarps * (int)sizeof(float2));
    if (e != cudaSuccess) return e;
  }
  return launch_after(k, grid, kAccThreads, smem, st, a);
}

template <int VEC>
cudaError_t accum_steps(int steps, const AccumArgs& a, dim3 grid, cudaStream_t st) {
  switch (steps) {
    case 1: return accum_launch<1, VEC>(a, grid, st);
    case 2: return accum_launch<2, VEC>(a, grid, st);
    case 3: return accum_launch<3, VEC>(a, grid, st);
    case 4: return accum_launch<4, VEC>(a, grid, st);
    default: return accum_launch<8, VEC>(a, grid, st);
  }
}

}  // namespace

cudaError_t launch_accum_obj_grad(const AccumArgs& args, cudaStream_t st) {
  AccumArgs a = args;
  const int ns = a.n_slices > 0 ? a.n_slices : a.S - a.s_begin;
  if (a.s_begin < 0 || ns <= 0 || a.s_begin + ns > a.S) return cudaErrorInvalidValue;
  // Tiles are bands of 8 rows (one per warp).  Their columns: the whole width
  // (up to kAccDefaultCols), halved while that leaves fewer than three blocks
  // per SM and still covers a window; a plan's tile may ask for other columns,
  // at least a window's.  (Halving measured: 230 blocks 4.73 -> 3.43 ms for the
  // patches above, 385 blocks at M = 96 374 -> 338 us; 552 blocks at M = 192 238
  // -> 284 us.)
  if (a.tile_w == 0) {
    const int n = (a.W + kAccDefaultCols - 1) / kAccDefaultCols;
    a.tile_w = (a.W + n - 1) / n;
    auto blocks = [&]() { return (int64_t)ns * ((a.H + kAccWarps - 1) / kAccWarps) * ((a.W + a.tile_w - 1) / a.tile_w); };
    while (blocks() < 3 * kSmCount && (a.tile_w + 1) / 2 >= a.M) a.tile_w = (a.tile_w + 1) / 2;
  } else {
    const int least = a.M < a.W ? a.M : a.W;
    if (a.tile_w < least) a.tile_w = least;
    if (a.tile_w > kAccMaxCols) a.tile_w = kAccMaxCols;
  }
  // Window rows start on 16 bytes for even M (the workspace is aligned).
  const int vec = a.M % 2 == 0 ? 2 : 1, step = 32 * vec;
  a.seg_w = a.tile_w;
  if (a.M > 8 * step && a.tile_w + vec - 1 > 8 * step) a.seg_w = 8 * step - vec + 1;
  const int span = a.seg_w + vec - 1 < a.M ? a.seg_w + vec - 1 : a.M;
  const int steps = (span + step - 1) / step;
  a.n_slices = ns;
  const int64_t blocks = (int64_t)ns * ((a.W + a.tile_w - 1) / a.tile_w) * ((a.H + kAccWarps - 1) / kAccWarps);
  if (blocks > INT32_MAX) return cudaErrorInvalidValue;
  const dim3 grid((unsigned)blocks);
  return vec == 2 ? accum_steps<2>(steps, a, grid, st) : accum_steps<1>(steps, a, grid, st);
}

cudaError_t launch_probe_loss(const float2* ws_gp, int n_pos, int M, float2* part, int n_split, float2* grad_probe,
                              const double* loss_part, int n_loss, double* loss, int accumulate, int* n_launches,
                              cudaStream_t st) {
  const int MM = M * M, blocks = (MM + 255) / 256;
  *n_launches = 1;
  const float2* src = ws_gp;
  int n = n_pos;
  void (*k)(const float2*, int, int, float2*, const double*, int, double*, int) =
      n_pos <= n_split ? k_probe_loss<1> : n_pos <= 2 * n_split ? k_probe_loss<2> : k_probe_loss<0>;
  if (n_pos > 2 * n_split) {
    *n_launches = 2;
    const cudaError_t e =
        launch_after(k_probe_grad_part, dim3(blocks, n_split), 256, 0, st, ws_gp, n_pos, MM, n_split, part);
    if (e != cudaSuccess) return e;
    src = part;
    n = n_split;
  }
  return launch_after(k, blocks + 1, 256, 0, st, src, n, MM, grad_probe, loss_part, n_loss, loss, accumulate);
}

cudaError_t launch_loss_accum(const double* loss_part, int n, double* acc, int accumulate, cudaStream_t st) {
  return launch_after(k_loss_accum, 1, 256, 0, st, loss_part, n, acc, accumulate);
}

cudaError_t launch_update(const UpdateArgs& u, cudaStream_t st) {
  const size_t n = u.n_obj > u.n_probe ? u.n_obj : u.n_probe;
  if (n == 0) return cudaSuccess;
  const size_t blocks = (n + 255) / 256;
  const unsigned grid = (unsigned)(blocks < 4096 ? blocks : 4096);
  return launch_after(u.acc ? k_update<true> : k_update<false>, grid, 256, 0, st, u);
}

cudaError_t launch_norm2(const float2* x, size_t n, double* part, int n_part, double* out, int slot,
                         cudaStream_t st) {
  k_norm2_part<<<n_part, 256, 0, st>>>(x, n, part);
  k_loss_accum<<<1, 256, 0, st>>>(part, n_part, out + slot, 0);
  return cudaGetLastError();
}

cudaError_t launch_potential_to_transmission(const float* V, float2* O, double sigma, size_t n, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  const size_t blocks = (n + 255) / 256;
  k_potential_to_transmission<<<(unsigned)(blocks < 4096 ? blocks : 4096), 256, 0, st>>>(V, O, (float)sigma, n);
  return cudaGetLastError();
}

cudaError_t launch_potential_grad(const float2* O, const float2* g, float* gV, double sigma, size_t n,
                                  cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  const size_t blocks = (n + 255) / 256;
  k_potential_grad<<<(unsigned)(blocks < 4096 ? blocks : 4096), 256, 0, st>>>(O, g, gV, (float)sigma, n);
  return cudaGetLastError();
}

cudaError_t launch_check_positions(const int2* pos, int n, int M, int H, int W, int* status, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  k_check_positions<<<(n + 255) / 256, 256, 0, st>>>(pos, n, M, H, W, status);
  return cudaGetLastError();
}

}  // namespace ptycho
