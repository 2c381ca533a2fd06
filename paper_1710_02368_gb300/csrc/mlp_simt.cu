// Kernels (a) and (b) on CUDA cores: the batched-over-workers MLP forward and
// backward with the fused local SGD step and gradient accumulation of
// Algorithm 1 (g = grad L; theta_k -= eta g; a_k += g) for AGN_GEMM_SIMT and
// nets without a hidden layer; and, for either GEMM path, the softmax
// cross-entropy of output layers the output-layer kernels do not take.
//
// One launch covers every worker of a wave: grid.z indexes the wave's slots,
// and slot z reads and updates the replica of worker slot_worker[z].  All
// three GEMM shapes use one tiled kernel (square tiles, double-buffered k
// slices); the element type T is float (fp32 mode) or bf16 (bf16 mode:
// operands bf16, accumulation fp32, master weights fp32).  Every output is one
// chain of fused multiply-adds over k in ascending order from zero, whatever
// the tile, so that the tile never changes a result.
#include <algorithm>

#include "mlp.cuh"

namespace agn {

namespace {

constexpr int kThreads = 256;   // 16 x 16, kTile / 16 rows and columns each
constexpr int64_t kShortK = 48;   // k up to which 32-square tiles take slices of 16

template <typename T>
__device__ __forceinline__ float to_f(T v);
template <>
__device__ __forceinline__ float to_f<float>(float v) { return v; }
template <>
__device__ __forceinline__ float to_f<bf16>(bf16 v) { return __bfloat162float(v); }

template <typename T>
__device__ __forceinline__ T from_f(float v);
template <>
__device__ __forceinline__ float from_f<float>(float v) { return v; }
template <>
__device__ __forceinline__ bf16 from_f<bf16>(float v) { return __float2bfloat16_rn(v); }

// The low-precision copy of an updated weight: one bf16, or its three exact
// pieces (fp32 mode on tensor cores).
__device__ __forceinline__ void write_copy(bf16* tb, int64_t plane, int64_t p, float t) {
  if (plane > 0) {
    bf16 q0, q1, q2;
    split3(t, q0, q1, q2);
    AGN_ST(tb + p, q0);
    AGN_ST(tb + plane + p, q1);
    AGN_ST(tb + 2 * plane + p, q2);
  } else {
    AGN_ST(tb + p, __float2bfloat16_rn(t));
  }
}

// C[M x N] (+)= sum_k A(m, k) B(k, n) for one slot; see GemmArgs for layouts.
// Bound by a block's chain over k (small launches) or by shared-memory reads:
// the next k slice's global loads are in flight while the current one is
// multiplied out of shared memory.  Against one 64 x 64 tile, one buffer and
// 4-byte shared loads: a forward of 613-301-150-26 at 5 slots of 100 samples
// 31.1 -> 16.4 us, dX 15.8 -> 9.9, dW 46 -> 19 (its three launches in one); the
// 784-1000-1000 forward of 10000 rows 20 -> 26 TFLOP/s.  A thread's rows are consecutive (its A
// values come in 16-byte loads), its columns 16 apart (coalesced epilogues).
// (kShort: a 32-square tile with at most kShortK k.)
template <typename T, typename TO, bool kAKMajor, bool kBKMajor, int kEpi, int kTile, bool kShort>
__device__ __forceinline__ void gemm_simt_tile(const GemmArgs& g, int tile_x, int tile_y) {
  constexpr int kBM = kTile, kBN = kTile;
  // k per slice.  Small tiles wait on the next slice's loads: 64 (32: 5 % slower on
  // 613-301-150-26's forwards).  32 for the fp32 dX at 64 x 64 (784-1001-1001-10, 8
  // slots of 128: a pass 2.70 -> 2.56 ms); elsewhere 32 cost blocks an SM (bf16
  // 333-777-29, 16 slots of 200: 1.87 -> 2.05 ms).
  // Few k take slices of 16: the rest of a longer one would be multiplied zeros
  // (16-344-4, 17 slots, us a run of ten steps with slices of 64 and 16: one sample
  // 312 and 250, 33 samples 338 and 318; 333-165-40-7, 8 slots of 48: 554 and 558).
  constexpr int kBK = kTile == 32 ? (kShort ? 16 : 64)
                      : kTile == 64 && kEpi == kEpiDX && sizeof(T) == 4 ? 32 : 16;
  constexpr int kTM = kTile / 16, kTN = kTile / 16;
  constexpr int kLoads = kTile * kBK / kThreads;   // per operand, thread and slice
  constexpr int kLd = kTile + 4;
  __shared__ __align__(16) float As[2][kBK][kLd];
  __shared__ __align__(16) float Bs[2][kBK][kLd];
  const int z = blockIdx.z;
  const int w = AGN_LD(g.slot_worker + z);
  const int64_t m0 = (int64_t)tile_y * kBM, n0 = (int64_t)tile_x * kBN;
  const T* A = reinterpret_cast<const T*>(g.a) + (g.a_by_worker ? (int64_t)w : z) * g.a_bstride;
  const T* B = reinterpret_cast<const T*>(g.b) + (g.b_by_worker ? (int64_t)w : z) * g.b_bstride;
  const int tid = threadIdx.x;
  const int tx = tid % 16, ty = tid / 16;

  float acc[kTM][kTN];
#pragma unroll
  for (int i = 0; i < kTM; ++i)
#pragma unroll
    for (int j = 0; j < kTN; ++j) acc[i][j] = 0.f;
  float bsum = 0.f;   // bias gradient (kEpi == kEpiDW, first column tile)
  const bool do_bias = (kEpi == kEpiDW) && tile_x == 0 && tid < kBM;

  // element r of this thread in a k slice: row (or column) o and k
  auto place = [&](bool k_major, int r, int& o, int& kk) {
    const int e = tid + r * kThreads;
    if (k_major) { o = e / kBK; kk = e % kBK; } else { kk = e / kTile; o = e % kTile; }
  };
  T ra[kLoads], rb[kLoads];
  auto load = [&](int64_t k0) {
#pragma unroll
    for (int r = 0; r < kLoads; ++r) {
      int o, kk;
      place(kAKMajor, r, o, kk);
      const int64_t gm = m0 + o, gk = k0 + kk;
      ra[r] = from_f<T>(0.f);
      if (gm < g.M && gk < g.K) ra[r] = AGN_LD(kAKMajor ? A + gm * g.lda + gk : A + gk * g.lda + gm);
    }
#pragma unroll
    for (int r = 0; r < kLoads; ++r) {
      int o, kk;
      place(kBKMajor, r, o, kk);
      const int64_t gn = n0 + o, gk = k0 + kk;
      rb[r] = from_f<T>(0.f);
      if (gn < g.N && gk < g.K) rb[r] = AGN_LD(kBKMajor ? B + gn * g.ldb + gk : B + gk * g.ldb + gn);
    }
  };
  auto stage = [&](int buf) {
#pragma unroll
    for (int r = 0; r < kLoads; ++r) {
      int o, kk;
      place(kAKMajor, r, o, kk);
      As[buf][kk][o] = to_f(ra[r]);
      place(kBKMajor, r, o, kk);
      Bs[buf][kk][o] = to_f(rb[r]);
    }
  };
  load(0);
  stage(0);
  __syncthreads();
  int buf = 0;
  for (int64_t k0 = 0; k0 < g.K; k0 += kBK) {
    const bool more = k0 + kBK < g.K;
    if (more) load(k0 + kBK);
#pragma unroll
    for (int kk = 0; kk < kBK; ++kk) {
      float a[kTM], b[kTN];
      const float* ar = &As[buf][kk][ty * kTM];
      if constexpr (kTM == 2) {
        const float2 v = *reinterpret_cast<const float2*>(ar);
        a[0] = v.x;
        a[1] = v.y;
      } else {
#pragma unroll
        for (int i = 0; i < kTM; i += 4) {
          const float4 v = *reinterpret_cast<const float4*>(ar + i);
          a[i] = v.x;
          a[i + 1] = v.y;
          a[i + 2] = v.z;
          a[i + 3] = v.w;
        }
      }
#pragma unroll
      for (int j = 0; j < kTN; ++j) b[j] = Bs[buf][kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < kTM; ++i)
#pragma unroll
        for (int j = 0; j < kTN; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    if (do_bias) {
#pragma unroll
      for (int kk = 0; kk < kBK; ++kk) bsum += As[buf][kk][tid];
    }
    if (more) {   // (the other buffer's readers passed the last barrier)
      stage(buf ^ 1);
      __syncthreads();
      buf ^= 1;
    }
  }

  // Epilogues.
  float* theta = g.theta + (int64_t)w * g.ld_param;
  if (kEpi == kEpiFwd) {
    const float* bias = theta + g.boff;
    TO* out = reinterpret_cast<TO*>(g.out) + (int64_t)z * g.out_bstride;
#pragma unroll
    for (int i = 0; i < kTM; ++i) {
      const int64_t m = m0 + ty * kTM + i;
      if (m >= g.M) continue;
#pragma unroll
      for (int j = 0; j < kTN; ++j) {
        const int64_t n = n0 + tx + 16 * j;
        if (n >= g.N) continue;
        float v = acc[i][j] + AGN_LD(bias + n);
        if (g.relu) v = fmaxf(v, 0.f);
        AGN_ST(out + m * g.ldo + n, from_f<TO>(v));
      }
    }
  } else if (kEpi == kEpiDX) {
    const T* mask = reinterpret_cast<const T*>(g.mask) + (int64_t)z * g.mask_bstride;
    TO* out = reinterpret_cast<TO*>(g.out) + (int64_t)z * g.out_bstride;
#pragma unroll
    for (int i = 0; i < kTM; ++i) {
      const int64_t m = m0 + ty * kTM + i;
      if (m >= g.M) continue;
#pragma unroll
      for (int j = 0; j < kTN; ++j) {
        const int64_t n = n0 + tx + 16 * j;
        if (n >= g.N) continue;
        const float h = to_f(AGN_LD(mask + m * g.ldo + n));
        AGN_ST(out + m * g.ldo + n, from_f<TO>(h > 0.f ? acc[i][j] : 0.f));
      }
    }
  } else if (g.grad_out) {   // kEpiDW, raw gradient out (the optimizer runs after)
    float* go = g.grad_out + (int64_t)w * g.ld_param;
#pragma unroll
    for (int i = 0; i < kTM; ++i) {
      const int64_t m = m0 + ty * kTM + i;
      if (m >= g.M) continue;
#pragma unroll
      for (int j = 0; j < kTN; ++j) {
        const int64_t n = n0 + tx + 16 * j;
        if (n < g.N) AGN_ST(go + g.woff + m * g.N + n, acc[i][j]);
      }
    }
    if (do_bias && m0 + tid < g.M) AGN_ST(go + g.boff + m0 + tid, bsum);
  } else {   // kEpiDW: theta_k -= eta g, a_k += g (unless elided), bf16 copy refresh
    const bool has_a = g.acc != nullptr;
    float* a = has_a ? g.acc + (int64_t)w * g.ld_param : theta;
    bf16* tb = g.theta_bf16 ? g.theta_bf16 + (int64_t)w * g.ld_param : nullptr;
    // loads of all outputs first, then the updates (memory-level parallelism)
    const float* __restrict__ th_in = theta;
    const float* __restrict__ a_in = a;
    float th[kTM][kTN], av[kTM][kTN];
#pragma unroll
    for (int i = 0; i < kTM; ++i) {
      const int64_t m = m0 + ty * kTM + i;
#pragma unroll
      for (int j = 0; j < kTN; ++j) {
        const int64_t n = n0 + tx + 16 * j;
        if (m < g.M && n < g.N) {
          const int64_t p = g.woff + m * g.N + n;
          th[i][j] = AGN_LDCS(th_in + p);
          av[i][j] = has_a ? AGN_LDCS(a_in + p) : 0.f;
        }
      }
    }
#pragma unroll
    for (int i = 0; i < kTM; ++i) {
      const int64_t m = m0 + ty * kTM + i;
      if (m >= g.M) continue;
#pragma unroll
      for (int j = 0; j < kTN; ++j) {
        const int64_t n = n0 + tx + 16 * j;
        if (n >= g.N) continue;
        const int64_t p = g.woff + m * g.N + n;
        const float gr = acc[i][j];
        const float t = local_step(th[i][j], g.eta, gr);
        AGN_ST(theta + p, t);
        if (has_a) AGN_ST(a + p, av[i][j] + gr);
        if (tb) write_copy(tb, g.piece_plane, p, t);
      }
    }
    if (do_bias && m0 + tid < g.M) {
      const int64_t p = g.boff + m0 + tid;
      const float t = local_step(AGN_LD(theta + p), g.eta, bsum);
      AGN_ST(theta + p, t);
      if (has_a) AGN_ST(a + p, AGN_LD(a + p) + bsum);
      if (tb) write_copy(tb, g.piece_plane, p, t);
    }
  }
}

template <typename T, typename TO, bool kAKMajor, bool kBKMajor, int kEpi, int kTile,
          bool kShort = false>
__global__ void __launch_bounds__(kThreads) gemm_simt_kernel(const GemmArgs g) {
  pdl_begin();
  gemm_simt_tile<T, TO, kAKMajor, kBKMajor, kEpi, kTile, kShort>(g, blockIdx.x, blockIdx.y);
}

// The weight gradients of several layers in one launch (they depend on no other
// layer's): layer i's tiles are blocks first[i] .. first[i + 1] - 1, columns
// fastest.
constexpr int kDwLayers = 8;
struct DwLayers {
  GemmArgs g[kDwLayers];
  int first[kDwLayers + 1];
  int n;
};
template <typename T, int kTile, bool kShort = false>
__global__ void __launch_bounds__(kThreads)
dw_simt_kernel(const __grid_constant__ DwLayers batch) {
  pdl_begin();
  int i = 0;
  while (i + 1 < batch.n && (int)blockIdx.x >= batch.first[i + 1]) ++i;
  const GemmArgs& g = batch.g[i];
  const int t = (int)blockIdx.x - batch.first[i], cols = (int)((g.N + kTile - 1) / kTile);
  gemm_simt_tile<T, T, false, false, kEpiDW, kTile, kShort>(g, t % cols, t / cols);
}

// Softmax cross-entropy (SoftmaxArgs).  A block takes a 32-sample chunk of a
// slot (one block per slot took 38 us a launch at 4 slots x 512 samples x 10
// classes): up to kXentClasses classes pass through shared memory, copied in
// and out by the whole block, and a thread sums its sample's classes in order;
// more classes pass through in tiles of as many, twice (maximum, then sum).  The
// chunk's loss is a fixed tree over its samples.  A thread reading its sample's
// classes from global memory instead took 215 us a launch at 16 slots x 128 samples x
// 1000 classes by itself, and a millisecond beside the dW launch waiting behind
// it, whose shared memory leaves the lines no room in L1; the tiles take 68.
constexpr int kXentThreads = 128, kXentClasses = 128;
template <typename T>
__global__ void __launch_bounds__(kXentThreads) softmax_xent_kernel(const SoftmaxArgs a) {
  pdl_begin();
  __shared__ float zs[32 * (kXentClasses + 1)];
  __shared__ float inv_s[32], mx_s[32];
  __shared__ int ys[32];
  const int z = blockIdx.y, chunk = blockIdx.x, tid = threadIdx.x;
  const int m = a.m, C = a.C, nj = min(32, m - 32 * chunk);
  const float inv_m = 1.0f / (float)m;
  const int64_t row0 = ((int64_t)z * m + 32 * chunk) * C;
  const float* Zc = a.Z + row0;
  T* dZc = static_cast<T*>(a.dZ) + row0;
  const bool staged = C <= kXentClasses;
  // odd row strides: no bank conflicts between the samples' rows
  const int ld = staged ? C + 1 - (C & 1) : kXentClasses + 1;
  float mx = -INFINITY, s = 0.f;   // of sample tid
  float* zr = zs + tid * ld;       // its row (tid < 32)
  if (staged) {
    for (int i = tid; i < nj * C; i += kXentThreads) zs[i / C * ld + i % C] = AGN_LD(Zc + i);
    __syncthreads();
  } else {
    const int warp = tid >> 5, lane = tid & 31;
    constexpr int kRowsPerWarp = 32 / (kXentThreads / 32), kLoads = kXentClasses / 32;
    for (int pass = 0; pass < 2; ++pass) {
      for (int c0 = 0; c0 < C; c0 += kXentClasses) {
        float v[kRowsPerWarp][kLoads];
#pragma unroll
        for (int r = 0; r < kRowsPerWarp; ++r)
#pragma unroll
          for (int q = 0; q < kLoads; ++q) {
            const int j = warp * kRowsPerWarp + r, c = c0 + 32 * q + lane;
            v[r][q] = j < nj && c < C ? AGN_LD(Zc + (int64_t)j * C + c) : 0.f;
          }
        __syncthreads();   // the tile before is read
#pragma unroll
        for (int r = 0; r < kRowsPerWarp; ++r)
#pragma unroll
          for (int q = 0; q < kLoads; ++q)
            zs[(warp * kRowsPerWarp + r) * ld + 32 * q + lane] = v[r][q];
        __syncthreads();
        if (tid < nj) {
          const int w = min(kXentClasses, C - c0);
          if (pass == 0)
            for (int c = 0; c < w; ++c) mx = fmaxf(mx, zr[c]);
          else
            for (int c = 0; c < w; ++c) s += expf(zr[c] - mx);
        }
      }
    }
  }
  if (tid < 32) {
    float ce = 0.f;
    if (tid < nj) {
      const int* yrow =
          a.x_shard > 0
              ? a.yb + (int64_t)AGN_LD(a.slot_worker + z) * (a.x_shard + m) +
                    batch_row0(a.slot_t0, z, a.step, m, a.x_shard)
              : a.yb + (int64_t)z * m;
      const int y = AGN_LD(yrow + 32 * chunk + tid);
      const float zy = staged ? zr[y] : AGN_LD(Zc + (int64_t)tid * C + y);
      if (staged) {
        for (int c = 0; c < C; ++c) mx = fmaxf(mx, zr[c]);
        for (int c = 0; c < C; ++c) {
          const float ex = expf(zr[c] - mx);
          zr[c] = ex;
          s += ex;
        }
      }
      ce = (logf(s) + mx) - zy;
      inv_s[tid] = 1.0f / s;
      mx_s[tid] = mx;
      ys[tid] = y;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) ce += __shfl_xor_sync(0xffffffffu, ce, off);
    if (tid == 0) {
      const float part = ce * inv_m;
      AGN_ST(a.loss_parts +
                 ((int64_t)AGN_LD(a.slot_commit + z) * a.lam + a.step) * gridDim.x + chunk,
             part);
      if (!isfinite(part)) atomicExch(a.flag, 1);
    }
  }
  __syncthreads();
  for (int i = tid; i < nj * C; i += kXentThreads) {
    const int j = i / C, c = i % C;
    float p = (staged ? zs[j * ld + c] : expf(AGN_LD(Zc + i) - mx_s[j])) * inv_s[j];
    if (c == ys[j]) p -= 1.0f;
    AGN_ST(dZc + i, from_f<T>(p * inv_m));
  }
}

// Minibatch gather (FetchNextMiniBatch of Algorithm 1): slot z, row j reads
// dataset row k S + ((t0 + i) m + j) mod S of worker k = slot_worker[z].
// With `pieces` (fp32 mode on tensor cores) the rows are also written as three
// exact bf16 pieces, planes `plane` apart.
template <typename T>
__global__ void gather_kernel(const T* __restrict__ X, const int* __restrict__ y, T* Xb, int* yb,
                              int d0, int m, int64_t S, const int* slot_worker,
                              const long long* slot_t0, int step, bf16* pieces, int64_t plane) {
  pdl_begin();
  const int z = blockIdx.y, j = blockIdx.x;
  const int w = AGN_LD(slot_worker + z);
  const long long t = AGN_LD(slot_t0 + z) + step;
  const int64_t row = (int64_t)w * S + (int64_t)(((unsigned long long)t * m + j) % (unsigned long long)S);
  const T* src = X + row * d0;
  const int64_t o = ((int64_t)z * m + j) * d0;
  T* dst = Xb + o;
  for (int c = threadIdx.x; c < d0; c += blockDim.x) {
    const T v = AGN_LD(src + c);
    AGN_ST(dst + c, v);
    if (pieces) {
      bf16 q0, q1, q2;
      split3(to_f(v), q0, q1, q2);
      AGN_ST(pieces + o + c, q0);
      AGN_ST(pieces + plane + o + c, q1);
      AGN_ST(pieces + 2 * plane + o + c, q2);
    }
  }
  if (threadIdx.x == 0) AGN_ST(yb + (int64_t)z * m + j, AGN_LD(y + row));
}

// The same gather, four consecutive elements per thread (d_0 a multiple of
// 4): a block per minibatch row, one 16-byte (fp32) or 8-byte (bf16) load and
// store per thread and group, and 8-byte piece stores.
//
// early = 1: the destination buffers are not read by the preceding kernel
// (the tensor-core operand alternates between two buffers by local step, and
// the labels' last reader finished before this launch could start), so the
// rows are copied before waiting for the preceding kernel; the wait at the
// end keeps this launch's completion ordered after it for the next kernel.
template <typename T>
__global__ void __launch_bounds__(256) gather4_kernel(const T* __restrict__ X,
                                                      const int* __restrict__ y, T* Xb, int* yb,
                                                      int d0, int m, int64_t S,
                                                      const int* slot_worker,
                                                      const long long* slot_t0, int step,
                                                      bf16* pieces, int64_t plane, int early) {
  if (early) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  else pdl_begin();
  struct alignas(4 * sizeof(T)) Vec { T v[4]; };
  struct alignas(8) Piece4 { bf16 v[4]; };
  const int r = blockIdx.x;                 // slot * m + j
  const int z = r / m, j = r - z * m;
  const int w = AGN_LD(slot_worker + z);
  const long long t = AGN_LD(slot_t0 + z) + step;
  const int64_t row =
      (int64_t)w * S + (int64_t)(((unsigned long long)t * m + j) % (unsigned long long)S);
  const T* src = X + row * d0;
  const int64_t o = (int64_t)r * d0;
  for (int c = threadIdx.x * 4; c < d0; c += blockDim.x * 4) {
    const Vec v = AGN_LD(reinterpret_cast<const Vec*>(src + c));
    if (Xb) AGN_ST(reinterpret_cast<Vec*>(Xb + o + c), v);
    if (pieces) {
      Piece4 p0, p1, p2;
#pragma unroll
      for (int e = 0; e < 4; ++e) split3(to_f(v.v[e]), p0.v[e], p1.v[e], p2.v[e]);
      AGN_ST(reinterpret_cast<Piece4*>(pieces + o + c), p0);
      AGN_ST(reinterpret_cast<Piece4*>(pieces + plane + o + c), p1);
      AGN_ST(reinterpret_cast<Piece4*>(pieces + 2 * plane + o + c), p2);
    }
  }
  if (threadIdx.x == 0) AGN_ST(yb + r, AGN_LD(y + row));
  if (early) asm volatile("griddepcontrol.wait;" ::: "memory");
}

int simt_sms() {
  static const int sms = [] {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      (void)cudaGetLastError();
    return std::max(n, 1);
  }();
  return sms;
}

// The largest tile (fewest shared-memory reads per multiply-add) that still
// gives every SM a block or, of 128, one and a half, and of 128 is not mostly
// padding; small launches take small tiles, since a block's chain over k is then
// what bounds them.  (785-2001-2001-10, 16 slots of one sample, us a run of six
// steps with tiles of 128 and 64: forward 4100 and 2660, dX 3155 and 1990.)
template <typename T, typename TO, bool kAK, bool kBK, int kEpi>
Status launch_gemm(const GemmArgs& g, int slots, cudaStream_t st) {
  const int sms = simt_sms();
  auto blocks = [&](int t) { return ceil_div(g.N, t) * ceil_div(g.M, t) * (int64_t)slots; };
  auto go = [&](auto kf, int t) -> Status {
    dim3 grid((unsigned)ceil_div(g.N, t), (unsigned)ceil_div(g.M, t), (unsigned)slots);
    AGN_TRY_CUDA(launch_pdl(kf, grid, kThreads, 0, st, g));
    AGN_TRY_CUDA(cudaGetLastError());
    return Status::Ok();
  };
  if (g.M > 64 && g.N > 64 && blocks(128) >= 3 * sms / 2)
    return go(gemm_simt_kernel<T, TO, kAK, kBK, kEpi, 128>, 128);
  if (blocks(64) >= sms) return go(gemm_simt_kernel<T, TO, kAK, kBK, kEpi, 64>, 64);
  if (g.K <= kShortK) return go(gemm_simt_kernel<T, TO, kAK, kBK, kEpi, 32, true>, 32);
  return go(gemm_simt_kernel<T, TO, kAK, kBK, kEpi, 32>, 32);
}

}  // namespace

template <typename T>
Status simt_forward(const GemmArgs& g, bool last, int slots, cudaStream_t st) {
  if (last) return launch_gemm<T, float, true, true, kEpiFwd>(g, slots, st);
  return launch_gemm<T, T, true, true, kEpiFwd>(g, slots, st);
}
template <typename T>
Status simt_backward_dx(const GemmArgs& g, int slots, cudaStream_t st) {
  return launch_gemm<T, T, true, false, kEpiDX>(g, slots, st);
}
template <typename T>
Status simt_backward_dw(const GemmArgs* layers, int n_layers, int slots, cudaStream_t st) {
  for (int l0 = 0; l0 < n_layers; l0 += kDwLayers) {
    DwLayers batch{};
    batch.n = std::min(kDwLayers, n_layers - l0);
    auto fill = [&](int tile) -> int64_t {   // the layers' tiles; their number
      int64_t tiles = 0;
      for (int i = 0; i < batch.n; ++i) {
        const GemmArgs& g = batch.g[i] = layers[l0 + i];
        batch.first[i] = (int)tiles;
        tiles += ceil_div(g.N, tile) * ceil_div(g.M, tile);
      }
      batch.first[batch.n] = (int)tiles;
      return tiles;
    };
    // tiles as in launch_gemm, but none of 128: bound by the update of theta_k
    // and a_k, whose 186 registers a thread would leave one block an SM (three
    // of 64).  us a run of six steps of 784-1000-1000-10 with 128 and 64: fp32, 16
    // slots of 128 samples 3430 and 1890, 4 slots 955 and 580; 785-1001-1001-10, 16
    // slots of 8 samples 2040 and 938 (bf16 2260 and 853)
    int tile = 64;
    int64_t tiles = fill(tile);
    if (tiles * slots < simt_sms()) tiles = fill(tile = 32);
    if (tiles > INT32_MAX) return Status::Err(AGN_E_UNSUPPORTED, "dW tile count overflows");
    auto kf = tile == 64               ? dw_simt_kernel<T, 64>
              : batch.g[0].K <= kShortK ? dw_simt_kernel<T, 32, true>
                                        : dw_simt_kernel<T, 32>;
    AGN_TRY_CUDA(launch_pdl(kf, dim3((unsigned)tiles, 1, (unsigned)slots), kThreads, 0, st, batch));
    AGN_TRY_CUDA(cudaGetLastError());
  }
  return Status::Ok();
}
template <typename T>
Status softmax_xent(const SoftmaxArgs& a, int slots, cudaStream_t st) {
  const dim3 grid((unsigned)ceil_div(a.m, 32), (unsigned)slots);
  auto kf = softmax_xent_kernel<T>;
  AGN_TRY_CUDA(launch_pdl(kf, grid, kXentThreads, 0, st, a));
  AGN_TRY_CUDA(cudaGetLastError());
  return Status::Ok();
}
template <typename T>
Status gather_batch(const T* X, const int* y, T* Xb, int* yb, int d0, int m, int64_t S,
                    const int* slot_worker, const long long* slot_t0, int step, int slots,
                    cudaStream_t st, bf16* pieces, int64_t plane, int early) {
  const bool vec = d0 % 4 == 0 && plane % 4 == 0 &&
                   ((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(Xb) |
                     reinterpret_cast<uintptr_t>(pieces)) & 15) == 0;
  if (slots <= 0 || m <= 0) return Status::Ok();
  if (vec) {
    const int threads = (int)std::min<int64_t>(256, round_up((int64_t)d0 / 4, 32));
    {
      auto kf = gather4_kernel<T>;
      AGN_TRY_CUDA(launch_pdl(kf, slots * m, threads, 0, st, X,
                              y, Xb, yb, d0, m, S, slot_worker, slot_t0, step, pieces, plane,
                              early));
    }
  } else {
    if (early) return Status::Err(AGN_E_INVALID, "internal: early gather needs d_0 % 4 == 0");
    dim3 grid((unsigned)m, (unsigned)slots);
    {
      auto kf = gather_kernel<T>;
      AGN_TRY_CUDA(launch_pdl(kf, grid, 128, 0, st, X,
                              y, Xb, yb, d0, m, S, slot_worker, slot_t0, step, pieces, plane));
    }
  }
  AGN_TRY_CUDA(cudaGetLastError());
  return Status::Ok();
}

#define AGN_INST(T)                                                                          \
  template Status simt_forward<T>(const GemmArgs&, bool, int, cudaStream_t);                 \
  template Status simt_backward_dx<T>(const GemmArgs&, int, cudaStream_t);                   \
  template Status simt_backward_dw<T>(const GemmArgs*, int, int, cudaStream_t);              \
  template Status softmax_xent<T>(const SoftmaxArgs&, int, cudaStream_t);                    \
  template Status gather_batch<T>(const T*, const int*, T*, int*, int, int, int64_t,          \
                                  const int*, const long long*, int, int, cudaStream_t,       \
                                  bf16*, int64_t, int);
AGN_INST(float)
AGN_INST(bf16)
#undef AGN_INST

AGN_BOUNDS_UNIT(simt)

}  // namespace agn
