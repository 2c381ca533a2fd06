// Kernel (b), weight-gradient half, on the tensor cores: D = H_{l-1}^T dZ_l
// for every slot of a wave and every hidden layer in one launch, fused with
// Algorithm 1's local step and accumulation (theta_k -= eta g, a_k += g, the
// bf16 copy of theta_k) for the weights and the biases.
//
// The GEMM is tiny next to its epilogue (K = m samples against 18-22 bytes
// of fp32 master weight and accumulator traffic per parameter), so the kernel
// is laid out around the parameter stream, not the MMA:
//
//   warp 0     operand producer: per tile, the GEMM operands (H^T and dZ^T
//              boxes, MN-major, 128-byte swizzle) into a ring of stages, as
//              fast as the MMA frees them, so the next tile's GEMM runs while
//              the current tile's epilogue drains.
//   last warp  parameter producer: each tile's theta_k rows (with Adam's moments;
//              with a_k's for waves whose accumulators exceed 64 MB, unless one
//              launch sums several steps' into a_k), 32 output features x
//              128 inputs per chunk, into a second ring.  Each slot is
//              refilled as soon as it frees, so DRAM reads of the next chunks
//              (and of the next tile) are in flight while the current one is
//              updated.  Smaller waves add g to a_k in the L2 (red.add) and
//              keep twice the theta_k chunks in flight.
//   warp 1     MMA issuer (one thread) and TMEM owner.  Two accumulators
//              (double buffer): the GEMM of the next tile runs while the
//              epilogue drains this one.
//   warps 2-9  (2-17 for Adam and for kept steps of short minibatches)
//              epilogue.  Warp w reads TMEM lanes 32 (w % 4) .. + 31, i.e.
//              32 consecutive inputs k of the tile, and 16 of the 32 features
//              of a chunk; it transposes them through shared memory so that
//              each lane updates four consecutive inputs of a feature at a
//              time (16-byte reads of theta_k and a_k from the chunk, 16-byte
//              coalesced stores).
//
// Bias gradients ride along: a layer with d_{l-1} = M inputs gets M + 1 GEMM
// rows, row M of H^T being all ones (written into the staged A tile by the
// MMA warp, over the zero fill of the out-of-range row), so D[M][f] =
// sum_j dZ_l[j][f] = g_b[f]; the epilogue updates b_l and its accumulator
// from that row, with their 32 values per chunk copied in by the producer.
//
// The local step rounds as Algorithm 1 computes it: g = fp32(-eta grad), then
// theta_k = fp32(theta_k + g) (local_step).
//
// The kernel is persistent (one CTA per SM: the rings take 210 KB of shared
// memory and the accumulators all 512 TMEM columns); tiles (layer, slot,
// feature tile, input tile) are dealt out round-robin with input tiles
// fastest, so neighbouring CTAs stream neighbouring parts of the same weight
// rows.  Every wait is bounded (2 s of global time): on expiry the CTA sets
// *err, stops issuing, drains its own copies and MMAs (bounded), frees TMEM
// and returns.
#include <cuda.h>

#include <algorithm>
#include <cstring>
#include <mutex>
#include <set>

#include "mlp.cuh"
#include "mlp_tc.cuh"
#include "tc_ptx.cuh"

namespace agn {

namespace {

constexpr int kChunkWarps = 8;                 // epilogue warps on one parameter chunk
constexpr int kCF = 32;                        // output features per parameter chunk
constexpr int kChunkBytes = kCF * 128 * 4;     // one fp32 chunk: 32 rows x 128 inputs
constexpr int kBiasHalf = kCF * 4;            // b_l (or its accumulator) for one chunk
constexpr uint64_t kWaitNs = 2000000000ull;    // 2 s
constexpr int kThrottleTiles = 8;              // tiles per CTA from which operands wait for chunks

// kBK samples per stage: one TMA box is 64 MN-elements x kBK samples of bf16
// (kBK rows of 128 bytes, 128-byte swizzle); A = two boxes (128 inputs),
// B = BN / 64 boxes.
// kMode: kDwUpdRed = the local step and accumulation, theta_k per chunk
// through the ring (6 slots in flight) and a_k += g as L2 adds (red.add,
// nothing read back into the SM); kDwSet = the same of a commit's first step,
// a_k = g; kDwRepull = either, with slots that only take a_k (args.slot_repull);
// kDwUpdAcc = kDwUpdRed with a_k's chunk read through the ring beside theta_k's
// and stored back (3 slots); kDwUpd = the local step without accumulator
// (elided: commits from a pull snapshot), theta_k alone (6 slots); kDwBlock =
// the same from several kept local steps' operands, or with slots that take
// nothing; kDwGrad = the raw gradient only, stored or added (no chunks): for a
// separate optimizer kernel, as a_k of workers about to pull, or as a_k of the
// kept local steps' operands; kDwKeep = kDwBlock that leaves theta_k at the base
// of its block of local steps (bf16 mode, args.theta_work; kDwKeep8 on eight
// epilogue warps); kDwAdam = Adam's step, theta_k and the two moments per chunk
// through the ring (2 slots of 49 KB), the steps added to a_k in the L2.
// (Modes, not arguments: an epilogue runs few times a launch on small waves, and
// the tests and code of the others cost 0.4-1.4 us a launch there.)
enum {
  kDwUpdAcc = 0, kDwUpd = 1, kDwGrad = 2, kDwUpdRed = 3, kDwKeep = 4, kDwAdam = 5, kDwKeep8 = 6,
  kDwSet = 7, kDwRepull = 8, kDwBlock = 9
};
constexpr bool is_keep(int mode) { return mode == kDwKeep || mode == kDwKeep8; }
template <int BN, int kSplit, int kStages, int kBKs, int kMode>
struct DwCfg {
  static constexpr bool kAcc =                                             // a_k += g
      kMode == kDwUpdAcc || kMode == kDwUpdRed || kMode == kDwSet || kMode == kDwRepull ||
      kMode == kDwAdam;
  static constexpr bool kAccRing = kMode == kDwUpdAcc;                     // a_k via the ring
  // Sixteen epilogue warps, every other chunk each, where eight are what bounds
  // the launch: Adam's divisions and square roots (91 us a launch with eight, 75
  // with sixteen), and theta_k kept at its base with minibatches to 128 (ten steps
  // of 16 slots of 784-4096-4096-10, GPU ms with eight and sixteen: m = 64 7.18 and
  // 7.00, m = 128 8.40 and 8.23, m = 192 9.84 and 9.90, m = 256 10.87 and 11.01).
  // The other modes are bound by DRAM or latency: no gain.
  static constexpr int kEpiWarps =
      kMode == kDwAdam || kMode == kDwKeep ? 2 * kChunkWarps : kChunkWarps;
  static constexpr int kWarps = kEpiWarps + 3;
  static constexpr int kThreads = 32 * kWarps;
  static constexpr int kArrays = kMode == kDwAdam ? 3 : kAccRing ? 2 : 1;
  static constexpr int kSlotBytes = kArrays * (kChunkBytes + kBiasHalf);
  static constexpr int kRing =                                             // (kDwGrad: unused)
      kMode == kDwGrad ? 1 : kMode == kDwAdam ? 2 : kAccRing ? 3 : kStages > 2 ? 4 : 6;
  static constexpr int kBK = kBKs;
  static constexpr int kBox = kBK * 128;
  static constexpr int kABytes = 2 * kBox;
  static constexpr int kBBytes = (BN / 64) * kBox;
  static constexpr int kStageBytes = kSplit * (kABytes + kBBytes);
  // one accumulator: BN columns, or two of BN in the split mode (the leading
  // piece products and the five smaller pairs, kept apart for accuracy)
  static constexpr uint32_t kAccCols = (kSplit == 1 ? 1 : 2) * BN;
  static constexpr uint32_t kTmemCols = 2 * kAccCols;
  static constexpr int kChunks = BN / kCF;
  static constexpr size_t kRingOff = (size_t)kStages * kStageBytes;
  static constexpr size_t kGOff = kRingOff + (size_t)kRing * kSlotBytes;   // gradient staging
  static constexpr size_t kBarOff = kGOff + (size_t)kEpiWarps * 16 * 32 * 4;
  static constexpr size_t kSmem = kBarOff + 256 + 1024;   // barriers, alignment slack
};

// Four floats as four bf16 (round to nearest even), packed for one 8-byte store.
__device__ __forceinline__ uint2 bf16x4(const float (&x)[4]) {
  const __nv_bfloat162 lo = __floats2bfloat162_rn(x[0], x[1]);
  const __nv_bfloat162 hi = __floats2bfloat162_rn(x[2], x[3]);
  return make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
}
// Piece pairs (i, j), i + j <= 2, of the split product (pair 0 = a0 b0).
__device__ __forceinline__ int pair_a(int q) { return q == 2 || q == 4 ? 1 : q == 5 ? 2 : 0; }
__device__ __forceinline__ int pair_b(int q) { return q == 1 || q == 4 ? 1 : q == 3 ? 2 : 0; }

constexpr int kMaxDwLayers = 8;   // layers per launch (more are split into launches)
struct DwLayer {
  int M, N;          // inputs d_{l-1}, outputs d_l
  int mt, nt;        // input tiles (M / 128 + 1: the last holds the bias row), feature tiles
  int tile_begin;    // first tile of this layer in the launch
  int a_direct;      // A = the padded shards' rows of the slot's minibatch (layer 1)
  int64_t woff, boff;
  int64_t wboff, wwoff;   // in theta_work
};
struct DwBatch {
  CUtensorMap a[kMaxDwLayers], b[kMaxDwLayers], th[kMaxDwLayers];
  CUtensorMap ac[kMaxDwLayers];    // accumulators, or Adam's first moments
  CUtensorMap ac2[kMaxDwLayers];   // Adam's second moments
  DwLayer layer[kMaxDwLayers];
  int n_layers, total_tiles;
};

struct TileIdx {
  int layer, m_tile, n_tile, slot;
};
__device__ __forceinline__ TileIdx decode(const DwBatch& B, int t) {
  int i = 0;
  while (i + 1 < B.n_layers && t >= B.layer[i + 1].tile_begin) ++i;
  const DwLayer& L = B.layer[i];
  const int u = t - L.tile_begin;
  TileIdx r;
  r.layer = i;
  r.m_tile = u % L.mt;
  const int rest = u / L.mt;
  r.n_tile = rest % L.nt;
  r.slot = rest / L.nt;
  return r;
}

// Row r (< 128) of H^T set to one in every sample of an A stage: two 64-input
// boxes of kBK 128-byte rows (one per sample), 16-byte chunks swizzled by
// row % 8.
template <int kBK>
__device__ __forceinline__ void write_ones_row(uint8_t* sa, int r) {
  uint8_t* box = sa + (r >> 6) * (kBK * 128);
  const int i = r & 63;
  for (int j = 0; j < kBK; ++j) {
    const int off = j * 128 + ((((i >> 3) ^ (j & 7))) << 4) + (i & 7) * 2;
    *reinterpret_cast<uint16_t*>(box + off) = 0x3F80;   // bf16 1.0
  }
}

template <int BN, int kSplit, int kStages, int kBKs, int kMode>
__global__ void __launch_bounds__(DwCfg<BN, kSplit, kStages, kBKs, kMode>::kThreads, 1)
tc_dw_kernel(const __grid_constant__ DwBatch B, const TcArgs args) {
  using Cfg = DwCfg<BN, kSplit, kStages, kBKs, kMode>;
  constexpr bool kAcc = Cfg::kAcc, kAccRing = Cfg::kAccRing, kGrad = kMode == kDwGrad;
  constexpr bool kAdam = kMode == kDwAdam;
  constexpr int kWarps = Cfg::kWarps, kEpiWarps = Cfg::kEpiWarps;
  constexpr int kRing = Cfg::kRing, kSlotBytes = Cfg::kSlotBytes;
  constexpr int kBK = Cfg::kBK, kABytes = Cfg::kABytes, kBox = Cfg::kBox;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + Cfg::kBarOff);
  uint64_t* empty = full + kStages;
  uint64_t* cfull = empty + kStages;     // parameter chunk landed
  uint64_t* cempty = cfull + kRing;      // parameter chunk consumed (its 8 epilogue warps)
  uint64_t* tfull = cempty + kRing;      // accumulator b complete
  uint64_t* tempty = tfull + 2;          // accumulator b drained (every epilogue warp)
  uint64_t* fin = tempty + 2;            // MMA drain on abort
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(fin + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_holder + 1);
  volatile int* chunk_tiles = abort_flag + 1;   // tiles whose chunks are all requested

  __shared__ int s_skip;
  if (threadIdx.x == 0) s_skip = *reinterpret_cast<volatile int*>(args.err);
  __syncthreads();
  if (s_skip != 0) return;   // an earlier launch gave up: uniform across the CTA

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int T = B.total_tiles;
  // a slot whose replica nothing reads before its next pull: a_k only (or,
  // where this launch keeps no a_k, nothing)
  constexpr bool kBlock = kMode == kDwBlock || is_keep(kMode);
  auto acc_only = [&](int slot) -> bool {
    return (kMode == kDwRepull || kBlock) && args.slot_repull &&
           AGN_LD(args.slot_repull + slot) != 0;
  };
  // a_k = g, whatever it held
  const bool acc_set = kMode == kDwSet || ((kMode == kDwRepull || kAdam) && args.acc_set);
  // k steps of one local step's minibatch, and of the whole launch
  const int KTs = (args.K + kBK - 1) / kBK;
  const int KT = KTs * (kGrad || kBlock ? max(1, args.hist_steps) : 1);

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      tc::mbar_init(&full[s], 1);
      tc::mbar_init(&empty[s], 1);
    }
    for (int r = 0; r < kRing; ++r) {
      tc::mbar_init(&cfull[r], 1);
      tc::mbar_init(&cempty[r], kChunkWarps);
    }
    for (int b = 0; b < 2; ++b) {
      tc::mbar_init(&tfull[b], 1);
      tc::mbar_init(&tempty[b], kEpiWarps);
    }
    tc::mbar_init(fin, 1);
    *abort_flag = 0;
    *chunk_tiles = 0;
    tc::fence_mbar_init();
    for (int i = 0; i < B.n_layers; ++i) {
      tc::tma_prefetch_desc(&B.a[i]);
      tc::tma_prefetch_desc(&B.b[i]);
      tc::tma_prefetch_desc(&B.th[i]);
      tc::tma_prefetch_desc(&B.ac[i]);
      if (kAdam) tc::tma_prefetch_desc(&B.ac2[i]);
    }
  }
  if (warp == 1) {
    tc::tmem_alloc(tmem_holder, Cfg::kTmemCols);
    tc::tmem_relinquish();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = *tmem_holder;
  // programmatic dependent launch: the setup above overlapped the preceding
  // kernel; global memory is touched only after it has completed, except the
  // producer's first parameter chunks (below)

  // (the next forward may read theta_k before its own dependency wait: this
  // kernel lets it launch only when all CTAs have exited, writes fenced)
  if (!((warp == 0 || warp == kWarps - 1) && lane == 0)) pdl_wait_only();
  if (warp == 0 || warp == kWarps - 1) {
    if (warp == 0 && lane == 0) {
      // operand producer (warp 0): the GEMM operands of every tile into the
      // stage ring, as fast as the MMA frees stages
      pdl_wait_only();
      uint32_t ml = 0;   // stage fills issued
      bool ok = true;
      // On a long stream of tiles (bound by DRAM) the operands of a tile are
      // requested only once the previous tile's parameter chunks are, so
      // those stay first in line; on a short one they run ahead.
      const bool throttle = !kGrad && T >= kThrottleTiles * (int)gridDim.x;
      int itp = 0;
      for (int t = blockIdx.x; ok && t < T; t += gridDim.x, ++itp) {
        const TileIdx ti = decode(B, t);
        const CUtensorMap* tmA = &B.a[ti.layer];
        const CUtensorMap* tmB = &B.b[ti.layer];
        // layer 1's A from the padded shards: the worker's shard at the slot's
        // minibatch row (samples past m multiply dZ rows that are zero fill)
        const bool a_direct = B.layer[ti.layer].a_direct && args.x_shard > 0;
        int a_row0 = 0, b_z = 0, a_z = 0;
        auto operands = [&](int st) {   // of local step st: batches and the first row
          b_z = args.z0 + st * args.z_step + ti.slot;
          a_z = a_direct ? AGN_LD(args.slot_worker + ti.slot) : b_z;
          if (a_direct)
            a_row0 = (int)batch_row0(args.slot_t0, ti.slot, args.step + st, args.K, args.x_shard);
        };
        // the first step's before the wait for chunks, not after it: the row's
        // 64-bit division stands before the tile's first copy (8 slots of 3072-
        // 2048x3-10 at m = 160: 204 and 199 us a launch)
        operands(0);
        if (throttle && itp > 0 && *chunk_tiles < itp) {
          const uint64_t t0 = tc::globaltimer_ns();
          while (*chunk_tiles < itp) {
            if (*abort_flag || tc::globaltimer_ns() - t0 > kWaitNs) {
              ok = false;
              break;
            }
            __nanosleep(64);
          }
          if (!ok) break;
        }
        for (int kt = 0, kr = 0, st = 0; kt < KT; ++kt) {
          const int s = ml % kStages;
          if (ml >= kStages &&
              !tc::wait_or_abort(&empty[s], ((ml / kStages) - 1) & 1, abort_flag, kWaitNs)) {
            ok = false;
            break;
          }
          uint8_t* sa0 = smem + s * Cfg::kStageBytes;
          uint8_t* sb0 = sa0 + kSplit * kABytes;
          tc::mbar_arrive_expect_tx(&full[s], Cfg::kStageBytes);
  #pragma unroll
          for (int p = 0; p < kSplit; ++p) {
            uint8_t* sa = sa0 + p * kABytes;
            uint8_t* sb = sb0 + p * Cfg::kBBytes;
            if (kSplit == 1) {
              tc::tma_load_3d(sa, tmA, &full[s], ti.m_tile * 128, kr * kBK + a_row0, a_z);
              tc::tma_load_3d(sa + kBox, tmA, &full[s], ti.m_tile * 128 + 64, kr * kBK + a_row0,
                              a_z);
  #pragma unroll
              for (int c = 0; c < BN / 64; ++c)
                tc::tma_load_3d(sb + c * kBox, tmB, &full[s], ti.n_tile * BN + c * 64, kr * kBK,
                                b_z);
            } else {
              tc::tma_load_4d(sa, tmA, &full[s], ti.m_tile * 128, kr * kBK + a_row0, a_z, p);
              tc::tma_load_4d(sa + kBox, tmA, &full[s], ti.m_tile * 128 + 64, kr * kBK + a_row0,
                              a_z, p);
  #pragma unroll
              for (int c = 0; c < BN / 64; ++c)
                tc::tma_load_4d(sb + c * kBox, tmB, &full[s], ti.n_tile * BN + c * 64, kr * kBK,
                                b_z, p);
            }
          }
          ++ml;
          if (++kr == KTs) {
            kr = 0;
            if (kt + 1 < KT) operands(++st);
          }
        }
      }
      if (!ok) {
        *abort_flag = 1;
        // drain (bounded) the copies armed but maybe not yet landed
        for (uint32_t j = ml > (uint32_t)kStages ? ml - kStages : 0; j < ml; ++j)
          tc::mbar_wait_bounded(&full[j % kStages], (j / kStages) & 1, kWaitNs);
      }
    } else if (lane == 0) {
      // parameter producer (the last warp): each tile's theta_k and a_k rows
      // into the chunk ring, as fast as the epilogue frees slots
      uint32_t ch = 0;   // chunk fills issued
      bool ok = true;
      // theta_k / a_k chunk c of tile ti into ring slot r
      auto issue_chunk = [&](const TileIdx& ti, int worker, int c, int r) {
        const DwLayer& L = B.layer[ti.layer];
        const bool bias_tile = ti.m_tile == L.M / 128;
        uint8_t* dst = smem + Cfg::kRingOff + (size_t)r * kSlotBytes;
        const int f0 = ti.n_tile * BN + c * kCF;
        constexpr int kA = Cfg::kArrays;
        tc::mbar_arrive_expect_tx(&cfull[r], kA * (kChunkBytes + (bias_tile ? kBiasHalf : 0)));
        tc::tma_load_3d(dst, &B.th[ti.layer], &cfull[r], ti.m_tile * 128, f0, worker);
        if (kAccRing || kAdam)
          tc::tma_load_3d(dst + kChunkBytes, &B.ac[ti.layer], &cfull[r], ti.m_tile * 128, f0,
                          worker);
        if (kAdam)
          tc::tma_load_3d(dst + 2 * kChunkBytes, &B.ac2[ti.layer], &cfull[r], ti.m_tile * 128, f0,
                          worker);
        if (bias_tile) {   // b_l[f0 .. f0 + 31] and its accumulator (within the replica)
          const int64_t pb = (int64_t)worker * args.ld_param + L.boff + f0;
          auto bias = [&](const float* src, int array) {
            if (AGN_BOUNDS_OK(src, kBiasHalf)) {
              tc::bulk_load(dst + kA * kChunkBytes + array * kBiasHalf, src, kBiasHalf, &cfull[r]);
            } else {   // bounds-checked build: account for the bytes, skip the copy
              AGN_BOUNDS_FAIL(src);
              tc::mbar_complete_tx(&cfull[r], kBiasHalf);
            }
          };
          bias(args.theta + pb, 0);
          if (kAccRing) bias(args.acc + pb, 1);
          if (kAdam) {
            bias(args.mom1 + pb, 1);
            bias(args.mom2 + pb, 2);
          }
        }
      };
      // theta_k and a_k were last written by this kernel's previous launch or
      // a pull, two or more launches back: the first tile's first chunks are
      // requested before waiting for the preceding kernel
      int npre = 0;
      if (!kGrad && (int)blockIdx.x < T && !acc_only(decode(B, blockIdx.x).slot)) {
        const TileIdx t0 = decode(B, blockIdx.x);
        const DwLayer& L0 = B.layer[t0.layer];
        npre = min(kRing, min(Cfg::kChunks, (L0.N - t0.n_tile * BN + kCF - 1) / kCF));
        const int w0 = AGN_LD(args.slot_worker + t0.slot);
        for (int c = 0; c < npre; ++c) {
          issue_chunk(t0, w0, c, (int)ch);
          ++ch;
        }
      }
      pdl_wait_only();
      for (int t = blockIdx.x; !kGrad && ok && t < T; t += gridDim.x) {
        const TileIdx ti = decode(B, t);
        const DwLayer& L = B.layer[ti.layer];
        const int worker = AGN_LD(args.slot_worker + ti.slot);
        const int nch = acc_only(ti.slot)
                            ? 0 : min(Cfg::kChunks, (L.N - ti.n_tile * BN + kCF - 1) / kCF);
        for (int c = t == (int)blockIdx.x ? npre : 0; c < nch; ++c) {
          const int r = ch % kRing;
          if (ch >= kRing &&
              !tc::wait_or_abort(&cempty[r], ((ch / kRing) - 1) & 1, abort_flag, kWaitNs)) {
            ok = false;
            break;
          }
          issue_chunk(ti, worker, c, r);
          ++ch;
        }
        *chunk_tiles = *chunk_tiles + 1;
      }
      if (!ok) {
        *abort_flag = 1;
        for (uint32_t j = ch > (uint32_t)kRing ? ch - kRing : 0; j < ch; ++j)
          tc::mbar_wait_bounded(&cfull[j % kRing], (j / kRing) & 1, kWaitNs);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t kIdesc = tc::idesc_bf16_f32(128, BN, true, true);
      uint32_t ml = 0;
      bool ok = true;
      int it = 0;
      for (int t = blockIdx.x; ok && t < T; t += gridDim.x, ++it) {
        const TileIdx ti = decode(B, t);
        const DwLayer& L = B.layer[ti.layer];
        const int b = it & 1;
        if (it >= 2 && !tc::wait_or_abort(&tempty[b], ((it >> 1) - 1) & 1, abort_flag, kWaitNs)) {
          ok = false;
          break;
        }
        tc::tc_fence_after();
        const uint32_t dbase = tmem + (uint32_t)b * Cfg::kAccCols;
        const int ones_row = L.M - ti.m_tile * 128;   // < 128 on the bias tile
        for (int kt = 0; kt < KT; ++kt) {
          const int s = ml % kStages;
          if (!tc::wait_or_abort(&full[s], (ml / kStages) & 1, abort_flag, kWaitNs)) {
            ok = false;
            break;
          }
          tc::tc_fence_after();
          if (ones_row < 128) {   // piece 0 of the out-of-range row := 1 (pieces 1, 2 stay 0)
            write_ones_row<kBK>(smem + s * Cfg::kStageBytes, ones_row);
            tc::fence_proxy_async_smem();
          }
          const uint32_t sa0 = tc::smem_u32(smem + s * Cfg::kStageBytes);
          const uint32_t sb0 = sa0 + kSplit * kABytes;
          constexpr int kPairs = kSplit == 1 ? 1 : 6;
#pragma unroll
          for (int kk = 0; kk < kBK / 16; ++kk) {
#pragma unroll
            for (int q = 0; q < kPairs; ++q) {
              const uint32_t sa = sa0 + (kSplit == 1 ? 0 : pair_a(q)) * kABytes;
              const uint32_t sb = sb0 + (kSplit == 1 ? 0 : pair_b(q)) * Cfg::kBBytes;
              const uint64_t ad = tc::smem_desc_sw128(sa + kk * 2048, kBox, 1024);
              const uint64_t bd = tc::smem_desc_sw128(sb + kk * 2048, kBox, 1024);
              const uint32_t dcol = (kSplit == 3 && q > 0) ? (uint32_t)BN : 0u;
              const bool acc_on = kSplit == 1 ? (kt | kk | q) != 0
                                              : (q == 0 ? (kt | kk) != 0
                                                        : ((kt | kk) != 0 || q > 1));
              tc::mma_bf16(dbase + dcol, ad, bd, kIdesc, acc_on ? 1u : 0u);
            }
          }
          tc::mma_commit(&empty[s]);
          ++ml;
        }
        if (!ok) break;
        tc::mma_commit(&tfull[b]);
      }
      if (!ok) {
        *abort_flag = 1;
        tc::mma_commit(fin);   // every MMA issued so far has completed once fin flips
        tc::mbar_wait_bounded(fin, 0, kWaitNs);
      }
    }
  } else {
    // epilogue warps (from 2): warp w reads TMEM lane quadrant w % 4 (inputs
    // 32 (w % 4) .. + 31 of the tile) and columns 16 hf .. + 15 of each chunk,
    // hf = (w - 2) / 4 mod 2.  It stages its 16 x 32 gradients in shared memory
    // (feature-major), then each lane updates four consecutive inputs of four
    // features with 16-byte shared loads and 16-byte global stores.
    // Of sixteen warps, the first eight take the even chunks (ch % 2 == 0): a ring
    // of an even number of slots keeps every slot with one half, which waits for
    // the slot's phases in order.
    const int g = warp & 3, hf = ((warp - 2) >> 2) & 1;
    constexpr bool kHalves = kEpiWarps > kChunkWarps;
    static_assert(!kHalves || kRing % 2 == 0, "one half of the warps per ring slot");
    const uint32_t odd = (uint32_t)(warp - 2) / kChunkWarps;
    float* gS = reinterpret_cast<float*>(smem + Cfg::kGOff) + (warp - 2) * (16 * 32);
    const float eta = args.eta;
    // theta_k left at its base: biases and W_L go to the working copy
    constexpr bool keep = is_keep(kMode);
    uint32_t ch = 0;
    bool ok = true;
    int it = 0;
    const int k4 = (lane & 7) * 4, i0 = lane >> 3;   // phase-2 position of this lane
    for (int t = blockIdx.x; ok && t < T; t += gridDim.x, ++it) {
      const TileIdx ti = decode(B, t);
      const DwLayer& L = B.layer[ti.layer];
      const int M = L.M, N = L.N;
      const int worker = AGN_LD(args.slot_worker + ti.slot);
      const float2 cc = kAdam ? AGN_LD(args.corr + (int64_t)ti.slot * args.lam + args.step)
                              : make_float2(0.f, 0.f);
      const int b = it & 1;
      // waits are warp-uniform: a lane that gave up takes its whole warp out
      // before the next .sync.aligned TMEM load
      ok = __all_sync(0xffffffffu, tc::wait_or_abort(&tfull[b], (it >> 1) & 1, abort_flag,
                                                      kWaitNs));
      if (!ok) break;
      tc::tc_fence_after();
      const int k0 = ti.m_tile * 128 + 32 * g;            // first input of this quadrant
      const bool quad_ok = k0 + k4 < M;                   // M % 8 == 0: all four or none
      const int kb = M - k0;                              // bias row, if 0 <= kb < 32
      const uint32_t tbase = tmem + ((uint32_t)(32 * g) << 16) + (uint32_t)b * Cfg::kAccCols +
                             (uint32_t)(16 * hf);
      const int64_t rbase = (int64_t)worker * args.ld_param;
      float* theta = args.theta + rbase;
      float* work = keep ? args.theta_work + (int64_t)worker * args.ld_work : nullptr;
      float* ww = keep && L.wwoff >= 0 ? work + L.wwoff : nullptr;
      float* acc = kAcc ? args.acc + rbase : nullptr;
      const bool has_acc = kAcc && (!kAdam || args.acc);   // (Adam elided: none)
      float *mom1 = args.mom1 + rbase, *mom2 = args.mom2 + rbase;   // Adam only
      auto adam = [&](float gr, float& m, float& v) {
        return adam_update(gr, m, v, eta, args.beta1, 1.0f - args.beta1, args.beta2,
                           1.0f - args.beta2, args.eps, cc.x, cc.y);
      };
      bf16* tb = args.theta_b ? args.theta_b + rbase : nullptr;   // bf16 mode only
      const bool grad_only = kGrad || acc_only(ti.slot);
      const int nch = grad_only && !kAcc && !kGrad
                          ? 0 : min(Cfg::kChunks, (N - ti.n_tile * BN + kCF - 1) / kCF);
      const bool grad_add = kGrad ? args.grad_add != 0 : !acc_set;
      for (int c = 0; c < nch; ++c) {
        if (kHalves && (ch & 1) != odd) {   // the other half's chunk
          ++ch;
          continue;
        }
        const int r = ch % kRing;
        uint32_t v[16];
        tc::tmem_ld_32x32b_x16(tbase + (uint32_t)(c * kCF), v);
        if (kSplit == 3) {
          uint32_t v2[16];
          tc::tmem_ld_32x32b_x16(tbase + (uint32_t)(BN + c * kCF), v2);
          tc::tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 16; ++i)
            v[i] = __float_as_uint(__fadd_rn(__uint_as_float(v[i]), __uint_as_float(v2[i])));
        } else {
          tc::tmem_ld_wait();
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) gS[i * 32 + lane] = __uint_as_float(v[i]);
        if (grad_only) {   // raw gradient out: grad (or a_k) = g or += g, coalesced 16 bytes
          __syncwarp();
          const int fbase = ti.n_tile * BN + c * kCF + 16 * hf;
          float* gout = kGrad ? args.grad_out + rbase : acc;
          if (quad_ok) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int i = i0 + 4 * u;
              if (fbase + i >= N) continue;
              float* go = gout + L.woff + (int64_t)(fbase + i) * M + k0 + k4;
              const float4 gv = *reinterpret_cast<const float4*>(gS + i * 32 + k4);
              if (grad_add) AGN_RED4(go, gv);
              else AGN_ST(reinterpret_cast<float4*>(go), gv);
            }
          }
          if (kb >= 0 && kb < 32 && lane < 16 && fbase + lane < N) {
            float* go = gout + L.boff + fbase + lane;
            if (grad_add) AGN_RED(go, gS[lane * 32 + kb]);
            else AGN_ST(go, gS[lane * 32 + kb]);
          }
          __syncwarp();
          continue;
        }
        ok = __all_sync(0xffffffffu,
                        tc::wait_or_abort(&cfull[r], (ch / kRing) & 1, abort_flag, kWaitNs));
        if (!ok) break;
        __syncwarp();
        const uint8_t* slot = smem + Cfg::kRingOff + (size_t)r * kSlotBytes;
        const int fbase = ti.n_tile * BN + c * kCF + 16 * hf;   // first feature of this warp
        if (quad_ok) {
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int i = i0 + 4 * u;                           // feature fbase + i
            if (fbase + i < N) {
              float4 gv = *reinterpret_cast<const float4*>(gS + i * 32 + k4);
              const int so = (16 * hf + i) * 128 + 32 * g + k4;   // in the fp32 chunks
              const float4 tv = *reinterpret_cast<const float4*>(
                  reinterpret_cast<const float*>(slot) + so);
              float tn[4];
              const int64_t p = L.woff + (int64_t)(fbase + i) * M + k0 + k4;
              if constexpr (kAdam) {   // g is then the step: a_k += g, theta_k += g
                const float4 m4 = *reinterpret_cast<const float4*>(
                    reinterpret_cast<const float*>(slot + kChunkBytes) + so);
                const float4 v4 = *reinterpret_cast<const float4*>(
                    reinterpret_cast<const float*>(slot + 2 * kChunkBytes) + so);
                float mm[4] = {m4.x, m4.y, m4.z, m4.w}, vv[4] = {v4.x, v4.y, v4.z, v4.w};
                gv.x = adam(gv.x, mm[0], vv[0]);
                gv.y = adam(gv.y, mm[1], vv[1]);
                gv.z = adam(gv.z, mm[2], vv[2]);
                gv.w = adam(gv.w, mm[3], vv[3]);
                AGN_ST(reinterpret_cast<float4*>(mom1 + p), make_float4(mm[0], mm[1], mm[2], mm[3]));
                AGN_ST(reinterpret_cast<float4*>(mom2 + p), make_float4(vv[0], vv[1], vv[2], vv[3]));
                tn[0] = tv.x + gv.x;
                tn[1] = tv.y + gv.y;
                tn[2] = tv.z + gv.z;
                tn[3] = tv.w + gv.w;
              } else {
                tn[0] = local_step(tv.x, eta, gv.x);
                tn[1] = local_step(tv.y, eta, gv.y);
                tn[2] = local_step(tv.z, eta, gv.z);
                tn[3] = local_step(tv.w, eta, gv.w);
              }
              if (!keep)
                AGN_ST(reinterpret_cast<float4*>(theta + p),
                       make_float4(tn[0], tn[1], tn[2], tn[3]));
              else if (ww)   // the output layer
                AGN_ST(reinterpret_cast<float4*>(ww + (p - L.woff)),
                       make_float4(tn[0], tn[1], tn[2], tn[3]));
              if (kAccRing) {
                const float4 av = *reinterpret_cast<const float4*>(
                    reinterpret_cast<const float*>(slot + kChunkBytes) + so);
                AGN_ST(reinterpret_cast<float4*>(acc + p),
                       make_float4(av.x + gv.x, av.y + gv.y, av.z + gv.z, av.w + gv.w));
              } else if (has_acc) {   // a_k += g in the L2 (one add per element and launch)
                if (acc_set) AGN_ST(reinterpret_cast<float4*>(acc + p), gv);
                else AGN_RED4(acc + p, gv);
              }
              // the bf16 copy (bf16 mode); the fp32 mode's GEMMs split the
              // fp32 weights themselves
              if (kSplit == 1) AGN_ST(reinterpret_cast<uint2*>(tb + p), bf16x4(tn));
            }
          }
        }
        if (kb >= 0 && kb < 32 && lane < 16 && fbase + lane < N) {   // bias row: b_l[f]
          const float* sTb =
              reinterpret_cast<const float*>(slot + Cfg::kArrays * kChunkBytes);
          float gb = gS[lane * 32 + kb];
          const int64_t pb = L.boff + fbase + lane;
          float tn;
          if constexpr (kAdam) {
            float mb = sTb[kCF + 16 * hf + lane], vb = sTb[2 * kCF + 16 * hf + lane];
            gb = adam(gb, mb, vb);
            AGN_ST(mom1 + pb, mb);
            AGN_ST(mom2 + pb, vb);
            tn = sTb[16 * hf + lane] + gb;
          } else {
            tn = local_step(sTb[16 * hf + lane], eta, gb);
          }
          AGN_ST(keep ? work + L.wboff + fbase + lane : theta + pb, tn);
          if (kAccRing) AGN_ST(acc + pb, sTb[kCF + 16 * hf + lane] + gb);
          else if (has_acc && acc_set) AGN_ST(acc + pb, gb);
          else if (has_acc) AGN_RED(acc + pb, gb);
          if (kSplit == 1) AGN_ST(tb + pb, __float2bfloat16_rn(tn));
        }
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&cempty[r]);
        ++ch;
      }
      if (!ok) break;
      tc::tc_fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&tempty[b]);
    }
    if (!ok) *abort_flag = 1;
  }
  __syncwarp();
  pdl_fence_exit();
  tc::tc_fence_before();
  __syncthreads();
  if (*abort_flag && threadIdx.x == 0) atomicExch(args.err, 1);
  if (warp == 1) tc::tmem_dealloc(tmem, Cfg::kTmemCols);
}

template <int BN, int kSplit, int kStages, int kBKs, int kMode>
Status launch_dw(const DwBatch& batch, const TcArgs& args, int num_sms, cudaStream_t st) {
  using Cfg = DwCfg<BN, kSplit, kStages, kBKs, kMode>;
  static_assert(Cfg::kSmem <= 232448, "shared memory");
  static_assert(Cfg::kSmem > 232448 / 2, "one CTA per SM (up to all 512 TMEM columns)");
  static_assert(Cfg::kTmemCols == 256 || Cfg::kTmemCols == 512, "TMEM columns");
  auto kern = tc_dw_kernel<BN, kSplit, kStages, kBKs, kMode>;
  static std::mutex mu;
  static std::set<int> done;
  {
    int dev = 0;
    AGN_TRY_CUDA(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lock(mu);
    if (!done.count(dev)) {
      AGN_TRY_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)Cfg::kSmem));
      done.insert(dev);
    }
  }
  if (batch.total_tiles <= 0) return Status::Ok();
  const int grid = std::min(batch.total_tiles, num_sms);
  {
    auto kf = kern;
    AGN_TRY_CUDA(launch_pdl(kf, grid, Cfg::kThreads, Cfg::kSmem, st, batch, args));
  }
  AGN_TRY_CUDA(cudaGetLastError());
  return Status::Ok();
}

}  // namespace

Status tc_backward_dw(const DwLayerMaps* layers, int n_layers, const TcArgs& args, int slots,
                      cudaStream_t st, bool split, int num_sms) {
  // Adam's chunks take longest: in bf16 mode too its tiles are 128 features wide,
  // which deals them out more evenly.  us a run of 64-512-10, 8 workers, 517 against
  // 670 with tiles of 256; 784-1000-1000-10, 4, m = 128 1344 and 1441; 2616-16-24-1400-5,
  // one, 412 and 494; 4 of 784-4096-4096-10 3961 and 3965
  const int bn = split || (args.mom1 && !args.grad_out) ? kTcDwBNSplit : kTcDwBN;
  for (int l0 = 0; l0 < n_layers; l0 += kMaxDwLayers) {
    DwBatch batch;
    std::memset(&batch, 0, sizeof(batch));
    int64_t tiles = 0, acc_bytes = 0;
    batch.n_layers = std::min(kMaxDwLayers, n_layers - l0);
    for (int i = 0; i < batch.n_layers; ++i) {
      const DwLayerMaps& d = layers[l0 + i];
      if (d.M <= 0 || d.N <= 0) return Status::Err(AGN_E_INVALID, "empty dW layer");
      batch.a[i] = *d.h_mn;
      batch.b[i] = *d.dz_mn;
      batch.th[i] = *d.theta;
      batch.ac[i] = args.mom1 ? *d.mom1 : *d.acc;
      if (args.mom1) batch.ac2[i] = *d.mom2;
      DwLayer& L = batch.layer[i];
      L.M = d.M;
      L.N = d.N;
      L.woff = d.woff;
      L.a_direct = d.a_direct;
      L.boff = d.boff;
      L.wboff = d.wboff;
      L.wwoff = d.wwoff;
      L.mt = d.M / 128 + 1;          // rows 0 .. M, row M the bias
      L.nt = (d.N + bn - 1) / bn;
      acc_bytes += ((int64_t)d.M + 1) * d.N * 4 * slots;
      L.tile_begin = (int)tiles;
      tiles += (int64_t)L.mt * L.nt * slots;
      if (tiles > INT32_MAX) return Status::Err(AGN_E_UNSUPPORTED, "dW tile count overflows");
    }
    batch.total_tiles = (int)tiles;
    // split mode: 32 samples per stage, so that two stages fit beside the
    // parameter ring (the next tile's operands land while this one multiplies)
    // grad_out: gradient only; else acc null: accumulator elided; else a_k
    // through L2 adds while the launch's accumulators fit well within the L2
    // (small waves, where the chunk ring's latency bounds the kernel and
    // half the ring's bytes per chunk buy twice the chunks in flight), or
    // through the ring (large waves, which stream theta_k and a_k from DRAM
    // at the copy bandwidth: there the L2's adds slowed the stream by 4 %;
    // and always with args.acc_ring)
    // (a first local step only stores a_k, and slots about to pull only add to
    // it: the ring stays with theta_k)
    const bool ring = !args.acc_set && !args.slot_repull &&
                      (args.acc_ring || acc_bytes > kTcRedAccBytes);
    const int mode = args.grad_out ? kDwGrad
                     : args.mom1  ? kDwAdam
                     : args.theta_work ? (args.K <= 128 ? kDwKeep : kDwKeep8)
                     : !args.acc  ? (args.hist_steps > 1 || args.slot_repull ? kDwBlock : kDwUpd)
                     : ring       ? kDwUpdAcc
                     : args.slot_repull ? kDwRepull
                     : args.acc_set     ? kDwSet
                                        : kDwUpdRed;
    if (split && (args.theta_work || mode == kDwBlock))
      return Status::Err(AGN_E_INVALID, "kept local steps: bf16 mode only");
    Status r = Status::Ok();
    // fp32, long minibatches (a tile's GEMM reads eight stages or more): a third
    // operand stage for two of the six chunks in flight.  784-1000-1000-10, 4 slots, us a launch at
    // m = 256, 300, 512: 43.0, 49.1, 70.0 with two stages, 40.5, 45.6, 61.5 with three
    // (42.9, 46.9, 60.9 with four stages and one chunk)
    const bool deep = ceil_div(args.K, 32) * std::max(1, args.hist_steps) >= 8;
#define AGN_DW_CASE(BN, SPLIT, STAGES, BK, MODE)                                 \
  case MODE:                                                                     \
    r = launch_dw<BN, SPLIT, STAGES, BK, MODE>(batch, args, num_sms, st);        \
    break
    if (split && deep && mode != kDwGrad && mode != kDwAdam && mode != kDwUpdAcc) {
      switch (mode) {
        AGN_DW_CASE(kTcDwBNSplit, 3, 3, 32, kDwUpd);
        AGN_DW_CASE(kTcDwBNSplit, 3, 3, 32, kDwSet);
        AGN_DW_CASE(kTcDwBNSplit, 3, 3, 32, kDwRepull);
        AGN_DW_CASE(kTcDwBNSplit, 3, 3, 32, kDwUpdRed);
      }
    } else if (split) {
      switch (mode) {
        AGN_DW_CASE(kTcDwBNSplit, 3, 4, 32, kDwGrad);
        AGN_DW_CASE(kTcDwBNSplit, 3, 2, 32, kDwAdam);
        AGN_DW_CASE(kTcDwBNSplit, 3, 2, 32, kDwUpd);
        AGN_DW_CASE(kTcDwBNSplit, 3, 2, 32, kDwUpdAcc);
        AGN_DW_CASE(kTcDwBNSplit, 3, 2, 32, kDwSet);
        AGN_DW_CASE(kTcDwBNSplit, 3, 2, 32, kDwRepull);
        AGN_DW_CASE(kTcDwBNSplit, 3, 2, 32, kDwUpdRed);
      }
    } else {
      switch (mode) {
        AGN_DW_CASE(kTcDwBN, 1, 4, 64, kDwGrad);
        AGN_DW_CASE(kTcDwBNSplit, 1, 2, 64, kDwAdam);
        AGN_DW_CASE(kTcDwBN, 1, 2, 64, kDwUpd);
        AGN_DW_CASE(kTcDwBN, 1, 2, 64, kDwBlock);
        AGN_DW_CASE(kTcDwBN, 1, 2, 64, kDwKeep);
        AGN_DW_CASE(kTcDwBN, 1, 2, 64, kDwKeep8);
        AGN_DW_CASE(kTcDwBN, 1, 2, 64, kDwUpdAcc);
        AGN_DW_CASE(kTcDwBN, 1, 2, 64, kDwSet);
        AGN_DW_CASE(kTcDwBN, 1, 2, 64, kDwRepull);
        AGN_DW_CASE(kTcDwBN, 1, 2, 64, kDwUpdRed);
      }
    }
#undef AGN_DW_CASE
    if (!r.ok()) return r;
  }
  return Status::Ok();
}

AGN_BOUNDS_UNIT(dw)

}  // namespace agn
