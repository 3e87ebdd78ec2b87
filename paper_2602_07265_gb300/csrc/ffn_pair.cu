// Expert SwiGLU FFN (step a8) for batches with many tokens per expert, on CTA
// pairs (tcgen05 cta_group::2).  Same operands, results and layouts as
// ffn_tc.cu:
//   gate/up phase: act[r, f] = silu(W_gate[e, f] . xp[r]) * (W_up[e, f] . xp[r])   (bf16)
//   down phase   : out[r, c] = W_down[e, c] . act[r]                                (fp32)
//
// What bounds it.  With hundreds of tokens per expert the layer is bound by the
// tensor cores, provided that the operands reach them: ffn_tc.cu's tile of 128
// weight rows x 128 tokens reads 94 bytes of operands per SM and cycle at full
// tensor rate, and its stream order spreads the running CTAs over all experts,
// so that weights come from HBM again for every 128 tokens.  Here
//   - a pair of CTAs shares a tile of 256 rows x up to 256 tokens: each SM loads
//     half of either operand, 62 bytes per cycle at full rate;
//   - the units are dealt to the pairs round robin, so that the pairs work on
//     neighbouring units (the same experts and tokens) and find them in L2;
//   - two 256-column TMEM accumulators let the epilogue of a unit run under
//     the MMAs of the next.
// Measured on GB300 (whole layer, ffn_tc.cu -> this): d = 2048, F = 1024, 48
// experts, B = 8192 (1365 tokens an expert) 1452 -> 702 us (gate/up 820 -> 333
// us, 1.65 PFLOP/s; down 440 -> 211 us, which also writes 537 MB of fp32 rows:
// 178 us without the stores); d = 2048, F = 768, 128 experts, B = 2048 (128
// tokens) 394 -> 278 us (gate/up 143 us for 805 MB of weights).  Four
// pipeline stages instead of six cost 5 %, tiles dealt expert by expert to all
// pairs (one row block at a time) 19 %.  With the loads left out the MMAs and
// the epilogue of the first case's gate/up phase take 254 us (2.2 PFLOP/s), of
// the second's 68 us (both with a faster, less exact silu; see silu()).
//
// Unit: (tile of up to 256 tokens of one expert, block of weight rows).  The
// weights are the MMA's M = 256 rows, 128 in each CTA; the tokens are its N
// (a multiple of 32, half of them in each CTA's shared memory).  In the
// gate/up phase the 128 rows of a CTA are 64 gate and 64 up rows of the same
// hidden units, alternating every 16 rows, so that gate and up of a hidden
// unit lie 16 lanes apart in one warp of the epilogue and meet by a shuffle.
// No unit is cut, so there are no partial sums and the result does not depend
// on the schedule.
//
// Roles inside a CTA (64 + 32 kEpiWarps threads): an elected lane of warp 0
// loads this CTA's half of both operands by TMA; in rank 0, one of warp 1
// issues the pair's MMAs; the other warps (two per TMEM lane quarter, taking
// turns at 32 columns) drain this CTA's accumulator.  Every mbarrier wait is
// bounded in time.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cstring>

#include "pair_rule.cuh"
#include "tc_ptx.cuh"
#include "tmap.cuh"
#include "xs_internal.cuh"

namespace xs {
namespace {

using namespace ptx;

constexpr int kBK = 64;                        // bf16 per K step (one 128-byte swizzle row)
constexpr int kEpiWarps = 8;                   // 12 and 16 measured up to 1 % slower
constexpr int kThreads = 64 + 32 * kEpiWarps;
constexpr int kABytes = 128 * kBK * 2;         // this CTA's weight rows of a step: 16 KB
constexpr int kStageBytes = 2 * kABytes;       // and up to 128 tokens
constexpr int kStages = 6;
constexpr int kAccCols = 256;                  // TMEM columns per accumulator
constexpr int kBarOffset = kStages * kStageBytes;
constexpr int kSmemBytes = kBarOffset + 256 + 1024;   // + barriers + alignment slack
constexpr uint64_t kWaitNs = 1000000000ull;    // 1 s per wait

struct PairParams {
  CUtensorMap tmA[2];   // weights: packed, [0]; plain, gate and up (or down in [0])
  CUtensorMap tmS[2];   // the same for the shared experts (experts >= n_routed)
  CUtensorMap tmB[8];   // xp or act [max_rows, K] bf16, boxes of 16, 32, ..., 128 rows x 64
  const Tile *tiles;
  Meta *meta;
  xs_stats *stats;
  uint16_t *act_out;    // gate/up output [max_rows, M]
  float *out;           // down output [max_rows, M]
  const uint16_t *drop; // down: nullable, the token rows [max_rows, M] that gate/up read
  int M;                // weight rows per expert: F (gate/up) or d (down)
  int K;                // reduction length: d (gate/up) or F (down)
  int n_routed;         // N: tiles of experts >= N use tmS
  int packed;
  int expert_base;      // routed expert e uses weights e - expert_base (expert parallelism)
};

template <bool kGateUp>
__global__ void __launch_bounds__(kThreads, 1) ffn_pair_kernel(const __grid_constant__ PairParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  const uint32_t sbase = smem_u32(smem);
  const uint32_t bar0 = sbase + kBarOffset;
  auto full_bar = [&](int s) { return bar0 + 8u * s; };                     // rank 0's is used
  auto empty_bar = [&](int s) { return bar0 + 8u * (kStages + s); };        // each CTA's own
  auto accfull_bar = [&](int b) { return bar0 + 8u * (2 * kStages + b); };  // each CTA's own
  auto accempty_bar = [&](int b) { return bar0 + 8u * (2 * kStages + 2 + b); };  // rank 0's is used
  const uint32_t drain_bar = bar0 + 8u * (2 * kStages + 4);
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + kBarOffset + 8 * (2 * kStages + 5));
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

  // The routing kernels that wrote meta and tiles finished before this grid
  // could start (see pdl_wait()); only the token operand and the outputs
  // depend on the kernel just before.
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int t0 = __ldcg(&p.meta->ffn_t0), n_rt = __ldcg(&p.meta->ffn_t1) - t0;
  const int s0 = __ldcg(&p.meta->ffn_s0), n_tiles = n_rt + __ldcg(&p.meta->ffn_s1) - s0;
  const int MB = kGateUp ? p.M / 128 : (p.M + 255) / 256, KI = p.K / kBK;
  const int n_units = n_tiles * MB;
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  if (pair >= n_units) {  // both CTAs of the pair
    pdl_wait();
    pdl_trigger();
    return;
  }

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(accfull_bar(b), 1);
      mbar_init(accempty_bar(b), 2 * kEpiWarps);   // the epilogue warps of both CTAs
    }
    mbar_init(drain_bar, 1);
    *abort_flag = 0;
    fence_mbar_init();
    prefetch_tmap(&p.tmB[0]);
    prefetch_tmap(&p.tmA[0]);
  }
  if (warp == 1) {
    tmem_alloc_pair(smem_u32(tmem_slot), 2 * kAccCols);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();   // both CTAs' barriers are ready
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  struct Unit {
    int ntok, row0, n_mma, mb;
    bool routed, single;
    int expert;      // among the weights of its kind
  };
  auto unit_at = [&](int u, bool early) {
    const int i = u / MB, ti = i < n_rt ? t0 + i : s0 + (i - n_rt);
    const int4 *tp = reinterpret_cast<const int4 *>(p.tiles) + ti;
    const int4 t4 = early ? __ldcg(tp) : *tp;
    Unit r;
    r.ntok = t4.z;
    r.row0 = t4.y;
    r.n_mma = (r.ntok + 31) & ~31;
    r.mb = u - i * MB;
    r.routed = t4.x < p.n_routed;
    r.single = t4.w != 0;
    r.expert = r.routed ? t4.x - p.expert_base : t4.x - p.n_routed;
    return r;
  };
  // In the last block of an odd number of 128-row down blocks rank 1 has no rows.
  auto rows_of = [&](const Unit &t, uint32_t rk) {
    return kGateUp || t.mb * 256 + static_cast<int>(rk) * 128 < p.M;
  };
  const uint32_t full0 = map_to_rank(full_bar(0), 0);

  // An expert's weights are read once if it has a single tile; its tokens are
  // read again for every block of weight rows (without these hints N = 64, d =
  // 2048, F = 1024, B = 512 took 166.3 instead of 155.9 us, B = 1024 189.6
  // instead of 180.0).
  const uint64_t pol_once = policy_evict_first(), pol_again = policy_evict_normal(), pol_tok = policy_evict_last();
  auto load_a = [&](const Unit &t, int kk, int stage) {
    const uint64_t pol = t.single ? pol_once : pol_again;
    const uint32_t dst = sbase + stage * kStageBytes, bar = full0 + 8u * stage;
    const CUtensorMap *m = t.routed ? p.tmA : p.tmS;
    if (kGateUp) {
      if (p.packed) {
        tma_load_5d_pair(dst, m, bar, 4 * static_cast<int>(rank), (t.expert * MB + t.mb) * KI + kk, pol);
      } else {
        const int row = t.expert * p.M + t.mb * 128 + static_cast<int>(rank) * 64;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          tma_load_2d_pair(dst + j * 4096, m, bar, kk * kBK, row + 16 * j, pol);
          tma_load_2d_pair(dst + j * 4096 + 2048, m + 1, bar, kk * kBK, row + 16 * j, pol);
        }
      }
    } else if (rows_of(t, rank)) {
      const int MT = p.M / 128, mt = t.mb * 2 + static_cast<int>(rank);
      if (p.packed)
        tma_load_2d_pair(dst, m, bar, 0, ((t.expert * MT + mt) * KI + kk) * 128, pol);
      else
        tma_load_2d_pair(dst, m, bar, kk * kBK, t.expert * p.M + mt * 128, pol);
    }
  };
  auto load_b = [&](const Unit &t, int kk, int stage) {
    const int half = t.n_mma / 2;
    tma_load_2d_pair(sbase + stage * kStageBytes + kABytes, &p.tmB[half / 16 - 1], full0 + 8u * stage,
                     kk * kBK, t.row0 + static_cast<int>(rank) * half, pol_tok);
  };
  // Bytes that both CTAs bring in for one step.
  auto step_bytes = [&](const Unit &t) {
    return static_cast<uint32_t>((rows_of(t, 1) ? 2 : 1) * kABytes + t.n_mma * kBK * 2);
  };
  auto fail = [&]() {
    atomicMax(&p.meta->status, XS_DEV_TIMEOUT);
    if (p.stats) atomicMax(&p.stats->status, XS_DEV_TIMEOUT);
    for (uint32_t r = 0; r < 2; ++r)  // both CTAs stop
      st_cluster_u32(map_to_rank(smem_u32(const_cast<int *>(abort_flag)), r), 1u);
  };

  const int n_mine = (n_units - pair + n_pairs - 1) / n_pairs;
  const long long steps = static_cast<long long>(n_mine) * KI;
  const int n_pre = steps < kStages ? static_cast<int>(steps) : kStages;
  if (warp == 0) {
    // Every stage is free at the start: its weights do not wait for the kernel before.
    Unit t = unit_at(pair, true);
    for (int i = 0, kk = 0, u = pair; i < n_pre; ++i) {
      if (elect_one()) {
        if (rank == 0) mbar_arrive_expect_tx(full_bar(i), step_bytes(t));
        load_a(t, kk, i);
      }
      __syncwarp();
      if (++kk == KI && i + 1 < n_pre) {
        kk = 0;
        u += n_pairs;
        t = unit_at(u, true);
      }
    }
  }
  pdl_wait();
  pdl_trigger();

  if (warp == 0) {
    // ------------------------------------------------ TMA producer
    int stage = 0, i = 0;
    uint32_t phase = 0;
    bool ok = true;
    for (int u = pair; ok && u < n_units; u += n_pairs) {
      const Unit t = unit_at(u, false);
      const uint32_t bytes = step_bytes(t);
      for (int kk = 0; kk < KI; ++kk, ++i) {
        if (i >= n_pre) {
          ok = mbar_wait_warp(empty_bar(stage), phase ^ 1u, kWaitNs, abort_flag);
          if (!ok) break;
        }
        if (elect_one()) {
          if (i >= n_pre) {
            if (rank == 0) mbar_arrive_expect_tx(full_bar(stage), bytes);
            load_a(t, kk, stage);
          }
          load_b(t, kk, stage);
        }
        __syncwarp();
        if (++stage == kStages) {
          stage = 0;
          phase ^= 1u;
        }
      }
    }
    // The last MMAs have read every stage, and this CTA got every signal that
    // is sent to it.
    for (int j = 0; ok && j < kStages; ++j) {
      ok = mbar_wait_warp(empty_bar(stage), phase ^ 1u, kWaitNs, abort_flag);
      if (++stage == kStages) {
        stage = 0;
        phase ^= 1u;
      }
    }
    if (!ok) {
      if (lane == 0) fail();
      // Copies may be in flight whose barrier no longer completes: they land
      // in microseconds; stay for two milliseconds.
      const uint64_t t_end = globaltimer() + 2000000ull;
      while (globaltimer() < t_end) __nanosleep(1000);
    }
  } else if (warp == 1) {
    // ------------------------------------------------ MMA issuer (rank 0)
    if (rank == 0) {
      // Stages and K blocks are added to the descriptor's address field.
      const uint64_t desc0 = sw128_desc(__shfl_sync(0xffffffffu, sbase, 0));
      const uint32_t acc0 = __shfl_sync(0xffffffffu, tmem, 0);
      int stage = 0, seq = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int u = pair; ok && u < n_units; u += n_pairs, ++seq) {
        const Unit t = unit_at(u, false);
        const uint32_t idesc = __shfl_sync(0xffffffffu, idesc_bf16(256, t.n_mma), 0);
        const int buf = seq & 1;
        ok = mbar_wait_warp(accempty_bar(buf), ((seq >> 1) & 1u) ^ 1u, kWaitNs, abort_flag);
        if (!ok) break;
        tc_fence_after();
        const uint32_t d0 = acc0 + buf * kAccCols;
        for (int kk = 0; kk < KI; ++kk) {
          ok = mbar_wait_warp(full_bar(stage), phase, kWaitNs, abort_flag);
          if (!ok) break;
          tc_fence_after();
          const uint64_t da = desc0 + static_cast<uint64_t>(stage * (kStageBytes >> 4));
          if (elect_one()) {
#pragma unroll
            for (int ks = 0; ks < kBK / 16; ++ks) {
              const uint64_t a = da + static_cast<uint64_t>((ks * 32) >> 4);
              mma_bf16_pair(d0, a, a + (kABytes >> 4), idesc, (kk > 0 || ks > 0) ? 1u : 0u);
            }
            mma_commit_pair(empty_bar(stage));
            if (kk + 1 == KI) mma_commit_pair(accfull_bar(buf));
          }
          __syncwarp();
          if (++stage == kStages) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
      if (!ok && lane == 0) fail();
      // All issued MMAs done before TMEM is released.
      if (elect_one()) mma_commit_pair_local(drain_bar);
      volatile int no_abort = 0;
      mbar_wait_warp(drain_bar, 0, kWaitNs, &no_abort);
    } else if (!kGateUp && p.drop != nullptr) {
      // The rows of all tiles, in equal shares over the pairs that have work.
      const Unit a = unit_at(0, false), b = unit_at(n_units - 1, false);
      const int lines = (b.row0 + b.ntok - a.row0) * (p.M / 64);
      const uint16_t *base = p.drop + static_cast<size_t>(a.row0) * p.M;
      const int step = 32 * (n_pairs < n_units ? n_pairs : n_units);
      for (int l = 32 * pair + lane; l < lines; l += step) discard_line(base + static_cast<size_t>(l) * 64);
    }
  } else {
    // ------------------------------------------------ epilogue
    const int q = warp & 3;                  // TMEM lane quarter of this warp
    const int row = q * 32 + lane;           // this thread's accumulator row
    const int first = (warp - 2) / 4 * 32;   // its first column; every other 8 kEpiWarps
    constexpr int kStep = 8 * kEpiWarps;
    const uint32_t accempty0 = map_to_rank(accempty_bar(0), 0);
    int seq = 0;
    for (int u = pair; u < n_units; u += n_pairs, ++seq) {
      const Unit t = unit_at(u, false);
      const int buf = seq & 1;
      if (!mbar_wait_warp(accfull_bar(buf), (seq >> 1) & 1u, kWaitNs, abort_flag)) {
        if (lane == 0) fail();
        break;
      }
      tc_fence_after();
      const uint32_t tacc = tmem + (static_cast<uint32_t>(q * 32) << 16) + buf * kAccCols;
      const int n_cols = rows_of(t, rank) ? t.n_mma : 0;   // columns this CTA finishes
      // The accumulator is free once this warp's last columns are in registers.
      auto release = [&]() {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(accempty0 + 8u * buf);
      };
      // Finishes columns [c0, c0 + 32): this thread's row of them in v.
      auto emit = [&](int c0, const float (&v)[32]) {
        if (kGateUp) {
          // Lanes 0-15 hold the gate rows of 16 hidden units, lanes 16-31 their
          // up rows; of every two tokens each half finishes one.
          const bool up_half = lane >= 16;
          const int f = t.mb * 128 + static_cast<int>(rank) * 64 + q * 16 + (lane & 15);
          uint16_t *dst = p.act_out + static_cast<size_t>(t.row0 + c0 + (up_half ? 1 : 0)) * p.M + f;
#pragma unroll
          for (int j = 0; j < 32; j += 2) {
            const float other = __shfl_xor_sync(0xffffffffu, up_half ? v[j] : v[j + 1], 16);
            const float gate = up_half ? other : v[j], up = up_half ? v[j + 1] : other;
            const __nv_bfloat16 h = __float2bfloat16_rn(silu(gate) * up);
            if (c0 + j + (up_half ? 1 : 0) < t.ntok)
              dst[static_cast<size_t>(j) * p.M] = *reinterpret_cast<const uint16_t *>(&h);
          }
        } else {
          float *dst = p.out + static_cast<size_t>(t.row0 + c0) * p.M + t.mb * 256 + static_cast<int>(rank) * 128 + row;
#pragma unroll
          for (int j = 0; j < 32; ++j)
            if (c0 + j < t.ntok) dst[static_cast<size_t>(j) * p.M] = v[j];
        }
      };
      if (first >= n_cols) release();
      for (int c0 = first; c0 < n_cols; c0 += kStep) {
        float v[32];
        tmem_ld32(tacc + c0, v);
        if (c0 + kStep >= n_cols) release();
        emit(c0, v);
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  cluster_sync();   // neither CTA leaves while the other may still signal it
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, 2 * kAccCols);
  }
}

// ---------------------------------------------------------------- host side

// Row-major [outer, inner] bf16 matrix, boxes of box_outer x 64, 128-byte swizzle.
bool make_map(CUtensorMap *m, const void *base, uint64_t inner, uint64_t outer, uint32_t box_outer) {
  return encode_tmap_2d(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, inner, outer,
                        static_cast<uint32_t>(kBK), box_outer, CU_TENSOR_MAP_SWIZZLE_128B);
}

// Packed gate/up blocks (pack.cu) as [block][16-row group][gate, up][16 rows][64]:
// a box is groups 4r .. 4r + 3 of a block, gate and up rows of a group side by
// side.  The tiles are swizzled already.
bool make_packed_gate_up(CUtensorMap *m, const void *base, uint64_t blocks) {
  const uint64_t dims[5] = {64, 16, 2, 8, blocks}, strides[4] = {128, 16384, 2048, 32768};
  const uint32_t box[5] = {64, 16, 2, 4, 1};
  return encode_tmap(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, base, 5, dims, strides, box,
                     CU_TENSOR_MAP_SWIZZLE_NONE);
}

// Packed down tiles as rows of 64.
bool make_packed_down(CUtensorMap *m, const void *base, uint64_t tiles) {
  return encode_tmap_2d(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, 64, tiles * 128, 64, 128,
                        CU_TENSOR_MAP_SWIZZLE_NONE);
}

template <bool kGateUp>
const void *kernel_ptr() {
  return reinterpret_cast<const void *>(ffn_pair_kernel<kGateUp>);
}

void pair_launch_config(cudaLaunchConfig_t *cfg, cudaLaunchAttribute *attr, int pairs, cudaStream_t s) {
  cfg->gridDim = dim3(2 * pairs);
  cfg->blockDim = dim3(kThreads);
  cfg->dynamicSmemBytes = kSmemBytes;
  cfg->stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg->attrs = attr;
  cfg->numAttrs = 2;
}

// CTA pairs of this kernel that the current device runs at once (cached per
// device; host threads that race on it store the same value); 0 if the query
// fails.
int resident_pairs() {
  constexpr int kDevs = 64;
  static std::atomic<int> cache[kDevs];   // the count + 1, 0 while unknown
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevs) return 0;
  const int known = cache[dev].load(std::memory_order_relaxed);
  if (known > 0) return known - 1;
  int n = 0;
  for (const void *k : {kernel_ptr<true>(), kernel_ptr<false>()})
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes) != cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  pair_launch_config(&cfg, attr, 1, nullptr);
  cfg.numAttrs = 1;
  if (cudaOccupancyMaxActiveClusters(&n, kernel_ptr<true>(), &cfg) != cudaSuccess) {
    n = 0;
    cudaGetLastError();  // a failed query leaves no sticky error
  }
  cache[dev].store(n + 1, std::memory_order_relaxed);
  return n;
}

template <bool kGateUp>
cudaError_t launch_phase(const FfnArgs &a, cudaStream_t s) {
  PairParams p;
  memset(&p, 0, sizeof(p));
  p.M = kGateUp ? a.F : a.d;
  p.K = kGateUp ? a.d : a.F;
  const void *tok = kGateUp ? static_cast<const void *>(a.xp) : static_cast<const void *>(a.act);
  for (int i = 0; i < 8; ++i)
    if (!make_map(&p.tmB[i], tok, p.K, a.max_rows, 16u * (i + 1))) return cudaErrorInvalidValue;
  const uint64_t blocks = static_cast<uint64_t>(p.M / 128) * (p.K / kBK);  // per expert
  p.packed = a.P_gate_up != nullptr;
  auto weights = [&](CUtensorMap *m, uint64_t n, const void *pk, const void *w0, const void *w1) {
    if (p.packed) return kGateUp ? make_packed_gate_up(m, pk, n * blocks) : make_packed_down(m, pk, n * blocks);
    const uint32_t rows = kGateUp ? 16 : 128;
    return make_map(m, w0, p.K, n * p.M, rows) && (!kGateUp || make_map(m + 1, w1, p.K, n * p.M, rows));
  };
  if (!weights(p.tmA, a.n_weights, kGateUp ? a.P_gate_up : a.P_down, kGateUp ? a.W_gate : a.W_down, a.W_up))
    return cudaErrorInvalidValue;
  const void *ps = kGateUp ? a.PS_gate_up : a.PS_down;
  if (a.n_shared > 0 && (!p.packed || ps != nullptr) &&
      !weights(p.tmS, a.n_shared, ps, kGateUp ? a.S_gate : a.S_down, a.S_up))
    return cudaErrorInvalidValue;
  p.tiles = a.tiles;
  p.meta = a.meta;
  p.stats = a.stats;
  p.act_out = a.act;
  p.out = a.out;
  p.drop = !kGateUp && a.drop_xp ? a.xp : nullptr;
  p.n_routed = a.N;
  p.expert_base = a.expert_base;
  cudaError_t e = cudaFuncSetAttribute(kernel_ptr<kGateUp>(), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kSmemBytes);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  pair_launch_config(&cfg, attr, resident_pairs(), s);
  return cudaLaunchKernelEx(&cfg, ffn_pair_kernel<kGateUp>, p);
}

}  // namespace

bool ffn_use_pairs(long long pairs, int experts, bool all, int ranks, int d, int F) {
  return pair_rule(pairs, experts, (experts + ranks - 1) / ranks, all || ranks == 1, resident_pairs(), d, F);
}

cudaError_t launch_ffn_pair_gate_up(const FfnArgs &a, cudaStream_t s) { return launch_phase<true>(a, s); }
cudaError_t launch_ffn_pair_down(const FfnArgs &a, cudaStream_t s) { return launch_phase<false>(a, s); }

}  // namespace xs
