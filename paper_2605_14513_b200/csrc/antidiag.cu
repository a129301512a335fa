// Strided antidiagonal block-importance estimator on the sm_100a tensor cores -- the estimator
// family of the paper's main backbone (appendix "XAttention and SVG2 Configurations": anti-diagonal
// scoring with stride 16; the paper gives the stride and the block size only, the definition is
// this library's):
//   groups of s = 16 consecutive tokens; only the Ns = floor(N / s) full groups are sampled;
//   S'(a, c) = (scale / s) * sum_t <q_{a s + t}, k_{c s + s-1-t}>      (antidiagonal mean of a tile)
//   P'(a, .) = softmax over the groups c;  importance(I, J) = sum of P' over the groups of the two
//   blocks / number of groups in I;  then the same top-p selection as the pooled estimator.
//
// The contraction is a bf16 GEMM per head on the very memory of Q and K: row a of the left operand
// is the 16 tokens of group a laid end to end (16 x 128 values), row c of the right operand the 16
// tokens of group c in reverse order.  A 5-D tensor map (dim, token in group, group, head, batch)
// lets one TMA box fetch "token t of 128 consecutive groups", which is exactly a K-major operand tile;
// reversing the key tokens is a change of one box coordinate.
//
// antidiag_scores_kernel: a tile is 256 query groups x 256 key groups of a head, the work of two CTAs of a cluster
// (cta_group::2): each loads its half of both operands, holds its half of the rows of the result and drains it.
// One CTA per SM; the tiles are dealt to the pairs, and the pipeline runs on across them.  Warp 0 issues the TMA
// loads into a six-stage ring (one stage = 64 dims of one token position: 16 KB of Q + 16 KB of K per CTA), warp 1 of
// the even CTA issues tcgen05.mma (M = 256, N = 256, 4 x K = 16 per stage, 32 stages per tile) into one of two
// 256-column accumulators in tensor memory, warps 2-5 drain the other accumulator: one thread per query group, and for
// every key block of the tile the pair (max, sum of 2^(x - max)) over the block's 4 or 8 groups goes to the workspace.
// What bounds it: a 128 x 256 tile per CTA asks the L2 for 96 bytes a clock and SM, which it does not give (197 us for
// 12 heads of 2048 groups); the pair asks for 64.  140 us now, 1470 TFLOP/s, the tensor pipe 81 % busy at the 1.5 GHz
// that the power limit leaves.
// antidiag_reduce_kernel (fp64) turns the pairs of the groups of one query block into the log of
// the block importances, which top_p_kernel consumes like pooled scores.
#include <cuda.h>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace heart {
using namespace tc;

namespace {

constexpr int kS = HEART_ANTIDIAG_STRIDE;  // tokens per group
constexpr int kMt = 256;                   // query groups per tile: 128 in each CTA of a pair
constexpr int kNt = 256;                   // key groups per tile
constexpr int kStagesAd = 6;
constexpr int kHalfBytes = 128 * 128;      // 128 groups x 64 dims: a CTA's half of either operand of a stage
constexpr int kStageBytes = 2 * kHalfBytes;
constexpr int kKSteps = kS * 2;            // ring stages per tile: 16 token positions x 2 halves of the head dim
constexpr int kThreadsAd = 192;

struct AdBars {
  uint64_t full[kStagesAd], empty[kStagesAd];  // full, acc_empty: the even CTA's count for both
  uint64_t acc_full[2], acc_empty[2];
  uint64_t drain;
  uint32_t tmem_base;
  int abort;
};

struct AdParams {
  float2 *pairs;          // [R][Ns][nb]: (max, sum) in the log2 domain per (query group, key block)
  const uint8_t *refresh;
  int32_t *status;
  int H, R, Ns, nb;
  float c2;               // (scale / s) * log2(e)
  int test_skip_copy;     // test-hook builds only: the first pair leaves out copies of its second stage
};

template <int G>  // groups per block: 4 (64-token blocks) or 8 (128-token blocks)
__global__ void __launch_bounds__(kThreadsAd, 1)
    antidiag_scores_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                           const AdParams p) {
  extern __shared__ unsigned char smem_dyn[];
  unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) &
                                                          ~static_cast<uintptr_t>(1023));
  AdBars *bars = reinterpret_cast<AdBars *>(smem + kStagesAd * kStageBytes);
  volatile int *abort = &bars->abort;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = cluster_ctarank();  // of the pair
  // Tiles of the refreshed heads (the others: reuse branch of Algorithm 1, nothing to predict), column tiles of a row
  // first, dealt to the pairs in turn.  Every role walks the same list.
  const int row_tiles = (p.Ns + kMt - 1) / kMt, col_tiles = (p.Ns + kNt - 1) / kNt, n_tiles = p.R * row_tiles * col_tiles;
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  auto each_tile = [&](auto body) {  // body(head, row tile, column tile) -> go on?
    for (int u = pair; u < n_tiles; u += n_pairs) {
      const int row = u / col_tiles, r = row / row_tiles;
      if (p.refresh != nullptr && p.refresh[r] == 0) continue;
      if (!body(r, row - r * row_tiles, u - row * col_tiles)) break;
    }
  };

  if (tid == 0) {
    for (int i = 0; i < kStagesAd; ++i) {
      mbar_init(&bars->full[i], 1);
      mbar_init(&bars->empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bars->acc_full[i], 1);
      mbar_init(&bars->acc_empty[i], 8);  // one arrival per draining warp of the pair
    }
    mbar_init(&bars->drain, 1);
    bars->abort = 0;
    mbar_fence_init();
  }
  if (warp == 1) tmem_alloc_pair(&bars->tmem_base, 512);
  pdl_wait();  // refresh flags, and the workspace that the kernel before this one may still read
  pdl_launch_dependents();
  tc_fence_before();
  cluster_sync();  // (the other CTA's barriers are there)
  tc_fence_after();
  const uint32_t tmem = bars->tmem_base;
  auto settle = [&](uint64_t *bar, uint32_t parity) {
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity) && clock64() - t0 < 40000000LL) {
    }
  };

  if (warp == 0) {
    if (lane == 0) {  // ===== TMA producer
      tma_prefetch_desc(&map_q);
      tma_prefetch_desc(&map_k);
      int it = 0;
      const uint32_t even_full = cluster_address(smem_u32(bars->full), 0);
      each_tile([&](int r, int row, int col) {
        const int bidx = r / p.H, hidx = r % p.H;
        for (int ks = 0; ks < kKSteps; ++ks, ++it) {
          const int st = it % kStagesAd, n = it / kStagesAd, t = ks >> 1, dh = ks & 1;
          if (n >= 1 && !mbar_wait(&bars->empty[st], (n - 1) & 1, abort)) return false;
          unsigned char *dst = smem + st * kStageBytes;
          if (rank == 0) mbar_expect_tx(&bars->full[st], 2 * kStageBytes);
#ifdef HEART_TEST_HOOKS
          // Test-only library: boxes whose bytes are expected are never asked for, so the waits that depend on the stage run
          // out, in both CTAs of the pair, and the abort path is taken.
          if (p.test_skip_copy && blockIdx.x == 0 && it == 1) continue;
#endif
          // this CTA's half of token t of the query groups, of token s-1-t of the key groups of the tile
          tma_load_5d_pair(dst, &map_q, even_full + 8 * st, dh * 64, t, row * kMt + rank * 128, hidx, bidx);
          tma_load_5d_pair(dst + kHalfBytes, &map_k, even_full + 8 * st, dh * 64, kS - 1 - t, col * kNt + rank * 128, hidx, bidx);
        }
        return true;
      });
    }
  } else if (warp == 1) {
    // ===== MMA issuer of the pair: the whole warp runs the loop, one elected lane issues
    if (rank == 0) {
      constexpr uint32_t idesc = idesc_bf16_f32(kMt, kNt, false, false);
      auto at = [](uint64_t desc, uint32_t off16) -> uint64_t {
        return (desc & 0xffffffff00000000ull) | (uint32_t)((uint32_t)desc + off16);
      };
      const bool leader = elect_one();
      const uint64_t a_desc0 = smem_desc_sw128(smem_u32(smem), 16, 1024);
      const uint64_t b_desc0 = smem_desc_sw128(smem_u32(smem + kHalfBytes), 16, 1024);
      int it = 0, tile = 0;
      each_tile([&](int, int, int) {
        const int buf = tile & 1, m = tile >> 1;
        ++tile;
        if (m >= 1 && !__all_sync(0xffffffffu, mbar_wait(&bars->acc_empty[buf], (m - 1) & 1, abort))) return false;
        tc_fence_after();
        const uint32_t d = tmem + buf * kNt;
        for (int ks = 0; ks < kKSteps; ++ks, ++it) {
          const int st = it % kStagesAd, n = it / kStagesAd;
          if (!__all_sync(0xffffffffu, mbar_wait(&bars->full[st], n & 1, abort))) return false;
          tc_fence_after();
          const uint64_t a_desc = at(a_desc0, st * (kStageBytes >> 4)), b_desc = at(b_desc0, st * (kStageBytes >> 4));
          if (leader) {
#pragma unroll
            for (int k = 0; k < 4; ++k) mma_ss_pair(d, at(a_desc, k * 2), at(b_desc, k * 2), idesc, (ks > 0 || k > 0) ? 1u : 0u);
            tc_commit_pair(&bars->empty[st]);
            if (ks == kKSteps - 1) tc_commit_pair(&bars->acc_full[buf]);
          }
          __syncwarp();
        }
        return true;
      });
      if (*abort) {  // tensor memory must not be released under a product in flight
        if (leader) tc_commit_pair(&bars->drain);
        __syncwarp();
        settle(&bars->drain, 0);
      }
    }
  } else {
    // ===== drain: thread = one query group; per key block of the tile a (max, sum) pair
    const int q = warp & 3;  // the lane quarter of tensor memory this warp may read
    const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16);
    int tile = 0;
    each_tile([&](int r, int row, int col) {
      const int buf = tile & 1, m = tile >> 1;
      ++tile;
      const int a = row * kMt + rank * 128 + q * 32 + lane;
      float2 *out = p.pairs + ((size_t)r * p.Ns + (a < p.Ns ? a : 0)) * p.nb;
      if (!__all_sync(0xffffffffu, mbar_wait(&bars->acc_full[buf], m & 1, abort))) return false;
      tc_fence_after();
      const int c0 = col * kNt;
#pragma unroll 1
      for (int ch = 0; ch < kNt / 32; ++ch) {
        if (c0 + ch * 32 >= p.Ns) break;  // (uniform) nothing but padding from here on
        uint32_t v[32];
        tmem_ld32(lane_addr + buf * kNt + ch * 32, v);
        tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 32 / G; ++j) {
          const int cb = c0 + ch * 32 + j * G;  // first group of this key block
          float mx = -INFINITY;
#pragma unroll
          for (int i = 0; i < G; ++i)
            if (cb + i < p.Ns) mx = fmaxf(mx, __uint_as_float(v[j * G + i]));
          float l = 0.f;
          const float mc = mx * p.c2;
#pragma unroll
          for (int i = 0; i < G; ++i)
            if (cb + i < p.Ns) l += ex2(fmaf(__uint_as_float(v[j * G + i]), p.c2, -mc));
          if (cb < p.Ns && a < p.Ns) out[cb / G] = make_float2(mc, l);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_in(&bars->acc_empty[buf], 0);
      return true;
    });
  }
  tc_fence_before();
  // Neither CTA leaves while the other one's products read its shared memory or arrivals are under way; after an
  // abort in either, copies in flight get time to land (bounded: a copy takes microseconds).
  cluster_sync();
  const uint32_t off_abort = smem_u32(&bars->abort);
  if ((cluster_ld1(cluster_address(off_abort, 0)) | cluster_ld1(cluster_address(off_abort, 1))) != 0u) {
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000LL) {
    }
  }
  cluster_sync();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, 512);
  }
  if (tid == 0 && bars->abort) atomicExch(p.status, HEART_ERR_DEVICE_CHECK);
}

// One CTA per (query block I, head r), fp64: the (max, sum) pairs of the block's groups become
// scores[r][I][J] = ln(importance(I, J)) (-inf for importance 0), which the top-p kernel reads like
// pooled scores.  A query block without a full group gets equal scores (uniform importance).
// One warp per group of the block (8, or 4 of a 64-token block): row maximum and row sum by shuffles, the weights of
// the lane's key blocks stay in registers in between; they meet in shared memory, where a thread adds up
// the groups of a key block one after the other.  Every reduction has a fixed shape: bit-reproducible.
template <int NJ, int G>  // NJ * 32 >= n_b, G groups per block
__global__ void __launch_bounds__(32 * G, 16 / G) antidiag_reduce_kernel(const float2 *__restrict__ pairs, int Ns, int nb,
                                                                 int pitch, const uint8_t *__restrict__ refresh,
                                                                 double *__restrict__ scores) {
  const int I = blockIdx.x, r = blockIdx.y;
  pdl_wait();
  pdl_launch_dependents();
  if (refresh != nullptr && refresh[r] == 0) return;
  extern __shared__ __align__(16) double wgt[];  // [G][NJ * 32]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int a0 = I * G, a1 = min(a0 + G, Ns);
  const int nJ = (Ns + G - 1) / G;  // key blocks that hold at least one full group
  double *srow = scores + ((size_t)r * nb + I) * pitch;
  if (a1 <= a0) {
    for (int J = tid; J < pitch; J += 32 * G) srow[J] = 0.0;
    return;
  }
  constexpr int kPerLane = NJ;
  const double ln2 = 0.6931471805599453;
  double e[kPerLane];
  const int a = a0 + warp;  // this warp's group
  if (a < a1) {
    const float2 *prow = pairs + ((size_t)r * Ns + a) * nb;
    float mxf = -INFINITY;
#pragma unroll
    for (int k = 0; k < kPerLane; ++k)
      if (lane + 32 * k < nJ) mxf = fmaxf(mxf, prow[lane + 32 * k].x);
    double mx = (double)mxf;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    double z = 0.0;
#pragma unroll
    for (int k = 0; k < kPerLane; ++k) {
      e[k] = 0.0;
      if (lane + 32 * k < nJ) {  // (the row is in L1 / L2 from the pass above)
        const float2 pr = prow[lane + 32 * k];
        e[k] = exp_nonpositive(((double)pr.x - mx) * ln2) * (double)pr.y;
      }
      z += e[k];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
    const double inv_z = 1.0 / z;
#pragma unroll
    for (int k = 0; k < kPerLane; ++k) wgt[(warp * kPerLane + k) * 32 + lane] = e[k] * inv_z;
  }
  __syncthreads();
  const double inv = 1.0 / (double)(a1 - a0);
  for (int J = tid; J < pitch; J += 32 * G) {
    double w = 0.0;
    for (int n = 0; n < a1 - a0; ++n) w += wgt[n * kPerLane * 32 + J];  // groups in ascending order: a fixed summation order
    w = (J < nJ) ? w * inv : 0.0;
    srow[J] = (w > 0.0) ? log(w) : -INFINITY;
  }
}

// bf16 [B,H,N,128] seen as (dim, token in group, group, head, batch); box = 64 dims of one token
// position of `rows` consecutive groups, 128-byte swizzle, groups past Ns read as zero.
bool make_group_map(CUtensorMap *m, const void *base, const Geom &g, int Ns, int rows) {
  EncodeTiledFn fn = encode_tiled_fn();
  if (!fn) return false;
  cuuint64_t dims[5] = {(cuuint64_t)kD, (cuuint64_t)kS, (cuuint64_t)Ns, (cuuint64_t)g.H, (cuuint64_t)g.B};
  cuuint64_t strides[4] = {(cuuint64_t)g.sn * 2, (cuuint64_t)g.sn * 2 * kS, (cuuint64_t)g.sh * 2, (cuuint64_t)g.sb * 2};
  cuuint32_t box[5] = {64, 1, (cuuint32_t)rows, 1, 1};
  cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void *>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int G>
cudaError_t launch_scores(const CUtensorMap &mq, const CUtensorMap &mk, const AdParams &prm, long long tiles, int smem, cudaStream_t s) {
  cudaError_t e = allow_shared_memory(antidiag_scores_kernel<G>, smem);
  if (e != cudaSuccess) return e;
  const int pairs = (int)(tiles < 74 ? tiles : 74);  // two of the 148 SMs each
  return launch_pdl(antidiag_scores_kernel<G>, dim3(2 * pairs), dim3(kThreadsAd), smem, s, Cluster{2}, mq, mk, prm);
}

template <int NJ, int G>
cudaError_t launch_reduce(const Geom &g, const float2 *pairs, int Ns, int pitch, const uint8_t *refresh, double *scores, cudaStream_t s) {
  constexpr int smem = G * NJ * 32 * (int)sizeof(double);
  cudaError_t e = allow_shared_memory(antidiag_reduce_kernel<NJ, G>, smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(antidiag_reduce_kernel<NJ, G>, dim3(g.nb, g.R), dim3(32 * G), (size_t)smem, s, pairs, Ns, g.nb, pitch, refresh, scores);
}
// The instance for the words of a row, an even number of them.  (With one for up to 8, 16, 24 or 32, and eight warps for the four groups
// of a 64-token block, whole calls, us, then / now: 12 heads x 512 blocks of 64 257.6 / 232.2, 40 x 200 174.7 / 165.7, 4 x 591 of 128
// 337.5 / 313.6.)
template <int G, int NJ = 2>
cudaError_t launch_reduce_of(int nj, const Geom &g, const float2 *pairs, int Ns, int pitch, const uint8_t *refresh, double *scores, cudaStream_t s) {
  if constexpr (NJ < HEART_MAX_BLOCKS / 32)
    if (nj > NJ) return launch_reduce_of<G, NJ + 2>(nj, g, pairs, Ns, pitch, refresh, scores, s);
  return launch_reduce<NJ, G>(g, pairs, Ns, pitch, refresh, scores, s);
}

}  // namespace

cudaError_t launch_antidiag_scores(const Geom &g, const Workspace &w, const void *Q, const void *K,
                                   const uint8_t *refresh, cudaStream_t s, int *launches) {
  const int Ns = g.N / kS, grp = g.block / kS, pitch = ((g.nb + 31) / 32) * 32;
  if (Ns > 0) {
    CUtensorMap mq, mk;
    if (!make_group_map(&mq, Q, g, Ns, 128) || !make_group_map(&mk, K, g, Ns, 128)) return cudaErrorInvalidValue;
    AdParams prm;
    prm.pairs = reinterpret_cast<float2 *>(w.pairs);
    prm.refresh = refresh;
    prm.status = w.status;
    prm.H = g.H;
    prm.Ns = Ns;
    prm.nb = g.nb;
    prm.R = g.R;
    prm.c2 = (float)(g.scale / (double)kS * 1.4426950408889634);
    prm.test_skip_copy = 0;
#ifdef HEART_TEST_HOOKS
    prm.test_skip_copy = (g.flags & 0x80000000u) ? 1 : 0;
#endif
    const int smem = kStagesAd * kStageBytes + 1024 + 256;
    const long long tiles = (long long)g.R * ((Ns + kMt - 1) / kMt) * ((Ns + kNt - 1) / kNt);
    cudaError_t e = grp == 4 ? launch_scores<4>(mq, mk, prm, tiles, smem, s) : launch_scores<8>(mq, mk, prm, tiles, smem, s);
    if (e != cudaSuccess) return e;
    ++*launches;
  }
  const float2 *pairs = reinterpret_cast<const float2 *>(w.pairs);
  const int nj = (g.nb + 31) / 32;
  cudaError_t e = grp == 4 ? launch_reduce_of<4>(nj, g, pairs, Ns, pitch, refresh, w.scores, s)
                           : launch_reduce_of<8>(nj, g, pairs, Ns, pitch, refresh, w.scores, s);
  ++*launches;
  return e;
}

}  // namespace heart
