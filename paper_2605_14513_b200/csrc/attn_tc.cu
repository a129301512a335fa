// Block-sparse attention with online softmax on the sm_100a tensor cores.
//
// A query tile is 128 rows of one head: one query block of 128 tokens, or two query blocks of 64 whose
// lists are merged (two flag bits per key block; rows of the half that does not list a key block get
// weight 0 there).  Keys are processed 128 at a time: a "key step" is one 128-token block or two listed
// 64-token blocks.
//
// What bounds it: for a 128 x 128 tile the tensor pipe needs 1024 clocks (512 for Q K^T, 512 for P V), the
// special-function units 1024 as well (ex2 issues every 8 clocks per sub-partition) and shared memory
// 1280 (operands of the products and the TMA writes, 128 bytes a clock).  The chain softmax -> products
// -> softmax of one step is about 3000 clocks long, hand-overs included, so it has to be off the critical
// path: one persistent CTA per SM works on one query tile at a time and two softmax warpgroups take its
// key steps (nearly) in turn.  Scores are double-buffered in tensor memory, and because P has columns of its own,
// S_{h+2} is computed as soon as the scores of step h sit in registers: a warpgroup finds its next
// scores ready when it ends a step.  (Two streams on different tiles with P over the scores, one
// warpgroup each, ran at 1870-2100 clocks per tile and step: each stream waited 1200-1500 of ~3900 clocks for
// its next scores.)  Tiles are drawn from a counter; the loads and the first scores of the next tile
// overlap the end of the present one.
//
// Warp roles (registers are moved from the helper warps to the softmax warps at start); g counts the key
// steps of a CTA over all its tiles, buffers and barriers go by g & 1:
//   warps 0-3, 4-7  softmax of a step: one thread per query row (lane quarter = warp & 3).  A
//               thread loads its row of S_g (128 columns), hands the buffer back, takes the max, agrees on the
//               row's reference with its partner in the other warpgroup, writes P_g = 2^(s*scale*log2e - m)
//               as bf16 and adds the row sum.  The warpgroup that does not have a tile's last step takes the first one of the
//               next tile and then writes O / l (and lse) of the tile, by a bulk copy from the place of its Q; meanwhile the
//               other one takes the second and the third.  (The warpgroup of the last step waited 1300 clocks for the last
//               products and wrote for 3300 more, with its partner waiting for its step of the next tile: 40 x 33k, 69 tiles a
//               CTA, 2860 us, now 2745; 2 x 12 x 2465 72.5, now 69.5.)  A tile of one step, with many tiles of two, is still written
//               by the warpgroup of its last step, before that one goes on.
//   warp 8      issues S_g = Q K_g^T once step g - 2 has emptied the buffer, warp 11 O += P_g V_g.
//   warp 9      V producer, warp 10 K and Q producer (draws the tiles and announces them): TMA loads
//               (cp.async.bulk.tensor, 128-byte swizzle, completion on mbarriers), two 32 KB buffers each.
// The reference: m_g = m_{g-1} unless the row's maximum of step g exceeds it by more than 2^8.  Each warp
// publishes the references of its 32 rows after the maximum of every step and reads those of the step
// before; a row whose reference moved gets its part of O rescaled by the warp that moved it, once the
// products of the steps before are complete, and both partners rescale their own row sums.
// Tensor memory: O (128 columns) | S[2] (2 x 128) | P[2] (2 x 64).
//
// Instructions: an SM keeps 32 KB of them (a loop of 24 KB runs at full rate, one of 48 KB at a third), the kernel has 60, and
// twelve warps are in different places of it.  So the loop over a softmax warp's steps holds only what every step needs, in one
// piece; what a step rarely needs (a wait that takes long, a ragged block, a reference that moves) stands outside and the loop is left
// for it.  With those in the loop 12 x 33k fetched 1.7 times as often and 2 x 12 x 2465 1.4 times, in 4 and 10 % more clocks.
// (A small launch goes through all of them once: there they stand where they are needed, 0.1 to 0.4 us of 13 to 24.)
//
// The step lists come from attn_plan_kernel (one warp per tile), which runs just before; the tiles are
// taken in the order of tile_order_kernel: head-major (the K/V of one or two heads stay in L2), within a
// head by the first key block of their lists once a head's K and V no longer fit one die's half of the L2,
// except for the launch's last tiles (up to 1024; all of a small launch), which go longest-list-first so that the
// launch does not end on a long tile that started late.
//
// Small launches (a tile per CTA at most) have an instance of their own, which plans its tile itself while Q comes in and, while
// tiles are few, shares its key steps among a cluster of 2 or 4 CTAs: each CTA copies the others their share of the rows of its
// part of O as soon as it has it, and puts its own share together.  2 heads x 2045 tokens, half of the blocks listed: 14.4 us when
// the CTAs read one another's parts behind a barrier, with the roles' first instructions and Q fetched behind the plan,
// 12.6 now.  (A first call of the merge code ahead of the wait, writing nothing, to have its instructions there: 12.9.)
//
// Every wait is bounded; a wait that runs out raises the CTA's abort flag and the status word, its roles
// drain and stop.  A tile whose products are complete is still written; the tile that the wait was for and those the CTA had drawn
// already, or was dealt, stay unwritten (as does a tile that a cluster shares); the other CTAs take the rest.
#include <cuda.h>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace heart {
using namespace tc;

constexpr int kAttnThreads = 384;
constexpr int kWarpQK = 8, kWarpV = 9, kWarpK = 10, kWarpPV = 11;
constexpr int kRegsSoftmax = 224, kRegsHelper = 56;  // 224 * 256 + 56 * 128 = the CTA's 384 x 168
constexpr int kTileBytes = 32768;  // 128 rows x 128 dims: [2 dim halves][128 rows][64] bf16, 128-byte swizzle
constexpr int kTileRing = 4;       // announced tiles
constexpr int kTileReaders = 11;   // softmax warps, issuers, V producer
constexpr float kNoReference = -3.0e38f;  // below every logit: the first step moves it
// A row's reference is set kHeadroom (log2) above the row's maximum, and moves when a maximum exceeds it by kMaxGrowth.
// A move costs a rescale of O behind the products in flight, so a row should climb far before its next one: 40 x 33k
// takes 3.47 ms if it moves 2^8 above the last maximum, 2.77 at 2^16, 2.69 at 2^24 and beyond.  Most of the room lies
// below 1: weights are at most 2^8, so n keys with values up to 2^120 / n cannot overflow O (all of it above 1, with
// weights up to 2^64, left 2^64 / n), and a weight of 2^-110 of the largest is still a normal number.
constexpr float kHeadroom = 16.f, kMaxGrowth = 8.f;
// ns that a softmax warp waits for its scores before it leaves the loop over its steps for a bounded wait.  (Nothing hangs on it: us with
// 20 and with 500, 24 x 119k 10941 and 10959, 40 x 76k 13146 and 13165, 16 x 8k 141.7 and 142.0, antidiagonal 12 x 33k 1073 and 1071, where
// two runs differ by as much.)
constexpr uint32_t kShortWait = 500;
constexpr int kMaxSplit = 4;  // CTAs that share a tile in a small launch

// Shared-memory plan (the dynamic allocation itself is 1024-byte aligned).
constexpr int kOffQ = 0, kOffK = 2 * kTileBytes, kOffV = 4 * kTileBytes;
constexpr int kOffPart = 6 * kTileBytes, kOffBar = kOffPart + kTileBytes / 2;  // small launches: the third part of a shared tile

struct AttnShared {
  uint64_t q_full[2], k_full[2], v_full[2];  // TMA -> issuer
  uint64_t s_full[2];      // S_g complete (K_g is free)
  uint64_t s_free[2];      // S_g is in registers (one arrival per softmax warp)
  uint64_t p_full[2];      // P_g written (one arrival per softmax warp)
  uint64_t pv_done[2];     // P_g V_g complete (V_g and P_g are free)
  uint64_t m_ready[2][4];  // references after step g, per lane quarter
  uint64_t o_full[2];      // the products of a tile are complete, per tile & 1 (a barrier of its own: the warpgroup that waits for it
                           // may be two phases of pv_done behind)
  uint64_t o_free;         // O of a tile has been read
  uint64_t out_done[2];    // a tile's output has left the place of its Q
  uint64_t tile_full[kTileRing], tile_empty[kTileRing];
  uint64_t drain[2];       // abort path: the issuers' products in flight have landed
  int4 tile[kTileRing];    // query tile of its head, listed key blocks, head, batch entry (-1: no tile left)
  uint32_t entry[4];       // the key steps in flight, for the softmax warps: entry[g & 3] is written before K_g is asked
                           // for and read before the scores of step g are handed back, which K_{g+4} waits for
  float m[2][128];         // references after step g
  float2 l[2][2][128];     // row sums and their references for the warpgroup that writes a tile: per tile & 1 and warpgroup; in a small
                           // launch the ones of the tile's last step, and those of the writer
  int4 written[2][8];      // that tile, per softmax warp
  uint32_t tmem_base;
  int abort;
  // small launches: the parts of a tile that this CTA puts together, the tile's plan
  uint64_t parts_full;     // the other CTAs' parts have arrived
  alignas(16) float2 part_l[128];      // row sums and references of this CTA's part (a row sum of -1: it gave up)
  alignas(16) float2 in_l[kMaxSplit - 1][128 / 2];  // of the rows that this CTA puts together, from the other CTAs
  uint32_t sets[2][32];
  uint32_t steps[HEART_MAX_BLOCKS];
};
constexpr int kAttnSmem = kOffBar + sizeof(AttnShared);

// A key step as the plan kernel writes it.  128-token blocks: the key block.  64-token blocks: two
// halves of 16 bits, key block | (flag of query block 0, flag of query block 1) << 10 | ragged block << 12; no
// flag: the keys do not count (the second half of the last step when the number of blocks is odd).
struct AttnParams {
  const uint32_t *steps;  // [B*H][tiles of a head][step_pitch]
  const uint4 *tiles;     // [tiles of the launch] (tile of the head | listed key blocks << 16, head of the launch,
                          // first step, first key block), in launch order
  int32_t *counter;       // tiles drawn beyond the first one of every CTA (zeroed by the plan kernel)
  uint16_t *O;
  float *lse;
  int32_t *status;
  long long sb, sh, sn;
  int H, N, nb, n_tiles, n_tiles_per_head, step_pitch, dense;
  int h0, hcount;  // this launch covers heads [h0, h0 + hcount) of every batch entry
  float scale_log2;
  int split;        // small launches: CTAs (one cluster) that share the key steps of a tile
  short at_once;    // a tile of at most so many steps is written by the warpgroup of its last step, before that one goes on
  short late;       // the warpgroup with a tile's first step takes its next one a step later: CTAs have several tiles
  // test-hook builds only: CTA 0 leaves out the V copy of its second key step (1) or the K copy of its second tile's first
  // step (2), CTA 1 does not send its part of a shared tile (4)
  int test_skip;
};

__device__ __forceinline__ float fmax3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

struct Sums {
  float a, b, c, d;
};
// Weights 2^(s*c - m) of 32 scores of a row, packed to bf16, and their sums.  The row sum is taken over the
// rounded weights, the ones the P V product really uses, so numerator and denominator carry the same
// rounding: O stays a weighted mean.
__device__ __forceinline__ void exp32(const uint32_t *s, uint64_t c2, uint64_t neg_m2, uint32_t *pk, Sums &sums) {
#pragma unroll
  for (int i = 0; i < 32; i += 4) {
    float x0, x1, x2, x3;
    unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(s[i]), __uint_as_float(s[i + 1])), c2, neg_m2), x0, x1);
    unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(s[i + 2]), __uint_as_float(s[i + 3])), c2, neg_m2), x2, x3);
    pk[i >> 1] = pack_bf16x2(ex2(x0), ex2(x1));
    pk[(i >> 1) + 1] = pack_bf16x2(ex2(x2), ex2(x3));
    add_bf16x2_to_f32(sums.a, sums.b, pk[i >> 1]);
    add_bf16x2_to_f32(sums.c, sums.d, pk[(i >> 1) + 1]);
  }
}
__device__ __forceinline__ float max64(const uint32_t *s) {
  float m[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
  for (int i = 0; i < 64; i += 8)
#pragma unroll
    for (int j = 0; j < 4; ++j) m[j] = fmax3(m[j], __uint_as_float(s[i + 2 * j]), __uint_as_float(s[i + 2 * j + 1]));
  return fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3]));
}

struct PlanParams {
  const int32_t *kv_idx, *kv_cnt;  // [B*H][nb][idx_stride], [B*H][nb]
  int nb, ncph, idx_stride;        // ncph: tiles of a head
  int H, h0, hcount;
  int ragged;                      // the last block is not whole
  int32_t *status;
};
// The step list of tile n of a launch, by one warp; it goes to out_of(tile among all heads).  The lists of the tile's query blocks (any
// order; entries out of range are skipped and reported, duplicates merged) become bit sets, and those the
// list of key steps.  64-token blocks: key blocks that both query blocks list come first, then blocks of
// query block 0 paired with blocks of query block 1, so that in such a step every row has 64 exponentials
// to take instead of half of the rows 128; ascending within each group.
// Returns the tile's word (see AttnParams), in lane 0.
template <int B, typename OutOf>
__device__ __forceinline__ uint4 plan_tile(const PlanParams &p, int n, int lane, uint32_t (*sets)[32], OutOf out_of) {
  constexpr int QBT = 128 / B;  // query blocks per tile
  const int rr = n / p.ncph, t = n % p.ncph;
  const int r = (rr / p.hcount) * p.H + p.h0 + rr % p.hcount;
#pragma unroll
  for (int q = 0; q < QBT; ++q) sets[q][lane] = 0u;
  __syncwarp();
  bool bad = false;
  // The counts and the first 64 entries of the lists are asked for together (entries beyond the count are not
  // looked at): one trip to memory for a short list instead of one for each query block's count and list.
  int cnt[QBT], head[QBT][2];
#pragma unroll
  for (int q = 0; q < QBT; ++q) {
    const size_t row = (size_t)r * p.nb + t * QBT + q;
    const bool real = t * QBT + q < p.nb;
    cnt[q] = real ? __ldcg(&p.kv_cnt[row]) : 0;
#pragma unroll
    for (int i = 0; i < 2; ++i) head[q][i] = real && lane + 32 * i < p.idx_stride ? __ldcg(&p.kv_idx[row * p.idx_stride + lane + 32 * i]) : 0;
  }
#pragma unroll
  for (int q = 0; q < QBT; ++q) {
    if (cnt[q] < 0 || cnt[q] > p.idx_stride) {
      bad = true;
      cnt[q] = cnt[q] < 0 ? 0 : p.idx_stride;
    }
    auto list = [&](int J) {
      if (J < 0 || J >= p.nb)
        bad = true;  // skipped, reported
      else
        atomicOr(&sets[q][J >> 5], 1u << (J & 31));
    };
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (lane + 32 * i < cnt[q]) list(head[q][i]);
    const int32_t *row = p.kv_idx + ((size_t)r * p.nb + t * QBT + q) * p.idx_stride;
#pragma unroll 4
    for (int k = lane + 64; k < cnt[q]; k += 32) list(__ldcg(&row[k]));
  }
  __syncwarp();
  if (bad) atomicExch(p.status, HEART_ERR_DEVICE_CHECK);
  auto sum = [](int v) { return (int)__reduce_add_sync(0xffffffffu, (unsigned)v); };
  uint32_t *out = out_of(r * p.ncph + t);
  const uint32_t a = sets[0][lane], b = QBT == 2 ? sets[QBT - 1][lane] : 0u;
  const uint32_t any = a | b;
  const int U = sum(__popc(any));
  // 32 key blocks at a time, one per lane.  (A lane per word of the set, bit after bit, made the whole call 15.6 us
  // instead of 14.7 for 2 heads of 32 key blocks and 55.2 instead of 51.3 for 24 of 39; sparse lists over 512 and more
  // take the same time either way.)
  const unsigned has = __ballot_sync(0xffffffffu, any != 0u);  // words of the set that are not empty
  const uint32_t bit = 1u << lane, below = bit - 1u;
  if (B == 128) {
    int pos = 0;
    for (unsigned todo = has; todo; todo &= todo - 1) {
      const int n = __ffs(todo) - 1;
      const uint32_t m = __shfl_sync(0xffffffffu, a, n);
      if (m & bit) out[pos + __popc(m & below)] = n * 32 + lane;
      pos += __popc(m);
    }
  } else {
    uint16_t *out16 = reinterpret_cast<uint16_t *>(out);
    const int D = sum(__popc(a & b));
    int S0 = sum(__popc(a & ~b)), S1 = sum(__popc(b & ~a));
    int start = D;
    int n_both = 0, n_a = 0, n_b = 0;  // blocks of each kind so far; the one that goes to D is number -1
    if ((D & 1) && S0 + S1 > 0) {      // one single next to the last shared block; pairs start on a step
      if (S0 >= S1) {
        n_a = -1;
        --S0;
      } else {
        n_b = -1;
        --S1;
      }
      ++start;
    }
    const int paired = min(S0, S1);
    int last = -1;  // the last listed block, in the lane that writes it
    for (unsigned todo = has; todo; todo &= todo - 1) {
      const int n = __ffs(todo) - 1;
      const uint32_t wa = __shfl_sync(0xffffffffu, a, n), wb = __shfl_sync(0xffffffffu, b, n);
      const uint32_t both = wa & wb, only_a = wa & ~wb, only_b = wb & ~wa;
      if ((wa | wb) & bit) {
        const int J = n * 32 + lane, q = (only_b & bit) ? 1 : 0;
        const int k = q ? n_b + __popc(only_b & below) : n_a + __popc(only_a & below);
        const int at = (both & bit) ? n_both + __popc(both & below) : k < 0 ? D : k < paired ? start + 2 * k + q : start + paired + k;
        const int flags = ((wa & bit) ? 1 : 0) | ((wb & bit) ? 2 : 0);
        out16[at] = (uint16_t)(J | flags << 10 | (p.ragged && J == p.nb - 1 ? 1 << 12 : 0));
        last = at == U - 1 ? J : last;
      }
      n_both += __popc(both);
      n_a += __popc(only_a);
      n_b += __popc(only_b);
    }
    if ((U & 1) && last >= 0) out16[U] = (uint16_t)last;  // second half of the last step: the same block, without flags
  }
  const int src = has ? __ffs(has) - 1 : 0;
  const int first = __shfl_sync(0xffffffffu, lane * 32 + __ffs(any) - 1, src);
  __syncwarp();  // the first step, written by some lane, is read back
  return make_uint4((uint32_t)t | (uint32_t)U << 16, rr, has ? *(volatile uint32_t *)out : 0u, has ? first : 0x3ff);
}

// Plans of all tiles of a launch, one warp per tile (a launch of at most one tile per SM makes them in the
// attention kernel instead).
constexpr int kPlanWarps = 8;

template <int B>
__global__ void __launch_bounds__(32 * kPlanWarps)
    attn_plan_kernel(const PlanParams p, int n_tiles, int step_pitch, uint32_t *__restrict__ steps, uint4 *__restrict__ tiles,
                     int32_t *__restrict__ counter) {
  __shared__ uint32_t sets[kPlanWarps][128 / B][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n = blockIdx.x * kPlanWarps + warp;
  pdl_wait();  // the lists come from the kernel before this one
  pdl_launch_dependents();
  if (blockIdx.x == 0 && threadIdx.x == 0) *counter = 0;
  if (n >= n_tiles) return;
  const uint4 word = plan_tile<B>(p, n, lane, sets[warp], [&](int tile) { return steps + (size_t)tile * step_pitch; });
  if (lane == 0) tiles[n] = word;
}

// Small launches: rows [rank * rows, (rank + 1) * rows) of a shared tile from the parts of the cluster's CTAs, by the
// softmax warps.
struct PartAddresses {
  uint32_t own, own_l, slot, slot2, in_l;  // in shared memory
};
__device__ __forceinline__ void merge_parts(const PartAddresses at, int rank, int split, int valid_rows, uint16_t *out, long long sn,
                                            float *lse) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, rows = 128 / split;
  // a warp: four rows at a time, eight lanes each, lane q of them pieces q, q + 8, q + 16 and q + 24 of four dims
#pragma unroll 1
  for (int i0 = warp * 4 + (lane >> 3); i0 < rows; i0 += 32) {
    const int row = rank * rows + i0, q = lane & 7;
    float l[kMaxSplit], m[kMaxSplit], m_all = kNoReference, l_all = 0.f;
    uint32_t src[kMaxSplit];
    bool gave_up = false;
#pragma unroll
    for (int i = 0; i < kMaxSplit; ++i) {
      // parts are held in the order of the CTAs behind this one, its own last
      const int place = (i - rank - 1 + split) & (split - 1);
      const bool own = place == split - 1;
      src[i] = own ? at.own + row * 512 : (place < 2 ? at.slot + place * (kTileBytes / 2) : at.slot2) + i0 * 512;
      const float2 lm = lds2(own ? at.own_l + row * 8 : at.in_l + place * (128 / 2 * 8) + i0 * 8);
      l[i] = i < split ? lm.x : 0.f;
      m[i] = l[i] != 0.f ? lm.y : kNoReference;  // (a part without keys)
      gave_up |= l[i] == -1.f;
      m_all = fmaxf(m_all, m[i]);
    }
    float4 o[4] = {};
#pragma unroll
    for (int i = 0; i < kMaxSplit; ++i) {
      if (i >= split) break;
      if (l[i] != 0.f) {  // (a part without keys has zeros; a sum that is not a number goes into the row's result)
        const float f = ex2(m[i] - m_all);
        l_all = fmaf(l[i], f, l_all);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float4 x = lds4(src[i] + (((q + 8 * k) ^ (row & 7)) << 4));
          o[k].x = fmaf(x.x, f, o[k].x);
          o[k].y = fmaf(x.y, f, o[k].y);
          o[k].z = fmaf(x.z, f, o[k].z);
          o[k].w = fmaf(x.w, f, o[k].w);
        }
      }
    }
    const float inv = l_all > 0.f ? 1.f / l_all : 0.f;
    if (row < valid_rows && !gave_up) {  // (a tile of which a part gave up is not written)
#pragma unroll
      for (int k = 0; k < 4; ++k)
        *reinterpret_cast<uint2 *>(out + row * sn + (q + 8 * k) * 4) = make_uint2(pack_bf16x2(o[k].x * inv, o[k].y * inv), pack_bf16x2(o[k].z * inv, o[k].w * inv));
      if (q == 0 && lse != nullptr) lse[row] = l_all > 0.f ? (m_all + log2f(l_all)) * 0.6931471805599453f : -INFINITY;
    }
  }
}

template <int B, bool Small>
__global__ void __launch_bounds__(kAttnThreads, 1)
    attn_tc_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                   const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_o, const AttnParams p,
                   const PlanParams plan) {
  extern __shared__ __align__(1024) unsigned char smem[];
  AttnShared &sh = *reinterpret_cast<AttnShared *>(smem + kOffBar);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool dense = B == 128 && p.dense;  // (dense calls come with blocks of 128)
  volatile int *abort = &sh.abort;

  // ------------------------------------------------------------------ set-up
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(&sh.q_full[i], 1);
      mbar_init(&sh.k_full[i], 1);
      mbar_init(&sh.v_full[i], 1);
      mbar_init(&sh.s_full[i], 1);
      mbar_init(&sh.s_free[i], 4);
      mbar_init(&sh.p_full[i], 4);
      mbar_init(&sh.pv_done[i], 1);
      for (int q = 0; q < 4; ++q) mbar_init(&sh.m_ready[i][q], 1);
    }
    for (int i = 0; i < kTileRing; ++i) {
      mbar_init(&sh.tile_full[i], 1);
      mbar_init(&sh.tile_empty[i], kTileReaders);
    }
    mbar_init(&sh.o_full[0], 1);
    mbar_init(&sh.o_full[1], 1);
    mbar_init(&sh.o_free, 4);
    mbar_init(&sh.out_done[0], 4);
    mbar_init(&sh.out_done[1], 4);
    mbar_init(&sh.drain[0], 1);
    mbar_init(&sh.drain[1], 1);
    mbar_init(&sh.parts_full, 1);
    if (Small) {  // this CTA's only tile, but for the number of its key blocks
      const int n = blockIdx.x / p.split, hr = n / p.n_tiles_per_head, b = hr / p.hcount;
      sh.tile[0] = make_int4(n - hr * p.n_tiles_per_head, p.nb, p.h0 + hr - b * p.hcount, b);
    }
    sh.abort = 0;
    mbar_fence_init();
  }
  if (warp == kWarpQK) {
    tmem_alloc(&sh.tmem_base, 512);
    tmem_relinquish();
  }
  if (warp == kWarpK && lane == 0) {
    tma_prefetch_desc(&map_q);
    tma_prefetch_desc(&map_k);
    tma_prefetch_desc(&map_v);
    tma_prefetch_desc(&map_o);
  }
  const int rank = Small ? (int)cluster_ctarank() : 0;
  const PartAddresses parts = {smem_u32(smem + kOffK), smem_u32(sh.part_l), smem_u32(smem + kOffQ + kTileBytes), smem_u32(smem + kOffPart),
                               smem_u32(sh.in_l)};
  if (Small) {  // the barriers are initialised: for the Q copy below, and for the other CTAs' parts
    if (p.split > 1) cluster_sync();
    else __syncthreads();
  }
  // Launched with programmatic stream serialisation: everything above overlaps the end of the kernels
  // before it.  A kernel that follows (the next layer-step's block-sum pass) may be scheduled once every
  // CTA of this launch has started: its CTAs then fill the SMs that finish first.
  // (In a small launch the roles wait where their code is: fetched only behind the plan, its first lines took 1 us.)
  if (!Small) pdl_wait();
  pdl_launch_dependents();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sh.tmem_base;

  // Key steps of a tile with U listed key blocks that this CTA takes, and the first one of them.  (A tile of fewer than four steps is
  // not shared: its cluster's first CTA takes it and the others leave.  64 tiles, us with two CTAs on each tile and with one: two steps
  // 10.0 and 9.2, three 10.6 and 10.2, four 10.7 and 10.9; 32 tiles with four CTAs 10.7 and 9.0, 10.6 and 10.1, 10.8 and 10.8.)
  bool shared_tile = false, at_barrier = false;
  int parts_of_tile = 1;
  auto first_step = [&](int U, int part) -> int { return Small ? (B == 128 ? U : (U + 1) / 2) * part / parts_of_tile : 0; };
  auto n_steps_of = [&](int U) -> int { return Small ? first_step(U, rank + 1) - first_step(U, rank) : B == 128 ? U : (U + 1) / 2; };
  auto steps_of = [&](const int4 &ti) -> const uint32_t * {
    if (Small) return sh.steps + first_step(ti.y, rank);
    return p.steps + ((size_t)(ti.w * p.H + ti.z) * p.n_tiles_per_head + ti.x) * p.step_pitch;
  };
  auto step_entry = [&](const uint32_t *steps, int h) -> uint32_t {
    if (!dense) return Small ? steps[h] : __ldcg(&steps[h]);
    return Small ? h + first_step(p.nb, rank) : h;
  };
  // Waits of a whole warp; ok turns false when one runs out or the CTA aborts.  The usual case is a barrier
  // that is complete already.
  bool ok = true;
  auto out_of_time = [&](uint32_t &since) -> bool {  // since: 0 at a wait's first call
    const uint32_t now = clock() | 1u;
    if (since == 0) since = now;
    if (*abort == 0 && now - since <= (uint32_t)kWaitLimitCycles) return false;
    *abort = 1;
    return true;
  };
  auto wait = [&](uint64_t *bar, uint32_t parity) {
    uint32_t since = 0;
#pragma unroll 1
    while (__builtin_expect(!__all_sync(0xffffffffu, mbar_try_wait(bar, parity)), 0))
      if (__any_sync(0xffffffffu, out_of_time(since))) return ok = false;
    return ok;
  };
  auto wait1 = [&](uint64_t *bar, uint32_t parity) {  // by one thread
    uint32_t since = 0;
#pragma unroll 1
    while (__builtin_expect(!mbar_try_wait(bar, parity), 0))
      if (out_of_time(since)) return ok = false;
    return ok;
  };
  auto small_tile = [&](int U) {
    shared_tile = p.split > 1 && (B == 128 ? U : (U + 1) / 2) >= 4;
    parts_of_tile = shared_tile ? p.split : 1;
  };
  // The announced tile t; false: none left (or abort).  Every lane of the warp gets the same answer.
  auto next_tile = [&](int t, int4 &ti) -> bool {
    if (Small) {
      if (t > 0 || !wait(&sh.tile_full[0], 0)) return false;
      ti = sh.tile[0];
      small_tile(ti.y);
      return rank < parts_of_tile;
    }
    const int i = t % kTileRing;
    if (!wait(&sh.tile_full[i], (t / kTileRing) & 1)) return false;
    ti = sh.tile[i];
    __syncwarp();
    if (lane == 0) mbar_arrive(&sh.tile_empty[i]);
    return ti.w >= 0;
  };
  // K of one key step into a 32 KB buffer: [dim half][128 keys][64 dims]
  auto load_k = [&](unsigned char *dst, uint64_t *bar, uint32_t e, int hidx, int bidx) {
    mbar_expect_tx(bar, kTileBytes);
    if (B == 128) {
      tma_load_5d(dst, &map_k, bar, 0, (int)e * 128, 0, hidx, bidx);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i)  // dim half i >> 1 of block i & 1
        tma_load_5d(dst + i * (kTileBytes / 4), &map_k, bar, 0, (int)((e >> (16 * (i & 1))) & 0x3ff) * 64, i >> 1, hidx, bidx);
    }
  };
  // V: [block][dim half][64 keys][64 dims] for blocks of 64.  A product takes 16 keys, so blocks may lie apart, and a copy
  // brings whole rows: two copies a step instead of four (whole steps of 40 x 33k 2839 us instead of 2882, 12 x 33k 1185 instead of
  // 1196, 8 x 33k 433 instead of 445; dense 12 x 33k 5744 instead of 5788).
  auto load_v = [&](unsigned char *dst, uint64_t *bar, uint32_t e, int hidx, int bidx) {
    mbar_expect_tx(bar, kTileBytes);
#pragma unroll
    for (int i = 0; i < 128 / B; ++i)
      tma_load_5d(dst + i * (kTileBytes / 2), &map_v, bar, 0, B == 128 ? (int)e * 128 : (int)((e >> (16 * i)) & 0x3ff) * 64, 0, hidx, bidx);
  };
  // Shared memory must not be released under a copy in flight: a producer that stops early (abort)
  // waits, bounded, for the copies it has issued.
  auto settle = [&](uint64_t *bar, uint32_t parity) {
    const uint32_t t0 = clock();
    while (!mbar_try_wait(bar, parity) && (uint32_t)clock() - t0 < 40000000u) {
    }
  };
  auto settle_pair = [&](uint64_t *bar, int issued) {  // the last two of `issued` copies on a pair of barriers
#pragma unroll 1
    for (int i = issued > 2 ? issued - 2 : 0; i < issued; ++i) settle(&bar[i & 1], (i >> 1) & 1);
  };

  // Descriptors differ only in the start-address field (low word, no carry out of it): base + an offset in
  // 16-byte units.
  auto desc_at = [](uint64_t desc, uint32_t off16) -> uint64_t {
    return (desc & 0xffffffff00000000ull) | (uint32_t)((uint32_t)desc + off16);
  };
  // Tensor memory must not be released under a product in flight either: after an abort a commit arrives
  // once everything the issuing lane has issued is complete; the wait for it is bounded like the others.
  auto drain_products = [&](bool leader, uint64_t *bar) {
    if (!*abort) return;
    if (leader) tc_commit(bar);
    __syncwarp();
    settle(bar, 0);
  };

  // ------------------------------------------------------------------ roles
  if (warp >= kWarpQK) setmaxnreg_dec<kRegsHelper>();
  if (warp == kWarpK) {
    if (Small) pdl_wait();
    if (lane == 0) {  // ===== K and Q producer
      int g = 0, nq = 0;     // key steps loaded, tiles with key steps
      if (Small) {
        // the launch's only tile of this CTA is known before its plan is: its Q comes in meanwhile
        int4 ti = sh.tile[0];
        mbar_expect_tx(&sh.q_full[0], kTileBytes);
        tma_load_5d(smem + kOffQ, &map_q, &sh.q_full[0], 0, ti.x * 128, 0, ti.z, ti.w);
        wait1(&sh.tile_full[0], 0);
        ti = sh.tile[0];
        small_tile(ti.y);
        const int n_steps = ok && rank < parts_of_tile ? n_steps_of(ti.y) : 0;
        const uint32_t *steps = steps_of(ti);
#pragma unroll 1
        for (; g < n_steps; ++g) {
          if (g >= 2) wait1(&sh.s_full[g & 1], ((g - 2) >> 1) & 1);
          if (!ok) break;
          const uint32_t e = step_entry(steps, g);
          sh.entry[g & 3] = e;
          load_k(smem + kOffK + (g & 1) * kTileBytes, &sh.k_full[g & 1], e, ti.z, ti.w);
        }
      }
      // The first tile of every CTA is fixed, the others are drawn.  Dense tiles are all
      // of one length: dealt in turn, so that dense calls share nothing and may overlap on one workspace.  (Drawn, the faster
      // SMs take the odd tiles: 12 x 33k 5604 us, dealt 5721.)
      int n = blockIdx.x;
#pragma unroll 1
      for (int t = 0; !Small; ++t) {
        int4 ti = make_int4(0, 0, 0, -1);
        uint32_t e = 0;  // its next key step, fetched ahead of time
        if (n < p.n_tiles) {
          uint4 word;
          if (dense) {
            word.y = n / p.n_tiles_per_head;
            word.x = (n - word.y * p.n_tiles_per_head) | (uint32_t)p.nb << 16;
            word.z = step_entry(nullptr, 0);
          } else {
            word = __ldcg(&p.tiles[n]);
          }
          e = word.z;
          ti.x = word.x & 0xffff;
          ti.y = word.x >> 16;
          ti.w = (int)word.y / p.hcount;
          ti.z = p.h0 + (int)word.y - ti.w * p.hcount;
        }
        const int i = t % kTileRing;
        if (t >= kTileRing && !wait1(&sh.tile_empty[i], (t / kTileRing - 1) & 1)) break;
        sh.tile[i] = ti;
        mbar_arrive(&sh.tile_full[i]);
        if (ti.w < 0) break;
        const int n_steps = n_steps_of(ti.y);
        const uint32_t *steps = steps_of(ti);
        int n_next = dense ? n + gridDim.x : 0;
        if (n_steps == 0 && !dense) n_next = gridDim.x + atomicAdd(p.counter, 1);
#pragma unroll 1
        for (int h = 0; h < n_steps; ++h, ++g) {
          const uint32_t e_next = h + 1 < n_steps ? step_entry(steps, h + 1) : 0u;
          if (g >= 2 && !wait1(&sh.s_full[g & 1], ((g - 2) >> 1) & 1)) break;
          sh.entry[g & 3] = e;
#ifdef HEART_TEST_HOOKS
          if (!((p.test_skip & 2) && blockIdx.x == 0 && t == 1 && h == 0))
#endif
          load_k(smem + kOffK + (g & 1) * kTileBytes, &sh.k_full[g & 1], e, ti.z, ti.w);
          if (h == 0) {
            // its buffer is free: the last step of the tile before the previous one is complete, its output gone
            if (nq >= 2 && !wait1(&sh.out_done[nq & 1], ((nq - 2) >> 1) & 1)) break;
            mbar_expect_tx(&sh.q_full[nq & 1], kTileBytes);
            tma_load_5d(smem + kOffQ + (nq & 1) * kTileBytes, &map_q, &sh.q_full[nq & 1], 0, ti.x * 128, 0, ti.z, ti.w);
            ++nq;
          }
          // The next tile is drawn at the last moment that hides the trip to memory: drawn with the first step, a
          // CTA on a long tile already owned another one while others ran out (2 x 12 x 2465: 56.9 us against 55.2).
          if (h == n_steps - 1 && !dense) n_next = gridDim.x + atomicAdd(p.counter, 1);
          e = e_next;
        }
        if (!ok) break;
        n = n_next;
      }
      if (Small) settle(&sh.q_full[0], 0);  // (a CTA without a step has not waited for it)
      if (*abort) {
        if (!Small) settle_pair(sh.q_full, nq);
        settle_pair(sh.k_full, g);
      }
    }
  } else if (warp == kWarpV) {
    // ===== V producer
    if (Small) pdl_wait();
    int g = 0;
    int4 ti;
#pragma unroll 1
    for (int t = 0; ok && next_tile(t, ti); ++t) {
      const int n_steps = n_steps_of(ti.y);
      const uint32_t *steps = steps_of(ti);
      uint32_t e_next = n_steps > 0 ? step_entry(steps, 0) : 0u;
#pragma unroll 1
      for (int h = 0; h < n_steps; ++h, ++g) {
        const uint32_t e = e_next;
        if (h + 1 < n_steps) e_next = step_entry(steps, h + 1);
        if (g >= 2 && !wait(&sh.pv_done[g & 1], ((g - 2) >> 1) & 1)) break;
#ifdef HEART_TEST_HOOKS
        // Test-only library: one V tile is never requested (neither the byte count nor the copy), so the
        // waits that depend on it run out and the abort path is taken.
        if ((p.test_skip & 1) && blockIdx.x == 0 && g == 1) continue;
#endif
        if (lane == 0) load_v(smem + kOffV + (g & 1) * kTileBytes, &sh.v_full[g & 1], e, ti.z, ti.w);
      }
    }
    if (*abort && lane == 0) settle_pair(sh.v_full, g);
  } else if (warp == kWarpQK) {
    // ===== issuer of the score products.  The whole warp runs the loop (uniform control flow keeps the
    // descriptors in uniform registers), one elected lane issues.  The two kinds of products have a warp
    // each: a step costs an issuing warp some 400 clocks of waits and hand-overs besides the products.
    constexpr uint32_t idesc = idesc_bf16_f32(128, 128, false, false);
    // Q, K (K-major): 64 dims = one 128-byte row; the dim halves are 128*128 B apart.
    const uint64_t q_desc = smem_desc_sw128(smem_u32(smem + kOffQ), 16, 1024);
    const uint64_t k_desc = smem_desc_sw128(smem_u32(smem + kOffK), 16, 1024);
    const bool leader = elect_one();  // the same lane every time: commits track its MMAs
    if (Small) pdl_wait();
    uint32_t g = 0, nq = 0;           // key steps and tiles with key steps so far
    int4 ti;
#pragma unroll 1
    for (int t = 0; ok && next_tile(t, ti); ++t) {
      const int n_steps = n_steps_of(ti.y);
      if (n_steps == 0) continue;
      wait(&sh.q_full[nq & 1], (nq >> 1) & 1);
      const uint64_t qd = desc_at(q_desc, (nq & 1) * (kTileBytes >> 4));
      ++nq;
#pragma unroll 1
      for (int h = 0; h < n_steps; ++h, ++g) {  // S_g = Q K_g^T
        const uint32_t b = g & 1;
        if (g >= 2) wait(&sh.s_free[b], ((g - 2) >> 1) & 1);
        if (!wait(&sh.k_full[b], (g >> 1) & 1)) break;
        tc_fence_after();
        if (leader) {
          const uint64_t kd = desc_at(k_desc, b * (kTileBytes >> 4));
#pragma unroll
          for (int ks = 0; ks < 8; ++ks)
            mma_ss(tmem + 128 + b * 128, desc_at(qd, (ks >> 2) * 1024 + (ks & 3) * 2), desc_at(kd, (ks >> 2) * 1024 + (ks & 3) * 2), idesc, ks > 0 ? 1u : 0u);
          tc_commit(&sh.s_full[b]);
        }
        __syncwarp();
      }
    }
    drain_products(leader, &sh.drain[0]);
  } else if (warp == kWarpPV) {
    // ===== issuer of the value products
    constexpr uint32_t idesc = idesc_bf16_f32(128, 128, false, true);
    // V (MN-major): 64 dims = one 128-byte row; dim halves B*128 B apart (the LBO); 16 keys = 16 rows = 2048 B per
    // k-step, the second block of 64 keys half a buffer on.
    const uint64_t v_desc = smem_desc_sw128(smem_u32(smem + kOffV), B * 128, 1024);
    const bool leader = elect_one();
    if (Small) pdl_wait();
    uint32_t g = 0, nt = 0;  // key steps and tiles with key steps so far
    int4 ti;
#pragma unroll 1
    for (int t = 0; ok && next_tile(t, ti); ++t) {
      const int n_steps = n_steps_of(ti.y);
      if (n_steps == 0) continue;
      if (nt > 0) wait(&sh.o_free, (nt - 1) & 1);
      ++nt;
#pragma unroll 1
      for (int h = 0; h < n_steps; ++h, ++g) {  // O (+)= P_g V_g
        const uint32_t b = g & 1;
        wait(&sh.v_full[b], (g >> 1) & 1);
        if (!wait(&sh.p_full[b], (g >> 1) & 1)) break;
        tc_fence_after();
        if (leader) {
          const uint64_t vd = desc_at(v_desc, b * (kTileBytes >> 4));
#pragma unroll
          for (int ks = 0; ks < 8; ++ks)
            mma_ts(tmem, tmem + 384 + b * 64 + ks * 8, desc_at(vd, B == 128 ? ks * 128 : (ks >> 2) * (kTileBytes >> 5) + (ks & 3) * 128), idesc, (h > 0 || ks > 0) ? 1u : 0u);
          if (h == n_steps - 1) tc_commit(&sh.o_full[(nt - 1) & 1]);
          tc_commit(&sh.pv_done[b]);
        }
        __syncwarp();
      }
    }
    drain_products(leader, &sh.drain[1]);
  } else if (warp < 8) {
    // ===== softmax / correction / epilogue: thread = one query row
    setmaxnreg_inc<kRegsSoftmax>();
    const uint32_t w = warp >> 2, quarter = warp & 3;
    const int row = quarter * 32 + lane;  // row inside the 128-row query tile
    const uint32_t o_addr = tmem + (quarter << 21), s_addr = o_addr + 128, p_addr = o_addr + 384;
    const float c = p.scale_log2;
    const uint64_t c2 = pack_f32x2(c, c);
    auto arrive = [&](uint64_t *bar) {  // this warp's tensor-memory accesses so far are ordered before it
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar);
    };
    if (Small) {
      pdl_wait();
      if (warp == 0) {
        uint32_t U = p.nb;
        if (!dense) {
          const uint4 word = plan_tile<B>(plan, blockIdx.x / p.split, lane, sh.sets, [&](int) { return sh.steps; });
          U = word.x >> 16;
        }
        __syncwarp();
        if (lane == 0) {
          sh.tile[0].y = U;
          mbar_arrive(&sh.tile_full[0]);
        }
      }
      named_barrier_sync(2, 256);
    }
    uint32_t g0 = 0, nt = 0;  // key steps before the present tile, tiles with key steps before it
    int n_steps = 0, h = 0;   // of the present tile; this warpgroup's next step of it
    bool leads = w == 0;      // takes the tile's first step
    uint32_t pending = 0;     // the tile before is this warpgroup's to write: 1 behind its first step of the next one, 2 before
    bool live = true;
    float m_ref = kNoReference, l_run = 0.f;
    // Why the loop over the steps was left: what a step rarely needs stands outside of it.
    enum { kNothing, kNotThere, kMask, kRescale } why = kNothing;
    bool masked = false;      // the keys of the step that do not count have been taken out
    float alpha = 1.f;        // O and the sums change scale by it
    auto advance = [&]() -> bool {  // to this warpgroup's next step; true if the output of the tile before comes first
      // Steps are taken in turn, but that the second and third go to one warpgroup: the other one writes the output of
      // the tile before meanwhile.  (In a CTA's first tile too: the order of a row's sum goes by the shape alone.)
      const bool first = h < 2;
      h += first && p.late ? 3 - 2 * h : 2;
      return first && pending != 0;
    };
    auto mask_keys = [&](uint32_t b, uint32_t e) {
      // Keys that do not count get a score of -inf in tensor memory, where a loop over columns is a loop;
      // the step is then like any other.  (As 128 selects between the loads and the weights it slowed all
      // steps by 7 %; a branch of its own, 32 columns at a time, took 5000-9000 clocks instead of 2600.)
      const uint32_t flags = (e >> (10 + (quarter >> 1))) & 0x10001u, s_at = s_addr + b * 128;
      int n0, n1;  // keys of each half that count
      if (B == 128) {
        n0 = p.N - (int)e * 128;
        n1 = n0 - 64;
      } else {
        n0 = (flags & 1u) ? p.N - (int)(e & 0x3ff) * 64 : 0;
        n1 = (flags >> 16) ? p.N - (int)((e >> 16) & 0x3ff) * 64 : 0;
      }
      tc_fence_after();
#pragma unroll 1
      for (int col = 0; col < 128; col += 8) {
        const int n = (col < 64 ? n0 : n1 + 64) - col;  // columns of these eight that count
        if (n <= 0) {
          tmem_st8_fill(s_at + col, 0xff800000u);
        } else {
#pragma unroll 1
          for (int i = n; i < 8; ++i) tmem_st1(s_at + col + i, 0xff800000u);
        }
      }
      tmem_wait_st();
    };
    auto end_tile = [&]() {
      if (n_steps == 0) return;  // (a tile without keys)
      const int last = n_steps - 1;
      const bool mine = leads == (p.late ? last == 0 || (last > 2 && (last & 1)) : !(last & 1));  // had the last step
      leads = !mine;
      const bool at_once = !Small && n_steps <= p.at_once;
      if (mine == at_once) {
        pending = at_once ? 2 : 1;
        if (Small) sh.l[1][w][row] = make_float2(l_run, m_ref);
        if (at_once && n_steps == 1) sh.l[nt & 1][w ^ 1][row] = make_float2(0.f, kNoReference);  // (the other one had no step)
      }
      g0 += n_steps;
      ++nt;
    };
    int t = 0;
    auto next = [&]() {  // tile
      int4 ti;
      live = next_tile(t++, ti);
      if (!live) return;
      if (lane == 0) sh.written[nt & 1][warp] = ti;
      __syncwarp();  // all lanes read it when they write the tile, in a small launch maybe with no step in between
      n_steps = n_steps_of(ti.y);
      h = leads ? 0 : 1;
      m_ref = kNoReference;  // (rows without a key keep it)
      l_run = 0.f;
      if (n_steps == 0) {  // rows without any key: 16 a warp, two at a time (a row a thread, by one warpgroup, took 42.8 us
                           // instead of 33.4 for 12 x 33k of such tiles)
        if (shared_tile) {
          if (leads) sh.part_l[row] = make_float2(0.f, kNoReference);  // (nothing else of this part is read)
        } else {
          int tok = ti.x * 128 + (int)warp * 16 + (lane >> 4);
          uint16_t *out = p.O + (long long)ti.w * p.sb + (long long)ti.z * p.sh + tok * p.sn + (lane & 15) * 8;
          float *lse = p.lse == nullptr ? nullptr : p.lse + (size_t)(ti.w * p.H + ti.z) * p.N;
#pragma unroll 1
          for (int i = 0; i < 8 && tok < p.N; ++i, tok += 2, out += 2 * p.sn) {
            *reinterpret_cast<uint4 *>(out) = make_uint4(0u, 0u, 0u, 0u);
            if (lse != nullptr && (lane & 15) == 0) lse[tok] = -INFINITY;
          }
        }
      }
    };
    if (Small) next();  // (the only one)
    for (;;) {
      if (Small || pending != 2)  // (a tile that is written at once comes before the steps of the next one)
#pragma unroll 1
      while (h < n_steps) {
        const uint32_t g = g0 + h, b = g & 1, s_at = s_addr + b * 128, p_at = p_addr + b * 64;
        // The scores, and the references after the step before (half a step old by now, as a rule), are asked for
        // together: a barrier that is complete costs ~170 clocks to ask, one after the other as many again.  (With the
        // same for P below, 24 x 119k: 15.95 to 15.3 M clocks.)  A parity tells two phases in a row apart: behind a step that
        // the other warpgroup took on this buffer, the answer for the scores holds once that step's partner has its reference.
        auto ask = [&](uint64_t *bar, uint32_t parity) { return Small ? mbar_test_wait(bar, parity) : mbar_try_wait(bar, parity, kShortWait); };
        const bool m_there = ask(&sh.m_ready[b ^ 1][quarter], ((g - 1) >> 1) & 1) || g == 0;
        const bool there = ask(&sh.s_full[b], (g >> 1) & 1) && m_there;
        if (__builtin_expect(!__all_sync(0xffffffffu, there), 0)) {
          if (!Small) {
            why = kNotThere;
            break;
          }
          // (a small launch waits for most of its few steps, and comes by all instructions for the first time)
          if (g > 0) wait(&sh.m_ready[b ^ 1][quarter], ((g - 1) >> 1) & 1);
          wait(&sh.s_full[b], (g >> 1) & 1);
        }
        const uint32_t e = sh.entry[g & 3];
        // which halves of the step this row's query block lists, whether the step holds the ragged last block
        const uint32_t flags = (e >> (10 + (quarter >> 1))) & 0x10001u;  // (64-token blocks)
        const bool ragged = B == 128 ? (int)(e + 1) * 128 > p.N : (e & 0x10001000u) != 0u;
        tc_fence_after();
        const float m_prev = h > 0 ? sh.m[b ^ 1][row] : kNoReference;  // the reference as the step before left it
        auto take_reference = [&]() {
          l_run *= ex2(m_ref - m_prev);
          m_ref = m_prev;
        };
        Sums sums = {0.f, 0.f, 0.f, 0.f};
        // Agrees on the reference of step g given the row's maximum; true if it moves (some row).
        bool moved = false;
        auto new_reference = [&](float x_max) -> bool {
          const bool grow = x_max > m_ref + kMaxGrowth;
          const float m_new = grow ? x_max + kHeadroom : m_ref;
          sh.m[b][row] = m_new;
          __syncwarp();
          if (lane == 0) mbar_arrive(&sh.m_ready[b][quarter]);
          if (__builtin_expect(!__any_sync(0xffffffffu, grow), 1)) return false;
          moved = true;
          alpha = ex2(m_ref - m_new);
          l_run *= alpha;
          m_ref = m_new;
          return true;
        };
        if (__builtin_expect(ragged && !masked, 0)) {
          if (!Small) {
            why = kMask;
            break;
          }
          mask_keys(b, e);
        }
        // the product that read this P two steps ago is complete
        auto p_free = [&]() {
          if (g >= 2) wait(&sh.pv_done[b], ((g - 2) >> 1) & 1);
          tc_fence_after();
        };
        if (__builtin_expect(B == 128 || flags == 0x10001u || ragged, 1)) {
          // The exponentials of the first 32 keys are taken with the reference as it was while the row maximum is
          // found, and once more, by the same instructions, in the rare step that moves it (a tile's first ones:
          // a copy of its own for them cost 2 % of the clocks of a tile with 10-20 steps, from cold instructions).
          uint32_t s[128], pk[32];
#pragma unroll
          for (int q = 0; q < 4; ++q) tmem_ld32(s_at + q * 32, *reinterpret_cast<uint32_t(*)[32]>(&s[q * 32]));
          take_reference();
          tmem_wait_ld();
          arrive(&sh.s_free[b]);
          uint64_t neg_m2;
          bool again = false;
#pragma unroll 1
          do {
            neg_m2 = pack_f32x2(-m_ref, -m_ref);
            sums = {0.f, 0.f, 0.f, 0.f};
            exp32(&s[0], c2, neg_m2, &pk[0], sums);
            const float x_max = fmaxf(max64(&s[0]), max64(&s[64])) * c;
            again = !again && new_reference(x_max);
          } while (__builtin_expect(again, 0));
          // p_free, asked for ahead of these exponentials
          const bool p_done = g < 2 || mbar_test_wait(&sh.pv_done[b], ((g - 2) >> 1) & 1);
          exp32(&s[32], c2, neg_m2, &pk[16], sums);
          if (__builtin_expect(!__all_sync(0xffffffffu, p_done), 0)) wait(&sh.pv_done[b], ((g - 2) >> 1) & 1);
          tc_fence_after();
          tmem_st32(p_at, pk);
          exp32(&s[64], c2, neg_m2, &pk[0], sums);
          exp32(&s[96], c2, neg_m2, &pk[16], sums);
          tmem_st32(p_at + 32, pk);
        } else {
          // This row's query block lists one of the step's two blocks or none.  The product reads all 128 keys of the
          // step: zeros for the others, in one store (eight keys at a time: 12 x 33k, 30 % of the blocks at random, 2658 us instead of
          // 2538, whole steps of 40 x 33k 0.4 % more).  The exponentials in a loop: unrolled, the random lists take 2 % less, short
          // ones, 24 x 2465, 0.6 % more.
          const uint32_t v = flags >> 16;
          uint32_t s[64], pk[16], zeros[32];
          tmem_ld32(s_at + v * 64, *reinterpret_cast<uint32_t(*)[32]>(&s[0]));
          tmem_ld32(s_at + v * 64 + 32, *reinterpret_cast<uint32_t(*)[32]>(&s[32]));
          take_reference();
          tmem_wait_ld();
          arrive(&sh.s_free[b]);
          const float x_max = max64(s) * c;
          new_reference(flags != 0u ? x_max : -INFINITY);
          p_free();
          const uint64_t neg_m2 = pack_f32x2(-m_ref, -m_ref);
          const uint32_t n_exp = flags != 0u ? 4 : 0;
#pragma unroll
          for (int i = 0; i < 32; ++i) zeros[i] = 0u;
          tmem_st32(p_at + (32 - v * 32), zeros);
          if (n_exp == 0) tmem_st32(p_at + v * 32, zeros);
#pragma unroll 1
          for (uint32_t i = 0; i < n_exp; i += 2) {
            exp32(&s[0], c2, neg_m2, &pk[0], sums);
            tmem_st16(p_at + v * 32 + i * 8, pk);
#pragma unroll
            for (int k = 0; k < 32; ++k) s[k] = s[32 + k];
          }
        }
        l_run += (sums.a + sums.b) + (sums.c + sums.d);
        // for the warpgroup that writes the tile (each one's last step is among the tile's last three)
        if (Small) {
          if (h == n_steps - 1) sh.l[0][nt & 1][row] = make_float2(l_run, m_ref);
        } else {
          if (h >= n_steps - 3) sh.l[nt & 1][w][row] = make_float2(l_run, m_ref);
        }
        if (!ok) break;
        if (__builtin_expect(moved && h > 0, 0)) {
          why = kRescale;
          break;
        }
        tmem_wait_st();
        arrive(&sh.p_full[b]);
        masked = false;
        if (__builtin_expect(advance(), 0)) break;
      }
      if (why != kNothing && ok) {
        const uint32_t g = g0 + h, b = g & 1;
        if (why == kNotThere) {
          if (g > 0) wait(&sh.m_ready[b ^ 1][quarter], ((g - 1) >> 1) & 1);
          wait(&sh.s_full[b], (g >> 1) & 1);
        } else if (why == kMask) {
          mask_keys(b, sh.entry[g & 3]);
          masked = true;
        } else {
          // O changes scale: the products of the steps before have to be complete
          if (wait(&sh.pv_done[b ^ 1], ((g - 1) >> 1) & 1)) {
            tc_fence_after();
            const uint64_t alpha2 = pack_f32x2(alpha, alpha);
#pragma unroll 1
            for (int ch = 0; ch < 8; ++ch) {
              uint32_t v[16];
              tmem_ld16(o_addr + ch * 16, v);
              tmem_wait_ld();
#pragma unroll
              for (int i = 0; i < 16; i += 2) {
                float lo, hi;
                unpack_f32x2(mul_f32x2(pack_f32x2(__uint_as_float(v[i]), __uint_as_float(v[i + 1])), alpha2), lo, hi);
                v[i] = __float_as_uint(lo);
                v[i + 1] = __float_as_uint(hi);
              }
              tmem_st16(o_addr + ch * 16, v);
            }
            tmem_wait_st();
            arrive(&sh.p_full[b]);
            masked = false;
            advance();
          }
        }
        const bool whole_step = why == kRescale;
        why = kNothing;
        if (ok && !whole_step) continue;
      }
      if (Small && !ok) break;
      if (Small && h >= n_steps) end_tile();
      if (pending) {
        // ===== the output of the tile before, O / l, one row per thread (when this CTA gives up, too, if the tile's products are
        // complete: it lacks nothing of what did not come)
        const uint32_t w_last = pending == 2 ? w : w ^ 1;
        pending = 0;
        const uint32_t q_buf = (nt - 1) & 1;
        const int4 to = sh.written[q_buf][warp];
        if (Small || ok ? !wait(&sh.o_full[q_buf], ((nt - 1) >> 1) & 1) : !__all_sync(0xffffffffu, mbar_test_wait(&sh.o_full[q_buf], ((nt - 1) >> 1) & 1))) break;
        tc_fence_after();
        // the sums of the warpgroup with the tile's last step, whose reference O has, and of the other one
        const float2 last = Small ? sh.l[0][q_buf][row] : sh.l[q_buf][w_last][row];
        const float2 other = Small ? sh.l[1][w][row] : sh.l[q_buf][w_last ^ 1][row];
        const float l = last.x + other.x * ex2(other.y - last.y), m = last.y;
        const float inv = l > 0.f ? 1.f / l : 0.f;
        const uint64_t inv2 = pack_f32x2(inv, inv);
        // Through the place of the tile's Q, a copy of 32 rows a warp; rows behind the last token are not written.
        unsigned char *out = smem + kOffQ + q_buf * kTileBytes + quarter * (kTileBytes / 4);
#pragma unroll 1
        for (int half = 0; half < 2; ++half) {  // of the dims (short code: it is fetched anew for every tile)
          uint32_t v[64];
          tmem_ld32(o_addr + half * 64, *reinterpret_cast<uint32_t(*)[32]>(&v[0]));
          tmem_ld32(o_addr + half * 64 + 32, *reinterpret_cast<uint32_t(*)[32]>(&v[32]));
          tmem_wait_ld();
          if (half == 1) arrive(&sh.o_free);
          if (shared_tile) {  // O as it is, where the keys were, with its row sums: the parts are put together below
            float4 *part = reinterpret_cast<float4 *>(smem + kOffK + row * 512) + half * 16;
#pragma unroll
            for (int i = 0; i < 16; ++i)
              part[i ^ (row & 7)] = make_float4(__uint_as_float(v[4 * i]), __uint_as_float(v[4 * i + 1]), __uint_as_float(v[4 * i + 2]), __uint_as_float(v[4 * i + 3]));
          } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) {  // eight dims: 16 bytes of a row of 64 dims, swizzled as the copy expects them
              uint32_t x[4];
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                float lo, hi;
                unpack_f32x2(mul_f32x2(pack_f32x2(__uint_as_float(v[i * 8 + 2 * k]), __uint_as_float(v[i * 8 + 2 * k + 1])), inv2), lo, hi);
                x[k] = pack_bf16x2(lo, hi);
              }
              *reinterpret_cast<uint4 *>(out + half * (kTileBytes / 8) + lane * 128 + ((i ^ (lane & 7)) << 4)) = make_uint4(x[0], x[1], x[2], x[3]);
            }
          }
        }
        if (shared_tile) {
          sh.part_l[row] = make_float2(l, m);
        } else {
          async_proxy_fence();
          __syncwarp();
          const int tok = to.x * 128 + row;
          if (lane == 0 && tok < p.N) tma_store_5d(&map_o, out, 0, tok, 0, to.z, to.w);
          if (p.lse != nullptr && tok < p.N)
            p.lse[(size_t)(to.w * p.H + to.z) * p.N + tok] = l > 0.f ? (m + log2f(l)) * 0.6931471805599453f : -INFINITY;
          if (lane == 0) {
            bulk_wait_read();
            mbar_arrive(&sh.out_done[q_buf]);
          }
          __syncwarp();
        }
      }
      if (!ok) break;
      if (h < n_steps) continue;
      if (Small || !live) break;
      end_tile();
      next();
    }
    if (shared_tile) {
      // ===== the parts of a tile: each CTA puts together 128 / split rows, its own part of them with those that the other
      // CTAs copy here: a bulk copy each as soon as a CTA has its part, into Q's second buffer, which a launch of one tile per CTA
      // does not use, and a place for the third one.
      const int rows = 128 / p.split;
      async_proxy_fence();
      named_barrier_sync(1, 256);
      const bool aborted = *abort != 0;
      if (tid == 0) mbar_expect_tx(&sh.parts_full, (p.split - 1) * rows * (512 + (int)sizeof(float2)));
#ifdef HEART_TEST_HOOKS
      const bool send = !((p.test_skip & 4) && blockIdx.x == 1);  // test-only library: one CTA's part never leaves
#else
      constexpr bool send = true;
#endif
      if (send && lane == 0 && warp < p.split - 1) {
        // to CTA `to`, which holds the parts of the CTAs behind it in order
        const int at = p.split - 2 - warp, to = (rank + 1 + warp) & (p.split - 1);
        if (aborted) {
          for (int i = 0; i < rows; ++i) sh.part_l[to * rows + i] = make_float2(-1.f, 0.f);
          async_proxy_fence();
        }
        const uint32_t bar = cluster_address(smem_u32(&sh.parts_full), to);
        bulk_copy_to_cluster(cluster_address(at < 2 ? parts.slot + at * (kTileBytes / 2) : parts.slot2, to), smem + kOffK + to * rows * 512, rows * 512, bar);
        bulk_copy_to_cluster(cluster_address(smem_u32(&sh.in_l[at][0]), to), &sh.part_l[to * rows], rows * (int)sizeof(float2), bar);
      }
      // (not cut short by an abort: nobody leaves with copies on their way.  A CTA that gives up sends its part all the same,
      // within the limit of one wait: only one that is later still makes this wait run out.  A warp decides for itself, and
      // the status word tells if any found the parts missing; a barrier for one answer cost 0.3 us of 17, steps of 8 blocks.)
      const long long t0 = clock64();
      bool there = mbar_try_wait(&sh.parts_full, 0);
      while (!there && clock64() - t0 < 2 * kWaitLimitCycles) there = mbar_try_wait(&sh.parts_full, 0);
      there = __all_sync(0xffffffffu, there);
      if (!there) *abort = 1;
      cluster_arrive();
      at_barrier = true;
      const int4 ti = sh.tile[0];
      if (there && *abort == 0)
        merge_parts(parts, rank, p.split, p.N - ti.x * 128,
                    p.O + (long long)ti.w * p.sb + (long long)ti.z * p.sh + (long long)ti.x * 128 * p.sn, p.sn,
                    p.lse != nullptr ? p.lse + (size_t)(ti.w * p.H + ti.z) * p.N + ti.x * 128 : nullptr);
    }
  }
  if (Small && p.split > 1) {  // the copies from this CTA's memory are complete: their receivers have them
    if (!at_barrier) cluster_arrive();
    cluster_wait();
  }

  // ------------------------------------------------------------------ tear-down
  tc_fence_before();
  __syncthreads();
  if (warp == kWarpQK) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
  if (tid == 0 && sh.abort) atomicExch(p.status, HEART_ERR_DEVICE_CHECK);
}

// Order of the tiles of a launch, one CTA per head and one for the launch's last tiles (at most 1024, whole heads;
// a small launch is all of it).
// Heads: index order while a head's K and V fit the L2 comfortably; beyond that ascending by the first key block that
// a tile's lists name (ties by tile index), every tile ranked against all others: tiles that read the same region
// of K and V run together.
// The last tiles: longest list first over all their heads, by counting the tiles of each length (ties in any order),
// so that the launch does not end on a long tile that started late.  (Head by head, the longest tile of the last head,
// 249 steps of 40 x 33k, started when 65 steps a CTA were left.  Ranking 1024 tiles against all others took 7.6 us,
// counting takes 1.1.)
__global__ void __launch_bounds__(1024) tile_order_kernel(const uint4 *__restrict__ tiles, int n_tiles, int per_head,
                                                          int by_first_key, uint4 *__restrict__ order) {
  __shared__ __align__(16) uint32_t key[1024];
  __shared__ int warp_sum[32];
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const bool tail = blockIdx.x == gridDim.x - 1;
  const int base = blockIdx.x * per_head, n = tail ? n_tiles - base : per_head;
  key[t] = tail ? 0u : 0xffffffffu;
  __syncthreads();
  pdl_wait();
  pdl_launch_dependents();
  uint4 word = make_uint4(0u, 0u, 0u, 0u);
  if (t < n) word = __ldcg(&tiles[base + t]);
  if (!tail) {
    int rank = t;
    if (by_first_key) {
      const uint32_t mine = word.w << 10 | (uint32_t)t;
      if (t < n) key[t] = mine;
      __syncthreads();
      rank = 0;
      const uint4 *k4 = reinterpret_cast<const uint4 *>(key);
#pragma unroll 4
      for (int u = 0; u < (n + 3) / 4; ++u) {
        const uint4 k = k4[u];
        rank += (k.x < mine ? 1 : 0) + (k.y < mine ? 1 : 0) + (k.z < mine ? 1 : 0) + (k.w < mine ? 1 : 0);
      }
    }
    if (t < n) order[base + rank] = word;
    return;
  }
  const int bin = 1023 - min((int)(word.x >> 16), 1023);
  uint32_t among = 0;  // place among the tiles of that length
  if (t < n) among = atomicAdd(&key[bin], 1u);
  __syncthreads();
  const int mine = (int)key[t];
  int before = mine;  // tiles in the bins up to this thread's, first of the warp's bins, then of all
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, before, o);
    if (lane >= o) before += u;
  }
  if (lane == 31) warp_sum[warp] = before;
  __syncthreads();
  if (warp == 0) {
    const int own = warp_sum[lane];
    int v = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += u;
    }
    warp_sum[lane] = v - own;
  }
  __syncthreads();
  key[t] = (uint32_t)(before - mine + warp_sum[warp]);
  __syncthreads();
  if (t < n) order[base + key[bin] + among] = word;
}

// ---------------------------------------------------------------------- host side
namespace {

constexpr int kSms = 148;
constexpr int kSplitCtas = 128;  // clusters of four do not fill the last SMs of every group of SMs

// bf16 [B,H,N,128] with element strides (sb, sh, sn, 1) as (64 dims, token, dim half, head, batch): box =
// 64 dims x `rows` tokens x `halves` dim halves, 128-byte swizzle, out-of-range rows read as zero.
bool make_map(CUtensorMap *m, const void *base, const Geom &g, int rows, int halves) {
  EncodeTiledFn fn = encode_tiled_fn();
  if (!fn) return false;
  cuuint64_t dims[5] = {64, (cuuint64_t)g.N, 2, (cuuint64_t)g.H, (cuuint64_t)g.B};
  cuuint64_t strides[4] = {(cuuint64_t)g.sn * 2, 128, (cuuint64_t)g.sh * 2, (cuuint64_t)g.sb * 2};
  cuuint32_t box[5] = {64, (cuuint32_t)rows, (cuuint32_t)halves, 1, 1};
  cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void *>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int B>
cudaError_t launch_bk(const Geom &g, const Workspace &w, const CUtensorMap &mq, const CUtensorMap &mk, const CUtensorMap &mv, const CUtensorMap &mo,
                      AttnParams prm, const int32_t *kv_idx, const int32_t *kv_cnt, cudaStream_t s, int *launches) {
  cudaError_t e;
  const int n_heads = g.B * prm.hcount;
  prm.n_tiles = n_heads * prm.n_tiles_per_head;
  const size_t all_tiles = (size_t)g.R * prm.n_tiles_per_head;
  uint4 *tiles = static_cast<uint4 *>(w.plan), *order = tiles + all_tiles;
  uint32_t *steps = reinterpret_cast<uint32_t *>(order + all_tiles);
  prm.step_pitch = (int)plan_steps_per_tile(g);
  prm.steps = steps;
  prm.tiles = tiles;
  PlanParams plan = {};
  plan.kv_idx = kv_idx;
  plan.kv_cnt = kv_cnt;
  plan.nb = g.nb;
  plan.ncph = prm.n_tiles_per_head;
  plan.idx_stride = g.idx_stride;
  plan.H = g.H;
  plan.h0 = prm.h0;
  plan.hcount = prm.hcount;
  plan.ragged = (int)(g.N % g.block != 0);
  plan.status = prm.status;
  // The other warpgroup has a step of a short tile or none, so most of the next tile would wait for the output behind its first step: us
  // at once, and behind a step of the next tile, for tiles of one step, 12 x 33k 71.5 and 98.9, 24 x 2465 20.8 and 23.1, 40 x 1000 19.8 and
  // 20.8; of two, 12 x 33k 91 and 110, 8 x 16000 39.1 and 44.0, 1200 tiles of 5000 tokens a head 44.8 and 50.3, but 520 tiles 26.4 and 26.0,
  // 320 tiles of 1000 24.0 and 22.1: with few tiles a CTA the way to the first output counts.
  prm.at_once = prm.n_tiles >= 5 * kSms ? 2 : 1;
  prm.late = all_tiles > (size_t)kSms;  // by the tiles of all heads, not of this launch: a call that runs its heads in groups gives the same bits
  if (prm.n_tiles <= kSms) {
    // Shared among CTAs as far as there are SMs (by the tiles of all heads as well).  The kernel shares tiles of four steps and more, as
    // planned; the launch goes by the steps a tile could have, because one as clusters costs by itself, 0.6 us with 28 CTAs to 1.3 with
    // 148 (launches back to back: the next one finds no room while it runs).  Dense calls have all their steps: pairs from four on, to all
    // SMs from eight on.  Lists, us with a CTA a tile and with two: up to 64 tiles, seven steps possible and all listed 11.9 and 11.4
    // (14 tiles) or 12.7 and 12.7 (63), two listed 7.5 and 7.9 or 8.0 and 9.2; 65 to 74 tiles, 36 possible: all 34.0 and 24.3, 70 % at
    // random 31.5 and 22.7, ten 14.5 and 13.9, eight 13.0 and 13.0, six 11.5 and 12.3, two 8.1 and 9.4; 22 possible, a third listed, 23.9
    // and 24.3.
    const int steps = prm.step_pitch;  // of a tile whose blocks list all
    prm.split = 1;
    if (all_tiles * 4 <= kSplitCtas && steps >= 8) prm.split = 4;
    else if (all_tiles * 2 <= kSplitCtas && steps >= (prm.dense ? 4 : 8)) prm.split = 2;
    else if (all_tiles * 2 <= kSms && steps >= (prm.dense ? 8 : 28)) prm.split = 2;
    e = allow_shared_memory(attn_tc_kernel<B, true>, kAttnSmem);
    if (e != cudaSuccess) return e;
    ++*launches;
    return launch_pdl(attn_tc_kernel<B, true>, dim3(prm.n_tiles * prm.split), dim3(kAttnThreads), kAttnSmem, s, Cluster{prm.split}, mq, mk,
                      mv, mo, prm, plan);
  }
  if (!prm.dense) {
    e = launch_pdl(attn_plan_kernel<B>, dim3((prm.n_tiles + kPlanWarps - 1) / kPlanWarps), dim3(32 * kPlanWarps), 0, s, plan, prm.n_tiles,
                   prm.step_pitch, steps, tiles, prm.counter);
    if (e != cudaSuccess) return e;
    ++*launches;
    // K + V of one head beyond 32 MB (about half of one die's share of the L2): order by key locality
    const int by_first_key = (size_t)g.N * kD * 2 * 2 > (size_t)(32u << 20) ? 1 : 0;
    const int tail_heads = 1024 / prm.n_tiles_per_head;  // (a head has at most 1024 tiles)
    const int heads = n_heads > tail_heads ? n_heads - tail_heads : 0;
    e = launch_pdl(tile_order_kernel, dim3(heads + 1), dim3(1024), 0, s, (const uint4 *)tiles, prm.n_tiles, prm.n_tiles_per_head, by_first_key, order);
    if (e != cudaSuccess) return e;
    ++*launches;
    prm.tiles = order;
  }
  e = allow_shared_memory(attn_tc_kernel<B, false>, kAttnSmem);
  if (e != cudaSuccess) return e;
  ++*launches;
  return launch_pdl(attn_tc_kernel<B, false>, dim3(kSms), dim3(kAttnThreads), kAttnSmem, s, mq, mk, mv, mo, prm, plan);
}

}  // namespace

cudaError_t launch_attention(const Geom &given, const Workspace &w, const void *Q, const void *K, const void *V,
                             const int32_t *kv_idx, const int32_t *kv_cnt, bool dense, void *O, float *lse,
                             cudaStream_t s, int *launches, int h0, int hcount) {
  if (hcount <= 0) {
    h0 = 0;
    hcount = given.H;
  }
  // A key step is 128 tokens either way: dense calls take blocks of 128, with a box where those of 64 take two, and half the
  // tests in a step (12 x 33k 5757 us with those of 64, 5665 so; the same bits).
  Geom g = given;
  if (dense) {
    g.block = 128;
    g.nb = (g.N + 127) / 128;
  }
  CUtensorMap mq, mk, mv, mo;
  if (!make_map(&mq, Q, g, 128, 2) || !make_map(&mo, O, g, 32, 2) || !make_map(&mk, K, g, g.block, g.block == 128 ? 2 : 1) || !make_map(&mv, V, g, g.block, 2))
    return cudaErrorInvalidValue;
  AttnParams prm = {};
  prm.O = static_cast<uint16_t *>(O);
  prm.lse = lse;
  prm.status = w.status;
  prm.counter = w.status + kStatusTileWord;
  prm.sb = g.sb;
  prm.sh = g.sh;
  prm.sn = g.sn;
  prm.H = g.H;
  prm.N = g.N;
  prm.nb = g.nb;
  prm.n_tiles_per_head = (g.N + 127) / 128;
  prm.dense = dense ? 1 : 0;
  prm.h0 = h0;
  prm.hcount = hcount;
  prm.scale_log2 = (float)(g.scale * 1.4426950408889634);
#ifdef HEART_TEST_HOOKS
  prm.test_skip = (g.flags & 0x80000000u ? 1 : 0) | (g.flags & 0x20000000u ? 2 : 0) | (g.flags & 0x40000000u ? 4 : 0);
#endif
  return g.block == 64 ? launch_bk<64>(g, w, mq, mk, mv, mo, prm, kv_idx, kv_cnt, s, launches)
                       : launch_bk<128>(g, w, mq, mk, mv, mo, prm, kv_idx, kv_cnt, s, launches);
}

}  // namespace heart
