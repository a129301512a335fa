// Block-sparse attention with online softmax on the sm_100a tensor cores.
//
// A query tile is 128 rows of one head: one query block of 128 tokens, or two query blocks of 64 whose
// lists are merged (two flag bits per key block; rows of the half that does not list a key block get
// weight 0 there).  Keys are processed 128 at a time: a "key step" is one 128-token block or two listed
// 64-token blocks.
//
// What bounds it: for a 128 x 128 tile the tensor pipe needs 1024 clocks (512 for Q K^T, 512 for P V)
// and the special-function units 1024 as well (ex2 issues every 8 clocks per sub-partition), and within
// a tile the products and the softmax of a step are serial.  So one persistent CTA per SM runs two
// independent streams on different query tiles, each with its own warps, barriers, buffers and half of
// the tensor memory: while one stream takes exponentials the other has its products running.  A stream
// draws its tiles from a counter; the loads and the first scores of its next tile overlap the end of
// the present one.
//
// Warp roles (registers are moved from the helper warps to the softmax warps at start):
//   warps 0-3, 4-7  softmax of stream 0, 1: one thread per query row (lane quarter = warp & 3).  Per key
//               step a thread reads its row of S (128 columns), takes the max, rescales its row of O only
//               when the max grew by more than 2^8, writes P = 2^(s*scale*log2e - m) as bf16 over the
//               first half of the S columns and adds the row sum; at the end it writes O / l (and lse).
//   warps 8, 9  MMA issuers: S_0 = Q K_0^T, then per step O += P_h V_h followed by S_{h+1} = Q K_{h+1}^T.
//               The tensor pipe executes a stream's products in issue order, so S_{h+1} may overwrite the
//               columns of P_h without a wait in between.  P V starts when 96 of the 128 keys of P_h are
//               written, while the softmax still works on the others.  A step has ONE commit (a commit
//               costs the issuing warp ~100 clocks): S_{h+1} complete, which also says that P_h V_h has
//               released its half of V and Q K_{h+1}^T its K.
//   warps 10, 11  producers: draw the tile, then TMA loads (cp.async.bulk.tensor, 128-byte swizzle,
//               completion on mbarriers) of Q and of the steps' K (one 32 KB buffer: S_h complete frees it a
//               whole softmax before the next product wants it) and V (first 64 keys double-buffered, last
//               64 single).
// Tensor memory (256 columns per stream): O (128) | S (128), P_h in the first 64 columns of S.
//
// The step lists come from attn_plan_kernel (one warp per tile), which runs just before; the tiles are
// taken head-major (the K/V of one or two heads stay in L2), within a head in the order of
// tile_order_kernel: by the first key block of their lists once a head's K and V no longer fit one die's
// half of the L2, except for the last two heads of the launch, whose tiles go longest-list-first so that
// the launch does not end on a long tile that started late.
//
// Every wait is bounded; a wait that runs out raises the stream's abort flag and the status word, the
// stream's roles drain and stop, the other streams take the remaining tiles.
#include <cuda.h>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace heart {
using namespace tc;

constexpr int kStreams = 2;
constexpr int kAttnThreads = 384;
constexpr int kWarpMma = 8, kWarpProd = 10;  // + stream
constexpr int kRegsSoftmax = 216, kRegsHelper = 72;  // 216 * 256 + 72 * 128 = the CTA's 384 x 168
constexpr int kHalfBytes = 16384;  // 64 dims of 128 keys of K, or 64 keys of V
constexpr int kQBytes = 2 * kHalfBytes;

// Shared-memory plan (the dynamic allocation itself is 1024-byte aligned), per stream.
constexpr int kOffQ = 0;                         // [2 dim halves][128 rows][64] bf16, 128-byte swizzle
constexpr int kOffK = kOffQ + kQBytes;           // [2 dim halves][128 keys][64]
constexpr int kOffVa = kOffK + 2 * kHalfBytes;   // two buffers [2 dim halves][64 keys][64]: keys 0-63 of a step
constexpr int kOffVb = kOffVa + 2 * kHalfBytes;  // keys 64-127
constexpr int kStreamBytes = kOffVb + kHalfBytes;
constexpr int kOffBar = kStreams * kStreamBytes;

struct AttnBars {
  uint64_t q_full, k_full, va_full[2], vb_full;  // TMA -> issuer
  uint64_t s_full;           // S_h complete, and with it every product issued before it
  uint64_t p_full[2];        // keys 0-95 / 96-127 of P_h written (one arrival per softmax warp)
  uint64_t o_done;           // the last product of a tile is complete
  uint64_t tile_full[2], tile_empty[2];  // the producer's announcements of tiles
  uint64_t drain;            // abort path: the issuer's products in flight have landed
  int4 tile[2];              // query tile of its head, listed key blocks, head of the launch, 1 (0: no tile left)
  int abort;
};
constexpr int kBarBytes = (sizeof(AttnBars) + 127) / 128 * 128;
constexpr int kAttnSmem = kOffBar + kStreams * kBarBytes + 128;

// A key step as the plan kernel writes it.  128-token blocks: the key block.  64-token blocks: two
// halves of 16 bits, key block | (flag of query block 0, flag of query block 1) << 10 | ragged block << 12; no
// flag: the keys do not count (the second half of the last step when the number of blocks is odd).
struct AttnParams {
  const uint32_t *steps;  // [B*H][tiles of a head][step_pitch]
  const uint32_t *tiles;  // [tiles of the launch] tile of the head | listed key blocks << 16, in launch order
  int32_t *counter;       // tiles drawn beyond the first one of every stream (zeroed by the plan kernel)
  uint16_t *O;
  float *lse;
  int32_t *status;
  long long sb, sh, sn;
  int H, N, nb, n_tiles, n_tiles_per_head, step_pitch, dense;
  int h0, hcount;  // this launch covers heads [h0, h0 + hcount) of every batch entry
  float scale_log2;
  int test_skip_v;  // test-hook builds only: stream 0 of CTA 0 leaves out one V copy of its first tile
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

template <int B>
__global__ void __launch_bounds__(kAttnThreads, 1)
    attn_tc_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                   const __grid_constant__ CUtensorMap map_v, const AttnParams p) {
  extern __shared__ __align__(1024) unsigned char smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int st = warp < 8 ? warp >> 2 : warp & 1;  // stream of this warp
  AttnBars *bars = reinterpret_cast<AttnBars *>(smem + kOffBar + st * kBarBytes);
  uint32_t *tmem_base = reinterpret_cast<uint32_t *>(smem + kOffBar + kStreams * kBarBytes);
  volatile int *abort = &bars->abort;
  unsigned char *mem = smem + st * kStreamBytes;

  // ------------------------------------------------------------------ set-up
  if (tid < kStreams) {
    AttnBars *b = reinterpret_cast<AttnBars *>(smem + kOffBar + tid * kBarBytes);
    mbar_init(&b->q_full, 1);
    mbar_init(&b->k_full, 1);
    mbar_init(&b->va_full[0], 1);
    mbar_init(&b->va_full[1], 1);
    mbar_init(&b->vb_full, 1);
    mbar_init(&b->s_full, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&b->p_full[i], 4);      // one arrival per softmax warp
      mbar_init(&b->tile_full[i], 1);
      mbar_init(&b->tile_empty[i], 5);  // the softmax warps and the issuer
    }
    mbar_init(&b->o_done, 1);
    mbar_init(&b->drain, 1);
    b->abort = 0;
    mbar_fence_init();
  }
  if (warp == kWarpMma) {
    tmem_alloc(tmem_base, 512);
    tmem_relinquish();
  }
  if (warp == kWarpProd && lane == 0) {
    tma_prefetch_desc(&map_q);
    tma_prefetch_desc(&map_k);
    tma_prefetch_desc(&map_v);
  }
  // Launched with programmatic stream serialisation: everything above overlaps the end of the kernels
  // before it.  A kernel that follows (the next layer-step's block-sum pass) may be scheduled once every
  // CTA of this launch has started: its CTAs then fill the SMs that finish first.
  pdl_wait();
  pdl_launch_dependents();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_base + st * 256;

  auto n_steps_of = [](int U) -> int { return B == 128 ? U : (U + 1) / 2; };
  auto step_entry = [&](const uint32_t *steps, int h) -> uint32_t {
    if (!p.dense) return __ldcg(&steps[h]);
    if (B == 128) return h;
    const uint32_t ragged = (p.N & 63) ? p.nb - 1 : 0x3ff + 1, a = 2 * h, b = 2 * h + 1;
    return (a | 3u << 10 | (a == ragged ? 1u << 12 : 0u)) | (b < (uint32_t)p.nb ? b | 3u << 10 | (b == ragged ? 1u << 12 : 0u) : a) << 16;
  };
  // The next announced tile; false: none left (or abort).  Every lane of the warp gets the same answer.
  auto next_tile = [&](int t, int4 &ti) -> bool {
    if (!__all_sync(0xffffffffu, mbar_wait(&bars->tile_full[t & 1], (t >> 1) & 1, abort))) return false;
    ti = bars->tile[t & 1];
    __syncwarp();
    if (lane == 0) mbar_arrive(&bars->tile_empty[t & 1]);
    return ti.w != 0;
  };
  // Shared memory must not be released under a copy in flight: a producer that stops early (abort)
  // waits, bounded, for the copies it has issued.
  auto settle = [&](uint64_t *bar, uint32_t parity) {
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity) && clock64() - t0 < 40000000LL) {
    }
  };

  // ------------------------------------------------------------------ roles
  if (warp >= kWarpMma) setmaxnreg_dec<kRegsHelper>();
  if (warp >= kWarpProd) {
    if (lane == 0) {  // ===== producer
      bool ok = true;
      int t = 0, n_q = 0, n_k = 0, n_va = 0, n_vb = 0;  // tiles announced, loads issued
      // the tile that is announced next, fetched ahead of time
      int nx = blockIdx.x + st * gridDim.x;  // the first tile of every stream is fixed, the others are drawn
      uint32_t nx_word = 0, nx_e = 0;
      const uint32_t *nx_steps = nullptr;
      auto fetch = [&]() {
        if (nx >= p.n_tiles) return;
        const int rr = nx / p.n_tiles_per_head;
        nx_word = p.dense ? (uint32_t)(nx - rr * p.n_tiles_per_head) | (uint32_t)p.nb << 16 : __ldcg(&p.tiles[nx]);
        const int r = rr / p.hcount * p.H + p.h0 + rr % p.hcount;
        nx_steps = p.steps + ((size_t)r * p.n_tiles_per_head + (nx_word & 0xffff)) * p.step_pitch;
        if (nx_word >> 16) nx_e = step_entry(nx_steps, 0);
      };
      auto draw = [&]() {
        nx = kStreams * gridDim.x + atomicAdd(p.counter, 1);
        fetch();
      };
      int tile = 0, n_steps = 0, bidx = 0, hidx = 0;
      const uint32_t *steps = nullptr;
      uint32_t e = 0;
      // announces tiles up to the next one that has key steps; false: none left
      auto next_with_steps = [&]() -> bool {
        for (;; draw()) {
          if (t >= 2) ok = mbar_wait(&bars->tile_empty[t & 1], ((t >> 1) - 1) & 1, abort);
          if (!ok) return false;
          const bool none = nx >= p.n_tiles;
          const int rr = none ? 0 : nx / p.n_tiles_per_head, U = nx_word >> 16;  // U = listed key blocks
          bars->tile[t & 1] = none ? make_int4(0, 0, 0, 0) : make_int4(nx_word & 0xffff, U, rr, 1);
          mbar_arrive(&bars->tile_full[t & 1]);
          ++t;
          if (none) return false;
          if (U == 0) continue;
          tile = nx_word & 0xffff;
          n_steps = n_steps_of(U);
          bidx = rr / p.hcount;
          hidx = p.h0 + rr % p.hcount;
          steps = nx_steps;
          e = nx_e;
          return true;
        }
      };
      auto key_of = [&](int half) -> int { return B == 128 ? (int)e * 128 + half * 64 : (int)((e >> (16 * half)) & 0x3ff) * 64; };
      auto load_q = [&]() {
        mbar_expect_tx(&bars->q_full, kQBytes);
        tma_load_5d(mem + kOffQ, &map_q, &bars->q_full, 0, tile * 128, 0, hidx, bidx);
        ++n_q;
      };
      auto load_k = [&]() {
        mbar_expect_tx(&bars->k_full, 2 * kHalfBytes);
        if (B == 128) {
          tma_load_5d(mem + kOffK, &map_k, &bars->k_full, 0, key_of(0), 0, hidx, bidx);
        } else {
#pragma unroll
          for (int i = 0; i < 4; ++i)  // dim half i >> 1 of block i & 1
            tma_load_5d(mem + kOffK + i * (kHalfBytes / 2), &map_k, &bars->k_full, 0, key_of(i & 1), i >> 1, hidx, bidx);
        }
        ++n_k;
      };
      auto load_va = [&]() {
        const int i = n_va & 1;
        ++n_va;
#ifdef HEART_TEST_HOOKS
        // Test-only library: one V tile is never requested (neither the byte count nor the copy), so the
        // waits that depend on it run out and the abort path is taken.
        if (p.test_skip_v && blockIdx.x == 0 && st == 0 && n_va == 2) return;
#endif
        mbar_expect_tx(&bars->va_full[i], kHalfBytes);
        tma_load_5d(mem + kOffVa + i * kHalfBytes, &map_v, &bars->va_full[i], 0, key_of(0), 0, hidx, bidx);
      };
      auto load_vb = [&]() {
        mbar_expect_tx(&bars->vb_full, kHalfBytes);
        tma_load_5d(mem + kOffVb, &map_v, &bars->vb_full, 0, key_of(1), 0, hidx, bidx);
        ++n_vb;
      };
      fetch();
      if (next_with_steps()) {
        load_q();
        load_k();
        load_va();
        load_vb();
        draw();
        int h = 0;
        for (uint32_t g = 0;; ++g) {  // g: key steps so far, over all tiles
          const uint32_t e_next = h + 1 < n_steps ? step_entry(steps, h + 1) : 0u;
          // S of step g complete: K is free, and the product of step g - 1 has released its V
          ok = mbar_wait(&bars->s_full, g & 1, abort);
          if (!ok) break;
          if (g > 0) load_vb();
          if (++h < n_steps) {
            e = e_next;
            load_k();
            load_va();
          } else {
            if (!next_with_steps()) break;
            h = 0;
            load_k();
            load_q();
            load_va();
            draw();
          }
        }
      }
      if (*abort) {
        if (n_q > 0) settle(&bars->q_full, (n_q - 1) & 1);
        if (n_k > 0) settle(&bars->k_full, (n_k - 1) & 1);
        if (n_vb > 0) settle(&bars->vb_full, (n_vb - 1) & 1);
        for (int i = n_va > 2 ? n_va - 2 : 0; i < n_va; ++i) settle(&bars->va_full[i & 1], (i >> 1) & 1);
      }
    }
  } else if (warp >= kWarpMma) {
    // ===== MMA issuer.  The whole warp runs the loop (uniform control flow keeps the descriptors in
    // uniform registers), one elected lane issues.
    constexpr uint32_t idesc_qk = idesc_bf16_f32(128, 128, false, false);
    constexpr uint32_t idesc_pv = idesc_bf16_f32(128, 128, false, true);
    // Descriptors differ only in the start-address field (low word, no carry out of it): base + a
    // compile-time offset per 16-element k-step, in 16-byte units.
    //   Q, K (K-major): 64 dims = one 128-byte row; the dim halves are 128*128 B apart.
    //   V (MN-major):   64 dims = one 128-byte row; dim halves 64*128 B apart (the LBO);
    //                   16 keys = 16 rows = 2048 B per k-step.
    auto at = [](uint64_t desc, uint32_t off16) -> uint64_t {
      return (desc & 0xffffffff00000000ull) | (uint32_t)((uint32_t)desc + off16);
    };
    const bool leader = elect_one();  // the same lane every time: commits track its MMAs
    const uint64_t q_desc = smem_desc_sw128(smem_u32(mem + kOffQ), 16, 1024);
    const uint64_t k_desc = smem_desc_sw128(smem_u32(mem + kOffK), 16, 1024);
    const uint64_t va_desc = smem_desc_sw128(smem_u32(mem + kOffVa), 64 * 128, 1024);
    const uint64_t vb_desc = smem_desc_sw128(smem_u32(mem + kOffVb), 64 * 128, 1024);
    const uint32_t t_o = tmem, t_s = tmem + 128;
    uint32_t g = 0, nq = 0;  // key steps and tiles with key steps so far
    bool ok = true;
    auto issue_qk = [&]() {  // S_g = Q K^T
      ok = mbar_wait(&bars->k_full, g & 1, abort);
      if (!ok) return;
      tc_fence_after();
      if (leader) {
#pragma unroll
        for (int ks = 0; ks < 8; ++ks)
          mma_ss(t_s, at(q_desc, (ks >> 2) * 1024 + (ks & 3) * 2), at(k_desc, (ks >> 2) * 1024 + (ks & 3) * 2), idesc_qk, ks > 0 ? 1u : 0u);
        tc_commit(&bars->s_full);
      }
      __syncwarp();
    };
    int4 ti;
    for (int t = 0; ok && next_tile(t, ti); ++t) {
      const int n_steps = n_steps_of(ti.y);
      if (n_steps == 0) continue;
      ok = mbar_wait(&bars->q_full, nq & 1, abort);
      ++nq;
      if (ok) issue_qk();
      for (int h = 0; h < n_steps && ok; ++h) {
        // O (+)= P_h V_h: keys 0-95, then 96-127
        const uint64_t va = at(va_desc, (g & 1) * (kHalfBytes >> 4));
        ok = mbar_wait(&bars->va_full[g & 1], (g >> 1) & 1, abort);
        if (ok) ok = mbar_wait(&bars->vb_full, g & 1, abort);
        if (ok) ok = mbar_wait(&bars->p_full[0], g & 1, abort);
        if (!ok) break;
        tc_fence_after();
        if (leader) {
#pragma unroll
          for (int ks = 0; ks < 4; ++ks) mma_ts(t_o, t_s + ks * 8, at(va, ks * 128), idesc_pv, (h > 0 || ks > 0) ? 1u : 0u);
#pragma unroll
          for (int ks = 0; ks < 2; ++ks) mma_ts(t_o, t_s + 32 + ks * 8, at(vb_desc, ks * 128), idesc_pv, 1u);
        }
        __syncwarp();
        ok = mbar_wait(&bars->p_full[1], g & 1, abort);
        if (!ok) break;
        tc_fence_after();
        if (leader) {
#pragma unroll
          for (int ks = 2; ks < 4; ++ks) mma_ts(t_o, t_s + 32 + ks * 8, at(vb_desc, ks * 128), idesc_pv, 1u);
        }
        __syncwarp();
        ++g;
        if (h + 1 < n_steps) {
          issue_qk();
        } else {
          if (leader) tc_commit(&bars->o_done);
          __syncwarp();
        }
      }
    }
    if (*abort) {
      // Tensor memory must not be released under a product in flight: a commit arrives once
      // everything this lane has issued is complete; the wait for it is bounded like the others.
      if (leader) tc_commit(&bars->drain);
      __syncwarp();
      settle(&bars->drain, 0);
    }
  } else {
    // ===== softmax / correction / epilogue: thread = one query row
    setmaxnreg_inc<kRegsSoftmax>();
    const int row = (warp & 3) * 32 + lane;  // row inside the 128-row query tile
    const uint32_t o_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16), s_addr = o_addr + 128;
    const float c = p.scale_log2;
    const uint64_t c2 = pack_f32x2(c, c);
    float m_ref, l_run;
    // Moves the reference of the rows whose maximum grew by more than 2^8 and rescales what they have
    // accumulated.  O is quiescent: its last product was issued before the scores of this step.
    auto move_reference = [&](float x_max, bool has_o, float &alpha) {
      if (x_max > m_ref + 8.f) {
        alpha = ex2(m_ref - x_max);
        m_ref = x_max;
      }
      if (has_o) {
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
      }
    };
    // part v of P_h is written: the product may read it
    auto arrive = [&](int v) {
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars->p_full[v]);
    };
    auto arrive_both = [&]() {
      arrive(0);
      if (lane == 0) mbar_arrive(&bars->p_full[1]);
    };
    uint32_t g = 0, nq = 0;
    bool ok = true;
    int4 ti;
    for (int t = 0; ok && next_tile(t, ti); ++t) {
      const int n_steps = n_steps_of(ti.y);
      const int bidx = ti.z / p.hcount, hidx = p.h0 + ti.z % p.hcount;
      const int r = bidx * p.H + hidx;
      const uint32_t *steps = p.steps + ((size_t)r * p.n_tiles_per_head + ti.x) * p.step_pitch;
      // below every logit: the first step moves it (and rows without a key keep it)
      m_ref = -3.0e38f;
      l_run = 0.f;
      uint32_t e_next = n_steps > 0 ? step_entry(steps, 0) : 0u;
      for (int h = 0; h < n_steps; ++h, ++g) {
        // whether all 128 keys of the step count for this row, or the 64 of one block (warp-uniform)
        const uint32_t e = e_next;
        if (h + 1 < n_steps) e_next = step_entry(steps, h + 1);
        const uint32_t qb = (warp & 3) >> 1, flags = (e >> (10 + qb)) & 0x10001u;  // (64-token blocks)
        const bool full = B == 128 ? (int)(e + 1) * 128 <= p.N : flags == 0x10001u && !(e & 0x10001000u);
        ok = __all_sync(0xffffffffu, mbar_wait(&bars->s_full, g & 1, abort));
        if (!ok) break;
        tc_fence_after();
        Sums sums = {0.f, 0.f, 0.f, 0.f};
        float alpha = 1.f;
        if (__builtin_expect(full, 1)) {
          // All 128 keys count.  The exponentials of the first 32 keys are taken with the running reference
          // as it stands while the row maximum is found, and once more in the rare step that moves it.
          uint32_t s[128], pk[32];
#pragma unroll
          for (int q = 0; q < 4; ++q) tmem_ld32(s_addr + q * 32, *reinterpret_cast<uint32_t(*)[32]>(&s[q * 32]));
          tmem_wait_ld();
          uint64_t neg_m2 = pack_f32x2(-m_ref, -m_ref);
          exp32(&s[0], c2, neg_m2, &pk[0], sums);
          const float x_max = fmaxf(max64(&s[0]), max64(&s[64])) * c;
          if (__any_sync(0xffffffffu, x_max > m_ref + 8.f)) {
            move_reference(x_max, h > 0, alpha);
            neg_m2 = pack_f32x2(-m_ref, -m_ref);
            sums = {0.f, 0.f, 0.f, 0.f};
            exp32(&s[0], c2, neg_m2, &pk[0], sums);
          }
          exp32(&s[32], c2, neg_m2, &pk[16], sums);
          tmem_st32(s_addr, pk);
          exp32(&s[64], c2, neg_m2, &pk[0], sums);
          tmem_st16(s_addr + 32, *reinterpret_cast<uint32_t(*)[16]>(&pk[0]));
          arrive(0);
          exp32(&s[96], c2, neg_m2, &pk[16], sums);
          tmem_st16(s_addr + 48, *reinterpret_cast<uint32_t(*)[16]>(&pk[16]));
          arrive(1);
        } else if (B == 64 && (flags == 1u || flags == 0x10000u) && !(e & 0x10001000u)) {
          // This row's query block lists one of the step's two blocks.  The product reads all 128 keys of
          // the step: zeros for the other one.
          const uint32_t v = flags >> 16;
          const uint32_t mine = s_addr + v * 64, p_mine = s_addr + v * 32, p_other = s_addr + (32 - v * 32);
          uint32_t s[64], pk[32];
          tmem_ld32(mine, *reinterpret_cast<uint32_t(*)[32]>(&s[0]));
          tmem_ld32(mine + 32, *reinterpret_cast<uint32_t(*)[32]>(&s[32]));
#pragma unroll
          for (int i = 0; i < 32; ++i) pk[i] = 0u;
          tmem_wait_ld();
          tmem_st32(p_other, pk);
          const float x_max = max64(s) * c;
          if (__any_sync(0xffffffffu, x_max > m_ref + 8.f)) move_reference(x_max, h > 0, alpha);
          const uint64_t neg_m2 = pack_f32x2(-m_ref, -m_ref);
          exp32(&s[0], c2, neg_m2, &pk[0], sums);
          exp32(&s[32], c2, neg_m2, &pk[16], sums);
          tmem_st32(p_mine, pk);
          arrive_both();
        } else if (B == 64 && flags == 0u) {
          // none of the step's blocks is listed by this row's query block
          uint32_t pk[32];
#pragma unroll
          for (int i = 0; i < 32; ++i) pk[i] = 0u;
          tmem_st32(s_addr, pk);
          tmem_st32(s_addr + 32, pk);
          arrive_both();
        } else {
          // The ragged last block: one half at a time, the scores read twice (the weights of the first half
          // only overwrite its own scores).
          int lim0, lim1;  // keys of each half that count
          if (B == 128) {
            const int rem = p.N - (int)e * 128;
            lim0 = min(rem, 64);
            lim1 = max(0, min(rem - 64, 64));
          } else {
            lim0 = (flags & 1u) ? min(64, p.N - (int)(e & 0x3ff) * 64) : 0;
            lim1 = (flags >> 16) ? min(64, p.N - (int)((e >> 16) & 0x3ff) * 64) : 0;
          }
          float x_max = -INFINITY;
#pragma unroll 1
          for (int pass = 0; pass < 4; ++pass) {
            const int v = pass & 1, n = v ? lim1 : lim0;
            uint32_t s[64], pk[32];
            tmem_ld32(s_addr + v * 64, *reinterpret_cast<uint32_t(*)[32]>(&s[0]));
            tmem_ld32(s_addr + v * 64 + 32, *reinterpret_cast<uint32_t(*)[32]>(&s[32]));
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 64; ++i)
              if (i >= n) s[i] = 0xff800000u;  // -inf: ignored by the max, 2^-inf = 0
            if (pass < 2) {
              x_max = fmaxf(x_max, max64(s) * c);
            } else {
              if (pass == 2 && __any_sync(0xffffffffu, x_max > m_ref + 8.f)) move_reference(x_max, h > 0, alpha);
              const uint64_t neg_m2 = pack_f32x2(-m_ref, -m_ref);
              exp32(&s[0], c2, neg_m2, &pk[0], sums);
              exp32(&s[32], c2, neg_m2, &pk[16], sums);
              tmem_st32(s_addr + v * 32, pk);
              tmem_wait_st();
            }
          }
          arrive_both();
        }
        l_run = l_run * alpha + ((sums.a + sums.b) + (sums.c + sums.d));
      }
      // epilogue: O / l, one row per thread
      const int tok = ti.x * 128 + row;
      const bool valid_row = tok < p.N;
      if (ok && n_steps > 0) {
        ok = __all_sync(0xffffffffu, mbar_wait(&bars->o_done, nq & 1, abort));
        ++nq;
      }
      if (ok) {
        tc_fence_after();
        const float inv = l_run > 0.f ? 1.f / l_run : 0.f;
        uint16_t *orow = p.O + (long long)bidx * p.sb + (long long)hidx * p.sh + (long long)tok * p.sn;
#pragma unroll 1
        for (int ch = 0; ch < 4; ++ch) {  // 32 output dims at a time
          uint32_t v[32];
          if (n_steps > 0) {
            tmem_ld32(o_addr + ch * 32, v);
            tmem_wait_ld();
          }
          if (valid_row) {
#pragma unroll
            for (int g4 = 0; g4 < 4; ++g4) {
              float o[8];
#pragma unroll
              for (int i = 0; i < 8; ++i) o[i] = n_steps > 0 ? __uint_as_float(v[g4 * 8 + i]) * inv : 0.f;
              uint4 w;
              w.x = pack_bf16x2(o[0], o[1]);
              w.y = pack_bf16x2(o[2], o[3]);
              w.z = pack_bf16x2(o[4], o[5]);
              w.w = pack_bf16x2(o[6], o[7]);
              *reinterpret_cast<uint4 *>(orow + ch * 32 + g4 * 8) = w;
            }
          }
        }
        if (valid_row && p.lse != nullptr)
          p.lse[(size_t)r * p.N + tok] = l_run > 0.f ? (m_ref + log2f(l_run)) * 0.6931471805599453f : -INFINITY;
        // (the first product of the next tile writes O only after this warp's next arrival on p_full)
      }
    }
  }

  // ------------------------------------------------------------------ tear-down
  tc_fence_before();
  __syncthreads();
  if (warp == kWarpMma) {
    tc_fence_after();
    tmem_dealloc(*tmem_base, 512);
  }
  if (tid < kStreams && reinterpret_cast<AttnBars *>(smem + kOffBar + tid * kBarBytes)->abort)
    atomicExch(p.status, HEART_ERR_DEVICE_CHECK);
}

// Step lists of the tiles of a launch: one warp per tile.  The lists of the tile's query blocks (any
// order; entries out of range are skipped and reported, duplicates merged) become bit sets, and those the
// list of key steps.  64-token blocks: key blocks that both query blocks list come first, then blocks of
// query block 0 paired with blocks of query block 1, so that in such a step every row has 64 exponentials
// to take instead of half of the rows 128; ascending within each group.
constexpr int kPlanWarps = 8;

template <int B>
__global__ void __launch_bounds__(32 * kPlanWarps)
    attn_plan_kernel(const int32_t *__restrict__ kv_idx, const int32_t *__restrict__ kv_cnt, int nb, int ncph, int idx_stride,
                     int H, int h0, int hcount, int n_tiles, int step_pitch, int ragged, uint32_t *__restrict__ steps,
                     uint32_t *__restrict__ tiles, uint32_t *__restrict__ firsts, int32_t *__restrict__ counter,
                     int32_t *__restrict__ status) {
  constexpr int QBT = 128 / B;  // query blocks per tile
  __shared__ uint32_t sets[kPlanWarps][QBT][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n = blockIdx.x * kPlanWarps + warp;
  pdl_wait();  // the lists come from the kernel before this one
  pdl_launch_dependents();
  if (blockIdx.x == 0 && threadIdx.x == 0) *counter = 0;
  if (n >= n_tiles) return;
  const int rr = n / ncph, t = n % ncph;
  const int r = (rr / hcount) * H + h0 + rr % hcount;
#pragma unroll
  for (int q = 0; q < QBT; ++q) sets[warp][q][lane] = 0u;
  __syncwarp();
  bool bad = false;
#pragma unroll
  for (int q = 0; q < QBT; ++q) {
    const int I = t * QBT + q;
    if (I >= nb) break;
    const size_t row = (size_t)r * nb + I;
    int cnt = __ldcg(&kv_cnt[row]);
    if (cnt < 0 || cnt > idx_stride) {
      bad = true;
      cnt = cnt < 0 ? 0 : idx_stride;
    }
    const int32_t *list = kv_idx + row * idx_stride;
#pragma unroll 4
    for (int k = lane; k < cnt; k += 32) {
      const int J = __ldcg(&list[k]);
      if (J < 0 || J >= nb)
        bad = true;  // skipped, reported
      else
        atomicOr(&sets[warp][q][J >> 5], 1u << (J & 31));
    }
  }
  __syncwarp();
  if (bad) atomicExch(status, HEART_ERR_DEVICE_CHECK);
  // exclusive prefix over the lanes of a count per lane
  auto prefix = [lane](int v) {
    int s = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += u;
    }
    return s - v;
  };
  auto sum = [](int v) { return (int)__reduce_add_sync(0xffffffffu, (unsigned)v); };
  uint32_t *out = steps + ((size_t)r * ncph + t) * step_pitch;
  const uint32_t a = sets[warp][0][lane], b = QBT == 2 ? sets[warp][QBT - 1][lane] : 0u;
  const uint32_t any = a | b;
  const int U = sum(__popc(any));
  if (B == 128) {
    int pos = prefix(__popc(a));
    for (uint32_t m = a; m; m &= m - 1) out[pos++] = lane * 32 + __ffs(m) - 1;
  } else {
    uint16_t *out16 = reinterpret_cast<uint16_t *>(out);
    // the word of key block J, listed by the query blocks in `flags`
    auto word = [&](int J, int flags) { return (uint16_t)(J | flags << 10 | (ragged && J == nb - 1 ? 1 << 12 : 0)); };
    int last = -1;  // the last listed block, in the lane that writes it
    const int D = sum(__popc(a & b));
    int pos = prefix(__popc(a & b));
    for (uint32_t m = a & b; m; m &= m - 1) {
      const int J = lane * 32 + __ffs(m) - 1;
      last = pos == U - 1 ? J : last;
      out16[pos++] = word(J, 3);
    }
    int S[2] = {sum(__popc(a & ~b)), sum(__popc(b & ~a))};
    int start = D, skip[2] = {0, 0};
    if ((D & 1) && S[0] + S[1] > 0) {  // one single next to the last shared block; pairs start on a step
      const int x = S[0] >= S[1] ? 0 : 1;
      skip[x] = 1;
      --S[x];
      ++start;
    }
    const int paired = min(S[0], S[1]);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const uint32_t only = q ? b & ~a : a & ~b;
      int k = prefix(__popc(only)) - skip[q];
      for (uint32_t m = only; m; m &= m - 1, ++k) {
        const int at = k < 0 ? D : k < paired ? start + 2 * k + q : start + paired + k;
        const int J = lane * 32 + __ffs(m) - 1;
        last = at == U - 1 ? J : last;
        out16[at] = word(J, 1 << q);
      }
    }
    if ((U & 1) && last >= 0) out16[U] = (uint16_t)last;  // second half of the last step: the same block, without flags
  }
  const unsigned has = __ballot_sync(0xffffffffu, any != 0u);
  const int src = has ? __ffs(has) - 1 : 0;
  const int first = __shfl_sync(0xffffffffu, lane * 32 + __ffs(any) - 1, src);
  if (lane == 0) {
    tiles[n] = (uint32_t)t | (uint32_t)U << 16;
    firsts[n] = has ? first : 0x3ff;
  }
}

// Order of the tiles of every head of a launch: rank by counting over at most 1024 distinct keys, 256
// tiles per CTA.  Heads before the last two: index order while a head's K and V fit the L2 comfortably;
// beyond that ascending by the first key block that the tile's lists name (ties by tile index) -- tiles
// that read the same region of K and V run together.  The last two heads: descending by the number of
// listed key blocks.
__global__ void __launch_bounds__(256) tile_order_kernel(const uint32_t *__restrict__ tiles, const uint32_t *__restrict__ firsts,
                                                         int ncph, int n_heads, int by_first_key, uint32_t *__restrict__ order) {
  __shared__ __align__(16) uint32_t key[1024];
  const int rr = blockIdx.y, t = blockIdx.x * 256 + threadIdx.x;
  pdl_wait();
  pdl_launch_dependents();
  const bool by_length = rr >= n_heads - 2;
  const size_t base = (size_t)rr * ncph;
  if (!by_length && !by_first_key) {
    if (t < ncph) order[base + t] = __ldcg(&tiles[base + t]);
    return;
  }
  uint32_t my_word = 0u;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int u = threadIdx.x + k * 256;
    uint32_t v = 0xffffffffu;
    if (u < ncph) {
      const uint32_t w = __ldcg(&tiles[base + u]);
      if (u == t) my_word = w;
      v = (by_length ? 0xffffu - (w >> 16) : __ldcg(&firsts[base + u])) << 10 | (uint32_t)u;
    }
    key[u] = v;
  }
  __syncthreads();
  if (t >= ncph) return;
  const uint32_t mine = key[t];
  int rank = 0;
  const uint4 *k4 = reinterpret_cast<const uint4 *>(key);
#pragma unroll 4
  for (int u = 0; u < (ncph + 3) / 4; ++u) {
    const uint4 w = k4[u];
    rank += (w.x < mine ? 1 : 0) + (w.y < mine ? 1 : 0) + (w.z < mine ? 1 : 0) + (w.w < mine ? 1 : 0);
  }
  order[base + rank] = my_word;
}

// ---------------------------------------------------------------------- host side
namespace {

constexpr int kSms = 148;

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
cudaError_t launch_bk(const Geom &g, const Workspace &w, const CUtensorMap &mq, const CUtensorMap &mk, const CUtensorMap &mv,
                      AttnParams prm, const int32_t *kv_idx, const int32_t *kv_cnt, cudaStream_t s, int *launches) {
  cudaError_t e;
  const int n_heads = g.B * prm.hcount;
  prm.n_tiles = n_heads * prm.n_tiles_per_head;
  // the plan lives where the pooled scores of the mask predictor were: [R][tiles][steps], then two words per tile
  uint32_t *steps = reinterpret_cast<uint32_t *>(w.scores);
  prm.step_pitch = B == 128 ? g.nb : (g.nb + 1) / 2;
  uint32_t *tiles = steps + (size_t)g.R * prm.n_tiles_per_head * prm.step_pitch;
  uint32_t *firsts = tiles + (size_t)g.R * prm.n_tiles_per_head;
  prm.steps = steps;
  prm.tiles = tiles;
  const int planned = prm.dense ? 0 : prm.n_tiles;  // (dense: the kernel only zeroes the counter)
  e = launch_pdl(attn_plan_kernel<B>, dim3(planned ? (planned + kPlanWarps - 1) / kPlanWarps : 1), dim3(32 * kPlanWarps), 0, s,
                 kv_idx, kv_cnt, g.nb, prm.n_tiles_per_head, g.idx_stride, g.H, prm.h0, prm.hcount, planned, prm.step_pitch,
                 (int)(g.N % g.block != 0), steps, tiles, firsts, prm.counter, prm.status);
  if (e != cudaSuccess) return e;
  ++*launches;
  if (planned > kStreams * kSms) {  // up to there every tile starts at once: no order to choose
    // K + V of one head beyond 32 MB (about half of one die's share of the L2): order by key locality
    const int by_first_key = (size_t)g.N * kD * 2 * 2 > (size_t)(32u << 20) ? 1 : 0;
    e = launch_pdl(tile_order_kernel, dim3((prm.n_tiles_per_head + 255) / 256, n_heads), dim3(256), 0, s,
                   (const uint32_t *)tiles, (const uint32_t *)firsts, prm.n_tiles_per_head, n_heads, by_first_key,
                   reinterpret_cast<uint32_t *>(w.order));
    if (e != cudaSuccess) return e;
    ++*launches;
    prm.tiles = reinterpret_cast<const uint32_t *>(w.order);
  }
  e = cudaFuncSetAttribute(attn_tc_kernel<B>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAttnSmem);
  if (e != cudaSuccess) return e;
  ++*launches;
  return launch_pdl(attn_tc_kernel<B>, dim3(prm.n_tiles < kSms ? prm.n_tiles : kSms), dim3(kAttnThreads), kAttnSmem, s, mq, mk,
                    mv, prm);
}

}  // namespace

cudaError_t launch_attention(const Geom &g, const Workspace &w, const void *Q, const void *K, const void *V,
                             const int32_t *kv_idx, const int32_t *kv_cnt, bool dense, void *O, float *lse,
                             cudaStream_t s, int *launches, int h0, int hcount) {
  if (hcount <= 0) {
    h0 = 0;
    hcount = g.H;
  }
  CUtensorMap mq, mk, mv;
  if (!make_map(&mq, Q, g, 128, 2) || !make_map(&mk, K, g, g.block, g.block == 128 ? 2 : 1) || !make_map(&mv, V, g, 64, 2))
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
  prm.test_skip_v = (g.flags & 0x80000000u) ? 1 : 0;
#endif
  return g.block == 64 ? launch_bk<64>(g, w, mq, mk, mv, prm, kv_idx, kv_cnt, s, launches)
                       : launch_bk<128>(g, w, mq, mk, mv, prm, kv_idx, kv_cnt, s, launches);
}

}  // namespace heart
