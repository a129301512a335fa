// Block-importance mask prediction for the refreshed heads (Observation II: rank candidate blocks by
// importance, retain until the accumulated importance reaches the head's threshold; the minimal
// cumulative-mass set of Observation I).  Importance = row softmax of the block-pooled Q.K^T scores.
//
// Two kernels, or one for the rows of a small layer-step (mask_rows_kernel, below).  pooled_scores_kernel contracts the
// pooled means with the fp64 matrix instruction (mma.m8n8k4.f64), the 128 dims in ascending order for every score; the
// means arrive by cp.async in shared-memory tiles.  The scores go to the workspace (they stay in L2).
// top_p_kernel gives each warp one row and finds the kept set WITHOUT a sort and without dividing by the
// row sum z: the blocks above a threshold plus the lowest-index ties at it, where the threshold is the
// largest element whose ">=" mass still reaches tau * z.  It decides in fp32 first: weights
// e = 2^((s - max) log2 e), a few rounds that narrow the threshold down, then a direct evaluation over the few blocks
// left.  That is final when the mass misses tau * z by more than 1.5e-5 z on both sides of the cut (the
// errors of weights and sums stay below 1.2e-5 z, derived at the kernel) and no other block may share the
// threshold's weight; otherwise (a few rows in a hundred) the row is decided in fp64: e = exp(s - max) and a search
// over the IEEE-754 pattern of e (positive doubles order like their bit patterns), starting below the
// leading bits that the largest and the smallest weight share, two bits a round over all blocks down to
// bit 48, the rest directly over the few blocks that share that prefix.  So the integer outputs (bit
// mask, ascending index list, count) agree with a plain fp64 sort-and-accumulate reference except when
// the cumulative mass is within rounding (1e-15) of tau.
#include "common.cuh"
#include "tc_ptx.cuh"

namespace heart {

using tc::ex2;
using tc::mma_f64;

// Rows (warps) per CTA of the top-p kernel.  A row that needs the fp64 search takes many times longer than the
// others and holds its CTA: 22296 rows of 929 take 121 us with eight rows a CTA,
// 108 with two; from 513 blocks on two are no slower anywhere (whole call, tau 0.97: 40 x 591 blocks 268 against 274 us, 16 x 735
// 161 against 167); short rows gain nothing and pay for the CTAs.
template <int NJ>
constexpr int kRowsPerCta = NJ > 16 ? 2 : 8;
// CTAs that an SM has to hold, which leaves 96 registers a thread for more than 16 words, 80 for 12 and more, 64 for 4, 48 for 2.  At 32
// words that spills a little and pays with many rows (24 heads x 929 blocks 280 us, 285 with 128 registers; one head 37 and 35).
// At 24 and 16 words another CTA would not pay for its spills (24 heads x 700 blocks 164 us with 12, 161 with 10).
template <int NJ>
constexpr int kCtasPerSm = NJ > 16 ? 10 : NJ >= 12 ? 3 : NJ >= 4 ? 4 : 5;
constexpr int kMaxCand = 64;    // candidates the direct threshold evaluation takes
constexpr float kMassBand = 1.5e-5f;  // of z: cuts whose mass is closer to tau * z are decided in fp64
// Blocks are ranked by their weight, lowest index first among equals.  Weights exp(s - max) round to the same double
// where s - max differ by less than 2^-52, and the fp32 value of s - max may then be the same or one step off: a cut with
// another block within a step of fp32 or 2^-51 is decided in fp64.  (One such row costs a launch of a few waves 10 us:
// 2^-22, two to three steps, sent one row in 20000 of nearly equal scores there.)
constexpr float kTieRel = 1.19209290e-7f, kTieAbs = 4.44089210e-16f;  // 2^-23, 2^-51

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;  // identical in every lane (each level adds the same two numbers in both partners)
}
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// 16-byte asynchronous copy global -> shared; src_bytes = 0 writes zeros instead
__device__ __forceinline__ void cp_async16(double *smem_dst, const double *src, int src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(smem_dst)),
               "l"(src), "r"(src_bytes)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// scores[r][I][J] = scale * <mean_q[r][I], mean_k[r][J]> for the refreshed heads r.  A CTA of four warps owns
// 2 WT x 2 WT scores of one head, a warp WT x WT; the dims come TD at a time through STAGES buffers.
// Bound by the fp64 rate (18.5 T fma/s measured, by the matrix instruction as by plain fma).  The matrix
// instruction is there for the operands: a warp reads 2 WT / 8 doubles per lane and k-step for (WT / 8)^2
// products of 256 fma; with plain fma the shared-memory reads took as long as the arithmetic (8.6 T fma/s).
// The row pitch is 4 (mod 16) doubles: the 8 x 4 fragments are read without bank conflicts.
template <int WT, int TD, int STAGES>
struct ScoreTile {
  static constexpr int kRows = 4 * WT, kPitch = TD + 4;  // 2 WT query rows, then 2 WT key rows
  static constexpr int kBytes = 8 * STAGES * kRows * kPitch;
};

template <int WT, int TD, int STAGES>
__global__ void __launch_bounds__(128) pooled_scores_kernel(const double *__restrict__ bmean, int R, int nb, int pitch,
                                                            double scale, const uint8_t *__restrict__ refresh,
                                                            double *__restrict__ scores, int32_t *__restrict__ status,
                                                            unsigned long long expect_sig) {
  using T = ScoreTile<WT, TD, STAGES>;
  constexpr int F = WT / 8;  // fragments per warp and side
  const int r = blockIdx.z;
  pdl_wait();  // refresh flags and block means come from the kernels before this one
  pdl_launch_dependents();
  if (expect_sig != 0 && *reinterpret_cast<const unsigned long long *>(status + kStatusSigWord) != expect_sig) {
    // the caller vouched for block means that this workspace does not hold: report, predict nothing
    if (threadIdx.x == 0) atomicExch(status, HEART_ERR_DEVICE_CHECK);
    return;
  }
  if (refresh != nullptr && refresh[r] == 0) return;  // reuse branch of Algorithm 1: nothing to predict
  const int I0 = blockIdx.y * 2 * WT, J0 = blockIdx.x * 2 * WT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double *tile = reinterpret_cast<double *>(smem_raw);  // [STAGES][kRows][kPitch]
  const double *bq = bmean + ((size_t)r * nb) * kD;
  const double *bk = bmean + (((size_t)R + r) * nb) * kD;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  auto stage_in = [&](int stage) {
    if (stage < kD / TD) {
      double *dst = tile + (size_t)(stage % STAGES) * T::kRows * T::kPitch;
#pragma unroll 8
      for (int e = tid; e < T::kRows * TD / 2; e += 128) {
        const int row = e / (TD / 2), dd = e % (TD / 2) * 2;
        const int blk = row < 2 * WT ? I0 + row : J0 + row - 2 * WT;
        const double *src = (row < 2 * WT ? bq : bk) + (size_t)min(blk, nb - 1) * kD + stage * TD + dd;
        cp_async16(dst + row * T::kPitch + dd, src, blk < nb ? 16 : 0);
      }
    }
    cp_async_commit();
  };
  double acc[F][F][2];
#pragma unroll
  for (int i = 0; i < F; ++i)
#pragma unroll
    for (int j = 0; j < F; ++j) acc[i][j][0] = acc[i][j][1] = 0.0;
#pragma unroll
  for (int i = 0; i < STAGES - 1; ++i) stage_in(i);
  const int ai = (warp >> 1) * WT + (lane >> 2), bj = 2 * WT + (warp & 1) * WT + (lane >> 2), kk = lane & 3;
  const bool idle = I0 + (warp >> 1) * WT >= nb || J0 + (warp & 1) * WT >= nb;  // nothing but padding
  for (int stage = 0; stage < kD / TD; ++stage) {
    stage_in(stage + STAGES - 1);  // its buffer was released by the barrier that ended stage - 1
    cp_async_wait<STAGES - 1>();
    __syncthreads();
    if (!idle) {
      const double *A = tile + (size_t)(stage % STAGES) * T::kRows * T::kPitch + ai * T::kPitch + kk;
      const double *Bt = tile + (size_t)(stage % STAGES) * T::kRows * T::kPitch + bj * T::kPitch + kk;
#pragma unroll 4
      for (int k = 0; k < TD; k += 4) {
        double a[F], b[F];
#pragma unroll
        for (int i = 0; i < F; ++i) a[i] = A[i * 8 * T::kPitch + k];
#pragma unroll
        for (int j = 0; j < F; ++j) b[j] = Bt[j * 8 * T::kPitch + k];
#pragma unroll
        for (int i = 0; i < F; ++i)
#pragma unroll
          for (int j = 0; j < F; ++j) mma_f64(acc[i][j], a[i], b[j]);
      }
    }
    __syncthreads();  // this stage's buffer may be refilled
  }
#pragma unroll
  for (int i = 0; i < F; ++i) {
    const int I = I0 + ai + i * 8;
    if (I >= nb) continue;
    double *srow = scores + ((size_t)r * nb + I) * pitch;
#pragma unroll
    for (int j = 0; j < F; ++j) {
      const int J = J0 + (warp & 1) * WT + j * 8 + 2 * kk;  // (pitch is even: the pair stays inside the row)
      if (J < pitch) *reinterpret_cast<double2 *>(srow + J) = make_double2(acc[i][j][0] * scale, acc[i][j][1] * scale);
    }
  }
}

// The kept set of one row of scores, by one warp.  `weights`: NJ * 32 doubles of shared memory, `cand`: kMaxCand of them.
template <int NJ>  // NJ*32 >= n_b
__device__ __forceinline__ void top_p_row(const double *__restrict__ srow, int nb, double tau_r, double *weights, double *cand,
                                          uint32_t *__restrict__ mask_row, int W, int32_t *__restrict__ idx_row, int32_t *cnt) {
  const int lane = threadIdx.x & 31;
  const unsigned lt_mask = (1u << lane) - 1u;
  // fp64 search: the row lives in shared memory (lane-major, conflict-free), and rolled loops over the NJ blocks
  // of a lane keep the kernel small -- fully unrolled over registers it was several times slower at n_b > 512.
  double *pw = weights + lane;
  const double neg_inf = __longlong_as_double(0xfff0000000000000LL);
  // fp32 search: in registers (from shared memory with rolled loops: 121 us instead of 115 for 22296 rows of 929).
  float x[NJ], e[NJ];  // s - max, exp of it
  double mx = neg_inf;
  {
    double v[NJ];
#pragma unroll
    for (int j = 0; j < NJ; ++j) v[j] = (j * 32 + lane < nb) ? srow[j * 32 + lane] : neg_inf;
#pragma unroll
    for (int j = 0; j < NJ; ++j) mx = fmax(mx, v[j]);
    mx = warp_max(mx);
#pragma unroll
    for (int j = 0; j < NJ; ++j) x[j] = (float)(v[j] - mx);
  }
  // Outputs: the mask words are gathered in registers (lane l keeps word l) and leave in one store.
  auto emit = [&](auto keep_of) {
    int base = 0;
    uint32_t my_word = 0u;
#pragma unroll 4
    for (int j = 0; j < NJ; ++j) {
      const int J = j * 32 + lane;
      const bool keep = keep_of(j, J < nb);
      const unsigned word = __ballot_sync(0xffffffffu, keep);
      if (lane == j) my_word = word;
      if (keep) idx_row[base + __popc(word & lt_mask)] = J;
      base += __popc(word);
    }
    if (lane < W) mask_row[lane] = my_word;
    if (lane == 0) *cnt = base;
  };

  // fp32.  Error of a weight: x rounds by |x| 2^-24, its product with log2 e by |x| (2^-24 + 2^-25), ex2 by
  // 2^-22 relative; over a row sum e (1.5e-7 |x| + 2.4e-7) <= 1.3e-6 z (sum e |x| <= z ln n_b).  tau * z
  // takes 38 roundings more, 2.3e-6, the mass at a cut at most 37 + 38 + 64 (row, list,
  // candidates), 8.3e-6: 1.2e-5 z together.
  if (tau_r > 0.0 && tau_r < 1.0) {
    float z = 0.f;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      e[j] = ex2(x[j] * 1.44269504f);
      z += e[j];
    }
    auto sum = [](float v) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      return v;
    };
    z = sum(z);
    const float t = (float)tau_r * z, band = kMassBand * z;
    // The threshold lies in [lo, hi): mass(x >= lo) reaches t, mass(x >= hi) = m_hi does not.  (All blocks below
    // -20 together hold less than 2.1e-6.)
    float lo = -20.f, hi = 1.f, m_hi = 0.f;
    float v1 = -10.f, v2 = -5.f, v3 = -2.5f;
    auto narrow = [&](float a1, float a2, float a3) {  // by the masses at v1 < v2 < v3
      if (a3 >= t) {
        lo = v3;
      } else {
        hi = v3, m_hi = a3;
        if (a2 >= t) {
          lo = v2;
        } else {
          hi = v2, m_hi = a2;
          if (a1 >= t) lo = v1;
          else hi = v1, m_hi = a1;
        }
      }
      const float step = 0.25f * (hi - lo);
      v1 = lo + step;
      v2 = lo + 2.f * step;
      v3 = hi - step;
    };
    for (int round = 0; round < 2; ++round) {
      float a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        a1 += x[j] >= v1 ? e[j] : 0.f;
        a2 += x[j] >= v2 ? e[j] : 0.f;
        a3 += x[j] >= v3 ? e[j] : 0.f;
      }
      narrow(sum(a1), sum(a2), sum(a3));
    }
    // The blocks of that interval (a tenth of the row, as a rule) go to shared memory, where the search goes on.
    float2 *list = reinterpret_cast<float2 *>(weights);
    int n_list = 0;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      const bool is_c = x[j] >= lo && x[j] < hi;
      const unsigned bal = __ballot_sync(0xffffffffu, is_c);
      if (is_c) list[n_list + __popc(bal & lt_mask)] = make_float2(x[j], e[j]);
      n_list += __popc(bal);
    }
    __syncwarp();
    float2 *close = reinterpret_cast<float2 *>(cand);
    int n_cand = 0;
    const float m_list = m_hi;  // mass above the list
    for (int round = 0; round < 12; ++round) {
      n_cand = 0;
#pragma unroll 4
      for (int k = lane; k - lane < n_list; k += 32) {
        const float2 c = k < n_list ? list[k] : make_float2(-INFINITY, 0.f);
        const bool is_c = c.x >= lo && c.x < hi;
        const unsigned bal = __ballot_sync(0xffffffffu, is_c);
        const int pos = n_cand + __popc(bal & lt_mask);
        if (is_c && pos < kMaxCand) close[pos] = c;
        n_cand += __popc(bal);
      }
      __syncwarp();
      if (n_cand <= kMaxCand) break;
      // More than the direct evaluation takes.  Equal ones (the first 64, at least) are left to fp64 at once: quarters do
      // not part them (12 rounds on rows of equal scores: 1147 us for 22296 of 929, 852 now; fp64 alone, before: 902).
      if (__all_sync(0xffffffffu, close[lane].x == close[0].x && close[lane + 32].x == close[0].x)) break;
      float a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll 4
      for (int k = lane; k < n_list; k += 32) {
        const float2 c = list[k];
        a1 += c.x >= v1 ? c.y : 0.f;
        a2 += c.x >= v2 ? c.y : 0.f;
        a3 += c.x >= v3 ? c.y : 0.f;
      }
      narrow(m_list + sum(a1), m_list + sum(a2), m_list + sum(a3));
    }
    if (n_cand <= kMaxCand) {
      // Each lane takes two candidates: is the cut at this one, clearly?
      if (lane == 0 && (n_cand & 1)) close[n_cand] = make_float2(-INFINITY, 0.f);  // (read in pairs; cand has room for one more)
      __syncwarp();
      float x_cut = 0.f;
      bool found = false;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        if (k * 32 >= n_cand) break;
        const bool have = lane + 32 * k < n_cand;
        const float2 mine = close[have ? lane + 32 * k : 0];
        float above = m_hi;
#pragma unroll 4
        for (int n = 0; n < n_cand; n += 2) {
          const float4 c = *reinterpret_cast<const float4 *>(&close[n]);
          above += c.x > mine.x ? c.y : 0.f;
          above += c.z > mine.x ? c.w : 0.f;
        }
        if (have && t - above > band && above + mine.y - t > band) found = true, x_cut = mine.x;
      }
      const unsigned who = __ballot_sync(0xffffffffu, found);
      bool clear = __popc(who) == 1;
      if (clear) {
        // ... and no other block may share its weight (with the interval's ends: no block outside is as near)
        x_cut = __shfl_sync(0xffffffffu, x_cut, __ffs(who) - 1);
        const float near = fmaf(fabsf(x_cut), kTieRel, kTieAbs);
        const unsigned same0 = __ballot_sync(0xffffffffu, lane < n_cand && fabsf(close[lane].x - x_cut) <= near);
        const unsigned same1 = __ballot_sync(0xffffffffu, lane + 32 < n_cand && fabsf(close[lane + 32].x - x_cut) <= near);
        clear = __popc(same0) + __popc(same1) == 1 && x_cut - near >= lo && x_cut + near < hi;
      }
      if (clear) {
        int base = 0;
        uint32_t my_word = 0u;
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
          const bool keep = j * 32 + lane < nb && x[j] >= x_cut;
          const unsigned word = __ballot_sync(0xffffffffu, keep);
          my_word = lane == j ? word : my_word;
          if (keep) idx_row[base + __popc(word & lt_mask)] = j * 32 + lane;
          base += __popc(word);
        }
        if (lane < W) mask_row[lane] = my_word;
        if (lane == 0) *cnt = base;
        return;
      }
    }
    __syncwarp();
  }

  // fp64
  double z = 0.0;
#pragma unroll 4
  for (int j = 0; j < NJ; ++j) {
    const int J = j * 32 + lane;
    pw[(j) * 32] = (J < nb) ? exp_nonpositive(srow[J] - mx) : 0.0;
    z += pw[(j) * 32];
  }
  z = warp_sum(z);
  // From here on p holds the unnormalised weights e = exp(s - max) <= 1 and every mass is compared
  // with tau * z instead of dividing the row by z: the same ranking, the same ties and the same
  // cumulative-mass test up to rounding, at 1/3 fewer fp64 instructions per block.
  // tau <= 0: every prefix reaches it, so the minimal one is the single largest block (lowest index
  // on ties): the smallest positive threshold gives exactly that
  const double t = (tau_r > 0.0 ? tau_r : 2.2250738585072014e-308) * z;
  const bool keep_all = !(tau_r < 1.0) || !(z >= t);
  long long theta = 0;
  int m_ties = 0, n_ties = 0;
  if (!keep_all) {
    // Rounds over all blocks, two bits of theta each: three trial thresholds per round, their three
    // reductions side by side (fixed split of the sums: same order on every run).
    auto round2 = [&](int bit) {
      // trial patterns theta | 01, 10, 11 at bits (bit+1, bit): the mass is non-increasing in them
      // (bit >= 32: the low words of the patterns are zero, so comparing the high words decides)
      const long long c1 = theta | (1LL << bit), c2 = theta | (2LL << bit), c3 = theta | (3LL << bit);
      const int h1 = (int)(c1 >> 32), h2 = (int)(c2 >> 32), h3 = (int)(c3 >> 32);
      double a1 = 0.0, a2 = 0.0, a3 = 0.0, b1 = 0.0, b2 = 0.0, b3 = 0.0;
#pragma unroll 2
      for (int j = 0; j < NJ; j += 2) {
        const int k0 = __double2hiint(pw[(j) * 32]), k1 = __double2hiint(pw[(j + 1) * 32]);
        if (k0 >= h1) a1 += pw[(j) * 32];
        if (k0 >= h2) a2 += pw[(j) * 32];
        if (k0 >= h3) a3 += pw[(j) * 32];
        if (k1 >= h1) b1 += pw[(j + 1) * 32];
        if (k1 >= h2) b2 += pw[(j + 1) * 32];
        if (k1 >= h3) b3 += pw[(j + 1) * 32];
      }
      double m1 = a1 + b1, m2 = a2 + b2, m3 = a3 + b3;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        m1 += __shfl_xor_sync(0xffffffffu, m1, o);
        m2 += __shfl_xor_sync(0xffffffffu, m2, o);
        m3 += __shfl_xor_sync(0xffffffffu, m3, o);
      }
      theta = (m3 >= t) ? c3 : (m2 >= t) ? c2 : (m1 >= t) ? c1 : theta;
    };
    static_assert(NJ % 2 == 0, "two blocks per step");
    // The exponent and the top four mantissa bits first (bits 61..48; bit 62 is clear for p <= 1) ...
    constexpr int low = 48;  // bits [low, 62) of theta are decided over all blocks
    static_assert(low >= 32, "the full-width rounds compare high words only");
    // theta is the value of one of the blocks, so it shares the leading bits that the largest and
    // the smallest weight of the row have in common: the rounds start below them.
    int first_bit = 60;
    {
      int hmax = 0, hmin = 0x7fffffff;
#pragma unroll 4
      for (int j = 0; j < NJ; ++j) {
        const int h = __double2hiint(pw[(j) * 32]);
        hmax = max(hmax, h);
        if (j * 32 + lane < nb) hmin = min(hmin, h);
      }
      hmax = __reduce_max_sync(0xffffffffu, hmax);
      hmin = __reduce_min_sync(0xffffffffu, hmin);
      const int top = 63 - __clz(hmax ^ hmin);  // highest bit (of the 64) in which they differ; 31 if none in the high word
      first_bit = min(60, top & ~1);            // the round at `bit` decides bits (bit + 1, bit)
      if (first_bit + 2 < 62) theta = ((long long)hmax << 32) & ~((1LL << (first_bit + 2)) - 1);
    }
    for (int bit = first_bit; bit >= low; bit -= 2) round2(bit);
    if (first_bit < low) theta &= ~((1LL << low) - 1);  // the whole searched prefix is common
    // ... then only the blocks whose pattern shares that prefix can still decide the remaining bits:
    // they are compacted into shared memory (the first kMaxCand of them; more than that takes the
    // slow path below, which does not read the list).  Blocks above the prefix enter as one constant.
    const long long hi = theta >> low;
    double *scr = cand;
    double ab0 = 0.0, ab1 = 0.0;
    int n_cand = 0;
    __syncwarp();
#pragma unroll 4
    for (int j = 0; j < NJ; ++j) {
      const long long kh = __double_as_longlong(pw[(j) * 32]) >> low;
      if (kh > hi) {
        if (j & 1) ab1 += pw[(j) * 32]; else ab0 += pw[(j) * 32];
      }
      const bool is_c = (kh == hi) && (j * 32 + lane < nb);
      const unsigned bal = __ballot_sync(0xffffffffu, is_c);
      if (is_c) {
        const int pos = n_cand + __popc(bal & lt_mask);
        if (pos < kMaxCand) scr[pos] = pw[(j) * 32];
      }
      n_cand += __popc(bal);
    }
    const double mass_above = warp_sum(ab0 + ab1);
    __syncwarp();
    if (n_cand <= kMaxCand) {
      // Few candidates: each lane takes two of them and adds up, over all candidates, the mass at
      // or above its own value; theta is the largest candidate whose mass still reaches tau (the
      // smallest candidate always does: that is what the prefix search established).
      const double c0 = (lane < n_cand) ? scr[lane] : 0.0, c1 = (lane + 32 < n_cand) ? scr[lane + 32] : 0.0;
      const long long k0 = __double_as_longlong(c0), k1 = __double_as_longlong(c1);
      double g0 = mass_above, g1 = mass_above;
      long long k_min = 0x7fffffffffffffffLL;
      for (int n = 0; n < n_cand; ++n) {
        const double v = scr[n];
        const long long kv = __double_as_longlong(v);
        if (kv >= k0) g0 += v;
        if (kv >= k1) g1 += v;
        k_min = kv < k_min ? kv : k_min;
      }
      long long best = k_min;
      if (lane < n_cand && g0 >= t && k0 > best) best = k0;
      if (lane + 32 < n_cand && g1 >= t && k1 > best) best = k1;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const long long other = __shfl_xor_sync(0xffffffffu, best, o);
        best = other > best ? other : best;
      }
      theta = best;
    } else {  // many near-equal blocks: keep searching over all of them, a bit at a time
      for (int bit = low - 1; bit >= 0; --bit) {
        const long long cnd = theta | (1LL << bit);
        double g0 = 0.0, g1 = 0.0, g2 = 0.0, g3 = 0.0;  // fixed 4-way split: same order on every run
#pragma unroll 1
        for (int j = 0; j < NJ; j += 4) {
          if (__double_as_longlong(pw[(j) * 32]) >= cnd) g0 += pw[(j) * 32];
          if (j + 1 < NJ && __double_as_longlong(pw[(j + 1) * 32]) >= cnd) g1 += pw[(j + 1) * 32];
          if (j + 2 < NJ && __double_as_longlong(pw[(j + 2) * 32]) >= cnd) g2 += pw[(j + 2) * 32];
          if (j + 3 < NJ && __double_as_longlong(pw[(j + 3) * 32]) >= cnd) g3 += pw[(j + 3) * 32];
        }
        if (warp_sum((g0 + g1) + (g2 + g3)) >= t) theta = cnd;
      }
    }
    double above = 0.0;
    int nties = 0;
#pragma unroll 4
    for (int j = 0; j < NJ; ++j) {
      const long long b = __double_as_longlong(pw[(j) * 32]);
      if (b > theta) above += pw[(j) * 32];
      nties += (b == theta && j * 32 + lane < nb) ? 1 : 0;
    }
    above = warp_sum(above);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nties += __shfl_xor_sync(0xffffffffu, nties, o);
    const double th = __longlong_as_double(theta);
    double c = above;
    do {  // ties enter in ascending index order, one at a time, until the mass reaches tau
      c += th;
      ++m_ties;
    } while (c < t && m_ties < nties);
    n_ties = nties;
  }

  int tie_seen = 0;
  // the usual case: every block equal to theta is kept (theta = 0 when all blocks are kept)
  const bool all_ties_kept = keep_all || m_ties == n_ties;
  emit([&](int j, bool valid) {
    const long long b = __double_as_longlong(pw[(j) * 32]);
    if (all_ties_kept) return valid && b >= theta;
    const bool is_tie = valid && b == theta;
    const unsigned tie_ballot = __ballot_sync(0xffffffffu, is_tie);
    const int tie_rank = tie_seen + __popc(tie_ballot & lt_mask);
    tie_seen += __popc(tie_ballot);
    return valid && (b > theta || (is_tie && tie_rank < m_ties));
  });
}

template <int NJ>  // NJ*32 >= n_b
__global__ void __launch_bounds__(32 * kRowsPerCta<NJ>, kCtasPerSm<NJ>) top_p_kernel(const double *__restrict__ scores, int nb, int pitch,
                                                                 const double *__restrict__ tau,
                                                                 const uint8_t *__restrict__ refresh,
                                                                 unsigned flags, uint32_t *__restrict__ mask_bits,
                                                                 int32_t *__restrict__ kv_idx,
                                                                 int32_t *__restrict__ kv_cnt, int idx_stride,
                                                                 int W, const int32_t *__restrict__ status,
                                                                 unsigned long long expect_sig) {
  const int r = blockIdx.y;
  pdl_wait();  // the scores come from the kernel before this one
  if (expect_sig != 0 && *reinterpret_cast<const unsigned long long *>(status + kStatusSigWord) != expect_sig)
    return;  // reported by the score kernel
  if (refresh != nullptr && refresh[r] == 0) return;  // reuse branch of Algorithm 1: mask untouched
  const int warp = threadIdx.x >> 5;
  extern __shared__ __align__(16) unsigned char smem_top[];
  double *weights = reinterpret_cast<double *>(smem_top);  // [kRowsPerCta<NJ>][NJ * 32]
  __shared__ __align__(16) double cand[kRowsPerCta<NJ>][kMaxCand];
  const int I = blockIdx.x * kRowsPerCta<NJ> + warp;
  if (I >= nb) return;
  const size_t row = (size_t)r * nb + I;
  top_p_row<NJ>(scores + row * pitch, nb, (flags & HEART_FORCE_DENSE) ? 1.0 : tau[r], weights + (size_t)warp * NJ * 32, cand[warp],
                mask_bits + row * W, W, kv_idx + row * idx_stride, kv_cnt + row);
}

// Small layer-steps: a CTA takes eight query blocks of a head from the pooled means to the lists, a warp per row, so that one
// launch does the work of two or three.  Bound by latency.  DECIDE (the smallest steps without the layer gate, a ticket for every
// head): every CTA of a head adds up the head's token means and decides for itself, bit for bit like mean_drift_kernel; the
// CTA that took the last of the head's tickets, when all of them have read the old anchor, moves it.
struct RowArgs {
  const double *bmean, *tau;
  int R, nb;
  double scale;
  unsigned flags;
  const uint8_t *refresh;  // kBefore
  const double *mean;      // kGateHere
  uint32_t *mask_bits;
  int32_t *kv_idx, *kv_cnt;
  int idx_stride, W;
  const double *psum;  // DECIDE
  int N, nchunks;
  DecideArgs decide;
};
constexpr int kRowsKernelThreads = 256, kRowsKernelPitch = kD + 4;
__host__ __device__ inline int rows_kernel_doubles(int nj, int nb) { return (8 + (nb + 7) / 8 * 8) * kRowsKernelPitch + 2 * 8 * nj * 32; }

// Where the decisions come from: mean_drift_kernel, this kernel, mean_drift_kernel with the layer gate applied here.
enum Decided { kBefore, kHere, kGateHere };
template <int NJ, Decided HOW>
__global__ void __launch_bounds__(kRowsKernelThreads) mask_rows_kernel(const RowArgs a) {
  constexpr bool DECIDE = HOW == kHere;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nb = a.nb, keys = (nb + 7) / 8 * 8, r = blockIdx.y, I0 = blockIdx.x * 8;
  double *tile = reinterpret_cast<double *>(smem_raw);  // 8 query rows, then the key rows
  double *scores = tile + (8 + keys) * kRowsKernelPitch, *weights = scores + 8 * NJ * 32;
  __shared__ __align__(16) double cand[8][kMaxCand];
  __shared__ double wsum[8], mean[2 * kD];
  __shared__ int sh_refresh;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  double anc = 0.0, dl = 0.0;
  bool had = false;
  if (DECIDE) {  // what does not come from the block-sum pass
    anc = ((tid >> 7) ? a.decide.anchor_k : a.decide.anchor_q)[(size_t)r * kD + (tid & (kD - 1))];
    if (tid == 0) {
      had = a.decide.has_anchor[r] != 0;
      dl = a.decide.delta[r];
    }
  }
  pdl_wait();
  pdl_launch_dependents();
  if (!DECIDE) {
    // Decided by mean_drift_kernel.  With the layer gate on, every CTA applies it to its head, from the head-wise decisions of the
    // batch entry, and the first one of a head moves the anchor: by the last CTA of mean_drift_kernel that was a chain of four
    // trips to memory in front of this kernel (2 x 12 heads x 2465 tokens: that kernel 8.1 us, 4.2 without; the step 67.2 and 64.5).
    bool rf = HOW == kBefore && a.refresh[r] != 0;
    if (HOW == kGateHere) {
      const int H = a.decide.H, b0 = r / H * H;
      int n = 0;
      for (int i = tid; i - tid < H; i += kRowsKernelThreads) n += __syncthreads_count(i < H && (__ldcg(&a.decide.pre_ws[b0 + i]) & 1));
      const int pre = __ldcg(&a.decide.pre_ws[r]);
      const double f = (double)n / (double)H;
      rf = (pre & 1) != 0;
      if (f < a.decide.gate_lo) rf = rf && !(pre & 2);
      else if (f > a.decide.gate_hi) rf = true;
      if (blockIdx.x == 0) {
        if (tid == 0) {
          a.decide.refresh_ws[r] = rf;
          if (a.decide.refresh_out) a.decide.refresh_out[r] = rf;
          if (rf) a.decide.has_anchor[r] = 1;
        }
        if (rf) ((tid >> 7) ? a.decide.anchor_k : a.decide.anchor_q)[(size_t)r * kD + (tid & (kD - 1))] = __ldcg(&a.mean[((size_t)(tid >> 7) * a.R + r) * kD + (tid & (kD - 1))]);
      }
    }
    if (!rf) return;
  }
  const double *bq = a.bmean + (size_t)r * nb * kD, *bk = a.bmean + ((size_t)a.R + r) * nb * kD;
#pragma unroll 8
  for (int e = tid; e < (8 + keys) * (kD / 2); e += kRowsKernelThreads) {
    const int row = e / (kD / 2), dd = e % (kD / 2) * 2, blk = row < 8 ? I0 + row : row - 8;
    cp_async16(tile + row * kRowsKernelPitch + dd, (row < 8 ? bq : bk) + (size_t)min(blk, nb - 1) * kD + dd, blk < nb ? 16 : 0);
  }
  cp_async_commit();
  if (DECIDE) {
    double s[4];
    sum_chunks(s, a.psum + ((size_t)(tid >> 7) * a.R + r) * a.nchunks * kD + (tid & (kD - 1)), a.nchunks);
    const double m = (((s[0] + s[1]) + s[2]) + s[3]) / (double)a.N;
    mean[tid] = m;
    double v = fabs(anc - m);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) wsum[warp] = v;
    __syncthreads();
    if (tid == 0) {
      const double pq = (wsum[0] + wsum[1]) + (wsum[2] + wsum[3]), pk = (wsum[4] + wsum[5]) + (wsum[6] + wsum[7]);
      const double dr = had ? (pq + pk) : __longlong_as_double(0x7ff0000000000000LL);
      const bool rf = !had || dr > dl || (a.decide.flags & HEART_FORCE_REFRESH) != 0;
      if (blockIdx.x == 0) {
        if (a.decide.drift_out) a.decide.drift_out[r] = dr;
        if (a.decide.refresh_out) a.decide.refresh_out[r] = rf;
        a.decide.refresh_ws[r] = rf;
      }
      sh_refresh = rf;
    }
  }
  cp_async_wait<0>();
  __syncthreads();
  if (DECIDE && !sh_refresh) return;
  int last = 0;
  if (DECIDE && warp == 7 && lane == 0) {
    // every warp has read its part of the anchor; asked for here, the answer has come when the lists are out
    __threadfence();
    last = atomicAdd(&a.decide.ticket[r], 1) == (int)gridDim.x - 1;
  }
  // 8 x 8 scores at a time, the 128 dims in ascending order as everywhere
  {
    const double *A = tile + (lane >> 2) * kRowsKernelPitch + (lane & 3), *B = A + (8 + warp * 8) * kRowsKernelPitch;
    double acc[(NJ + 1) / 2][2];
#pragma unroll
    for (int i = 0; i < (NJ + 1) / 2; ++i) acc[i][0] = acc[i][1] = 0.0;
#pragma unroll 8
    for (int k = 0; k < kD; k += 4) {
      const double q = A[k];
#pragma unroll
      for (int i = 0; i < (NJ + 1) / 2; ++i)
        if ((warp + 8 * i) * 8 < keys) mma_f64(acc[i], q, B[i * 64 * kRowsKernelPitch + k]);
    }
#pragma unroll
    for (int i = 0; i < (NJ + 1) / 2; ++i)
      if ((warp + 8 * i) * 8 < keys)
        *reinterpret_cast<double2 *>(scores + (lane >> 2) * NJ * 32 + (warp + 8 * i) * 8 + 2 * (lane & 3)) =
            make_double2(acc[i][0] * a.scale, acc[i][1] * a.scale);
  }
  __syncthreads();
  const int I = I0 + warp;
  const size_t row = (size_t)r * nb + I;
  if (I < nb)
    top_p_row<NJ>(scores + warp * NJ * 32, nb, (a.flags & HEART_FORCE_DENSE) ? 1.0 : a.tau[r], weights + warp * NJ * 32, cand[warp],
                  a.mask_bits + row * a.W, a.W, a.kv_idx + row * a.idx_stride, a.kv_cnt + row);
  if (DECIDE && warp == 7 && __shfl_sync(0xffffffffu, last, 0)) {
    if (lane == 0) a.decide.ticket[r] = 0, a.decide.has_anchor[r] = 1;
#pragma unroll
    for (int i = lane; i < 2 * kD; i += 32) (i >= kD ? a.decide.anchor_k : a.decide.anchor_q)[(size_t)r * kD + (i & (kD - 1))] = mean[i];
  }
}

template <int NJ>
static cudaError_t launch_nj(const Geom &g, const Workspace &w, const double *tau, const uint8_t *refresh,
                             heart_state st, int pitch, cudaStream_t s, unsigned long long expect_sig) {
  dim3 grid((g.nb + kRowsPerCta<NJ> - 1) / kRowsPerCta<NJ>, g.R);
  const size_t smem = sizeof(double) * kRowsPerCta<NJ> * NJ * 32;
  cudaError_t e = allow_shared_memory(top_p_kernel<NJ>, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(top_p_kernel<NJ>, grid, dim3(32 * kRowsPerCta<NJ>), smem, s, (const double *)w.scores, g.nb, pitch, tau,
                    refresh, g.flags, st.mask_bits, st.kv_idx, st.kv_cnt, g.idx_stride, g.W, (const int32_t *)w.status,
                    expect_sig);
}

// The instance for the words of a row, an even number of them.  (With one for up to 2, 8, 16, 24 or 32, whole calls, us, then / now:
// 9 heads x 100 blocks 11.1 / 9.4, 12 x 300 34.8 / 32.6, 24 x 520 123.0 / 113.2, 24 x 820 267.2 / 248.4, 24 x 929 335.4 / 327.1.)
template <int NJ = 2>
static cudaError_t launch_top_p_of(int nj, const Geom &g, const Workspace &w, const double *tau, const uint8_t *refresh, heart_state st,
                                   int pitch, cudaStream_t s, unsigned long long expect_sig) {
  if constexpr (NJ < HEART_MAX_BLOCKS / 32)
    if (nj > NJ) return launch_top_p_of<NJ + 2>(nj, g, w, tau, refresh, st, pitch, s, expect_sig);
  return launch_nj<NJ>(g, w, tau, refresh, st, pitch, s, expect_sig);
}

template <int WT, int TD, int STAGES>
static cudaError_t launch_scores(const Geom &g, const Workspace &w, const uint8_t *refresh, cudaStream_t s,
                                 unsigned long long expect_sig) {
  constexpr int smem = ScoreTile<WT, TD, STAGES>::kBytes;
  cudaError_t e = allow_shared_memory(pooled_scores_kernel<WT, TD, STAGES>, smem);
  if (e != cudaSuccess) return e;
  const unsigned t = (g.nb + 2 * WT - 1) / (2 * WT);
  return launch_pdl(pooled_scores_kernel<WT, TD, STAGES>, dim3(t, t, g.R), dim3(128), (size_t)smem, s, (const double *)w.bmean,
                    g.R, g.nb, ((g.nb + 31) / 32) * 32, g.scale, refresh, w.scores, w.status, expect_sig);
}

cudaError_t launch_pooled_scores(const Geom &g, const Workspace &w, const uint8_t *refresh, cudaStream_t s,
                                 int *launches, unsigned long long expect_sig) {
  ++*launches;
  // Tiles of 64 x 64 scores read their operands half as often as tiles of 32 x 32, which leave less of the chip idle: up to half a wave
  // of large ones (a tile an SM) small ones with all dims loaded at once, up to three waves of small ones these in three stages,
  // beyond that these where their waves, at 0.35 of a large one's time, are shorter: few waves, or much padding.  Whole calls timed
  // both ways on 354 shapes (129 to 1000 blocks, 1 to 40 heads), against the first kind up to a wave and large ones beyond: 0.978 in
  // the mean, us, before / now: 24 heads x 130 blocks 21.6 / 17.4, 30 x 200 36.4 / 32.3, 3 x 600 39.1 / 36.2.  One wave of large ones
  // against four of small ones, 31 shapes: 0.96 in the mean, 768 blocks 14.3 / 16.8, 8 x 256 12.7 / 14.3, largest 14.4 / 13.9 (5 x 289);
  // against three, 56 shapes: 1.17, 12 x 192 12.5 / 10.6.
  const long long n64 = (g.nb + 63) / 64, n32 = (g.nb + 31) / 32, tiles64 = n64 * n64 * g.R, tiles32 = n32 * n32 * g.R;
  auto waves = [](long long tiles) { return (tiles + 147) / 148; };
  if (tiles64 <= 74) return launch_scores<16, 128, 1>(g, w, refresh, s, expect_sig);
  if (tiles32 <= 3 * 148 || 35 * waves(tiles32) < 100 * waves(tiles64)) return launch_scores<16, 32, 3>(g, w, refresh, s, expect_sig);
  return launch_scores<32, 16, 3>(g, w, refresh, s, expect_sig);
}

cudaError_t launch_top_p(const Geom &g, const Workspace &w, const double *tau, const uint8_t *refresh,
                         heart_state st, cudaStream_t s, int *launches, unsigned long long expect_sig) {
  ++*launches;
  const int nj = (g.nb + 31) / 32, pitch = nj * 32;
  return launch_top_p_of(nj, g, w, tau, refresh, st, pitch, s, expect_sig);
}

// About one wave of CTAs, by their shared memory: three an SM at 32 blocks, two at 64, one at 128 (up to six at 16 and fewer, of which
// the registers hold five).  A second wave would read every head's key means once more for each eight rows, which the tiles
// of pooled_scores_kernel do not.  Steps that refresh every head, us, with separate kernels / with this one: 37 heads x 64 blocks
// 95.5 / 92.5, 9 x 128 82.5 / 80.6, 111 x 32 120.2 / 119.9; beyond the line 45 x 64 111.9 / 111.4, 12 x 128 88.1 / 89.3, 16 x 96
// 74.3 / 77.0.
bool rows_kernel_fits(const Geom &g) {
  const int nj = (g.nb + 31) / 32;
  if (nj > 4 || (g.flags & HEART_ESTIMATOR_ANTIDIAG)) return false;
  const size_t bytes = sizeof(double) * rows_kernel_doubles(nj <= 2 ? 2 : 4, g.nb);
  const long long per_sm = (long long)(224 * 1024 / (bytes + 8 * 1024));
  return (long long)g.R * ((g.nb + 7) / 8) <= 148 * per_sm;
}

// Whether the row kernel decides too.  Every CTA of a head adds up all of the head's partial sums then: that pays while there are
// few CTAs, the sums take one trip to memory (a chunk is one block in such a step) and the attention behind them is a small launch,
// which starts a launch earlier.  Steps in which every head refreshes (reuses) its mask, us, so and with mean_drift_kernel:
// 8 heads x 20 blocks 20.1 (16.8), 19.6 (17.9); 2 x 40 23.3 (20.3), 22.8 (22.4); beyond the line 24 x 24 31.4 (27.3), 28.8 (25.7);
// 16 x 64 52.2 (48.6), 47.4 (43.1).
static bool rows_kernel_decides(const Geom &g) {
  const bool gate_on = g.gate_lo > 0.0 || g.gate_hi < 1.0;
  return !gate_on && g.R * ((g.nb + 7) / 8) <= kStatusHeadTickets && g.nb <= 4 * kRangeLoads && g.R * ((g.N + 127) / 128) <= 148;
}

template <int NJ, Decided HOW>
static cudaError_t launch_rows(const Geom &g, const RowArgs &a, cudaStream_t s) {
  const int smem = (int)sizeof(double) * rows_kernel_doubles(NJ, g.nb);
  cudaError_t e = allow_shared_memory(mask_rows_kernel<NJ, HOW>, (int)sizeof(double) * rows_kernel_doubles(NJ, NJ * 32));
  if (e != cudaSuccess) return e;
  return launch_pdl(mask_rows_kernel<NJ, HOW>, dim3((g.nb + 7) / 8, g.R), dim3(kRowsKernelThreads), (size_t)smem, s, a);
}

static RowArgs row_args(const Geom &g, const Workspace &w, const double *tau, heart_state st) {
  RowArgs a = {};
  a.bmean = w.bmean;
  a.tau = tau;
  a.R = g.R;
  a.nb = g.nb;
  a.scale = g.scale;
  a.flags = g.flags;
  a.mask_bits = st.mask_bits;
  a.kv_idx = st.kv_idx;
  a.kv_cnt = st.kv_cnt;
  a.idx_stride = g.idx_stride;
  a.W = g.W;
  return a;
}

cudaError_t launch_decide_and_predict(const Geom &g, const Workspace &w, const DecideArgs &decide, const double *tau, heart_state st,
                                      cudaStream_t s, int *launches) {
  RowArgs a = row_args(g, w, tau, st);
  ++*launches;
  if (!rows_kernel_decides(g)) {
    a.decide = decide;
    a.decide.gate_later = g.gate_lo > 0.0 || g.gate_hi < 1.0;
    a.mean = w.mean;
    a.refresh = w.refresh;
    cudaError_t e = launch_decide(g, w, a.decide, s);
    if (e != cudaSuccess) return e;
    ++*launches;
    if (a.decide.gate_later) return g.nb <= 64 ? launch_rows<2, kGateHere>(g, a, s) : launch_rows<4, kGateHere>(g, a, s);
    return g.nb <= 64 ? launch_rows<2, kBefore>(g, a, s) : launch_rows<4, kBefore>(g, a, s);
  }
  a.psum = w.psum;
  a.N = g.N;
  a.nchunks = g.nchunks;
  a.decide = decide;
  a.decide.ticket = w.status + kStatusHeadTicketWord;
  return launch_rows<2, kHere>(g, a, s);
}

cudaError_t launch_predict_mask(const Geom &g, const Workspace &w, const double *tau,
                                const uint8_t *refresh, heart_state st, cudaStream_t s, int *launches,
                                unsigned long long expect_sig) {
  cudaError_t e = launch_pooled_scores(g, w, refresh, s, launches, expect_sig);
  if (e != cudaSuccess) return e;
  return launch_top_p(g, w, tau, refresh, st, s, launches, expect_sig);
}

}  // namespace heart
