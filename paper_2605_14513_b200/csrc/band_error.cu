// Frequency-aware velocity error of the offline calibration (Eq. calibration error; appendix
// "Frequency-aware velocity error"): the spectral energy of err = y_sparse - y_dense in four bands
// of its 3-D DFT over (t, y, x), weighted and divided by the energy of y_dense.
//
// A real-valued DFT is taken axis by axis, all in fp64: along an axis of length n the coefficients
//   c_k = sum_j x_j cos(2 pi k j / n), k = 0 .. n/2,   and   s_k = sum_j x_j sin(2 pi k j / n), k = 1 .. (n-1)/2.
// |X_k|^2 + |X_{n-k}|^2 = 2 (c_k^2 + s_k^2), so a product coefficient counts once for every axis with k = 0 or
// k = n/2 and twice for every other: the four bands are sums of squares with weights 1, 2, 4, 8, each from
// its own coefficients (no subtraction of energies).  Low along an axis: k <= floor(n/4).
//
// Each axis is a contraction with the fp64 matrix instruction.  Folding x_j +- x_{n-j} halves it: cosines see the
// even part, sines the odd one.  For 16 x 21 x 60 x 104 that is 1.9e8 fma (10 us at 18.5 T fma/s).  Two ways through it:
// planes that a CTA holds are transformed along y and x in one kernel, another goes over t (39 us); where that is not the
// faster way (planes_pay), axis by axis through the workspace, in five launches (53 us for that one).
#include <math.h>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace heart {

namespace {

using tc::mma_f64;

constexpr int kLines = 16;        // lines of an axis per warp
constexpr int kMaxChunk = 160;    // folded samples of a line in shared memory at a time
constexpr int kMaxSharedTable = 1024;
constexpr int kBandThreads = 128, kBandWarps = kBandThreads / 32;

// Warps of a CTA that share their lines and split the frequencies (8 at a time); the others take lines of
// their own.
__host__ __device__ inline int frequency_warps(int n) {
  const int groups = (n / 2 + 1 + 7) / 8;
  return groups <= 1 ? 1 : groups <= 2 ? 2 : kBandWarps;
}
__host__ __device__ inline int lines_per_cta(int n) { return kLines * (kBandWarps / frequency_warps(n)); }

// Folded samples of a CTA's lines in shared memory, `rows` of them at a time (a multiple of 4): along the line
// contiguous on the axis whose samples are (the copies then go along it), across the lines otherwise.  The
// pitch is 4 or 12 (mod 16) doubles either way: 8 x 4 fragments are read without bank conflicts.
struct FoldLayout {
  int chunk, line_step, row_step, doubles;
};
__host__ __device__ inline FoldLayout fold_layout(int n, bool contiguous) {
  FoldLayout f;
  const int rows = (n / 2 + 1 + 3) / 4 * 4, lines = lines_per_cta(n);
  f.chunk = rows < kMaxChunk ? rows : kMaxChunk;
  f.line_step = contiguous ? f.chunk + (f.chunk % 8 == 0 ? 4 : 0) : 1;
  f.row_step = contiguous ? 1 : lines + 4;
  f.doubles = contiguous ? lines * f.line_step : f.chunk * f.row_step;
  return f;
}

// tables[axis][m] = (cos, sin)(2 pi m / n) for the three axes, one after the other
__global__ void trig_tables_kernel(int n0, int n1, int n2, double2 *__restrict__ tables) {
  pdl_launch_dependents();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n0 + n1 + n2) return;
  const int n = i < n0 ? n0 : i < n0 + n1 ? n1 : n2, m = i < n0 ? i : i < n0 + n1 ? i - n0 : i - n0 - n1;
  double sn, cs;
  sincospi(2.0 * (double)m / (double)n, &sn, &cs);
  tables[i] = make_double2(cs, sn);
}

// Sums over the CTA of kBandThreads threads, in a fixed order; valid in thread 0.
template <int NV>
__device__ __forceinline__ void cta_sums(double (&v)[NV], double *red /* [kBandWarps * NV] */) {
#pragma unroll
  for (int q = 0; q < NV; ++q) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
    if ((threadIdx.x & 31) == 0) red[(threadIdx.x >> 5) * NV + q] = v[q];
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < NV; ++q) v[q] = (red[q] + red[NV + q]) + (red[2 * NV + q] + red[3 * NV + q]);
}

struct AxisArgs {
  const double *src;      // passes 1, 2
  const float *ys, *yd;   // pass 0: err = ys - yd
  const double2 *table;   // of this axis
  double *dst;            // passes 0, 1: coefficients, c_0 .. c_{n/2}, s_1 .. in place of the samples
  double *partial;        // pass 0: |y_dense|^2 per CTA of the first frequencies; pass 2: [CTA][4] energies
  unsigned lines, inner;  // (their product with n is at most 2^31)
  int n;
  int ny, nx;             // pass 2: lengths of the other axes (inner = ny * nx)
};

// One pass over an axis of a [outer, n, inner] view; a CTA takes lines_per_cta(n) of the outer * inner lines and, of their
// rounds of 8 * frequency_warps(n) frequencies, every gridDim.y-th.
template <int PASS>
__global__ void __launch_bounds__(kBandThreads, 8) axis_kernel(const AxisArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int n = a.n, h = n / 2, m = (n - 1) / 2;
  const int fw = frequency_warps(n), lines = lines_per_cta(n);
  const FoldLayout f = fold_layout(n, a.inner == 1);
  const int chunk = f.chunk, n_chunks = (h + chunk) / chunk;
  double *even = reinterpret_cast<double *>(smem_raw), *odd = even + f.doubles;
  double2 *tab = reinterpret_cast<double2 *>(odd + f.doubles);
  __shared__ double red[kBandWarps * 4];
  __shared__ unsigned line_at[kLines * kBandWarps];  // offset of a line's first sample
  __shared__ int line_band[kLines * kBandWarps];     // pass 2: low along y and x | log2 of the weight << 1
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const unsigned l0 = blockIdx.x * (unsigned)lines;
  const int n_lines = (int)min((unsigned)lines, a.lines - l0);
  double dense = 0.0;
  for (int i = tid; i < n_lines; i += kBandThreads) {
    const unsigned l = l0 + i, o = l / a.inner;
    line_at[i] = o * n * a.inner + (l - o * a.inner);
    if (PASS == 2) {
      const int in = (int)(l - o * a.inner), iy = in / a.nx, ix = in % a.nx;
      const int ky = iy <= a.ny / 2 ? iy : iy - a.ny / 2, kx = ix <= a.nx / 2 ? ix : ix - a.nx / 2;
      const int wy = ky == 0 || 2 * ky == a.ny ? 0 : 1, wx = kx == 0 || 2 * kx == a.nx ? 0 : 1;
      line_band[i] = (ky <= a.ny / 4 && kx <= a.nx / 4 ? 1 : 0) | (wy + wx) << 1;
    }
  }
  __syncthreads();
  // folded samples [j0, j0 + chunk) of the lines; consecutive threads take consecutive addresses
  auto fold = [&](int line, int jj, int j) {
    double x = 0.0, y = 0.0;
    const bool pair = j >= 1 && j <= m;
    if (line < n_lines && j <= h) {
      const unsigned at = line_at[line] + j * a.inner, mirror = line_at[line] + (n - j) * a.inner;
      if (PASS == 0) {
        const float d = a.yd[at], v = a.ys[at];
        float d2 = 0.f, v2 = 0.f;
        if (pair) d2 = a.yd[mirror], v2 = a.ys[mirror];
        x = (double)v - (double)d;
        y = (double)v2 - (double)d2;
        dense = fma((double)d, (double)d, fma((double)d2, (double)d2, dense));
      } else {
        x = __ldcg(&a.src[at]);
        if (pair) y = __ldcg(&a.src[mirror]);
      }
    }
    even[jj * f.row_step + line * f.line_step] = x + y;
    odd[jj * f.row_step + line * f.line_step] = pair ? x - y : 0.0;
  };
  auto stage = [&](int j0) {
    if (a.inner == 1) {
      // a warp per line, its lanes along the line
      for (int jj = lane; jj < chunk; jj += 32)
#pragma unroll 4
        for (int line = warp; line < lines; line += kBandWarps) fold(line, jj, j0 + jj);
    } else {
      const int line = tid % lines;  // (lines divides the number of threads)
#pragma unroll 4
      for (int jj = tid / lines; jj < chunk; jj += kBandThreads / lines) fold(line, jj, j0 + jj);
    }
  };
  if (PASS == 0 && n_chunks == 1) stage(0);  // (the caller's tensors do not come from the kernel before)
  pdl_wait();
  pdl_launch_dependents();
  if (PASS != 0 && n_chunks == 1) stage(0);
  const double2 *table = a.table;
  if (n <= kMaxSharedTable) {
    for (int i = tid; i < n; i += kBandThreads) tab[i] = __ldcg(&a.table[i]);
    table = tab;
  }
  __syncthreads();
  double energy[4] = {0.0, 0.0, 0.0, 0.0};  // LL, LH, HL, HH
  const int jl = lane & 3, kl = lane >> 2, line0 = warp / fw * kLines;
  for (int kg = 8 * fw * blockIdx.y; kg <= h; kg += 8 * fw * gridDim.y) {  // a warp: 8 frequencies of its 16 lines
    const int k0 = kg + 8 * (warp % fw), k = k0 + kl;
    double c[kLines / 8][2], s[kLines / 8][2];
#pragma unroll
    for (int i = 0; i < kLines / 8; ++i) c[i][0] = c[i][1] = s[i][0] = s[i][1] = 0.0;
    // (k * j) mod n, advanced by 4 k (mod n) from one four-sample step to the next
    int idx = (int)((long long)min(k, h) * jl % n);
    const int inc = (int)(4LL * min(k, h) % n);
    for (int ch = 0; ch < n_chunks; ++ch) {
      if (n_chunks > 1) {
        __syncthreads();
        const double counted = dense;
        stage(ch * chunk);
        if (kg > 0) dense = counted;  // (|y_dense|^2: in the first round only)
        __syncthreads();
      }
      if (k0 <= h) {
        const int at = jl * f.row_step + (line0 + kl) * f.line_step;
        const double *E = even + at, *O = odd + at;
#pragma unroll 2
        for (int j = 0; j < chunk; j += 4, E += 4 * f.row_step, O += 4 * f.row_step) {
          const double2 t = table[idx];
          idx += inc;
          idx -= idx >= n ? n : 0;
#pragma unroll
          for (int i = 0; i < kLines / 8; ++i) {
            mma_f64(c[i], E[8 * i * f.line_step], t.x);
            mma_f64(s[i], O[8 * i * f.line_step], t.y);
          }
        }
      }
    }
    if (k0 > h) continue;
    // lane: line line0 + 8 i + kl, frequencies k0 + 2 jl + {0, 1}
#pragma unroll
    for (int i = 0; i < kLines / 8; ++i) {
      const int line = line0 + 8 * i + kl;
      if (line >= n_lines) continue;
      double *out = PASS == 2 ? nullptr : a.dst + line_at[line];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int kk = k0 + 2 * jl + u;
        if (kk > h) continue;
        if (PASS == 2) {
          const int band = line_band[line];
          const double w = (double)(1 << ((band >> 1) + (kk == 0 || 2 * kk == n ? 0 : 1)));
          const double e = w * (kk >= 1 && kk <= m ? fma(c[i][u], c[i][u], s[i][u] * s[i][u]) : c[i][u] * c[i][u]);
          const int q = (kk <= n / 4 ? 0 : 2) + ((band & 1) ? 0 : 1);
#pragma unroll
          for (int b = 0; b < 4; ++b) energy[b] += b == q ? e : 0.0;
        } else {
          out[kk * a.inner] = c[i][u];
          if (kk >= 1 && kk <= m) out[(h + kk) * a.inner] = s[i][u];
        }
      }
    }
  }
  if (PASS == 2) {
    cta_sums<4>(energy, red);
    if (tid == 0) {
#pragma unroll
      for (int b = 0; b < 4; ++b) a.partial[((size_t)blockIdx.y * gridDim.x + blockIdx.x) * 4 + b] = energy[b];
    }
  }
  if (PASS == 0) {
    double v[1] = {dense};
    cta_sums<1>(v, red);
    if (tid == 0 && blockIdx.y == 0) a.partial[blockIdx.x] = v[0];
  }
}

// out = (e, E_LL, E_LH, E_HL, E_HH, denominator); the denominator is N |y_dense|^2 + eps (Parseval).
__global__ void __launch_bounds__(1024) band_final_kernel(const double *__restrict__ energies, long long n_energies,
                                                          const double *__restrict__ dense, long long n_dense, double n_freq,
                                                          double w0, double w1, double w2, double w3, double eps,
                                                          double *__restrict__ out) {
  __shared__ double red[32][5];
  pdl_wait();
  double v[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  for (long long i = threadIdx.x; i < n_energies; i += 1024)
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] += __ldcg(&energies[i * 4 + q]);
  for (long long i = threadIdx.x; i < n_dense; i += 1024) v[4] += __ldcg(&dense[i]);
#pragma unroll
  for (int q = 0; q < 5; ++q) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][q] = v[q];
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    double tot[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      tot[q] = red[threadIdx.x][q];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) tot[q] += __shfl_xor_sync(0xffffffffu, tot[q], o);
    }
    if (threadIdx.x == 0) {
      const double denom = tot[4] * n_freq + eps;
      out[0] = (w0 * tot[0] + w1 * tot[1] + w2 * tot[2] + w3 * tot[3]) / denom;
      out[1] = tot[0];
      out[2] = tot[1];
      out[3] = tot[2];
      out[4] = tot[3];
      out[5] = denom;
    }
  }
}

// ------------------------------------------------------------------ planes that fit in shared memory
// The usual latent: a [y, x] plane of one channel and time is transformed along both of its axes by two CTAs, one for
// the part that is even along y and one for the odd one, without a trip to the workspace in between; a second kernel
// goes over t, and its last CTA puts the result together.  Two launches instead of five, 34 MB of traffic in the L2 less:
// 16 x 21 x 60 x 104 takes 39.1 us instead of 55.3.  The products run at the rate of the fp64 matrix pipe, but the 672 CTAs,
// three an SM, fold and multiply at about the same time; a third of the first kernel is the fold.  (Each CTA of a pair folding
// the whole plane for its own half: 40.6 us.  64-bit remainders and the cosine and sine of an entry side by side, so that
// a warp's entries collide in twice as many banks: 50.2.)

constexpr int kPlaneThreads = 256, kPlaneWarps = kPlaneThreads / 32;
constexpr int kPlaneMaxShared = 200 * 1024;  // of a CTA, in bytes
constexpr int kTilesX = 4, kTilesY = 7;      // tiles of 8 lines that share the table entries of a warp, along x and y
constexpr int kTimeThreads = 128, kTimeLines = 64, kTimePitch = kTimeLines + 4, kTimeMax = 96, kTimeCtas = 148 * 4;

__host__ __device__ inline int round_up(int v, int m) { return (v + m - 1) / m * m; }

// A: folded rows, [rows rounded to 8][even part along x | odd part], B: [x coefficients rounded to 8][rows].  The pitches are
// 4 (mod 8) doubles: 8 x 4 fragments are read without bank conflicts.
struct PlaneLayout {
  int even_cols, pitch_a, rows, pitch_b, doubles;
};
__host__ __device__ inline PlaneLayout plane_layout(int ny, int nx) {
  PlaneLayout f;
  f.even_cols = round_up(nx / 2 + 1, 4);
  const int cols = f.even_cols + round_up((nx - 1) / 2, 4);
  f.pitch_a = cols + (cols % 8 == 0 ? 4 : 0);
  f.rows = round_up(ny / 2 + 1, 8);
  f.pitch_b = f.rows + 4;
  f.doubles = f.rows * f.pitch_a + round_up(nx, 8) * f.pitch_b;
  return f;
}
inline size_t plane_shared_bytes(int ny, int nx) { return sizeof(double) * plane_layout(ny, nx).doubles + sizeof(double2) * ((size_t)ny + nx); }

// cos 2 pi m / n, then sin 2 pi m / n (apart: a warp's entries collide in fewer banks); entry i0 of the CTA's first thread
__device__ __forceinline__ void fill_trig_table(double *tab, int n, int i0 = 0) {
  for (int m = (int)threadIdx.x - i0; m < n; m += blockDim.x)
    if (m >= 0) sincospi(2.0 * (double)m / (double)n, &tab[n + m], &tab[m]);
}

__device__ __forceinline__ int mod_small(int v, int n) {  // v mod n for 0 <= v < 3 n
  v -= v >= n ? n : 0;
  return v - (v >= n ? n : 0);
}
// acc[i] = lines of tile t0 + i (of n_tiles, 8 lines each) times 8 frequencies over `samples` samples, the first of which is
// sample j0 (0 or 1) of the axis; tab: the cosines or the sines of the axis.  lane: frequency k <= n / 2.
template <int TILES>
__device__ __forceinline__ void contract(double (&acc)[TILES][2], const double *lines, int pitch, int t0, int n_tiles, int samples,
                                         const double *tab, int n, int k, int j0) {
  const int lane = threadIdx.x & 31, jl = lane & 3;
  const double *a = lines + (t0 * 8 + (lane >> 2)) * pitch + jl;
  int idx = mod_small(k * (j0 + jl), n);  // (at most n / 2 * 4)
  const int inc = mod_small(4 * k, n);
#pragma unroll
  for (int i = 0; i < TILES; ++i) acc[i][0] = acc[i][1] = 0.0;
  if (t0 + TILES <= n_tiles) {
#pragma unroll 2
    for (int j = 0; j < samples; j += 4) {
      const double t = tab[idx];
      idx += inc;
      idx -= idx >= n ? n : 0;
#pragma unroll
      for (int i = 0; i < TILES; ++i) mma_f64(acc[i], a[i * 8 * pitch + j], t);
    }
  } else {
    for (int j = 0; j < samples; j += 4) {
      const double t = tab[idx];
      idx += inc;
      idx -= idx >= n ? n : 0;
#pragma unroll
      for (int i = 0; i < TILES; ++i)
        if (t0 + i < n_tiles) mma_f64(acc[i], a[i * 8 * pitch + j], t);
    }
  }
}

__device__ __forceinline__ void cluster_store(uint32_t addr, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}

// CTA 2 * plane + parity along y.
__global__ void __launch_bounds__(kPlaneThreads, 3) plane_kernel(const float *__restrict__ ys, const float *__restrict__ yd, int ny, int nx,
                                                                 double *__restrict__ dst, double *__restrict__ dense_out,
                                                                 int *__restrict__ ticket) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const PlaneLayout f = plane_layout(ny, nx);
  double *tab_x = reinterpret_cast<double *>(smem_raw), *tab_y = tab_x + 2 * nx;
  double *A = tab_y + 2 * ny, *Bm = A + f.rows * f.pitch_a;
  __shared__ double red[kPlaneWarps];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int odd = blockIdx.x & 1;
  const size_t plane = (size_t)(blockIdx.x >> 1) * ny * nx;
  const int hx = nx / 2, mx = (nx - 1) / 2, hy = ny / 2, my = (ny - 1) / 2;
  const int rows = odd ? my : hy + 1;  // samples along y of this parity: odd ones start at 1
  fill_trig_table(tab_x, nx);
  fill_trig_table(tab_y, ny, nx < kPlaneThreads ? nx : 0);  // (by the threads that have no entry of x)
  tc::cluster_sync();  // (the other CTA has started: its memory is there)
  pdl_wait();
  pdl_launch_dependents();
  if (blockIdx.x == 0 && threadIdx.x == 0) *ticket = 0;

  // Folded along both axes, a warp per row.  The pair of CTAs shares the rows: a CTA takes every other row, with its mirror,
  // and puts the even sums into the even CTA's memory and the odd ones into the other's.
  double dense = 0.0;
  const int row_tiles = (rows + 7) / 8, odd_cols = round_up(mx, 4);
  const float *s0 = ys + plane, *d0 = yd + plane;
  const uint32_t even_a = tc::cluster_address(tc::smem_u32(A), 0), odd_a = tc::cluster_address(tc::smem_u32(A), 1);
  for (int j = lane; j < f.even_cols; j += 32) {
    const bool in = j <= hx, xpair = j >= 1 && j <= mx;
#pragma unroll 2
    for (int jy = 2 * warp + odd; jy <= hy; jy += 2 * kPlaneWarps) {
      const bool pair = jy >= 1 && jy <= my;
      const int at = jy * nx, mirror = (ny - jy) * nx;
      float s1[4], d1[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int off = (q < 2 ? at : mirror) + ((q & 1) ? nx - j : j);
        const bool load = in && (q < 2 || pair) && ((q & 1) == 0 || xpair);
        s1[q] = load ? __ldg(&s0[off]) : 0.f;
        d1[q] = load ? __ldg(&d0[off]) : 0.f;
      }
      double e[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const double d = (double)d1[q];
        e[q] = (double)s1[q] - d;
        dense = fma(d, d, dense);
      }
      const double u = e[0] + e[2], v = e[1] + e[3];
      const uint32_t to_even = even_a + (jy * f.pitch_a + j) * 8;
      cluster_store(to_even, u + v);
      if (xpair) cluster_store(to_even + (f.even_cols - 1) * 8, u - v);
      if (pair) {
        const double x = e[0] - e[2], y = e[1] - e[3];
        const uint32_t to_odd = odd_a + ((jy - 1) * f.pitch_a + j) * 8;
        cluster_store(to_odd, x + y);
        if (xpair) cluster_store(to_odd + (f.even_cols - 1) * 8, x - y);
      }
    }
  }
  // zeros: the columns that fill the last step of four, the rows that fill the last tile
  for (int i = warp; i < row_tiles * 8; i += kPlaneWarps) {
    for (int j = mx + lane; j < odd_cols; j += 32) A[i * f.pitch_a + f.even_cols + j] = 0.0;
    if (i >= rows)
      for (int j = lane; j < f.even_cols + odd_cols; j += 32) A[i * f.pitch_a + j] = 0.0;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) dense += __shfl_xor_sync(0xffffffffu, dense, o);
  if (lane == 0) red[warp] = dense;
  tc::cluster_sync();
  if (threadIdx.x == 0) {  // |y_dense|^2 of the rows that this CTA read
    double sum = 0.0;
#pragma unroll
    for (int i = 0; i < kPlaneWarps; ++i) sum += red[i];
    dense_out[blockIdx.x] = sum;
  }

  // along x: lines are the rows; cosines of the even part, then sines of the odd one
  constexpr int TX = kTilesX, TY = kTilesY;
  const int cos_x = (hx + 8) / 8, sin_x = (mx + 7) / 8;
  for (int t0 = 0; t0 < row_tiles; t0 += TX) {
    for (int kt = warp; kt < cos_x + sin_x; kt += kPlaneWarps) {
      const bool sine = kt >= cos_x;
      const int k0 = sine ? 1 + (kt - cos_x) * 8 : kt * 8, k_last = sine ? mx : hx;
      double acc[TX][2];
      contract<TX>(acc, A + (sine ? f.even_cols : 0), f.pitch_a, t0, row_tiles, sine ? odd_cols : f.even_cols, tab_x + (sine ? nx : 0), nx,
                   min(k0 + (lane >> 2), k_last), sine ? 1 : 0);
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int k = k0 + 2 * (lane & 3) + u;
        if (k > k_last) continue;
        double *col = Bm + (sine ? hx + k : k) * f.pitch_b + t0 * 8 + (lane >> 2);
#pragma unroll
        for (int i = 0; i < TX; ++i)
          if (t0 + i < row_tiles) col[i * 8] = acc[i][u];
      }
    }
  }
  __syncthreads();

  // along y: lines are the coefficients of x
  const int kts = odd ? (my + 7) / 8 : (hy + 8) / 8, col_tiles = (nx + 7) / 8, k_last = odd ? my : hy;
  const int samples = round_up(rows, 4);
  for (int e = warp; e < kts * ((col_tiles + TY - 1) / TY); e += kPlaneWarps) {
    const int t0 = e / kts * TY, k0 = e % kts * 8 + odd;
    double acc[TY][2];
    contract<TY>(acc, Bm, f.pitch_b, t0, col_tiles, samples, tab_y + (odd ? ny : 0), ny, min(k0 + (lane >> 2), k_last), odd);
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int k = k0 + 2 * (lane & 3) + u, col = t0 * 8 + (lane >> 2);
      if (k > k_last) continue;
      double *out = dst + plane + (size_t)((odd ? hy + k : k) * nx + col);
#pragma unroll
      for (int i = 0; i < TY; ++i)
        if (col + i * 8 < nx) out[i * 8] = acc[i][u];
    }
  }
}

struct TimeArgs {
  const double *src;    // [C][n][inner]
  double *energies;     // [gridDim.x][4]
  const double *dense;  // [planes], two a plane
  int *ticket;
  double *out;
  int n, ny, nx, units_per_c, units, planes;
  double n_freq, w0, w1, w2, w3, eps;
};

// The pass over t: 64 lines at a time, their samples brought in while those before are worked on; the energies are added
// up over all of a CTA's lines, and the CTA that finishes last adds those of all CTAs in a fixed order and writes the result.
__global__ void __launch_bounds__(kTimeThreads, 4) time_kernel(const TimeArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int n = a.n, h = n / 2, m = (n - 1) / 2, inner = a.ny * a.nx;
  double *tab = reinterpret_cast<double *>(smem_raw), *raw = tab + 2 * n;  // samples: [2][n + 1][kTimePitch], the last row zero
  const int stage = (n + 1) * kTimePitch;
  __shared__ int line_band[2][kTimeLines];  // low along y and x | log2 of the weight << 1 (no line: 0x100)
  __shared__ double red[(kTimeThreads / 32) * 5];
  __shared__ int last;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  fill_trig_table(tab, n);
  for (int i = tid; i < kTimePitch; i += kTimeThreads) raw[n * kTimePitch + i] = raw[stage + n * kTimePitch + i] = 0.0;
  const int line = tid & (kTimeLines - 1), part = tid / kTimeLines;
  pdl_wait();
  pdl_launch_dependents();
  auto bring = [&](int unit, int buf) {
    if (unit < a.units) {
      const int c = unit / a.units_per_c, in = (unit - c * a.units_per_c) * kTimeLines + line;
      const bool real = in < inner;
      const double *src = a.src + (size_t)c * n * inner + (real ? in : 0);
      const uint32_t dst = (uint32_t)__cvta_generic_to_shared(raw + buf * stage + line);
      for (int j = part; j < n; j += kTimeThreads / kTimeLines)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst + j * kTimePitch * 8), "l"(src + (size_t)j * inner), "r"(real ? 8 : 0) : "memory");
      if (part == 0) {
        const int iy = in / a.nx, ix = in - iy * a.nx;
        const int ky = iy <= a.ny / 2 ? iy : iy - a.ny / 2, kx = ix <= a.nx / 2 ? ix : ix - a.nx / 2;
        const int wy = ky == 0 || 2 * ky == a.ny ? 0 : 1, wx = kx == 0 || 2 * kx == a.nx ? 0 : 1;
        line_band[buf][line] = real ? (ky <= a.ny / 4 && kx <= a.nx / 4 ? 1 : 0) | (wy + wx) << 1 : 0x100;
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  double energy[4] = {0.0, 0.0, 0.0, 0.0};  // LL, LH, HL, HH
  const int l0 = warp * 16 + (lane >> 2), jl = lane & 3;
  bring(blockIdx.x, 0);
  int buf = 0;
  for (int unit = blockIdx.x; unit < a.units; unit += gridDim.x, buf ^= 1) {
    bring(unit + gridDim.x, buf ^ 1);  // (free since the barrier that ended the unit before)
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    // a warp: 16 lines; cosines and sines of 8 frequencies at a time
    const double *x = raw + buf * stage + l0;
    double low[2] = {0.0, 0.0}, high[2] = {0.0, 0.0};  // energy below and above n / 4, per line
    for (int k0 = 0; k0 <= h; k0 += 8) {
      const int k = min(k0 + (lane >> 2), h);
      double cs[2][2] = {}, sn[2][2] = {};
      int idx = mod_small(k * jl, n);
      const int inc = mod_small(4 * k, n);
#pragma unroll 3
      for (int j = jl; j - jl <= h; j += 4) {
        const bool pair = j >= 1 && j <= m;
        const double *p = x + (j <= h ? j : n) * kTimePitch, *q = x + (pair ? n - j : n) * kTimePitch;
        const double c = tab[idx], s = tab[n + idx];
        idx += inc;
        idx -= idx >= n ? n : 0;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const double u = p[8 * i], v = q[8 * i];
          mma_f64(cs[i], u + v, c);
          mma_f64(sn[i], pair ? u - v : 0.0, s);
        }
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int kk = k0 + 2 * jl + u;
        if (kk > h) continue;
        const double w = kk == 0 || 2 * kk == n ? 1.0 : 2.0;
        const bool sine = kk >= 1 && kk <= m, below = kk <= n / 4;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const double e = sine ? fma(cs[i][u], cs[i][u], sn[i][u] * sn[i][u]) : cs[i][u] * cs[i][u];
          if (below) low[i] = fma(w, e, low[i]);
          else high[i] = fma(w, e, high[i]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int band = line_band[buf][l0 + 8 * i];
      if (band >> 8) continue;
      const double w = (double)(1 << (band >> 1));
      if (band & 1) {
        energy[0] = fma(w, low[i], energy[0]);
        energy[2] = fma(w, high[i], energy[2]);
      } else {
        energy[1] = fma(w, low[i], energy[1]);
        energy[3] = fma(w, high[i], energy[3]);
      }
    }
    __syncthreads();
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  auto sums = [&](auto &v, int nv) {  // over the CTA, in a fixed order; valid in thread 0
#pragma unroll
    for (int q = 0; q < nv; ++q) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
      if (lane == 0) red[warp * nv + q] = v[q];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < nv; ++q) v[q] = (red[q] + red[nv + q]) + (red[2 * nv + q] + red[3 * nv + q]);
  };
  sums(energy, 4);
  if (tid == 0) {
#pragma unroll
    for (int b = 0; b < 4; ++b) __stcg(&a.energies[(size_t)blockIdx.x * 4 + b], energy[b]);
    __threadfence();
    last = atomicAdd(a.ticket, 1) == (int)gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double tot[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
  for (int i = tid; i < (int)gridDim.x; i += kTimeThreads) {
    const double2 x = __ldcg(reinterpret_cast<const double2 *>(a.energies) + 2 * i), y = __ldcg(reinterpret_cast<const double2 *>(a.energies) + 2 * i + 1);
    tot[0] += x.x, tot[1] += x.y, tot[2] += y.x, tot[3] += y.y;
  }
#pragma unroll 4
  for (int i = tid; i < a.planes; i += kTimeThreads) tot[4] += __ldcg(&a.dense[i]);
  sums(tot, 5);
  if (tid == 0) {
    const double denom = tot[4] * a.n_freq + a.eps;
    a.out[0] = (a.w0 * tot[0] + a.w1 * tot[1] + a.w2 * tot[2] + a.w3 * tot[3]) / denom;
    a.out[1] = tot[0];
    a.out[2] = tot[1];
    a.out[3] = tot[2];
    a.out[4] = tot[3];
    a.out[5] = denom;
  }
}

// Planes of 512 points and more that a CTA holds, and time axes whose samples of 64 lines it holds.
bool planes_fit(int T, int H, int W) {
  return (long long)H * W >= 512 && (long long)H * W <= kPlaneMaxShared / 8 && plane_shared_bytes(H, W) <= kPlaneMaxShared && T <= kTimeMax;
}

// Products that a warp of plane_kernel takes one after the other: along x, then along y.
int plane_steps(int ny, int nx) {
  const int row_tiles = (ny / 2 + 8) / 8, col_tiles = (nx + 7) / 8;
  const int rounds_x = (row_tiles + kTilesX - 1) / kTilesX * ((nx / 2 + 8) / 8 + ((nx - 1) / 2 + 7) / 8);
  const int rounds_y = (ny / 2 + 8) / 8 * ((col_tiles + kTilesY - 1) / kTilesY);
  const int each_x = round_up(nx / 2 + 1, 4) / 4 * (row_tiles < kTilesX ? row_tiles : kTilesX);
  const int each_y = round_up(ny / 2 + 1, 4) / 4 * (col_tiles < kTilesY ? col_tiles : kTilesY);
  return (rounds_x + kPlaneWarps - 1) / kPlaneWarps * each_x + (rounds_y + kPlaneWarps - 1) / kPlaneWarps * each_y;
}

// Whether plane by plane is the faster way, by 15 000 shapes measured both ways (C 1-32, T 1-96, 8 x 64 to 96 x 200 and 300 x 24
// points).  Taken always, it was 2.5 % slower in the mean than the faster way of each shape and up to 2.2 times; by these lines
// 0.4 % and up to 1.5 times, and 98 % of usual latents (C 4 or 16, T 5-33, 30-96 x 40-170) are within 5 %.  The CTAs of
// plane_kernel hide each other's folds and chains while an SM has two or three.  Times in us, axis by axis / plane by plane:
//  - a plane that fills an SM pays only while the planes make about one wave (16 x 21 x 90 x 160 134 / 140, one plane of it
//    18 / 26, 4 x 17 x 88 x 160 40 / 32);
//  - fewer CTAs than SMs run alone: the chain of a warp has to be short (4 x 7 x 72 x 144 24 / 33, 520 steps; 4 x 7 x 60 x 104
//    18 / 14, 168), and while only some SMs have a second one (4 x 21 x 68 x 104 26 / 32);
//  - a CTA costs some 3 us however small its plane, and tiles of eight lines of a narrow plane are padding in part: few of them
//    are welcome, many are not (1 x 5 x 23 x 23 13.7 / 7.9, 16 x 96 x 23 x 23 32 / 52; 16 x 21 x 8 x 200 32 / 48,
//    3 x 57 x 5 x 178 20 / 30, 3 x 2048 x 1 68 / 583).
bool planes_pay(int C, int T, int H, int W) {
  if (!planes_fit(T, H, W)) return false;
  const long long ctas = 2LL * C * T;
  const int steps = plane_steps(H, W), per_sm = (int)(226 * 1024 / (plane_shared_bytes(H, W) + 1100));  // (three, by registers)
  if (per_sm == 1) return ctas > 60 && ctas <= 148;
  if (H < 24 || W < 24) return ctas <= 148 ? steps <= 150 : ctas <= 592 && steps <= 100 && H >= 8;
  if (steps <= 50) return ctas <= 888;
  if (ctas <= 148) return steps <= 400;
  return steps <= 340 || ctas > 222 || per_sm == 2;
}
int time_units(int C, int H, int W) { return C * ((H * W + kTimeLines - 1) / kTimeLines); }
int time_ctas(int C, int H, int W) { return time_units(C, H, W) < kTimeCtas ? time_units(C, H, W) : kTimeCtas; }
size_t time_shared_bytes(int n) { return sizeof(double) * (2 * n + 2 * (n + 1) * kTimePitch); }

cudaError_t launch_planes(const float *ys, const float *yd, int C, int T, int H, int W, const double *weights, double eps, double *out,
                          char *p, cudaStream_t s, int *launches) {
  TimeArgs a = {};
  a.ticket = reinterpret_cast<int *>(p);
  p += 256;
  double *coef = reinterpret_cast<double *>(p);
  p += align256(sizeof(double) * (size_t)C * T * H * W);
  a.energies = reinterpret_cast<double *>(p);
  p += align256(sizeof(double) * 4 * time_ctas(C, H, W));
  double *dense = reinterpret_cast<double *>(p);  // of the CTAs of the first kernel
  cudaError_t e = allow_shared_memory(plane_kernel, kPlaneMaxShared);
  if (e != cudaSuccess) return e;
  e = launch_pdl(plane_kernel, dim3(2u * C * T), dim3(kPlaneThreads), plane_shared_bytes(H, W), s, Cluster{2}, ys, yd, H, W, coef, dense, a.ticket);
  if (e != cudaSuccess) return e;
  ++*launches;
  a.src = coef;
  a.dense = dense;
  a.out = out;
  a.n = T;
  a.ny = H;
  a.nx = W;
  a.units_per_c = time_units(1, H, W);
  a.units = time_units(C, H, W);
  a.planes = 2 * C * T;
  a.n_freq = (double)T * H * W;
  a.w0 = weights[0];
  a.w1 = weights[1];
  a.w2 = weights[2];
  a.w3 = weights[3];
  a.eps = eps;
  e = allow_shared_memory(time_kernel, (int)time_shared_bytes(kTimeMax));
  if (e != cudaSuccess) return e;
  e = launch_pdl(time_kernel, dim3(time_ctas(C, H, W)), dim3(kTimeThreads), time_shared_bytes(T), s, a);
  ++*launches;
  return e;
}

size_t n_ctas(long long lines, int n) { return (size_t)((lines + lines_per_cta(n) - 1) / lines_per_cta(n)); }

// CTAs that share the frequencies of a set of lines: as many as there are rounds, while lines alone leave SMs without a
// CTA.  (One line of 4096 samples, 65 rounds over 13 chunks: 6466 us in one CTA.)
int frequency_splits(long long lines, int n) {
  const size_t ctas = n_ctas(lines, n), per_round = 8 * frequency_warps(n), rounds = (n / 2 + per_round) / per_round;
  return ctas >= 148 ? 1 : (int)(rounds < 296 / ctas ? rounds : 296 / ctas);
}
// CTAs of the pass over t: each leaves four sums.
size_t n_energies(int C, int T, int H, int W) { return n_ctas((long long)C * H * W, T) * frequency_splits((long long)C * H * W, T); }

template <int PASS>
cudaError_t launch_axis(const AxisArgs &a, cudaStream_t s) {
  const size_t smem = sizeof(double) * 2 * fold_layout(a.n, a.inner == 1).doubles + (a.n <= kMaxSharedTable ? sizeof(double2) * a.n : 0);
  constexpr int kMost = sizeof(double) * 2 * kMaxChunk * (kLines + 4) + sizeof(double2) * kMaxSharedTable;
  cudaError_t e = allow_shared_memory(axis_kernel<PASS>, kMost);
  if (e != cudaSuccess) return e;
  const dim3 grid((unsigned)n_ctas(a.lines, a.n), (unsigned)frequency_splits(a.lines, a.n));
  return launch_pdl(axis_kernel<PASS>, grid, dim3(kBandThreads), smem, s, a);
}

}  // namespace

// What the way axis by axis takes, also where the other one does with half of it: a buffer made for some tensor goes on
// serving every smaller one, whichever way that takes.
size_t band_error_workspace_bytes(int C, int T, int H, int W) {
  const size_t n = (size_t)C * T * H * W;
  return align256(sizeof(double2) * ((size_t)T + H + W)) + 2 * align256(sizeof(double) * n) +
         align256(sizeof(double) * 4 * n_energies(C, T, H, W)) + align256(sizeof(double) * n_ctas((long long)C * T * H, W));
}

cudaError_t launch_band_error(const float *ys, const float *yd, int C, int T, int H, int W, const double *weights,
                              double eps, double *out, void *workspace, cudaStream_t s, int *launches) {
  const long long n = (long long)C * T * H * W;
  char *p = static_cast<char *>(workspace);
  if (planes_pay(C, T, H, W)) return launch_planes(ys, yd, C, T, H, W, weights, eps, out, p, s, launches);
  double2 *tables = reinterpret_cast<double2 *>(p);  // of x, y, t
  p += align256(sizeof(double2) * ((size_t)T + H + W));
  double *A = reinterpret_cast<double *>(p);
  p += align256(sizeof(double) * n);
  double *Bm = reinterpret_cast<double *>(p);
  p += align256(sizeof(double) * n);
  double *energies = reinterpret_cast<double *>(p);
  p += align256(sizeof(double) * 4 * n_energies(C, T, H, W));
  double *dense = reinterpret_cast<double *>(p);
  trig_tables_kernel<<<(unsigned)(((long long)T + H + W + 127) / 128), 128, 0, s>>>(W, H, T, tables);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  AxisArgs a = {};
  a.ys = ys;
  a.yd = yd;
  a.table = tables;
  a.dst = A;
  a.partial = dense;
  a.lines = (unsigned)C * T * H;
  a.inner = 1;
  a.n = W;
  if ((e = launch_axis<0>(a, s)) != cudaSuccess) return e;
  a.src = A;
  a.table = tables + W;
  a.dst = Bm;
  a.partial = nullptr;
  a.lines = (unsigned)C * T * W;
  a.inner = W;
  a.n = H;
  if ((e = launch_axis<1>(a, s)) != cudaSuccess) return e;
  a.src = Bm;
  a.table = tables + W + H;
  a.dst = nullptr;
  a.partial = energies;
  a.lines = (unsigned)C * H * W;
  a.inner = (unsigned)H * W;
  a.n = T;
  a.ny = H;
  a.nx = W;
  if ((e = launch_axis<2>(a, s)) != cudaSuccess) return e;
  e = launch_pdl(band_final_kernel, dim3(1), dim3(1024), 0, s, (const double *)energies, (long long)n_energies(C, T, H, W),
                 (const double *)dense, (long long)n_ctas((long long)C * T * H, W), (double)T * H * W, weights[0], weights[1],
                 weights[2], weights[3], eps, out);
  *launches += 5;
  return e;
}

}  // namespace heart
