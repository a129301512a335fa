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
// even part, sines the odd one.  x and y write their coefficients to the workspace (they stay in L2), t only
// adds up energies.  For 16 x 21 x 60 x 104 that is 1.9e8 fma (10 us at 18.5 T fma/s) and 84 MB of L2 traffic in
// three passes (58 us; 16 lines a warp and 8 CTAs an SM, against 64 us with 32 and 4); the full circulant projections used
// before took 4.3e8 fma with two loads for each (0.45 ms).
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

size_t band_error_workspace_bytes(int C, int T, int H, int W) {
  const size_t n = (size_t)C * T * H * W;
  return align256(sizeof(double2) * ((size_t)T + H + W)) + 2 * align256(sizeof(double) * n) +
         align256(sizeof(double) * 4 * n_energies(C, T, H, W)) + align256(sizeof(double) * n_ctas((long long)C * T * H, W));
}

cudaError_t launch_band_error(const float *ys, const float *yd, int C, int T, int H, int W, const double *weights,
                              double eps, double *out, void *workspace, cudaStream_t s, int *launches) {
  const long long n = (long long)C * T * H * W;
  char *p = static_cast<char *>(workspace);
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
