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
// three passes; the full circulant projections used before took 4.3e8 fma with two loads for each (0.45 ms).
#include <math.h>

#include "common.cuh"

namespace heart {

namespace {

constexpr int kLines = 32;        // lines of an axis per CTA
constexpr int kLinePitch = 36;    // 4 (mod 16) doubles: 8 x 4 fragments are read without bank conflicts
constexpr int kMaxChunk = 160;    // folded samples of a line in shared memory at a time
constexpr int kMaxSharedTable = 1024;
constexpr int kBandThreads = 128;

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

__device__ __forceinline__ void mma_f64(double (&d)[2], double a, double b) {
  asm("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(d[0]), "+d"(d[1]) : "d"(a), "d"(b));
}

// Sums over the CTA of kBandThreads threads, in a fixed order; valid in thread 0.
template <int NV>
__device__ __forceinline__ void cta_sums(double (&v)[NV], double *red /* [kBandThreads / 32 * NV] */) {
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
  double *partial;        // pass 0: |y_dense|^2 per CTA; pass 2: [CTA][4] energies
  long long lines, inner;
  int n;
  int ny, nx;             // pass 2: lengths of the other axes (inner = ny * nx)
};

// One pass over an axis of a [outer, n, inner] view; a CTA takes kLines of the outer * inner lines.
template <int PASS>
__global__ void __launch_bounds__(kBandThreads) axis_kernel(const AxisArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int n = a.n, h = n / 2, m = (n - 1) / 2;
  const int rows = (h + 1 + 3) / 4 * 4, chunk = min(rows, kMaxChunk), n_chunks = (rows + chunk - 1) / chunk;
  double *even = reinterpret_cast<double *>(smem_raw), *odd = even + chunk * kLinePitch;
  double2 *tab = reinterpret_cast<double2 *>(odd + chunk * kLinePitch);
  __shared__ double red[kBandThreads / 32 * 4];
  __shared__ int line_band[kLines];      // pass 2: low along y and x | log2 of the weight << 1
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const long long l0 = (long long)blockIdx.x * kLines;
  const int n_lines = (int)min((long long)kLines, a.lines - l0);
  double dense = 0.0;
  // folded samples [j0, j0 + chunk) of the lines
  auto stage = [&](int j0) {
    for (int e = tid; e < chunk * kLines; e += kBandThreads) {
      const int jj = a.inner == 1 ? e % chunk : e / kLines, line = a.inner == 1 ? e / chunk : e % kLines;
      const int j = j0 + jj;
      double x = 0.0, y = 0.0;
      if (line < n_lines && j <= h) {
        const long long l = l0 + line, o = a.inner == 1 ? l : l / a.inner;
        const long long at = o * n * a.inner + (l - o * a.inner) + (long long)j * a.inner;
        const long long mirror = at + (long long)(n - 2 * j) * a.inner;
        const bool pair = j >= 1 && j <= m;
        if (PASS == 0) {
          const double d = (double)a.yd[at];
          x = (double)a.ys[at] - d;
          dense = fma(d, d, dense);
          if (pair) {
            const double d2 = (double)a.yd[mirror];
            y = (double)a.ys[mirror] - d2;
            dense = fma(d2, d2, dense);
          }
        } else {
          x = __ldcg(&a.src[at]);
          if (pair) y = __ldcg(&a.src[mirror]);
        }
        even[jj * kLinePitch + line] = x + y;
        odd[jj * kLinePitch + line] = pair ? x - y : 0.0;
      } else {
        even[jj * kLinePitch + line] = 0.0;
        odd[jj * kLinePitch + line] = 0.0;
      }
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
  if (PASS == 2 && tid < kLines) {
    const int in = (int)((l0 + tid) % a.inner), iy = in / a.nx, ix = in % a.nx;
    const int ky = iy <= a.ny / 2 ? iy : iy - a.ny / 2, kx = ix <= a.nx / 2 ? ix : ix - a.nx / 2;
    const int wy = ky == 0 || 2 * ky == a.ny ? 0 : 1, wx = kx == 0 || 2 * kx == a.nx ? 0 : 1;
    line_band[tid] = (ky <= a.ny / 4 && kx <= a.nx / 4 ? 1 : 0) | (wy + wx) << 1;
  }
  __syncthreads();
  double energy[4] = {0.0, 0.0, 0.0, 0.0};  // LL, LH, HL, HH
  const int jl = lane & 3, kl = lane >> 2;
  for (int k0 = 0; k0 <= h; k0 += 8 * (kBandThreads / 32)) {  // warp w: frequencies k0 + 8 w ... + 7
    const int k = k0 + 8 * warp + kl;
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
        if (k0 > 0) dense = counted;  // (|y_dense|^2: in the first round only)
        __syncthreads();
      }
      if (k0 + 8 * warp <= h) {
        const double *E = even + jl * kLinePitch + kl, *O = odd + jl * kLinePitch + kl;
#pragma unroll 2
        for (int j = 0; j < chunk; j += 4, E += 4 * kLinePitch, O += 4 * kLinePitch) {
          const double2 t = table[idx];
          idx += inc;
          idx -= idx >= n ? n : 0;
#pragma unroll
          for (int i = 0; i < kLines / 8; ++i) {
            mma_f64(c[i], E[8 * i], t.x);
            mma_f64(s[i], O[8 * i], t.y);
          }
        }
      }
    }
    if (k0 + 8 * warp > h) continue;
    // lane: line 8 i + kl, frequencies k0 + 8 warp + 2 jl + {0, 1}
#pragma unroll
    for (int i = 0; i < kLines / 8; ++i) {
      const int line = 8 * i + kl;
      if (line >= n_lines) continue;
      const long long l = l0 + line, o = a.inner == 1 ? l : l / a.inner;
      double *out = PASS == 2 ? nullptr : a.dst + o * n * a.inner + (l - o * a.inner);
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int kk = k0 + 8 * warp + 2 * jl + u;
        if (kk > h) continue;
        if (PASS == 2) {
          const int band = line_band[line];
          const double w = (double)(1 << ((band >> 1) + (kk == 0 || 2 * kk == n ? 0 : 1)));
          const double e = w * (kk >= 1 && kk <= m ? fma(c[i][u], c[i][u], s[i][u] * s[i][u]) : c[i][u] * c[i][u]);
          const int q = (kk <= n / 4 ? 0 : 2) + ((band & 1) ? 0 : 1);
#pragma unroll
          for (int b = 0; b < 4; ++b) energy[b] += b == q ? e : 0.0;
        } else {
          out[(long long)kk * a.inner] = c[i][u];
          if (kk >= 1 && kk <= m) out[(long long)(h + kk) * a.inner] = s[i][u];
        }
      }
    }
  }
  if (PASS == 2) {
    cta_sums<4>(energy, red);
    if (tid < 4) a.partial[(size_t)blockIdx.x * 4 + tid] = energy[tid];
  }
  if (PASS == 0) {
    double v[1] = {dense};
    cta_sums<1>(v, red);
    if (tid == 0) a.partial[blockIdx.x] = v[0];
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

size_t n_ctas(long long lines) { return (size_t)((lines + kLines - 1) / kLines); }

template <int PASS>
cudaError_t launch_axis(const AxisArgs &a, cudaStream_t s) {
  const int rows = (a.n / 2 + 1 + 3) / 4 * 4, chunk = rows < kMaxChunk ? rows : kMaxChunk;
  const size_t smem = sizeof(double) * 2 * chunk * kLinePitch + (a.n <= kMaxSharedTable ? sizeof(double2) * a.n : 0);
  cudaError_t e = cudaFuncSetAttribute(axis_kernel<PASS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)(sizeof(double) * 2 * kMaxChunk * kLinePitch + sizeof(double2) * kMaxSharedTable));
  if (e != cudaSuccess) return e;
  return launch_pdl(axis_kernel<PASS>, dim3((unsigned)n_ctas(a.lines)), dim3(kBandThreads), smem, s, a);
}

}  // namespace

size_t band_error_workspace_bytes(int C, int T, int H, int W) {
  const size_t n = (size_t)C * T * H * W;
  return align256(sizeof(double2) * ((size_t)T + H + W)) + 2 * align256(sizeof(double) * n) +
         align256(sizeof(double) * 4 * n_ctas((long long)C * H * W)) + align256(sizeof(double) * n_ctas((long long)C * T * H));
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
  p += align256(sizeof(double) * 4 * n_ctas((long long)C * H * W));
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
  a.lines = (long long)C * T * H;
  a.inner = 1;
  a.n = W;
  if ((e = launch_axis<0>(a, s)) != cudaSuccess) return e;
  a.src = A;
  a.table = tables + W;
  a.dst = Bm;
  a.partial = nullptr;
  a.lines = (long long)C * T * W;
  a.inner = W;
  a.n = H;
  if ((e = launch_axis<1>(a, s)) != cudaSuccess) return e;
  a.src = Bm;
  a.table = tables + W + H;
  a.dst = nullptr;
  a.partial = energies;
  a.lines = (long long)C * H * W;
  a.inner = (long long)H * W;
  a.n = T;
  a.ny = H;
  a.nx = W;
  if ((e = launch_axis<2>(a, s)) != cudaSuccess) return e;
  e = launch_pdl(band_final_kernel, dim3(1), dim3(1024), 0, s, (const double *)energies, (long long)n_ctas((long long)C * H * W),
                 (const double *)dense, (long long)n_ctas((long long)C * T * H), (double)T * H * W, weights[0], weights[1],
                 weights[2], weights[3], eps, out);
  *launches += 5;
  return e;
}

}  // namespace heart
