// FP64 log-domain Gibbs operator for point clouds (cost |x_i - y_j|^2):
//
//   z_i = log sum_j exp(L_j - |x_i - y_j|^2 / eps),   L_j = W_j/eps + log w_j.
//
// Two forms.
//
// rows64, on the fly: an FP32 sweep finds a shift M_i close to the largest
// exponent (FP64 has a thousand powers of two to spare, so its error does not
// matter), an FP64 sweep sums the exponentials.  Bound: FP64 issue, 2 lanes per
// clock and SM.  The exponential is table-driven (P. T. P. Tang, ACM TOMS 15,
// 1989): the exponent in units of 1/256 bit, split by adding a large constant
// into an integer, read from the sum's low bits by integer instructions, and a
// remainder of at most half a unit, whose power needs four terms of the series;
// 2^(k/256) comes from shared memory.  15 FP64 instructions a term in two
// dimensions, against about 28 with two FP64 sweeps and exp().
//
// Stored kernel, for the solvers: the first pass of an eps stores its terms
//   K_ij = exp(beta_j - |x_i - y_j|^2/eps - M_i),  beta = L at that time
// (Algorithm 2's stabilised kernel), and later passes of that eps are products,
//   rows     z_i = M_i + log sum_j K_ij e^{L_j - beta_j},
//   columns  z_j = -beta_j + log sum_i K_ij e^{L_i + M_i},
// one FP64 multiply-add and 8 bytes a term, in both directions from one copy.
// A row is stored with a shift that puts its sum between 1e-30 and 1e30 (the FP32
// shift where it does, else the FP64 maximum), so K_ij < 1e30.  A result is used
// only where neither underflow nor overflow can have touched it: with all weights
// below e^300 the terms that K_ij lost are below e^300 2^-1022 nin in sum, so a sum
// above 1e-150 is exact to rounding, and no sum comes near 1e300; any other row or
// column is redone on the fly.  A weight above e^300 (the potentials moved by 300
// eps) makes the next row pass store the kernel anew.
//
// Measured, 3001 x 2477 points in 2-D: 20 iterations and the objective 31.9 ms
// with two FP64 sweeps and exp() per pass (705 us), 2.76 ms here.
#include <string.h>

#include <algorithm>

#include "exp_table.cuh"
#include "uot_internal.cuh"

namespace uot {
namespace {

constexpr double kDrift = 300.0;                  // largest log weight before a new kernel
constexpr double kLeastSum = 1e-150, kMostSum = 1e300;  // sums of products that are used

// The line L and its FP32 copy; with a stored kernel the weights e^{L - beta},
// and *drift raised where one is too large or a point that had no mass when the
// kernel was stored has some now.
__global__ void __launch_bounds__(128) points64_line(const double* __restrict__ W, const double* __restrict__ logw,
                                                     int nin, double inv_eps, double* __restrict__ Ls,
                                                     float* __restrict__ L32, const double* __restrict__ beta,
                                                     double* __restrict__ w, int* __restrict__ drift) {
  pdl_wait();
  pdl_launch_dependents();
  const int j = blockIdx.x * 128 + threadIdx.x;
  if (j >= nin) return;
  const double v = W[j];
  const double L = (v == -kInf) ? -kInf : fma(v, inv_eps, logw[j]);
  Ls[j] = L;
  if (L32) L32[j] = (float)L;
  if (w) {
    const double b = beta[j];
    double q = 0.0;
    if (L != -kInf) {
      const double d = L - b;
      if (b == -kInf || !(d <= kDrift)) *drift = 1;
      else q = exp(d);
    }
    w[j] = q;
  }
}

struct Rows64 {
  const double* x;   // [nrows][d]
  const double* y;   // [nin][d]
  const float* x32;  // FP32 copies, or NULL: the shift is found in FP64
  const float* y32;
  const double* Ls;  // [nin] the line, L32 its FP32 copy
  const float* L32;
  int d, nrows, nin;
  double inv_eps;
  // stored kernel (K NULL: on the fly)
  double* K;         // [nrows][ld]
  int64_t ld;
  double* M;         // [nrows]
  double* beta;      // [nin] (-inf: no mass then)
  const double* w;   // [nin] weights of this pass
  const int* drift;  // store the kernel anew when set (or when force)
  int force;
};

// One row by one warp, on the fly; STORE writes its terms.  Returns the sum and
// the shift (-inf for an empty row).
template <int D, bool STORE>
__device__ __forceinline__ void row64(const Rows64& a, int i, const double* tab, double& S, double& M) {
  const int lane = threadIdx.x & 31;
  const int d = D ? D : a.d;
  const double k = a.inv_eps;
  double xi[D ? D : 8];
#pragma unroll
  for (int c = 0; c < (D ? D : 8); ++c) xi[c] = (c < d) ? a.x[(int64_t)i * d + c] : 0.0;
  auto cost = [&](int j) {
    double q = 0.0;
#pragma unroll
    for (int c = 0; c < (D ? D : 8); ++c)
      if (c < d) {
        const double t = xi[c] - a.y[(int64_t)j * d + c];
        q = fma(t, t, q);
      }
    return q;
  };
  // the shift: from the FP32 copies, and once more in FP64 where that left the
  // sum empty or out of range (exponents beyond FP32's reach, or no mass at all).
  // Stored terms meet weights up to e^300, so their range is narrower: coordinates
  // with an offset large against their spread move the FP32 shift by hundreds.
  constexpr double least = STORE ? 1e-30 : 1e-270, most = STORE ? 1e30 : 1e290;
  for (int attempt = a.x32 ? 0 : 1; attempt < 2; ++attempt) {
    double m;
    if (attempt == 0) {
      float xf[D ? D : 8], mf = -INFINITY;
#pragma unroll
      for (int c = 0; c < (D ? D : 8); ++c) xf[c] = (c < d) ? a.x32[(int64_t)i * d + c] : 0.0f;
      const float kf = -(float)k;
#pragma unroll 4
      for (int j = lane; j < a.nin; j += 32) {
        float q = 0.0f;
#pragma unroll
        for (int c = 0; c < (D ? D : 8); ++c)
          if (c < d) {
            const float t = xf[c] - a.y32[(int64_t)j * d + c];
            q = fmaf(t, t, q);
          }
        mf = fmaxf(mf, fmaf(kf, q, a.L32[j]));
      }
      m = (double)warp_maxf(mf);
    } else {
      m = -kInf;
      for (int j = lane; j < a.nin; j += 32) m = fmax(m, fma(-k, cost(j), a.Ls[j]));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
      if (m == -kInf) {  // every input is empty (or NaN: then the sum below says so)
        bool nan = false;
        for (int j = lane; j < a.nin; j += 32) nan = nan || a.Ls[j] != a.Ls[j];
        nan = __any_sync(0xffffffffu, nan);
        if (STORE)
          for (int j = lane; j < a.nin; j += 32) a.K[i * a.ld + j] = 0.0;
        S = nan ? __longlong_as_double(0x7ff8000000000000ll) : 0.0;
        M = nan ? 0.0 : -kInf;
        return;
      }
    }
    M = m;
    double s = 0.0;
#pragma unroll 2
    for (int j = lane; j < a.nin; j += 32) {
      const double t = exp_tab(fma(-k, cost(j), a.Ls[j]) - m, tab);
      if (STORE) a.K[i * a.ld + j] = t;
      s += t;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    S = s;
    if (s >= least && s <= most) return;
  }
}

constexpr int kRowWarps = 8;

// Row pass: a warp per row, then the CTA's epilogues (log, Table 1 row) side by
// side in the lanes of one warp.
template <int D>
__global__ void __launch_bounds__(kRowWarps * 32) points64_rows(Rows64 a, Epilogue epi) {
  static_assert(kRowWarps * 32 == kExpUnits, "one table entry a thread");
  __shared__ double tab[kExpUnits];
  __shared__ double sS[kRowWarps], sM[kRowWarps];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x * kRowWarps + warp;
  pdl_wait();
  pdl_launch_dependents();
  const bool build = a.K && (a.force || *a.drift);
  if (build) {  // beta becomes this pass's line
    const int j = blockIdx.x * (kRowWarps * 32) + threadIdx.x;
    for (int64_t q = j; q < a.nin; q += (int64_t)gridDim.x * (kRowWarps * 32)) a.beta[q] = a.Ls[q];
  }
  double S = 0.0, M = 0.0;
  bool done = i >= a.nrows;
  if (!done && a.K && !build) {
    const double* row = a.K + i * a.ld;  // ld is even
    double s0 = 0.0, s1 = 0.0;
#pragma unroll 4
    for (int j = 2 * lane; j + 1 < a.nin; j += 64) {
      const double2 kv = *reinterpret_cast<const double2*>(row + j);
      const double2 wv = *reinterpret_cast<const double2*>(a.w + j);
      s0 = fma(kv.x, wv.x, s0);
      s1 = fma(kv.y, wv.y, s1);
    }
    if ((a.nin & 1) && lane == 0) s0 = fma(row[a.nin - 1], a.w[a.nin - 1], s0);
    s0 += s1;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s0 += __shfl_xor_sync(0xffffffffu, s0, o);
    S = s0;
    M = a.M[i];
    done = S >= kLeastSum && S <= kMostSum && M != -kInf;  // (a NaN is recomputed and stays one)
  }
  if (__syncthreads_or(!done)) {  // block-uniform
    exp_table_load(tab);
    __syncthreads();
    if (!done) {
      if (build) row64<D, true>(a, i, tab, S, M);
      else row64<D, false>(a, i, tab, S, M);
      if (build && lane == 0) a.M[i] = M;
    }
  }
  if (lane == 0 && i < a.nrows) {
    sS[warp] = S;
    sM[warp] = M;
  }
  __syncthreads();
  double num = 0.0, den = 0.0;
  if (warp == 0 && lane < kRowWarps) {
    const int r = blockIdx.x * kRowWarps + lane;
    if (r < a.nrows) {
      const double M = sM[lane];
      apply_epilogue(epi, 0, r, (M == -kInf) ? -kInf : M + log(sS[lane]), num, den);
    }
  }
  if (epi.err) block_add2<kRowWarps * 32>(num, den, epi.err);
}

// Column pass over the stored kernel: CTA = 256 columns x kColRows rows, all in the
// launch grid's first dimension (the others end at 65535: 4.2 million rows).  The
// rows' weights e^{L_i + M_i - s} are formed here, s their largest log in this
// chunk of rows (16 KB of exponentials per chunk, repeated per column tile).
constexpr int kColRows = 64, kColTile = 256;

__global__ void __launch_bounds__(kColTile / 2) points64_cols(const double* __restrict__ K, int64_t ld, int nrows,
                                                              int ncols, const double* __restrict__ W,
                                                              const double* __restrict__ logw, double inv_eps,
                                                              const double* __restrict__ M, double* __restrict__ part,
                                                              double* __restrict__ shift) {
  __shared__ double v[kColRows];
  __shared__ double sh;
  const int ntiles = (ncols + kColTile - 1) / kColTile;
  const int chunk = blockIdx.x / ntiles, tile = blockIdx.x - chunk * ntiles;
  const int r0 = chunk * kColRows, nr = min(kColRows, nrows - r0);
  pdl_wait();
  pdl_launch_dependents();
  if (threadIdx.x < 32) {
    double l[2], mx = -kInf;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int r = threadIdx.x + 32 * u;
      l[u] = -kInf;
      if (r < nr) {
        const double w = W[r0 + r], m = M[r0 + r];
        if (w != -kInf && m != -kInf) l[u] = fma(w, inv_eps, logw[r0 + r]) + m;
      }
      mx = (l[u] > mx || l[u] != l[u]) ? l[u] : mx;  // keeps NaN
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double q = __shfl_xor_sync(0xffffffffu, mx, o);
      mx = (q > mx || q != q) ? q : mx;
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) v[threadIdx.x + 32 * u] = (l[u] == -kInf) ? 0.0 : exp(l[u] - mx);
    if (threadIdx.x == 0) {
      sh = mx;
      if (tile == 0) shift[chunk] = mx;
    }
  }
  __syncthreads();
  const int c = tile * kColTile + 2 * threadIdx.x;
  if (c >= ncols) return;
  double s0 = 0.0, s1 = 0.0;
  if (sh != -kInf) {
    const double* k = K + r0 * ld + c;  // ld is even and covers c + 1
#pragma unroll 8
    for (int r = 0; r < nr; ++r) {
      const double2 kv = *reinterpret_cast<const double2*>(k + r * ld);
      s0 = fma(kv.x, v[r], s0);
      s1 = fma(kv.y, v[r], s1);
    }
  }
  double* p = part + (int64_t)chunk * ld + c;
  *reinterpret_cast<double2*>(p) = make_double2(s0, s1);
}

// Sums the chunks of 32 columns, a share of them by each of 8 warps, then the
// epilogues in the lanes of one warp.  A column that the stored kernel cannot
// give is redone on the fly (a = the column as a row: x its point, y the rows'
// points, Ls their line).
template <int D>
__global__ void __launch_bounds__(256) points64_cols_end(Rows64 a, const double* __restrict__ part,
                                                         const double* __restrict__ shift, int nchunks,
                                                         const double* __restrict__ beta, int* __restrict__ drift,
                                                         Epilogue epi) {
  constexpr int kMaxF = 256;
  __shared__ double tab[kExpUnits];
  __shared__ double f[kMaxF], red[8][32], zc[32], smx[8];
  __shared__ unsigned bad_mask;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int c = blockIdx.x * 32 + lane;
  pdl_wait();
  pdl_launch_dependents();
  if (blockIdx.x == 0 && threadIdx.x == 0) *drift = 0;  // read by the row pass before this one
  double smax = -kInf;
  for (int k = threadIdx.x; k < nchunks; k += 256) {
    const double q = shift[k];
    smax = (q > smax || q != q) ? q : smax;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double q = __shfl_xor_sync(0xffffffffu, smax, o);
    smax = (q > smax || q != q) ? q : smax;
  }
  if (lane == 0) smx[warp] = smax;
  __syncthreads();
  for (int w = 0; w < 8; ++w) smax = (smx[w] > smax || smx[w] != smx[w]) ? smx[w] : smax;
  double s = 0.0;
  for (int k0 = 0; k0 < nchunks; k0 += kMaxF) {
    const int nk = min(kMaxF, nchunks - k0);
    if (k0) __syncthreads();
    if (threadIdx.x < nk) {
      const double d = shift[k0 + threadIdx.x] - smax;  // NaN only if a shift is (or all are -inf)
      f[threadIdx.x] = (smax == -kInf) ? 0.0 : exp(d);
    }
    __syncthreads();
    if (c < a.nrows) {
#pragma unroll 4
      for (int k = warp; k < nk; k += 8) s = fma(part[(int64_t)(k0 + k) * a.ld + c], f[k], s);
    }
  }
  red[warp][lane] = s;
  __syncthreads();
  if (warp == 0) {
    s = 0.0;
#pragma unroll
    for (int w = 0; w < 8; ++w) s += red[w][lane];
    const double b = (c < a.nrows) ? beta[c] : 0.0;
    const bool bad = c < a.nrows && (!(s >= kLeastSum && s <= kMostSum) || b == -kInf);
    zc[lane] = smax - b + log(s);
    const unsigned m = __ballot_sync(0xffffffffu, bad);
    if (lane == 0) bad_mask = m;
  }
  __syncthreads();
  if (bad_mask) {  // block-uniform
    exp_table_load(tab);
    __syncthreads();
    for (int q = warp; q < 32; q += 8) {
      if (!((bad_mask >> q) & 1u)) continue;
      double S, M;
      row64<D, false>(a, blockIdx.x * 32 + q, tab, S, M);
      if (lane == 0) zc[q] = (M == -kInf) ? -kInf : M + log(S);
    }
    __syncthreads();
  }
  double num = 0.0, den = 0.0;
  if (warp == 0 && c < a.nrows) apply_epilogue(epi, 0, c, zc[lane], num, den);
  if (epi.err) block_add2<256>(num, den, epi.err);
}

}  // namespace

int64_t points64_ld(int m) { return ((int64_t)m + 1) & ~(int64_t)1; }
size_t points64_part_elems(int n, int m) {
  return (size_t)((n + kColRows - 1) / kColRows) * (points64_ld(m) + 1);
}

cudaError_t launch_points64(const Points64& p, int dir, const double* W, const double* logw, double eps,
                            bool first, const Epilogue& epi, cudaStream_t s) {
  Rows64 a;
  memset(&a, 0, sizeof(a));
  a.x = dir == 0 ? p.x : p.y;
  a.y = dir == 0 ? p.y : p.x;
  a.x32 = dir == 0 ? p.x32 : p.y32;
  a.y32 = dir == 0 ? p.y32 : p.x32;
  a.d = p.d;
  a.nrows = dir == 0 ? p.n : p.m;
  a.nin = dir == 0 ? p.m : p.n;
  a.Ls = p.Ls;
  a.L32 = p.L32;
  a.inv_eps = 1.0 / eps;
  const bool rows = p.K && dir == 0;             // row pass over (or storing) the kernel
  const bool cols = p.K && dir == 1 && !first;   // column pass over it
  const dim3 line_grid((a.nin + 127) / 128);
  const bool have = rows && !first;
  count_launches(1);
  cudaError_t e = launch_pdl(points64_line, line_grid, dim3(128), 0, s, W, logw, a.nin, a.inv_eps, p.Ls, p.L32,
                             (const double*)p.beta, have ? p.w : (double*)nullptr, p.drift);
  if (e != cudaSuccess) return e;
  prof_mark_begin(PROF_ROWS, s);
  if (cols) {
    const int nchunks = (p.n + kColRows - 1) / kColRows;
    const int64_t ld = points64_ld(p.m);
    double* shift = p.part + (int64_t)nchunks * ld;
    a.ld = ld;
    count_launches(2);
    // (a stored kernel has at most 2^29 entries: the product fits)
    e = launch_pdl(points64_cols, dim3((p.m + kColTile - 1) / kColTile * nchunks), dim3(kColTile / 2), 0, s,
                   (const double*)p.K, ld, p.n, p.m, W, logw, a.inv_eps, (const double*)p.M, p.part, shift);
    if (e != cudaSuccess) return e;
    auto end = [&](auto kern) {
      return launch_pdl(kern, dim3((p.m + 31) / 32), dim3(256), 0, s, a, (const double*)p.part, (const double*)shift,
                        nchunks, (const double*)p.beta, p.drift, epi);
    };
    e = p.d == 1 ? end(points64_cols_end<1>) : p.d == 2 ? end(points64_cols_end<2>)
        : p.d == 3 ? end(points64_cols_end<3>) : end(points64_cols_end<0>);
  } else {
    if (rows) {
      a.K = p.K;
      a.ld = points64_ld(p.m);
      a.M = p.M;
      a.beta = p.beta;
      a.w = p.w;
      a.drift = p.drift;
      a.force = first ? 1 : 0;
    }
    count_launches(1);
    const dim3 grid((a.nrows + kRowWarps - 1) / kRowWarps), block(kRowWarps * 32);
    e = p.d == 1 ? launch_pdl(points64_rows<1>, grid, block, 0, s, a, epi)
        : p.d == 2 ? launch_pdl(points64_rows<2>, grid, block, 0, s, a, epi)
        : p.d == 3 ? launch_pdl(points64_rows<3>, grid, block, 0, s, a, epi)
                   : launch_pdl(points64_rows<0>, grid, block, 0, s, a, epi);
  }
  if (e != cudaSuccess) return e;
  prof_mark_end(PROF_ROWS, s);
  return cudaGetLastError();
}

}  // namespace uot
