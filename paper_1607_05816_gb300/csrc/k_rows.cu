// Row-wise Gibbs operators for explicit cost matrices and point clouds.
//
// Log domain (Sec. 4.3, absorption after every update):
//   z_i = log sum_j exp(L_j - C_ij/eps),   L_j = W_j/eps + log w_j,
// with C_ij read from a dense row-major matrix or recomputed as |x_i - y_j|^2
// (point clouds; the cost is never stored).  One warp per row: a max sweep and
// a sum sweep over j, lanes strided over j, then warp reductions.  L is first
// shifted by its FP64 maximum (prepare_L) so the FP32 variant only ever sees
// values <= 0.
//
// Algorithm 1 (Sec. 4.2): a_i = proxdiv_F(sum_j K_ij b_j w_j, eps) on a stored
// FP64 kernel K = exp(-C/eps), with the proxdiv column of Table 1 (u = 0).
#include <string.h>

#include <cooperative_groups.h>

#include <algorithm>

#include "exp_table.cuh"
#include "uot_internal.cuh"

namespace uot {
namespace {


template <typename T>
__device__ __forceinline__ T wmax(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
template <typename T>
__device__ __forceinline__ T wsum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// L_j = W_j/eps + log w_j in FP64; then Lt_j = (L_j - max L) in T, scaled by
// log2(e) for the FP32 variant.  Single block; *Lmax receives max L.
template <typename T, int NT>
__global__ void __launch_bounds__(NT) prepare_L(const double* __restrict__ W,
                                                const double* __restrict__ logw, int nin,
                                                double eps, T* __restrict__ Lt,
                                                double* __restrict__ Lmax) {
  __shared__ double red[NT / 32];
  const double inv_eps = 1.0 / eps;
  double mx = -kInf;
  // L_j is stored unshifted first, then shifted in place (one FP64 evaluation each)
  for (int j = threadIdx.x; j < nin; j += NT) {
    const double w = W[j];
    const double L = (w == -kInf) ? -kInf : fma(w, inv_eps, logw[j]);
    mx = fmax(mx, L);
    if (sizeof(T) == 8) reinterpret_cast<double*>(Lt)[j] = L;
  }
  mx = wmax(mx);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x < 32) {
    double v = (threadIdx.x < NT / 32) ? red[threadIdx.x] : -kInf;
    v = wmax(v);
    if (threadIdx.x == 0) red[0] = v;
  }
  __syncthreads();
  mx = red[0];
  for (int j = threadIdx.x; j < nin; j += NT) {
    double L;
    if (sizeof(T) == 8) {
      L = reinterpret_cast<const double*>(Lt)[j];
    } else {
      const double w = W[j];
      L = (w == -kInf) ? -kInf : fma(w, inv_eps, logw[j]);
    }
    double v = (mx == -kInf) ? -kInf : L - mx;
    if (sizeof(T) == 4) v *= (double)kLog2e;
    Lt[j] = (T)v;
  }
  if (threadIdx.x == 0) *Lmax = mx;
}

template <typename T, int DMAX>
struct RowCtx {
  T xi[DMAX];
};

// Cost of entry (i, j) in "cost/eps" units scaled as the variant requires.
template <typename T, int DMAX>
__device__ __forceinline__ T cost_ij(int kind, const T* __restrict__ C, const T* __restrict__ y,
                                     int d, int64_t rowbase, int j, const RowCtx<T, DMAX>& c) {
  if (kind == UOT_GEOM_DENSE) return C[rowbase + j];
  T acc = 0;
#pragma unroll
  for (int k = 0; k < DMAX; ++k) {
    if (k < d) {
      const T t = c.xi[k] - y[(int64_t)j * d + k];
      acc = fma(t, t, acc);
    }
  }
  return acc;
}

template <typename T, int DMAX, int WARPS>
__global__ void __launch_bounds__(WARPS * 32)
    rows_lse(int kind, const T* __restrict__ C, const T* __restrict__ x, const T* __restrict__ y,
             int d, int nrows, int nin, const T* __restrict__ Lt,
             const double* __restrict__ Lmax_p, double eps, Epilogue epi) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x * WARPS + warp;
  double num = 0.0, den = 0.0;
  const double Lmax = *Lmax_p;
  if (i < nrows) {
    if (Lmax == -kInf) {
      if (lane == 0) apply_epilogue(epi, 0, i, -kInf, num, den);
    } else {
      RowCtx<T, DMAX> c;
      if (kind == UOT_GEOM_POINTS) {
#pragma unroll
        for (int k = 0; k < DMAX; ++k) c.xi[k] = (k < d) ? x[(int64_t)i * d + k] : T(0);
      }
      const int64_t rowbase = (int64_t)i * nin;
      // FP32 works in log2 units, FP64 in natural units.
      const T k2 = (sizeof(T) == 4) ? T((double)kLog2e / eps) : T(1.0 / eps);
      T m = -INFINITY;
      for (int j = lane; j < nin; j += 32)
        m = fmax(m, fma(-k2, cost_ij<T, DMAX>(kind, C, y, d, rowbase, j, c), Lt[j]));
      m = wmax(m);
      T s = 0;
      // m = -inf: every term vanishes (C = +inf where the input is finite)
      if (m != -INFINITY)
        for (int j = lane; j < nin; j += 32) {
          const T a = fma(-k2, cost_ij<T, DMAX>(kind, C, y, d, rowbase, j, c), Lt[j] - m);
          if (sizeof(T) == 4)
            s += ex2_approx((float)a);
          else if (a > -746.0)  // below, e^a is 0 in FP64: skip the FP64 exponential
            s += exp((double)a);
        }
      s = wsum(s);
      if (lane == 0 && m == -INFINITY) {
        apply_epilogue(epi, 0, i, -kInf, num, den);
      } else if (lane == 0) {
        const double z = Lmax + ((sizeof(T) == 4) ? (double)kLn2 * (double)m : (double)m) +
                         log((double)s);
        apply_epilogue(epi, 0, i, z, num, den);
      }
    }
  }
  if (epi.err) block_add2<WARPS * 32>(num, den, epi.err);
}

// ---------------------------------------------------------------------------
// FP64 rows of a dense cost by chunks of 32 columns.  GB300's FP64 pipe issues
// 2 operations per clock per SM against 128 for FP32, and at small eps few
// terms of a row matter.  Terms below e^-(50 + log nin) of the row's largest add
// less than e^-50 = 2^-72 of the sum together and are left out, by conservative
// FP32 tests: first per chunk, from the chunk's least cost (chunkmin32, built
// once with the FP32 copy of C) and the largest input (prepare_L_chunks), then
// per column on the FP32 copies.  What is left is evaluated in FP64, 32 terms at
// a time with every lane active.
//
// A pass reads the row's least costs (1/32 of the FP32 cost) and the chunks that
// matter, where the kernel before it read the whole FP32 cost (36 MB at
// 3000 x 3000) into shared memory and kept every term above e^-746.  WF flow of
// 3000 samples, eps = 1e-8: 28 -> 16 us a half-step (two kernels and the growth
// step's share).  20 iterations, 3000 random points in 2-D: eps = 1e-1 16.5 -> 13.2
// ms (FP64 terms: all of them count), 1e-2 16.4 -> 12.0, 1e-3 16.2 -> 4.3, 1e-4
// 5.5 -> 2.3.
// ---------------------------------------------------------------------------

// L_j = W_j/eps + log w_j in FP64 (L64) and as a float-float pair (Lff); the
// largest L of each chunk of 32 columns as a pair (Lch), +inf where one is NaN: the
// maximum of a line then says so without a test of its own.
__global__ void __launch_bounds__(256) prepare_L_chunks(const double* __restrict__ W, const double* __restrict__ logw,
                                                        int nin, double inv_eps, double* __restrict__ L64,
                                                        float2* __restrict__ Lff, float2* __restrict__ Lch) {
  pdl_wait();  // W is the preceding kernel's output
  pdl_launch_dependents();
  const int j = blockIdx.x * 256 + threadIdx.x;
  auto pair = [](double L) {
    const float hi = (float)L;
    return make_float2(hi, (L == -kInf) ? 0.0f : (float)(L - (double)hi));
  };
  double L = -kInf;
  if (j < nin) {
    const double w = W[j];
    L = (w == -kInf) ? -kInf : fma(w, inv_eps, logw[j]);
    L64[j] = L;
    Lff[j] = pair(L);
  }
  const double mx = wmax(L);
  const bool nan = __any_sync(0xffffffffu, L != L);
  if ((threadIdx.x & 31) == 0 && j < nin) Lch[j >> 5] = nan ? make_float2(INFINITY, 0.0f) : pair(mx);
}

// C32 = C rounded to FP32 and the least C32 of each chunk (-inf where one is NaN);
// one warp per (row, chunk).
__global__ void __launch_bounds__(256) chunkmin32(const double* __restrict__ C, int64_t nrows, int nin, int nchunk,
                                                  float* __restrict__ C32, float* __restrict__ Cmin) {
  const int lane = threadIdx.x & 31;
  for (int64_t t = blockIdx.x * (int64_t)8 + (threadIdx.x >> 5); t < nrows * nchunk; t += (int64_t)gridDim.x * 8) {
    const int64_t i = t / nchunk;
    const int j = (int)(t - i * nchunk) * 32 + lane;
    float c = INFINITY;
    if (j < nin) {
      c = (float)C[i * nin + j];
      C32[i * nin + j] = c;
      if (c != c) c = -INFINITY;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c = fminf(c, __shfl_xor_sync(0xffffffffu, c, o));
    if (lane == 0) Cmin[t] = c;
  }
}

// WPR warps per row, NW / WPR rows per CTA (rows b, b + G, ... of G CTAs: neighbouring
// rows with hundreds of terms each, 12 us of one SM's FP64 pipe for ten of them,
// go to different SMs); chunk c belongs to warp c mod WPR of its row.  The row's
// shift m is the largest exponent
// of the chunk with the largest bound, then of any chunk whose bound lies more
// than 30 above it, so every exponent stays below 30 plus the FP32 error.  Where that
// error is in the hundreds (exponents of 1e9 and more) terms can leave the FP64
// range; the warp of such a row redoes it with its FP64 maximum.
// Surviving columns are collected per warp (ballot, shared-memory list of
// kRowList, drained 32 at a time when full); the lists are then evaluated by the
// whole CTA, so a row with hundreds of terms among rows of five (the edge of a
// density at small eps) does not wait for one warp's loads, and every sum is taken
// in a fixed order.
// Rows of at most kShort (8 or 10) chunks a warp need no bounds: all their
// exponents fit in registers, with the costs loaded before the preceding kernel has
// ended (WF flow of 400 samples, two species, eps = 1e-8: 4.0 -> 3.5 ms).
//
// At small eps a pass is a chain of latencies and of FP64 instructions of one
// warp, the CTA's epilogue (some 150 of 16 clocks each), so many rows share a CTA
// where there are many.
constexpr int kRowList = 352;
constexpr int kShortChunks = 8, kShortWide = 10;  // kShort: chunks per warp in registers (0: by bounds)
constexpr float kRowFarTol = 200.0f;  // an error that keeps every term between e^-200 and e^430
constexpr unsigned kRowLeastHi = 123u << 20, kRowMostHi = 0x7ff00000u;  // high words of 2^-900 and infinity

// Chunks' maxima kept in shared memory (48 KB, 393,216 columns); those of later chunks
// are read from L2 where they are used.
constexpr int kStagedChunks = 12288;

// pval [nw][kRowList + 32], slist likewise, and the chunks' maxima
size_t rows_chunks_smem(int nw, int nchunk) {
  return (size_t)nw * (kRowList + 32) * (sizeof(double) + sizeof(int)) +
         (size_t)std::min(nchunk, kStagedChunks) * sizeof(float);
}

template <int NW, int WPR, int kShort>
__global__ void __launch_bounds__(NW * 32)
    rows_lse_f64_chunks(const double* __restrict__ C, const float* __restrict__ C32, const float* __restrict__ Cmin,
                        int nrows, int nin, int nchunk, const double* __restrict__ L64,
                        const float2* __restrict__ Lff, const float2* __restrict__ Lch, double k2, float cut,
                        Epilogue epi) {
  constexpr int NT = NW * 32, RPC = NW / WPR;
  static_assert(NW <= 32 && NT >= kExpUnits, "a table entry a thread, a warp's lanes cover the rows");
  static_assert(32 * kShort <= kRowList, "a short row's columns fit its warp's list without draining it");
  extern __shared__ double pval[];  // the terms of the lists, row by row
  int* slist = reinterpret_cast<int*>(pval + NW * (kRowList + 32));  // [NW][kRowList + 32] columns
  float* sLc = reinterpret_cast<float*>(slist + NW * (kRowList + 32));  // largest inputs, relative to the line's
  __shared__ float sm_m[NW];        // the rows' shifts
  __shared__ double sm_s[NW];
  __shared__ double sm_lmax;
  __shared__ int woff[33];          // exclusive prefix sum of the list lengths
  __shared__ double tab[kExpUnits];
  __shared__ float sm_best[NW];     // WPR > 1: the warps' parts of what a row needs
  __shared__ int sm_at[NW];
  __shared__ float sm_neg[NW], sm_mx[NW];
  __shared__ unsigned sm_hi[NW];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rloc = warp / WPR, part = warp % WPR;
  const int i = blockIdx.x + rloc * gridDim.x;
  const float* cmin = Cmin + (int64_t)(i < nrows ? i : 0) * nchunk;
  // before the preceding kernel has ended: the table and the least costs of the first 128 chunks
  exp_table_load(tab);
  constexpr int kOwn = kShort ? kShort : 1;
  float q4[4], cs[kOwn];
#pragma unroll
  for (int u = 0; u < (kShort ? 0 : 4); ++u) {
    const int c = part + WPR * (lane + 32 * u);
    q4[u] = c < nchunk ? cmin[c] : INFINITY;
  }
#pragma unroll
  for (int u = 0; u < (kShort ? kOwn : 0); ++u) {
    const int j = 32 * (part + WPR * u) + lane;
    cs[u] = (i < nrows && j < nin) ? C32[(int64_t)i * nin + j] : INFINITY;
  }
  pdl_wait();
  pdl_launch_dependents();
  float2 ls[kOwn];
#pragma unroll
  for (int u = 0; u < (kShort ? kOwn : 0); ++u) {
    const int j = 32 * (part + WPR * u) + lane;
    ls[u] = j < nin ? Lff[j] : make_float2(-INFINITY, 0.0f);
  }
  // mhi: the FP32 rounding of max L (the shift of the whole line)
  const float2 l0 = (threadIdx.x < nchunk) ? Lch[threadIdx.x] : make_float2(-INFINITY, 0.0f);
  float mhi = l0.x;
  for (int c = threadIdx.x + NT; c < nchunk; c += NT) mhi = fmaxf(mhi, Lch[c].x);
  mhi = wmax(mhi);
  if (lane == 0) sm_m[warp] = mhi;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < NW; ++w) mhi = fmaxf(mhi, sm_m[w]);
  auto shifted = [&](float2 l) { return (mhi == -INFINITY || l.x == -INFINITY) ? -INFINITY : (l.x - mhi) + l.y; };
  if (threadIdx.x == 0) sm_lmax = (mhi == -INFINITY) ? -kInf : (double)mhi;  // (a conversion takes the FP64 pipe)
  if (!kShort) {
    if (threadIdx.x < nchunk) sLc[threadIdx.x] = shifted(l0);
    for (int c = threadIdx.x + NT; c < min(nchunk, kStagedChunks); c += NT) sLc[c] = shifted(Lch[c]);
  }
  __syncthreads();
  // the pairs carry |L| 2^-47 of representation error besides the FP32 rounding
  const float lerr = (mhi == -INFINITY) ? 4.0f : fmaf(fabsf(mhi), 0x1p-44f, 4.0f);
  const float k2f = (float)k2;
  // (mhi = +inf, a NaN on the line: no chunk has a finite bound below, and the epilogue says NaN)
  const bool live = i < nrows && mhi != -INFINITY;  // warp-uniform
  const float* crow = C32 + (int64_t)(live ? i : 0) * nin;
  // The warp's chunks are part, part + WPR, ...: bound of its e-th one (e = lane mod 32) and
  // its FP32 error (the roundings of k2, c, l and the fma).
  auto bound = [&](int e, float& tol, float& q) {
    const int c = part + WPR * e;
    if (c >= nchunk) return -INFINITY;
    const float l = c < kStagedChunks ? sLc[c] : shifted(Lch[c]);
    q = e < 64 ? (e < 32 ? q4[0] : q4[1]) : e < 128 ? (e < 96 ? q4[2] : q4[3]) : cmin[c];
    const float b = fmaf(-k2f, q, l);
    tol = fmaf(fabsf(b) + fmaf(k2f, fabsf(q), fabsf(l)), 0x1p-22f, lerr);
    return b;
  };
  // exponents of column j[u] (-inf where j[u] is none); every load is issued before the first
  // is used (conditional loads wait for one another: 2.6 us for eight)
  auto exponents = [&](auto& j, auto& t, auto& mag) {
    constexpr int G = sizeof(j) / sizeof(int);
    float cv[G];
    float2 lv[G];
#pragma unroll
    for (int u = 0; u < G; ++u) {
      const int q = (unsigned)j[u] < (unsigned)nin ? j[u] : 0;
      cv[u] = crow[q];
      lv[u] = Lff[q];
    }
#pragma unroll
    for (int u = 0; u < G; ++u) {
      const float l = shifted(lv[u]);
      t[u] = (unsigned)j[u] < (unsigned)nin ? fmaf(-k2f, cv[u], l) : -INFINITY;
      mag[u] = fmaf(k2f, fabsf(cv[u]), fabsf(l));
    }
  };
  double s = 0.0;
  bool drained = false, far = false;
  int cnt = 0;  // warp-uniform
  int* lst = slist + warp * (kRowList + 32);
  float m = -INFINITY, best = -INFINITY;
  float mneg = 0.0f;  // costs below zero: the parts of the shift's exponent may cancel
  int jj[8];
  float tt[8], mg[8];
  auto largest = [&]() {
    exponents(jj, tt, mg);
    float g = tt[0];
#pragma unroll
    for (int u = 1; u < 8; ++u) g = fmaxf(g, tt[u]);
    return wmax(g);
  };
  int at = 0;
  float ts[kOwn];
  if (kShort) {  // every exponent of the row in registers
    float qmin = 0.0f;
    bool nan = false;
#pragma unroll
    for (int u = 0; u < kOwn; ++u) {
      const bool in = 32 * (part + WPR * u) + lane < nin;
      ts[u] = in ? fmaf(-k2f, cs[u], shifted(ls[u])) : -INFINITY;
      nan = nan || ts[u] != ts[u];
      m = fmaxf(m, ts[u]);
      qmin = fminf(qmin, cs[u]);
    }
    m = wmax(m);
    if (__any_sync(0xffffffffu, nan)) m = fmaxf(m, 0.0f);  // (the row is NaN, with any shift)
    if (__any_sync(0xffffffffu, qmin < 0.0f)) mneg = 2.0f * k2f * wmax(-qmin) * 0x1p-22f;
    if (WPR > 1 && lane == 0) sm_neg[warp] = mneg;
  } else if (live) {
    float qmin = 0.0f;
    for (int e = lane; part + WPR * e < nchunk; e += 32) {
      float tol, q;
      const float b = bound(e, tol, q);
      qmin = fminf(qmin, q);
      if (b > best) {
        best = b;
        at = part + WPR * e;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float b = __shfl_xor_sync(0xffffffffu, best, o);
      const int c = __shfl_xor_sync(0xffffffffu, at, o);
      if (b > best || (b == best && c < at)) {
        best = b;
        at = c;
      }
    }
    if (__any_sync(0xffffffffu, qmin < 0.0f)) mneg = 2.0f * k2f * wmax(-qmin) * 0x1p-22f;
  }
  if (WPR > 1 && !kShort) {
    if (lane == 0) {
      sm_best[warp] = best;
      sm_at[warp] = at;
      sm_neg[warp] = mneg;
    }
    __syncthreads();
#pragma unroll
    for (int w = 0; w < WPR; ++w) {
      const float b = sm_best[rloc * WPR + w];
      const int c = sm_at[rloc * WPR + w];
      if (b > best || (b == best && c < at)) {
        best = b;
        at = c;
      }
      mneg = fmaxf(mneg, sm_neg[rloc * WPR + w]);
    }
  }
  if (!kShort && live) {
    if (best != -INFINITY) {
      // that chunk and its neighbours: on a steep line over sorted points all bounds near the
      // largest are loose, and the row's maximum lies a few chunks away
#pragma unroll
      for (int u = 0; u < 8; ++u) jj[u] = 32 * (at + u - 4) + lane;
      m = largest();
      for (int c0 = 0; part + WPR * c0 < nchunk; c0 += 32) {
        float tol = 0.0f, q;
        const float b = bound(c0 + lane, tol, q);
        unsigned mask = __ballot_sync(0xffffffffu, b - tol > m + 30.0f);
        while (mask) {  // eight chunks at a time for loads in flight
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            jj[u] = mask ? 32 * (part + WPR * (c0 + __ffs(mask) - 1)) + lane : nin;
            mask &= mask - 1;  // 0 stays 0
          }
          m = fmaxf(m, largest());
        }
      }
    }
  }
  if (WPR > 1) {
    if (lane == 0) sm_mx[warp] = m;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < WPR; ++w) {
      m = fmaxf(m, sm_mx[rloc * WPR + w]);
      if (kShort) mneg = fmaxf(mneg, sm_neg[rloc * WPR + w]);
    }
  }
  if (m == -INFINITY && best == INFINITY) m = 0.0f;  // NaN costs and nothing else
  // FP64 term of column j of the row of warp r, relative to that row's shift mr
  auto term = [&](int r, int j, float mr) {
    const int64_t ri = (int64_t)(blockIdx.x + r / WPR * gridDim.x);
    return exp_tab(fma(-k2, C[ri * nin + j], L64[j] - sm_lmax) - (double)mr, tab);
  };
  far = !(mneg <= kRowFarTol);
  const float lowest = -cut - mneg;
  // |t - t_FP64| and the error of m are below (k2 |c| + |l| + |t| + |d|) 2^-22 plus lerr
  // (and mneg): |m| <= |t| + |d|, and the two parts of an exponent have one sign
  auto list = [&](bool in, float t, float mag, int j) {
    const float d = t - m;
    const float tol = fmaf(fabsf(t) + fabsf(d) + mag, 0x1p-22f, lerr);
    const bool keep = in && !(d <= lowest - tol);
    const unsigned km = __ballot_sync(0xffffffffu, keep);
    if (!km) return;  // warp-uniform, and the usual case at small eps
    far = far || (keep && !(tol <= kRowFarTol));
    if (keep) lst[cnt + __popc(km & ((1u << lane) - 1u))] = j;
    cnt += __popc(km);
  };
  if (kShort && m != -INFINITY) {
#pragma unroll
    for (int u = 0; u < kOwn; ++u) {
      const int j = 32 * (part + WPR * u) + lane;
      list(j < nin, ts[u], fmaf(k2f, fabsf(cs[u]), fabsf(shifted(ls[u]))), j);
    }
  }
  if (!kShort && live && m != -INFINITY) {
    // warp-uniform sweep over the surviving chunks
    constexpr int G = 4;
    for (int c0 = 0; part + WPR * c0 < nchunk; c0 += 32) {
      float ctol = 0.0f, q;
      const float b = bound(c0 + lane, ctol, q);
      const float a = b - m;
      unsigned mask = __ballot_sync(0xffffffffu, !(a <= lowest - fmaf(fabsf(a), 0x1p-22f, ctol)));  // (NaN counts)
      while (mask) {
        int cj[G];
        float t[G], mag[G];
#pragma unroll
        for (int u = 0; u < G; ++u) {
          cj[u] = mask ? 32 * (part + WPR * (c0 + __ffs(mask) - 1)) + lane : nin;
          mask &= mask - 1;  // 0 stays 0
        }
        exponents(cj, t, mag);
#pragma unroll
        for (int u = 0; u < G; ++u) {
          list(cj[u] < nin, t[u], mag[u], cj[u]);
          if (cnt > kRowList) {  // a full batch from the list's end: every lane evaluates one term
            __syncwarp();
            cnt -= 32;
            s += term(warp, lst[cnt + lane], m);
            drained = true;
            __syncwarp();
          }
        }
      }
    }
  }
  if (drained) s = wsum(s);
  if (lane == 0) {
    sm_m[warp] = m;  // (the maxima there were read before the last barrier)
    sm_s[warp] = s;
    woff[warp] = cnt;
  }
  __syncthreads();
  if (warp == 0) {
    const int c = lane < NW ? woff[lane] : 0;
    int o = c;
#pragma unroll
    for (int k = 1; k < 32; k <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, o, k);
      if (lane >= k) o += v;
    }
    woff[lane + 1] = o;  // (lanes from NW on repeat the total)
    if (lane == 0) woff[0] = 0;
  }
  __syncthreads();
  const int np = woff[NW];
  for (int k = threadIdx.x; k < np; k += NT) {
    int r = 0;  // the last row that starts at or before k
#pragma unroll
    for (int h = 16; h > 0; h >>= 1)
      if (r + h < NW && woff[r + h] <= k) r += h;
    pval[k] = term(r, slist[r * (kRowList + 32) + k - woff[r]], sm_m[r]);
  }
  __syncthreads();
  // Lists of more than kLaneTerms terms are summed by their warps; where a row has one warp, the
  // others by the epilogue's lanes (a warp's sum takes five FP64 instructions whatever its length).
  constexpr int kLaneTerms = WPR > 1 ? 0 : 8;
  if (cnt > kLaneTerms) {
    double t = 0.0;
    for (int k = woff[warp] + lane; k < woff[warp + 1]; k += 32) t += pval[k];
    t = wsum(t);
    if (lane == 0) sm_s[warp] = s + t;
  }
  auto redo_outside_range = [&](unsigned hi) {  // hi: the high word of the row's largest term
    if (hi >= kRowLeastHi && hi < kRowMostHi) return;
    const double* c64 = C + (int64_t)i * nin;
    double mx = -kInf, t = 0.0;
    bool nan = false;
    for (int j = lane; j < nin; j += 32) {
      const double a = fma(-k2, c64[j], L64[j] - sm_lmax);
      nan = nan || a != a;
      mx = fmax(mx, a);
    }
    mx = wmax(mx);
    nan = __any_sync(0xffffffffu, nan);
    if (mx != -kInf && !nan)
      for (int j = lane; j < nin; j += 32) t += exp_tab(fma(-k2, c64[j], L64[j] - sm_lmax) - mx, tab);
    t = wsum(t);
    if (lane == 0) {
      sm_m[warp] = NAN;  // sm_s holds the row's result
      sm_s[warp] = nan ? (double)NAN : mx == -kInf ? -kInf : sm_lmax + mx + log(t);
    }
  };
  auto largest_hi = [&]() {  // of the warp's terms (not negative; integer instructions only)
    unsigned hi = drained ? (unsigned)__double2hiint(s) : 0u;
    for (int k = woff[warp] + lane; k < woff[warp + 1]; k += 32) hi = max(hi, (unsigned)__double2hiint(pval[k]));
    return __reduce_max_sync(0xffffffffu, hi);
  };
  if (WPR == 1) {
    if (__any_sync(0xffffffffu, far)) redo_outside_range(largest_hi());
    __syncthreads();
  } else if (__syncthreads_or(far)) {
    const unsigned hi = largest_hi();
    if (lane == 0) sm_hi[warp] = hi;
    __syncthreads();
    if (part == 0 && live && m != -INFINITY) {
      unsigned top = hi;
#pragma unroll
      for (int w = 1; w < WPR; ++w) top = max(top, sm_hi[rloc * WPR + w]);
      redo_outside_range(top);
    }
    __syncthreads();
  }
  // the CTA's row epilogues (FP64 log and Table 1 row) side by side in the
  // lanes of warp 0: one warp instruction stream for RPC rows instead of one
  // per row on the narrow FP64 pipe
  double num = 0.0, den = 0.0;
  if (warp == 0 && lane < RPC) {
    const int r = blockIdx.x + lane * gridDim.x;
    if (r < nrows) {
      double z = -kInf;
      const float mr = sm_m[lane * WPR];
      double t = sm_s[lane * WPR];
      if (sm_lmax == kInf) {
        z = NAN;
      } else if (mr != mr) {
        z = t;
      } else if (mr != -INFINITY) {
        if (WPR == 1) {
          if (woff[lane + 1] - woff[lane] <= kLaneTerms)
            for (int k = woff[lane]; k < woff[lane + 1]; ++k) t += pval[k];
        } else {
#pragma unroll
          for (int w = 1; w < WPR; ++w) t += sm_s[lane * WPR + w];
        }
        z = sm_lmax + (double)mr + log(t);
      }
      apply_epilogue(epi, 0, r, z, num, den);
    }
  }
  if (epi.err) block_add2<NT>(num, den, epi.err);
}

// FP32 path: L_j = W_j/eps + log w_j in float-float; Lt_j = (L_j - max) log2(e)
// in FP32; *Lmax (a float) receives the maximum of the high parts.
template <int NT>
__global__ void __launch_bounds__(NT) prepare_L_ff(const float2* __restrict__ W,
                                                   const float2* __restrict__ logw, int nin,
                                                   float2 inv_eps, float* __restrict__ Lt,
                                                   float* __restrict__ Lmax) {
  __shared__ float red[NT / 32];
  float mx = -INFINITY;
  for (int j = threadIdx.x; j < nin; j += NT) {
    const ff w = ffl(W[j]);
    const ff L = (w.hi == -INFINITY) ? ff_ninf() : ff_add(ff_mul(w, ffl(inv_eps)), ffl(logw[j]));
    mx = fmaxf(mx, L.hi);
  }
  mx = wmax(mx);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x < 32) {
    float v = (threadIdx.x < NT / 32) ? red[threadIdx.x] : -INFINITY;
    v = wmax(v);
    if (threadIdx.x == 0) red[0] = v;
  }
  __syncthreads();
  mx = red[0];
  for (int j = threadIdx.x; j < nin; j += NT) {
    const ff w = ffl(W[j]);
    const ff L = (w.hi == -INFINITY) ? ff_ninf() : ff_add(ff_mul(w, ffl(inv_eps)), ffl(logw[j]));
    Lt[j] = (mx == -INFINITY || L.hi == -INFINITY) ? -INFINITY : ((L.hi - mx) + L.lo) * kLog2e;
  }
  if (threadIdx.x == 0) *Lmax = mx;
}

template <int DMAX, int WARPS>
__global__ void __launch_bounds__(WARPS * 32)
    rows_lse_f32(int kind, const float* __restrict__ C, const float* __restrict__ x,
                 const float* __restrict__ y, int d, int nrows, int nin,
                 const float* __restrict__ Lt, const float* __restrict__ Lmax_p, float k2,
                 Epilogue epi) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x * WARPS + warp;
  float num = 0.0f, den = 0.0f;
  const float Lmax = *Lmax_p;
  if (i < nrows) {
    if (Lmax == -INFINITY) {
      if (lane == 0) apply_epilogue_ff(epi, 0, i, ff_ninf(), num, den);
    } else {
      RowCtx<float, DMAX> c;
      if (kind == UOT_GEOM_POINTS) {
#pragma unroll
        for (int k = 0; k < DMAX; ++k) c.xi[k] = (k < d) ? x[(int64_t)i * d + k] : 0.0f;
      }
      const int64_t rowbase = (int64_t)i * nin;
      float m = -INFINITY;
      for (int j = lane; j < nin; j += 32)
        m = fmaxf(m, fmaf(-k2, cost_ij<float, DMAX>(kind, C, y, d, rowbase, j, c), Lt[j]));
      m = wmax(m);
      float s = 0.0f;
      // m = -inf: every term vanishes (C = +inf where the input is finite)
      if (m != -INFINITY)
        for (int j = lane; j < nin; j += 32)
          s += ex2_approx(fmaf(-k2, cost_ij<float, DMAX>(kind, C, y, d, rowbase, j, c), Lt[j] - m));
      s = wsum(s);
      if (lane == 0 && m == -INFINITY) {
        apply_epilogue_ff(epi, 0, i, ff_ninf(), num, den);
      } else if (lane == 0) {
        const ff ln2 = ln2_ff();
        float lg;
        asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(lg) : "f"(s));
        const ff z = ff_add_f(ff_add_f(ff_mul_f(ln2, m), Lmax), kLn2 * lg);
        apply_epilogue_ff(epi, 0, i, z, num, den);
      }
    }
  }
  if (epi.err) block_add2f<WARPS * 32>(num, den, epi.err);
}

// Table 1 proxdiv column with u = 0 (non-log form), 0/0 = 0.
__device__ inline double proxdiv_plain(const DivParams& F, double p, double s, double eps) {
  if (!(s > 0.0)) return 0.0;
  const double ps = p / s;
  switch (F.kind) {
    case UOT_DIV_EQ:
      return ps;
    case UOT_DIV_KL:
      return pow(ps, F.lam / (F.lam + eps));
    case UOT_DIV_TV:
      return fmin(exp(F.lam / eps), fmax(exp(-F.lam / eps), ps));
    default: {
      const double lo = exp(F.log_alpha) * ps;
      const double inner = fmax(lo, 1.0);
      return (F.log_beta == kInf) ? inner : fmin(exp(F.log_beta) * ps, inner);
    }
  }
}

template <int WARPS>
__global__ void __launch_bounds__(WARPS * 32)
    alg1_half(const double* __restrict__ K, int nrows, int nin, const double* __restrict__ b,
              const double* __restrict__ w, const double* __restrict__ p, DivParams F, double eps,
              double* __restrict__ a, const double* __restrict__ wout, double* err) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x * WARPS + warp;
  double num = 0.0, den = 0.0;
  if (i < nrows) {
    const double* row = K + (int64_t)i * nin;
    double s = 0.0;
    for (int j = lane; j < nin; j += 32) s = fma(row[j], b[j] * w[j], s);
    s = wsum(s);
    if (lane == 0) {
      const double aold = a[i];
      const double anew = proxdiv_plain(F, p[i], s, eps);
      a[i] = anew;
      if (err) {
        num = wout[i] * fabs(aold * s - anew * s);
        den = wout[i] * anew * s;
      }
    }
  }
  if (err) block_add2<WARPS * 32>(num, den, err);
}

// Algorithm 1 for one eps with the stored kernel resident in the shared memory
// of one thread-block cluster (CL CTAs, all iterations in one launch).  CTA r
// holds rows [r R, r R + R) of K and rows [r Q, r Q + Q) of K^T (R = ceil(n/CL),
// Q = ceil(m/CL)) and full copies of b (.) dy and a (.) dx.  A half-step is
// alg1_half's arithmetic (one warp per row, lane-strided FMAs, warp sum), so a
// and b are bit for bit those of the per-launch path.  After each half-step a
// cluster barrier, then every CTA copies the other CTAs' new entries out of
// their shared memory.  The violation sums of a checked iteration are reduced
// per CTA, and every CTA adds the CTAs' sums in the same order, so all of them
// take the same stop decision; there is no spin loop, only hardware barriers.
constexpr int kAlg1Warps = 16;

struct Alg1ClusterArgs {
  const double* K;
  const double* KT;
  int n, m, R, Q;
  const double *p, *dx, *q, *dy;
  DivParams F1, F2;
  double eps;
  double* a;  // [n] in/out
  double* b;  // [m] in/out
  int iters, check_every;  // check_every = 0: no checks
  double tol;
  double* res;  // [3]: violation of the last check, iterations run, converged (0/1)
};

__global__ void __launch_bounds__(kAlg1Warps * 32) alg1_cluster(Alg1ClusterArgs A) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  extern __shared__ double sh[];
  __shared__ double cpart[2];  // this CTA's violation sums, read by every CTA
  const int CL = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, NT = kAlg1Warps * 32;
  const int n = A.n, m = A.m, R = A.R, Q = A.Q;
  const int r0 = rank * R, nr = max(0, min(R, n - r0));
  const int c0 = rank * Q, nc = max(0, min(Q, m - c0));
  double* sK = sh;                      // [R][m]
  double* sKT = sK + (size_t)R * m;     // [Q][n]
  double* sbw = sKT + (size_t)Q * n;    // [m] b (.) dy
  double* saw = sbw + m;                // [n] a (.) dx
  double* sa = saw + n;                 // [R] this CTA's a
  double* sb = sa + R;                  // [Q] this CTA's b
  double* ssum = sb + Q;                // [max(R, Q)] row sums of the current half-step
  for (size_t t = threadIdx.x; t < (size_t)nr * m; t += NT) sK[t] = A.K[(size_t)r0 * m + t];
  for (size_t t = threadIdx.x; t < (size_t)nc * n; t += NT) sKT[t] = A.KT[(size_t)c0 * n + t];
  for (int j = threadIdx.x; j < m; j += NT) sbw[j] = A.b[j] * A.dy[j];
  for (int i = threadIdx.x; i < nr; i += NT) sa[i] = A.a[r0 + i];
  for (int j = threadIdx.x; j < nc; j += NT) sb[j] = A.b[c0 + j];
  __syncthreads();
  double err = INFINITY;
  int done = 0, conv = 0;
  for (int k = 0; k < A.iters; ++k) {
    const bool check = A.check_every > 0 && ((k + 1) % A.check_every == 0 || k == A.iters - 1);
    // a-update on this CTA's rows: the sums, then Table 1 one row per lane of
    // warp 0 (one FP64 instruction stream for all rows on the narrow FP64 pipe)
    for (int r = warp; r < nr; r += kAlg1Warps) {
      const double* row = sK + (size_t)r * m;
      double sacc = 0.0;
      for (int j = lane; j < m; j += 32) sacc = fma(row[j], sbw[j], sacc);
      sacc = wsum(sacc);
      if (lane == 0) ssum[r] = sacc;
    }
    __syncthreads();
    if (warp == 0) {
      double num = 0.0, den = 0.0;
      for (int r = lane; r < nr; r += 32) {
        const int i = r0 + r;
        const double sv = ssum[r], aold = sa[r];
        const double anew = proxdiv_plain(A.F1, A.p[i], sv, A.eps);
        sa[r] = anew;
        saw[i] = anew * A.dx[i];
        if (check) {
          num += A.dx[i] * fabs(aold * sv - anew * sv);
          den += A.dx[i] * anew * sv;
        }
      }
      if (check) {
        num = wsum(num);
        den = wsum(den);
        if (lane == 0) {
          cpart[0] = num;
          cpart[1] = den;
        }
      }
    }
    cluster.sync();
    // the other CTAs' a (.) dx
    for (int i = threadIdx.x; i < n; i += NT) {
      const int owner = i / R;
      if (owner != rank) saw[i] = *cluster.map_shared_rank(saw + i, owner);
    }
    if (check) {
      double tn = 0.0, td = 0.0;
      for (int c = 0; c < CL; ++c) {
        const double* pc = cluster.map_shared_rank(cpart, c);
        tn += pc[0];
        td += pc[1];
      }
      err = (td > 0.0) ? tn / td : 0.0;
    }
    __syncthreads();
    // b-update on this CTA's columns
    for (int r = warp; r < nc; r += kAlg1Warps) {
      const double* row = sKT + (size_t)r * n;
      double sacc = 0.0;
      for (int i = lane; i < n; i += 32) sacc = fma(row[i], saw[i], sacc);
      sacc = wsum(sacc);
      if (lane == 0) ssum[r] = sacc;
    }
    __syncthreads();
    if (warp == 0) {
      for (int r = lane; r < nc; r += 32) {
        const int j = c0 + r;
        const double bnew = proxdiv_plain(A.F2, A.q[j], ssum[r], A.eps);
        sb[r] = bnew;
        sbw[j] = bnew * A.dy[j];
      }
    }
    cluster.sync();
    for (int j = threadIdx.x; j < m; j += NT) {
      const int owner = j / Q;
      if (owner != rank) sbw[j] = *cluster.map_shared_rank(sbw + j, owner);
    }
    __syncthreads();
    done = k + 1;
    if (check && done > 1 && A.tol > 0.0 && err <= A.tol) {  // the same decision in every CTA
      conv = 1;
      break;
    }
  }
  for (int i = threadIdx.x; i < nr; i += NT) A.a[r0 + i] = sa[i];
  for (int j = threadIdx.x; j < nc; j += NT) A.b[c0 + j] = sb[j];
  if (rank == 0 && threadIdx.x == 0) {
    A.res[0] = err;
    A.res[1] = (double)done;
    A.res[2] = (double)conv;
  }
  cluster.sync();  // no CTA leaves while another may still read its shared memory
}

}  // namespace

// L64 | Lff | Lch of prepare_L_chunks
size_t rows_chunks_scratch_bytes(int64_t nin) {
  return 2 * (((size_t)nin * 8 + 255) & ~(size_t)255) + ((size_t)rows_chunks(nin) * 8 + 255);
}

cudaError_t launch_chunkmin32(const double* C, int64_t nrows, int nin, float* C32, float* Cmin, cudaStream_t s) {
  const int nchunk = (int)rows_chunks(nin);
  count_launches(1);
  chunkmin32<<<(unsigned)std::min<int64_t>((nrows * nchunk + 7) / 8, 64 * sm_count()), 256, 0, s>>>(C, nrows, nin, nchunk, C32,
                                                                                         Cmin);
  return cudaGetLastError();
}

cudaError_t launch_rows(int prec, const RowsGeom& g, int nrows, int nin, const double* W,
                        const double* logw, double eps, void* scratch_L, const Epilogue& epi,
                        cudaStream_t s, float* zprev, float zscale, void* part, int precise) {
  if ((precise || precise_forced()) && prec == UOT_F32 && g.kind == UOT_GEOM_POINTS && g.d <= 3)
    return launch_points_ffp((const float*)g.x, (const float*)g.y, g.d, nrows, nin, W, logw, eps,
                             (float*)scratch_L, zprev, epi, s);
  // scratch_L: nin elements of the precision's type followed by one double
  // (Lmax); FP64 dense rows: rows_chunks_scratch_bytes.
  constexpr int WARPS = 8;
  const int grid = (nrows + WARPS - 1) / WARPS;
  if (g.kind == UOT_GEOM_POINTS && (g.d < 1 || g.d > 8)) return cudaErrorInvalidValue;
  count_launches(2);
  if (prec == UOT_F32 && g.kind == UOT_GEOM_POINTS && g.d <= 3 && part) {
    // chunked point-cloud kernels; scratch_L holds the block maxima
    count_launches(-2);
    return launch_points((const float*)g.x, (const float*)g.y, g.d, nrows, nin, W, logw, eps,
                         (float*)scratch_L, zprev, zscale, reinterpret_cast<float2*>(part), epi, s);
  }
  if (prec == UOT_F32) {
    float* Lt = (float*)scratch_L;
    float* Lmax = (float*)((char*)scratch_L + (((size_t)nin * 4 + 255) & ~(size_t)255));
    prepare_L_ff<1024><<<1, 1024, 0, s>>>(reinterpret_cast<const float2*>(W),
                                           reinterpret_cast<const float2*>(logw), nin,
                                           ff2(ff_make(1.0 / eps)), Lt, Lmax);
    prof_mark_begin(PROF_ROWS, s);
    const float* C = (const float*)g.C;
    const float* x = (const float*)g.x;
    const float* y = (const float*)g.y;
    const float k2 = (float)((double)kLog2e / eps);
    if (g.kind == UOT_GEOM_DENSE || g.d <= 4)
      rows_lse_f32<4, WARPS><<<grid, WARPS * 32, 0, s>>>(g.kind, C, x, y, g.d, nrows, nin, Lt, Lmax, k2, epi);
    else
      rows_lse_f32<8, WARPS><<<grid, WARPS * 32, 0, s>>>(g.kind, C, x, y, g.d, nrows, nin, Lt, Lmax, k2, epi);
  } else {
    double* Lt = (double*)scratch_L;
    double* Lmax = (double*)((char*)scratch_L + (((size_t)nin * 8 + 255) & ~(size_t)255));
    const double* C = (const double*)g.C;
    // dense rows with an FP32 copy of C (k2 = 1/eps must stay an FP32 number)
    if (g.kind == UOT_GEOM_DENSE && g.C32 && 1.0 / eps < 1e30) {
      char* base = (char*)scratch_L;
      const size_t r8 = ((size_t)nin * 8 + 255) & ~(size_t)255;
      double* L64 = (double*)base;
      float2* Lff = (float2*)(base + r8);
      float2* Lch = (float2*)(base + 2 * r8);
      const int nchunk = (int)rows_chunks(nin);
      cudaError_t e = launch_pdl(prepare_L_chunks, dim3((nin + 255) / 256), dim3(256), 0, s, W, logw, nin, 1.0 / eps,
                                 L64, Lff, Lch);
      if (e != cudaSuccess) return e;
      prof_mark_begin(PROF_ROWS, s);
      auto run = [&](auto kern, int nw, int rpc) -> cudaError_t {
        const size_t smem = rows_chunks_smem(nw, nchunk);
        const cudaError_t e0 = smem_at_least(kern, smem);
        if (e0 != cudaSuccess) return e0;
        const double* l64 = L64;
        const float2 *lff = Lff, *lch = Lch;
        return launch_pdl(kern, dim3((nrows + rpc - 1) / rpc), dim3(nw * 32), smem, s, C, g.C32,
                          g.Cmin, nrows, nin, nchunk, l64, lff, lch, 1.0 / eps, 50.0f + logf((float)nin), epi);
      };
      // Warps per row, as many as keep the CTAs at one per SM, so that few rows still fill the
      // GPU (one warp a row left 1 x 300000 at 2.3 times the time of the four-warp kernel before,
      // 300 x 300 at 1.17).  Times of 20 iterations with 1, 2, 4 warps: 300 rows 1.19, 0.90,
      // 0.80 ms; 450 rows (WF, eps 1e-3) 2.87, 2.19, 2.2; 784 rows (WF, 1e-8) 2.12, 2.25; 3000 rows
      // (WF, 1e-8) 3.2, 4.1, 5.0.  152 rows of 30000 columns: 4 warps 1.16 ms, 16 0.69.
      // Four to eight rows per SM that fit registers take CTAs of 32 warps, eight rows of four:
      // 700 x 700 at eps 1 1.84 -> 1.70 ms, 1128 rows (WF, 1e-3) 4.43 -> 4.21, (1e-8) 2.15 both;
      // eight SMs stay free for the kernels before and after, which such a CTA leaves no
      // registers (1216 rows, one on every SM, WF at 1e-8: 2.36 against 2.25 ms).
      const int sms = sm_count();
      auto by_length = [&](auto shrt, auto lng, int nw, int wpr) {
        return nchunk <= kShortChunks * wpr ? run(shrt, nw, nw / wpr) : run(lng, nw, nw / wpr);
      };
      if (nrows <= sms && nchunk >= 128)
        e = run(&rows_lse_f64_chunks<16, 16, 0>, 16, 1);
      else if (nrows <= 2 * sms)
        e = by_length(&rows_lse_f64_chunks<8, 4, kShortChunks>, &rows_lse_f64_chunks<8, 4, 0>, 8, 4);
      else if (nrows <= 4 * sms)
        e = by_length(&rows_lse_f64_chunks<8, 2, kShortChunks>, &rows_lse_f64_chunks<8, 2, 0>, 8, 2);
      else if (nrows <= 8 * (sms - 8) && nchunk <= 4 * kShortWide)
        e = nchunk <= 4 * kShortChunks ? run(&rows_lse_f64_chunks<32, 4, kShortChunks>, 32, 8)
                                       : run(&rows_lse_f64_chunks<32, 4, kShortWide>, 32, 8);
      else
        e = by_length(&rows_lse_f64_chunks<8, 1, kShortChunks>, &rows_lse_f64_chunks<8, 1, 0>, 8, 1);
      if (e != cudaSuccess) return e;
      prof_mark_end(PROF_ROWS, s);
      return cudaGetLastError();
    }
    prepare_L<double, 1024><<<1, 1024, 0, s>>>(W, logw, nin, eps, Lt, Lmax);
    prof_mark_begin(PROF_ROWS, s);
    const double* x = (const double*)g.x;
    const double* y = (const double*)g.y;
    if (g.kind == UOT_GEOM_DENSE || g.d <= 4)
      rows_lse<double, 4, WARPS><<<grid, WARPS * 32, 0, s>>>(g.kind, C, x, y, g.d, nrows, nin,
                                                            Lt, Lmax, eps, epi);
    else
      rows_lse<double, 8, WARPS><<<grid, WARPS * 32, 0, s>>>(g.kind, C, x, y, g.d, nrows, nin,
                                                            Lt, Lmax, eps, epi);
  }
  prof_mark_end(PROF_ROWS, s);
  return cudaGetLastError();
}

size_t alg1_cluster_smem(int n, int m, int CL) {
  const size_t R = (n + CL - 1) / CL, Q = (m + CL - 1) / CL;
  return 8 * (R * m + Q * n + m + n + R + Q + std::max(R, Q));
}

cudaError_t launch_alg1_cluster(const double* K, const double* KT, int n, int m, const double* p,
                                const double* dx, const double* q, const double* dy, DivParams F1,
                                DivParams F2, double eps, double* a, double* b, int iters, int check_every,
                                double tol, double* res, cudaStream_t s, bool* launched) {
  *launched = false;
  for (int CL : {16, 8}) {
    const size_t smem = alg1_cluster_smem(n, m, CL);
    if (smem > 200 * 1024) continue;
    if (CL > 8 && cudaFuncSetAttribute(alg1_cluster, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
      (void)cudaGetLastError();
      continue;
    }
    if (smem_at_least(alg1_cluster, smem) != cudaSuccess) {
      (void)cudaGetLastError();
      continue;
    }
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(CL);
    cfg.blockDim = dim3(kAlg1Warps * 32);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CL;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int nclusters = 0;
    if (cudaOccupancyMaxActiveClusters(&nclusters, alg1_cluster, &cfg) != cudaSuccess || nclusters < 1) {
      (void)cudaGetLastError();
      continue;
    }
    Alg1ClusterArgs A;
    A.K = K;
    A.KT = KT;
    A.n = n;
    A.m = m;
    A.R = (n + CL - 1) / CL;
    A.Q = (m + CL - 1) / CL;
    A.p = p;
    A.dx = dx;
    A.q = q;
    A.dy = dy;
    A.F1 = F1;
    A.F2 = F2;
    A.eps = eps;
    A.a = a;
    A.b = b;
    A.iters = iters;
    A.check_every = check_every;
    A.tol = tol;
    A.res = res;
    count_launches(1);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, alg1_cluster, A);
    if (e == cudaSuccess) *launched = true;
    return e;
  }
  return cudaSuccess;  // does not fit: the caller runs the per-launch path
}

cudaError_t launch_alg1_half(const double* K, int nrows, int nin, const double* b,
                             const double* w, const double* p, DivParams F, double eps,
                             double* a, const double* wout, double* err, cudaStream_t s) {
  count_launches(1);
  // one row per warp; with few rows, one warp per CTA so that every SM's
  // (narrow) FP64 pipe takes part
  if (nrows < 8 * 152) {
    alg1_half<1><<<nrows, 32, 0, s>>>(K, nrows, nin, b, w, p, F, eps, a, wout, err);
  } else {
    constexpr int WARPS = 8;
    alg1_half<WARPS><<<(nrows + WARPS - 1) / WARPS, WARPS * 32, 0, s>>>(K, nrows, nin, b, w, p, F, eps, a, wout,
                                                                        err);
  }
  return cudaGetLastError();
}

}  // namespace uot
