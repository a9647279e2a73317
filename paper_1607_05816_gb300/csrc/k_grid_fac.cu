// FP64 separable grid pass as a product with a stored kernel (Sec. 4.4 in the
// log domain of Sec. 4.3):
//
//   z[i][l] = log sum_j exp(L[l][j] - (x_i - y_j)^2 / eps)
//           = M + log sum_j A_j G_ij,
//   A_j  = exp(L[l][j] - (c - y_j)^2 / eps - M),  M the largest exponent,
//   G_ij = exp(-((x_i - y_j)^2 - (c - y_j)^2) / eps),
//
// for a block of outputs with centre c.  G does not depend on the line, so it
// is stored once per eps and axis, and a term costs one FP64 multiply-add
// where the log-sum-exp pays an FP64 exponential (about 15 FP64 instructions
// on a pipe that issues 2 lanes per clock and SM); A costs one exponential per
// input and block of 64 outputs.  Centring keeps both factors inside the FP64
// range: with reach = (d^2 + 2 d D) / eps (d the block's half width, D the
// largest |c - y_j|), exp(-reach) <= G <= exp(reach) and the input of the
// largest exponent alone gives a sum >= exp(-reach), while an A that underflows
// loses less than exp(reach - 708).  At reach <= 320 the loss is below
// exp(-60) of any sum, so the result is the log-sum-exp to FP64 rounding and
// needs no check and no shift from an earlier pass.  A tile of 64 outputs is
// cut into 2 to 16 blocks where its own reach is larger; where that is not
// enough (an eps far below the grid spacing) its outputs take the plain
// log-sum-exp, in the same kernel, so the host never reads the axes.
//
// Bound: FP64 FMA issue (nlines nin nout / (2 x 152 x 2.07e9 /s): 26.7 us for a
// 256 x 256 grid pass).
#include <string.h>

#include <algorithm>

#include "uot_internal.cuh"

namespace uot {
namespace {

constexpr int kTile = kFacTile;  // outputs per tile
constexpr int kChunk = 256;      // inputs staged at a time (fewer where a tile has over 4 blocks)
constexpr double kMaxReach = 320.0;

__device__ __forceinline__ double wmax_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// G [nin][ld] (ld = 64 x tiles, zero beyond nout) and the tiles' blocks.
// CTA (tile, 16 inputs); every CTA of a tile finds the same blocks.
__global__ void __launch_bounds__(256) fac64_build(const double* __restrict__ xo, int nout,
                                                   const double* __restrict__ yi, int nin, double inv_eps,
                                                   double* __restrict__ G, FacTile* __restrict__ tiles) {
  __shared__ double s_lo[8], s_hi[8], s_xl[kFacMaxSub], s_xh[kFacMaxSub];
  __shared__ FacTile s_t;
  const int tile = blockIdx.x, i0 = tile * kTile;
  const int tid = threadIdx.x;
  double lo = kInf, hi = -kInf;
  for (int j = tid; j < nin; j += 256) {
    lo = fmin(lo, yi[j]);
    hi = fmax(hi, yi[j]);
  }
  lo = -wmax_d(-lo);
  hi = wmax_d(hi);
  if ((tid & 31) == 0) {
    s_lo[tid >> 5] = lo;
    s_hi[tid >> 5] = hi;
  }
  // the tile's outputs in 16 blocks of 4: least and largest coordinate
  constexpr int kLeast = kTile / kFacMaxSub;
  if (tid < kFacMaxSub) {
    double xl = kInf, xh = -kInf;
#pragma unroll
    for (int u = 0; u < kLeast; ++u) {
      const int i = i0 + tid * kLeast + u;
      if (i < nout) {
        xl = fmin(xl, xo[i]);
        xh = fmax(xh, xo[i]);
      }
    }
    s_xl[tid] = xl;
    s_xh[tid] = xh;
  }
  __syncthreads();
  // Lane p of the first warp tries block s of a cut into sub blocks, p = sub - 1 + s
  // (31 of them; one thread trying all took 46 us at 64 outputs: an operator call on 64 x 64
  // at eps 1e-4 0.42 ms, 0.33 here).
  if (tid < 32) {
    for (int w = 0; w < 8; ++w) {
      lo = fmin(lo, s_lo[w]);
      hi = fmax(hi, s_hi[w]);
    }
    const int sub = 1 << (31 - __clz(tid + 1)), s = tid + 1 - sub, per = kFacMaxSub / sub;
    bool ok = true;
    double c = 0.0;
    if (sub <= kFacMaxSub) {
      double xl = kInf, xh = -kInf;
      for (int u = 0; u < per; ++u) {
        xl = fmin(xl, s_xl[s * per + u]);
        xh = fmax(xh, s_xh[s * per + u]);
      }
      const bool some = i0 + s * (kTile / sub) < nout;
      c = some ? 0.5 * (xl + xh) : xo[i0];
      const double d = some ? fmax(xh - c, c - xl) : 0.0;
      const double D = fmax(fabs(c - lo), fabs(c - hi));
      ok = (d * d + 2.0 * d * D) * inv_eps <= kMaxReach;  // false for NaN as well
    }
    const unsigned fits = __ballot_sync(0xffffffffu, ok);
    int best = 0;  // the fewest blocks that all fit
    for (int k = kFacMaxSub; k; k /= 2) {
      const unsigned all = ((1u << k) - 1u) << (k - 1);
      if ((fits & all) == all) best = k;
    }
    if (tid == 0) s_t.sub = best;
    if (sub == best) s_t.c[s] = c;
  }
  __syncthreads();
  if (blockIdx.y == 0 && tid == 0) tiles[tile] = s_t;
  if (s_t.sub == 0) return;
  const int o = tid & (kTile - 1), i = i0 + o;
  const int64_t ld = (int64_t)gridDim.x * kTile;
  const double c = s_t.c[o / (kTile / s_t.sub)];
  const double x = xo[min(i, nout - 1)], d = x - c;
  for (int j = blockIdx.y * 16 + tid / kTile; j < min(nin, (int)blockIdx.y * 16 + 16); j += 256 / kTile) {
    const double y = yi[j];
    G[j * ld + i] = (i < nout) ? exp(-d * ((x - y) + (c - y)) * inv_eps) : 0.0;
  }
}

struct Fac64Args {
  const double* in;
  const double* logw;  // in_is_pot
  int in_is_pot, nlines, nin, nout;
  const double* yi;
  const double* xo;
  double inv_eps;
  const double* G;       // NULL: every tile takes the plain log-sum-exp
  const FacTile* tiles;
  float* zprev;          // plain log-sum-exp: the previous results, its shifts with use_prev
  int use_prev;
};

// CTA = TL lines x one tile; thread = (slice of the inputs, line, output).
template <int TL, int KS>
__global__ void __launch_bounds__(kTile * TL * KS) grid_pass_f64(Fac64Args a, Epilogue epi) {
  constexpr int NT = kTile * TL * KS, NW = NT / 32;
  __shared__ double sL[TL][kChunk], sy[kChunk];
  __shared__ double sA[TL * 4 * kChunk];  // A of every (line, block) pair, kc inputs each
  __shared__ double sM[TL * kFacMaxSub], sScale[TL * kFacMaxSub];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int o = tid & (kTile - 1), ln = (tid / kTile) % TL, ks = tid / (kTile * TL);
  const int i = blockIdx.x * kTile + o, l0 = blockIdx.y * TL, l = l0 + ln;
  const int64_t bz = blockIdx.z;
  const int nin = a.nin;
  const double inv_eps = a.inv_eps;
  pdl_wait();
  pdl_launch_dependents();
  const double* in = a.in + bz * (int64_t)a.nlines * nin;
  auto stage = [&](int j0, int nc) {
    for (int t = tid; t < TL * nc; t += NT) {
      const int r = t / nc, j = t - r * nc;
      double v = -kInf;
      if (l0 + r < a.nlines) {
        const int64_t idx = (int64_t)(l0 + r) * nin + j0 + j;
        v = in[idx];
        if (a.in_is_pot) v = (v == -kInf) ? -kInf : v * inv_eps + a.logw[idx];
      }
      sL[r][j] = v;
      if (r == 0) sy[j] = a.yi[j0 + j];
    }
  };
  FacTile t;
  t.sub = 0;
  if (a.G) t = a.tiles[blockIdx.x];
  double z = -kInf;
  if (t.sub) {
    const int pair = ln * t.sub + o / (kTile / t.sub);
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    const int64_t ld = (int64_t)gridDim.x * kTile;
    const int kc = t.sub <= 4 ? kChunk : 4 * kChunk / t.sub;
    for (int j0 = 0; j0 < nin; j0 += kc) {
      const int nc = min(kc, nin - j0);
      if (j0) __syncthreads();
      stage(j0, nc);
      __syncthreads();
      // One warp per (line, block) pair.  Spreading a pair's inputs over all warps
      // (segment maxima merged through shared memory) measured slower, 60 against
      // 51 us: the extra FP64 maxima cost more than the idle warps, since other
      // CTAs' FMAs fill the pipe meanwhile.
      for (int p = warp; p < TL * t.sub; p += NW) {
        const double c = t.c[p % t.sub];
        const double* Lp = sL[p / t.sub];
        double* A = sA + p * kc;
        const double m_old = j0 ? sM[p] : -kInf;
        double m = m_old;
        for (int j = lane; j < nc; j += 32) {
          const double d = c - sy[j], e = Lp[j] - d * d * inv_eps;
          A[j] = e;
          m = fmax(m, e);
        }
        m = wmax_d(m);
        for (int j = lane; j < nc; j += 32) {
          const double e = A[j];
          A[j] = (m == -kInf && e == e) ? 0.0 : exp(e - m);  // (a line of NaN alone has no maximum)
        }
        __syncwarp();
        if (lane == 0) {
          sM[p] = m;
          sScale[p] = (m_old == -kInf) ? 0.0 : exp(m_old - m);
        }
      }
      __syncthreads();
      if (j0) {
        const double f = sScale[pair];
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[u] *= f;
      }
      const int len = ((nc + KS - 1) / KS + 3) & ~3;
      const int ja = min(nc, ks * len), jb = min(nc, ja + len);
      const double* A = sA + pair * kc;
      const double* Gp = a.G + (int64_t)(j0 + ja) * ld + i;
      int j = ja;
      for (; j + 8 <= jb; j += 8, Gp += 8 * ld) {
        double g[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) g[u] = __ldg(Gp + u * ld);
#pragma unroll
        for (int u = 0; u < 8; ++u) acc[u & 3] = fma(A[j + u], g[u], acc[u & 3]);
      }
      for (; j < jb; ++j, Gp += ld) acc[0] = fma(A[j], __ldg(Gp), acc[0]);
    }
    double s = (acc[0] + acc[1]) + (acc[2] + acc[3]);
    if (KS > 1) {
      __syncthreads();
      double* red = sA;  // TL * 4 * kChunk >= NT
      red[tid] = s;
      __syncthreads();
      if (ks == 0)
        for (int q = 1; q < KS; ++q) s += red[tid + q * kTile * TL];
    }
    const double m = sM[pair];
    if (ks == 0 && (m != -kInf || s != s)) z = m + log(s);
  } else {
    // plain log-sum-exp: shifted by the previous result where there is one (one
    // sweep), redone with running maxima if a sum leaves [1e-290, 1e290]
    const double x = a.xo[min(i, a.nout - 1)];
    float* zp = a.zprev ? a.zprev + bz * (int64_t)a.nout * a.nlines + (int64_t)i * a.nlines + l : nullptr;
    const bool own = i < a.nout && l < a.nlines;
    const double shift = (a.use_prev && zp && own) ? (double)*zp : 0.0;
    bool exact = !(a.use_prev && a.zprev) || __syncthreads_or(!(shift > -kInf));
    for (int attempt = 0; attempt < 2; ++attempt) {
      double m = exact ? -kInf : shift, s = 0.0;
      for (int j0 = 0; j0 < nin; j0 += kChunk) {
        const int nc = min(kChunk, nin - j0);
        __syncthreads();
        stage(j0, nc);
        __syncthreads();
        const int len = (nc + KS - 1) / KS;
        const int ja = min(nc, ks * len), jb = min(nc, ja + len);
        const double* Lp = sL[ln];
        if (exact) {
          double cm = m;
          for (int j = ja; j < jb; ++j) {
            const double d = x - sy[j];
            cm = fmax(cm, Lp[j] - d * d * inv_eps);
          }
          if (cm > m) {
            s = (m == -kInf && s == s) ? 0.0 : s * exp(m - cm);
            m = cm;
          }
        }
        if (m != -kInf) {
#pragma unroll 2
          for (int j = ja; j < jb; ++j) {
            const double d = x - sy[j];
            s += exp((Lp[j] - m) - d * d * inv_eps);
          }
        } else {
          for (int j = ja; j < jb; ++j) {
            const double d = x - sy[j], e = Lp[j] - d * d * inv_eps;
            if (e != e) s = e;  // NaN has no maximum
          }
        }
      }
      if (KS > 1) {
        double* rm = sA;
        double* rs = rm + NT;
        static_assert(KS == 1 || 2 * NT <= TL * 4 * kChunk, "reduction buffer");
        __syncthreads();
        rm[tid] = m;
        rs[tid] = s;
        __syncthreads();
        if (ks == 0) {
          for (int q = 1; q < KS; ++q) m = fmax(m, rm[tid + q * kTile * TL]);
          s = 0.0;
          for (int q = 0; q < KS; ++q) {
            const double mq = rm[tid + q * kTile * TL];
            const double sq = rs[tid + q * kTile * TL];
            if (mq == -kInf) s += (sq != sq) ? sq : 0.0;
            else s += (mq == m) ? sq : sq * exp(mq - m);
          }
        }
      }
      if (!exact && __syncthreads_or(own && ks == 0 && !(s >= 1e-290 && s <= 1e290))) {
        exact = true;
        continue;
      }
      if (ks == 0 && (m != -kInf || s != s)) z = m + log(s);
      break;
    }
    if (zp && own && ks == 0) *zp = (float)z;
  }
  double num = 0.0, den = 0.0;
  if (ks == 0 && i < a.nout && l < a.nlines) apply_epilogue(epi, bz, (int64_t)i * a.nlines + l, z, num, den);
  if (epi.err) block_add2<NT>(num, den, epi.err + 2 * bz);
}

// A few outputs without a stored kernel (the operator on one short line): one
// warp per output, lanes over the inputs, so that the exponentials of a single
// line spread over the chip; a tile of 64 outputs per CTA leaves them to a few
// SMs' FP64 pipes (1 x 256 points: 126 us a call against 30).
__global__ void __launch_bounds__(128) grid_pass_f64_few(Fac64Args a, Epilogue epi) {
  const int lane = threadIdx.x & 31;
  const int64_t w = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
  const int64_t per = (int64_t)a.nlines * a.nout;
  const int64_t bz = blockIdx.y;
  double num = 0.0, den = 0.0;
  pdl_wait();
  pdl_launch_dependents();
  if (w < per) {
    const int l = (int)(w % a.nlines), i = (int)(w / a.nlines);
    const double* in = a.in + (bz * a.nlines + l) * (int64_t)a.nin;
    const double* lw = a.logw + (int64_t)l * a.nin;
    const double x = a.xo[i];
    auto expo = [&](int j) {
      double v = in[j];
      if (a.in_is_pot) v = (v == -kInf) ? -kInf : v * a.inv_eps + lw[j];
      const double d = x - a.yi[j];
      return v - d * d * a.inv_eps;
    };
    double m = -kInf, s = 0.0;
    for (int j = lane; j < a.nin; j += 32) m = fmax(m, expo(j));
    m = wmax_d(m);
    double z = -kInf;
    if (m == -kInf) {  // every input is empty, or NaN, which has no maximum
      bool nan = false;
      for (int j = lane; j < a.nin; j += 32) nan = nan || expo(j) != expo(j);
      if (__any_sync(0xffffffffu, nan)) z = NAN;
    } else {
      for (int j = lane; j < a.nin; j += 32) s += exp(expo(j) - m);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      z = m + log(s);
    }
    if (lane == 0) apply_epilogue(epi, bz, w, z, num, den);
  }
  if (epi.err) block_add2<128>(num, den, epi.err + 2 * bz);
}

template <int TL, int KS>
cudaError_t launch_pass(const Fac64Args& a, const Epilogue& epi, int nbatch, cudaStream_t s) {
  const dim3 grid((a.nout + kTile - 1) / kTile, (a.nlines + TL - 1) / TL, nbatch);
  if (grid.y > 65535 || grid.z > 65535) return cudaErrorInvalidConfiguration;
  return launch_pdl(grid_pass_f64<TL, KS>, grid, dim3(kTile * TL * KS), 0, s, a, epi);
}

}  // namespace

cudaError_t launch_fac64_build(const double* xo, int nout, const double* yi, int nin, double eps, double* G,
                               FacTile* tiles, cudaStream_t s) {
  count_launches(1);
  const dim3 grid((nout + kTile - 1) / kTile, (nin + 15) / 16);
  fac64_build<<<grid, 256, 0, s>>>(xo, nout, yi, nin, 1.0 / eps, G, tiles);
  return cudaGetLastError();
}

cudaError_t launch_grid_pass_f64(const double* in, const double* logw, int in_is_pot, int nlines, int nin,
                                 const double* yi, int nout, const double* xo, double eps, int nbatch,
                                 const Epilogue& epi, const double* G, const FacTile* tiles, float* zprev,
                                 int use_prev, cudaStream_t s) {
  Fac64Args a;
  a.in = in;
  a.logw = logw;
  a.in_is_pot = in_is_pot;
  a.nlines = nlines;
  a.nin = nin;
  a.nout = nout;
  a.yi = yi;
  a.xo = xo;
  a.inv_eps = 1.0 / eps;
  a.G = G;
  a.tiles = tiles;
  a.zprev = zprev;
  a.use_prev = use_prev;
  const int64_t outs = (int64_t)nlines * nout;
  if (!G && outs * nbatch <= 64 * sm_count() && nbatch <= 65535)
    return launch_pdl(grid_pass_f64_few, dim3((unsigned)((outs + 3) / 4), nbatch), dim3(128), 0, s, a, epi);
  // Four slices of the inputs per output: 256 x 256, 51 us a pass (one slice 49,
  // eight 66); 300 x 300, 88 (one slice 128: the short last chunk's exponentials
  // are not hidden); 64 x 64, 7.6 (9.1).
  return launch_pass<1, 4>(a, epi, nbatch, s);
}

}  // namespace uot
