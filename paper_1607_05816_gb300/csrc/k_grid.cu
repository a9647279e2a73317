// Separable log-domain Gibbs operator on Cartesian grids (Sec. 4.4): for the
// cost |x - y|^2 the kernel is a product of 1-D kernels, so K(b.dy) is taken
// one axis at a time.  In the log domain each axis pass is a batch of 1-D
// log-sum-exp convolutions
//
//   z[i][l] = log sum_j exp(L[l][j] - (xo[i] - yi[j])^2 / eps)
//
// over `nlines` independent lines l.  The result is written transposed
// (point index i*nlines + l), so that d successive passes over the last axis
// cycle a row-major d-dimensional array back to row-major order.
//
// This file holds the FP32 passes, nlines * nout * nin exponentials each, bound
// by the FP32 pipe; the FP64 pass is in k_grid_fac.cu.
#include <string.h>

#include <algorithm>
#include <atomic>
#include <map>
#include <mutex>
#include <string>

#include "k_grid_pass.cuh"

namespace uot {
namespace {

// FP32 grid pass.  One CTA = one line x (32 * OPL) consecutive outputs; its NW
// warps split the contraction index j into NW contiguous ranges and combine
// their partial (max, sum) pairs through shared memory.  Each lane owns OPL
// outputs handled as OPL/2 f32x2 pairs.  (NW, OPL) is the tile shape; the
// shapes below are all compiled and one is picked per pass shape (nlines, nin,
// nout, batch) by timing them on the device (see the tuner further down).
//
// The log-sum-exp needs a shift m per output; any m with every term's
// exponent <= ~100 and the largest >= ~-90 gives the full FP32 accuracy, and
// the result does not depend on m.  When `zprev` holds this pass's result
// from the previous call at the same eps (potentials move little between
// iterations), that value is used as the shift and each term costs one sweep.
// If any combined sum of the CTA falls outside [2^-90, 2^100], the CTA redoes
// its outputs with the exact per-range maximum (a max sweep and a sum sweep).
constexpr int kNW = 8;                    // tile of the persistent solve: warps per CTA
constexpr int kOutCTA = 128;              // ... and outputs per CTA (4 per lane)

// Compile-time quantities of a tile shape.
template <int NW, int OPL>
struct Tile {
  static_assert(OPL == 2 || OPL == 4, "outputs per lane");
  static constexpr int kOut = 32 * OPL;                          // outputs per CTA
  static constexpr int kThreads = 32 * NW;
  static constexpr int kOwn = (kOut + kThreads - 1) / kThreads;  // outputs per thread in the epilogue
  static constexpr int kLineRegs = NW >= 2 ? 4 : 8;              // line elements held per thread
};

// Shared-memory workspace of one work item.
struct ItemSmem {
  float4* sline;  // nin x {t, t, y, y}
  float2* part;   // [NW][kOut] partial (max, sum) pairs
  float* sshift;  // [kOut]
  float* sred;    // [NW]
};

// One work item of a grid pass: line l of batch entry bz, outputs i0 .. i0+kOut-1.
// With kPDL the item waits for the preceding kernel after its independent
// prologue (programmatic dependent launch) and clears the violation
// accumulators when asked.  Returns the item's violation terms in num, den.
template <int NW, int OPL, bool kPDL>
__device__ __forceinline__ void grid_item_f32(const PassArgs& a, const Epilogue& epi, int l, int64_t bz,
                                              int i0, const ItemSmem& sm, float& num, float& den) {
  typedef Tile<NW, OPL> T;
  constexpr int OUT = T::kOut, NT = T::kThreads, OWN = T::kOwn, LR = T::kLineRegs, P = OPL / 2;
  float4* sline = sm.sline;
  float2* part = sm.part;
  float* sshift = sm.sshift;
  float* sred = sm.sred;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nin = a.nin, nout = a.nout, nlines = a.nlines;
  const float2* in = a.in + bz * (int64_t)nlines * nin;
  const int64_t base = (int64_t)l * nin;
  float* zprev = a.zprev ? a.zprev + bz * (int64_t)nout * nlines : nullptr;
  const bool spec = a.use_prev && zprev;

  // ---- prologue independent of the preceding kernel ----
  bool owns[OWN];
  int64_t my_pt[OWN];
  float zp[OWN];
  EpiPre pre[OWN];
#pragma unroll
  for (int r = 0; r < OWN; ++r) {
    const int o = tid + r * NT;
    const int i = i0 + o;
    owns[r] = (o < OUT) && (i < nout);
    my_pt[r] = (int64_t)i * nlines + l;
    zp[r] = 0.0f;
    if (owns[r]) {
      if (spec) zp[r] = zprev[my_pt[r]];
      epilogue_prefetch(epi, bz, my_pt[r], pre[r]);
    }
  }
  float yv[LR];
#pragma unroll
  for (int r = 0; r < LR; ++r) {
    const int j = tid + r * NT;
    yv[r] = (j < nin) ? a.yi[j] : 0.0f;
  }
  float xq[OPL];
#pragma unroll
  for (int q = 0; q < OPL; ++q) {
    const int i = i0 + lane + 32 * q;
    xq[q] = a.xo[i < nout ? i : nout - 1];
  }

  if (kPDL) {
    pdl_wait();
    if (a.zero_acc && blockIdx.x == 0 && blockIdx.y == 0 && tid < 2) a.zero_acc[2 * bz + tid] = 0.0;
    pdl_launch_dependents();
  }

  // ---- line values: one read, kept in registers when the line is short ----
  ff lv[LR];
  const bool in_regs = nin <= LR * NT;
  float mx = -INFINITY;
  if (in_regs) {
#pragma unroll
    for (int r = 0; r < LR; ++r) {
      const int j = tid + r * NT;
      lv[r] = (j < nin) ? load_L_ff(a, in, base + j) : ff_ninf();
      mx = fmaxf(mx, lv[r].hi);
    }
  } else {
    for (int j = tid; j < nin; j += NT) mx = fmaxf(mx, load_L_ff(a, in, base + j).hi);
  }
  mx = warp_maxf(mx);
  if (lane == 0) sred[warp] = mx;
  __syncthreads();
  mx = sred[0];
#pragma unroll
  for (int w = 1; w < NW; ++w) mx = fmaxf(mx, sred[w]);

  num = 0.0f;
  den = 0.0f;
  if (mx == -INFINITY) {
    // b = 0 on the whole line: every sum is empty.
#pragma unroll
    for (int r = 0; r < OWN; ++r) {
      if (owns[r]) {
        if (zprev) zprev[my_pt[r]] = -INFINITY;
        float n1, d1;
        epilogue_apply(epi, bz, my_pt[r], ff_ninf(), pre[r], n1, d1);
        num += n1;
        den += d1;
      }
    }
    return;
  }
  if (in_regs) {
#pragma unroll
    for (int r = 0; r < LR; ++r) {
      const int j = tid + r * NT;
      if (j < nin) {
        const float t = (lv[r].hi == -INFINITY) ? -INFINITY : ((lv[r].hi - mx) + lv[r].lo) * kLog2e;
        sline[j] = make_float4(t, t, yv[r], yv[r]);
      }
    }
  } else {
    for (int j = tid; j < nin; j += NT) {
      const ff v = load_L_ff(a, in, base + j);
      const float t = (v.hi == -INFINITY) ? -INFINITY : ((v.hi - mx) + v.lo) * kLog2e;
      const float y = a.yi[j];
      sline[j] = make_float4(t, t, y, y);
    }
  }
  // speculative shifts in log2 units relative to the staged line
#pragma unroll
  for (int r = 0; r < OWN; ++r) {
    const int o = tid + r * NT;
    if (o < OUT) sshift[o] = (!owns[r] || zp[r] == -INFINITY) ? 0.0f : (zp[r] - mx) * kLog2e;
  }
  __syncthreads();

  const f2p nk2 = pk(-a.k2, -a.k2);
  const int J = (nin + NW - 1) / NW;
  const int j0 = warp * J, j1 = min(nin, j0 + J);
  f2p X[P];
#pragma unroll
  for (int p = 0; p < P; ++p) X[p] = pk(xq[2 * p], xq[2 * p + 1]);

  bool exact = !spec;
  for (int attempt = 0; attempt < 2; ++attempt) {
    float mq[OPL];
    if (!exact) {
#pragma unroll
      for (int q = 0; q < OPL; ++q) mq[q] = sshift[lane + 32 * q];
    } else {
      // exact per-range maximum
#pragma unroll
      for (int q = 0; q < OPL; ++q) mq[q] = -INFINITY;
#pragma unroll 4
      for (int j = j0; j < j1; ++j) {
        const float4 v = sline[j];
        const f2p Tv = pk(v.x, v.y), Y = pk(v.z, v.w);
#pragma unroll
        for (int p = 0; p < P; ++p) {
          const f2p D = sub2(X[p], Y);
          const float2 A = upk(fma2(nk2, mul2(D, D), Tv));
          mq[2 * p] = fmaxf(mq[2 * p], A.x);
          mq[2 * p + 1] = fmaxf(mq[2 * p + 1], A.y);
        }
      }
    }
    // sum sweep relative to the shifts (a -inf shift means an empty range)
    f2p MS[P], S[P];
#pragma unroll
    for (int p = 0; p < P; ++p) {
      MS[p] = pk(mq[2 * p] == -INFINITY ? 0.0f : mq[2 * p], mq[2 * p + 1] == -INFINITY ? 0.0f : mq[2 * p + 1]);
      S[p] = pk(0.0f, 0.0f);
    }
#pragma unroll 4
    for (int j = j0; j < j1; ++j) {
      const float4 v = sline[j];
      const f2p Tv = pk(v.x, v.y), Y = pk(v.z, v.w);
#pragma unroll
      for (int p = 0; p < P; ++p) {
        const f2p D = sub2(X[p], Y);
        const float2 A = upk(fma2(nk2, mul2(D, D), sub2(Tv, MS[p])));
        S[p] = add2(S[p], pk(ex2_approx(A.x), ex2_approx(A.y)));
      }
    }
#pragma unroll
    for (int p = 0; p < P; ++p) {
      const float2 s = upk(S[p]);
      const float m0 = mq[2 * p], m1 = mq[2 * p + 1];
      part[warp * OUT + lane + 64 * p] = make_float2(m0 == -INFINITY ? 0.0f : m0, m0 == -INFINITY ? 0.0f : s.x);
      part[warp * OUT + lane + 64 * p + 32] = make_float2(m1 == -INFINITY ? 0.0f : m1, m1 == -INFINITY ? 0.0f : s.y);
    }
    __syncthreads();

    // combine the NW ranges of each output
    bool bad = false;
    float Mo[OWN], So[OWN];
#pragma unroll
    for (int r = 0; r < OWN; ++r) {
      const int o = tid + r * NT;
      Mo[r] = -INFINITY;
      So[r] = 0.0f;
      if (o < OUT) {
#pragma unroll
        for (int w = 0; w < NW; ++w) {
          const float2 pr = part[w * OUT + o];
          if (pr.y > 0.0f) Mo[r] = fmaxf(Mo[r], pr.x);
        }
        if (Mo[r] != -INFINITY) {
#pragma unroll
          for (int w = 0; w < NW; ++w) {
            const float2 pr = part[w * OUT + o];
            if (pr.y > 0.0f) So[r] += pr.y * ex2_approx(pr.x - Mo[r]);
          }
        }
        if (owns[r] && !exact) bad = bad || !(So[r] >= 0x1p-90f && So[r] <= 0x1p100f);
      }
    }
    const int any_bad = __syncthreads_or(bad ? 1 : 0);
    if (any_bad && !exact) {
      exact = true;
      continue;  // block-uniform: redo with exact maxima
    }
#pragma unroll
    for (int r = 0; r < OWN; ++r) {
      if (!owns[r]) continue;
      ff z = ff_ninf();
      if (So[r] > 0.0f) {
        z = pass_result(mx, Mo[r], So[r]);
      }
      if (zprev) zprev[my_pt[r]] = z.hi;
      float n1, d1;
      epilogue_apply(epi, bz, my_pt[r], z, pre[r], n1, d1);
      num += n1;
      den += d1;
    }
    break;
  }
}

template <int NW, int OPL>
__global__ void __launch_bounds__(NW * 32, NW == 1 ? 16 : 32 / NW)
    grid_pass_f32(PassArgs a, Epilogue epi) {
  extern __shared__ float4 sline[];
  __shared__ float2 part[NW * 32 * OPL];
  __shared__ float sshift[32 * OPL];
  __shared__ float sred[NW];
  const ItemSmem sm{sline, part, sshift, sred};
  float num, den;
  grid_item_f32<NW, OPL, true>(a, epi, blockIdx.y, blockIdx.z, blockIdx.x * (32 * OPL), sm, num, den);
  if (epi.err) block_add2f<NW * 32>(num, den, epi.err + 2 * (int64_t)blockIdx.z);
}

// Four lines per CTA: 4 consecutive lines x (32 * OPL) outputs, the contraction
// index split over the NW warps as above.  Two things bound the one-line CTA where
// there are many lines.  The result is stored transposed (point i*nlines + l), so
// its epilogue uses 8 bytes of every 32-byte sector that it touches (old and new
// potential, log density, shifts); here the epilogue's threads run over the lines
// first and use whole sectors.  And of the 5 FP32-pipe operations of a term two,
// the squared distance, do not depend on the line: a warp computes them once for
// its 4 lines (3.5 operations a term; the exponential, 32 a clock and SM, becomes
// the bound).  Arithmetic and summation order are grid_pass_f32's.
constexpr int kMlLines = 4;

template <int NW, int OPL>
struct MlTile {
  static constexpr int kOut = 32 * OPL;
  static constexpr int kThreads = 32 * NW;
  static constexpr int kOwn = (kMlLines * kOut + kThreads - 1) / kThreads;
  static_assert(NW % kMlLines == 0, "whole warps per line in the loading phase");
  static constexpr int kWarpsPerLine = NW / kMlLines;
  static constexpr int kLineRegs = 4;
  // partial sums of a line; 4 float2 of padding put the lines 8 banks apart
  static constexpr int kPartStride = NW * kOut + 4;
  static size_t smem(int nin) {
    return (size_t)nin * (sizeof(float4) + sizeof(float2)) +
           (size_t)kMlLines * (kPartStride * sizeof(float2) + kOut * sizeof(float));
  }
};

template <int NW, int OPL>
__global__ void __launch_bounds__(MlTile<NW, OPL>::kThreads, (OPL == 4 ? 24 : 32) / NW)
    grid_pass_f32_ml(PassArgs a, Epilogue epi) {
  typedef MlTile<NW, OPL> T;
  constexpr int NL = kMlLines, OUT = T::kOut, NT = T::kThreads, WPL = T::kWarpsPerLine, OWN = T::kOwn,
                LR = T::kLineRegs, P = OPL / 2;
  extern __shared__ float4 sml[];  // [nin] the lines' values at j
  __shared__ float sred[NL][WPL];
  const int nin = a.nin, nout = a.nout, nlines = a.nlines;
  float2* sy = reinterpret_cast<float2*>(sml + nin);                             // [nin] {y, y}
  float2* part = sy + nin;                                                       // [NL][kPartStride]
  float* sshift = reinterpret_cast<float*>(part + (size_t)NL * T::kPartStride);  // [NL][OUT]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int i0 = blockIdx.x * OUT, l0 = blockIdx.y * NL;
  const int64_t bz = blockIdx.z;
  const float2* in = a.in + bz * (int64_t)nlines * nin;
  float* zprev = a.zprev ? a.zprev + bz * (int64_t)nout * nlines : nullptr;
  const bool spec = a.use_prev && zprev;
  // loading phase: line la, elements jl, jl + JS, ...
  const int la = warp / WPL, l = l0 + la, jl = (warp % WPL) * 32 + lane;
  constexpr int JS = 32 * WPL;

  // ---- prologue independent of the preceding kernel ----
  // output o = tid + r NT of the CTA: line o % NL, output i0 + o / NL
  const int oline = tid % NL;
  bool owns[OWN];
  int64_t my_pt[OWN];
#pragma unroll
  for (int r = 0; r < OWN; ++r) {
    const int oi = (tid + r * NT) / NL;
    owns[r] = oi < OUT && i0 + oi < nout && l0 + oline < nlines;
    my_pt[r] = (int64_t)(i0 + oi) * nlines + l0 + oline;
  }
  float zp[OWN];
#pragma unroll
  for (int r = 0; r < OWN; ++r) zp[r] = (owns[r] && spec) ? zprev[my_pt[r]] : 0.0f;
  for (int j = tid; j < nin; j += NT) {
    const float y = a.yi[j];
    sy[j] = make_float2(y, y);
  }
  float xq[OPL];
#pragma unroll
  for (int q = 0; q < OPL; ++q) {
    const int i = i0 + lane + 32 * q;
    xq[q] = a.xo[i < nout ? i : nout - 1];
  }
  pdl_wait();
  if (a.zero_acc && blockIdx.x == 0 && blockIdx.y == 0 && tid < 2) a.zero_acc[2 * bz + tid] = 0.0;
  pdl_launch_dependents();

  // ---- line values ----
  const bool in_regs = nin <= LR * JS;
  const int64_t base = (int64_t)l * nin;
  ff lv[LR];
  float mx = -INFINITY;
#pragma unroll
  for (int r = 0; r < LR; ++r) lv[r] = ff_ninf();
  if (l < nlines) {
    if (in_regs) {
#pragma unroll
      for (int r = 0; r < LR; ++r) {
        const int j = jl + r * JS;
        if (j < nin) lv[r] = load_L_ff(a, in, base + j);
        mx = fmaxf(mx, lv[r].hi);
      }
    } else {
      for (int j = jl; j < nin; j += JS) mx = fmaxf(mx, load_L_ff(a, in, base + j).hi);
    }
  }
  mx = warp_maxf(mx);
  if (lane == 0) sred[la][warp % WPL] = mx;
  __syncthreads();
  float mxo = sred[oline][0];  // of the line whose outputs this thread finishes
#pragma unroll
  for (int w = 1; w < WPL; ++w) mxo = fmaxf(mxo, sred[oline][w]);
#pragma unroll
  for (int w = 0; w < WPL; ++w) mx = fmaxf(mx, sred[la][w]);
  auto stage = [&](int j, ff v) {
    reinterpret_cast<float*>(sml)[4 * j + la] = (v.hi == -INFINITY) ? -INFINITY : ((v.hi - mx) + v.lo) * kLog2e;
  };
  if (in_regs) {
#pragma unroll
    for (int r = 0; r < LR; ++r) {
      const int j = jl + r * JS;
      if (j < nin) stage(j, lv[r]);
    }
  } else {
    for (int j = jl; j < nin; j += JS) stage(j, l < nlines ? load_L_ff(a, in, base + j) : ff_ninf());
  }
  // speculative shifts in log2 units relative to the staged line
#pragma unroll
  for (int r = 0; r < OWN; ++r) {
    const int oi = (tid + r * NT) / NL;
    if (oi < OUT)
      sshift[oline * OUT + oi] = (!owns[r] || zp[r] == -INFINITY || mxo == -INFINITY) ? 0.0f : (zp[r] - mxo) * kLog2e;
  }
  __syncthreads();

  const f2p nk2 = pk(-a.k2, -a.k2);
  const int J = (nin + NW - 1) / NW;
  const int j0 = warp * J, j1 = min(nin, j0 + J);
  f2p X[P];
#pragma unroll
  for (int p = 0; p < P; ++p) X[p] = pk(xq[2 * p], xq[2 * p + 1]);

  bool exact = !spec;
  float num = 0.0f, den = 0.0f;
  for (int attempt = 0; attempt < 2; ++attempt) {
    float mq[NL][OPL];
    if (!exact) {
#pragma unroll
      for (int u = 0; u < NL; ++u)
#pragma unroll
        for (int q = 0; q < OPL; ++q) mq[u][q] = sshift[u * OUT + lane + 32 * q];
    } else {
#pragma unroll
      for (int u = 0; u < NL; ++u)
#pragma unroll
        for (int q = 0; q < OPL; ++q) mq[u][q] = -INFINITY;
#pragma unroll 2
      for (int j = j0; j < j1; ++j) {
        const float4 t4 = sml[j];
        const float2 y2 = sy[j];
        const f2p Y = pk(y2.x, y2.y);
        const float t[NL] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
        for (int p = 0; p < P; ++p) {
          const f2p D = sub2(X[p], Y);
          const f2p Q = mul2(D, D);
#pragma unroll
          for (int u = 0; u < NL; ++u) {
            const float2 A = upk(fma2(nk2, Q, pk(t[u], t[u])));
            mq[u][2 * p] = fmaxf(mq[u][2 * p], A.x);
            mq[u][2 * p + 1] = fmaxf(mq[u][2 * p + 1], A.y);
          }
        }
      }
    }
    f2p MS[NL][P], S[NL][P];
#pragma unroll
    for (int u = 0; u < NL; ++u)
#pragma unroll
      for (int p = 0; p < P; ++p) {
        const float m0 = mq[u][2 * p], m1 = mq[u][2 * p + 1];
        MS[u][p] = pk(m0 == -INFINITY ? 0.0f : m0, m1 == -INFINITY ? 0.0f : m1);
        S[u][p] = pk(0.0f, 0.0f);
      }
#pragma unroll 2
    for (int j = j0; j < j1; ++j) {
      const float4 t4 = sml[j];
      const float2 y2 = sy[j];
      const f2p Y = pk(y2.x, y2.y);
      const float t[NL] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
      for (int p = 0; p < P; ++p) {
        const f2p D = sub2(X[p], Y);
        const f2p Q = mul2(D, D);
#pragma unroll
        for (int u = 0; u < NL; ++u) {
          const float2 A = upk(fma2(nk2, Q, sub2(pk(t[u], t[u]), MS[u][p])));
          S[u][p] = add2(S[u][p], pk(ex2_approx(A.x), ex2_approx(A.y)));
        }
      }
    }
#pragma unroll
    for (int u = 0; u < NL; ++u)
#pragma unroll
      for (int p = 0; p < P; ++p) {
        const float2 sv = upk(S[u][p]), m = upk(MS[u][p]);
        // (a maximum of -inf: every staged value of the range is -inf, and so the sum 0)
        float2* dst = part + (size_t)u * T::kPartStride + warp * OUT + lane + 64 * p;
        dst[0] = make_float2(m.x, sv.x);
        dst[32] = make_float2(m.y, sv.y);
      }
    __syncthreads();

    // combine the NW ranges of each output
    const float2* opart = part + (size_t)oline * T::kPartStride;
    bool bad = false;
    float Mo[OWN], So[OWN];
#pragma unroll
    for (int r = 0; r < OWN; ++r) {
      const int oi = (tid + r * NT) / NL;
      Mo[r] = -INFINITY;
      So[r] = 0.0f;
      if (oi < OUT) {
#pragma unroll
        for (int w = 0; w < NW; ++w) {
          const float2 pr = opart[w * OUT + oi];
          if (pr.y > 0.0f) Mo[r] = fmaxf(Mo[r], pr.x);
        }
        if (Mo[r] != -INFINITY) {
#pragma unroll
          for (int w = 0; w < NW; ++w) {
            const float2 pr = opart[w * OUT + oi];
            if (pr.y > 0.0f) So[r] += pr.y * ex2_approx(pr.x - Mo[r]);
          }
        }
        if (owns[r] && !exact && mxo != -INFINITY) bad = bad || !(So[r] >= 0x1p-90f && So[r] <= 0x1p100f);
      }
    }
    if (!exact && __syncthreads_or(bad ? 1 : 0)) {
      exact = true;
      continue;  // block-uniform: redo with exact maxima
    }
#pragma unroll
    for (int r = 0; r < OWN; ++r) {
      if (!owns[r]) continue;
      EpiPre pre;
      epilogue_prefetch(epi, bz, my_pt[r], pre);
      ff z = ff_ninf();
      if (So[r] > 0.0f) z = pass_result(mxo, Mo[r], So[r]);
      if (zprev) zprev[my_pt[r]] = z.hi;
      float n1, d1;
      epilogue_apply(epi, bz, my_pt[r], z, pre, n1, d1);
      num += n1;
      den += d1;
    }
    break;
  }
  if (epi.err) block_add2f<NT>(num, den, epi.err + 2 * bz);
}

// ---------------------------------------------------------------------------
// Persistent solve: the whole iteration of a single FP32 grid problem in one
// cooperative launch (all CTAs co-resident).  Each pass is a set of work items
// (line, 128 outputs) spread over the CTAs, followed by a grid barrier; the
// eps-scaling stages and the convergence test run on the device, so the host
// waits only for the end of the solve.  Barrier waits are bounded in time
// (status[0] = 1 and every CTA returns if one expires).
// ---------------------------------------------------------------------------

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Waits until *p != v, for at most limit_ns nanoseconds of the global timer;
// on expiry sets *status = 1 and returns false.  Every device-side wait on
// another CTA's progress goes through here.
__device__ bool bounded_wait_change(const volatile unsigned* p, unsigned v, unsigned long long limit_ns,
                                    int* status) {
  const unsigned long long t0 = global_ns();
  while (*p == v) {
    __nanosleep(64);
    if (global_ns() - t0 > limit_ns) {
      atomicExch(status, 1);
      return false;
    }
  }
  return true;
}

constexpr unsigned long long kBarrierLimitNs = 2000000000ull;  // 2 s

// Generation-counting barrier: bar[0] arrivals, bar[1] generation.
__device__ bool grid_barrier(unsigned* bar, int* status) {
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile unsigned* gen = bar + 1;
    const unsigned g = *gen;
    __threadfence();
    if (atomicAdd(bar, 1u) == gridDim.x - 1) {
      bar[0] = 0;
      __threadfence();
      atomicAdd(bar + 1, 1u);
    } else {
      bounded_wait_change(gen, g, kBarrierLimitNs, status);
    }
    __threadfence();
  }
  __syncthreads();
  return *(volatile int*)status == 0;
}

// The bounded wait on a flag that nothing sets: exercises the expiry path of
// bounded_wait_change (status set, kernel returns, context stays usable).
__global__ void wait_selftest(const unsigned* flag, unsigned long long limit_ns, int* status) {
  if (threadIdx.x == 0 && blockIdx.x == 0) bounded_wait_change(flag, 0u, limit_ns, status);
}

struct PersistArgs {
  int ndim;
  int shape_x[UOT_MAX_DIM], shape_y[UOT_MAX_DIM];
  const float* axes_x[UOT_MAX_DIM];
  const float* axes_y[UOT_MAX_DIM];
  float2* U;
  float2* V;
  const float2* logp;
  const float2* logq;
  const float2* logdx;
  const float2* logdy;
  float2* pass[2];
  float* zbuf[2][UOT_MAX_DIM];
  int nstage, iters_per_stage, max_iter, check_every;
  double tol;
  const float2* eps_ff;      // [nstage+1]
  const float2* inv_eps_ff;  // [nstage+1]
  const float* k2;           // [nstage+1]
  const DivFF* F;            // [nstage+1][2]
  double* acc;               // [2] violation accumulators
  unsigned* bar;             // [2] barrier state (zero before the launch)
  int* status;               // [4] timeout, converged, final iterations, total iterations
  double* err_out;           // last measured violation
};

__global__ void __launch_bounds__(kNW * 32, 4)
    grid_solve_persistent(PersistArgs P) {
  extern __shared__ float4 sline[];
  __shared__ float2 part[kNW * kOutCTA];
  __shared__ float sshift[kOutCTA];
  __shared__ float sred[kNW];
  const ItemSmem sm{sline, part, sshift, sred};
  const int d = P.ndim;
  if (blockIdx.x == 0 && threadIdx.x < 2) P.acc[threadIdx.x] = 0.0;
  if (!grid_barrier(P.bar, P.status)) return;
  int total = 0, it_final = 0;
  bool stop = false;
  for (int s = 0; s <= P.nstage && !stop; ++s) {
    const int iters = (s < P.nstage) ? P.iters_per_stage : P.max_iter;
    const bool final_stage = (s == P.nstage);
    for (int it = 0; it < iters; ++it) {
      const bool check = final_stage && (((it + 1) % P.check_every == 0) || it == iters - 1);
      for (int pidx = 0; pidx < 2 * d; ++pidx) {
        const int dir = pidx / d, k = pidx % d, ax = d - 1 - k;
        const int* in_shape = dir == 0 ? P.shape_y : P.shape_x;
        const int* out_shape = dir == 0 ? P.shape_x : P.shape_y;
        int nlines = 1;
        for (int t = 0; t < ax; ++t) nlines *= in_shape[t];
        for (int t = ax + 1; t < d; ++t) nlines *= out_shape[t];
        PassArgs a;
        a.in = (k == 0) ? (dir == 0 ? P.V : P.U) : P.pass[(k - 1) & 1];
        a.logw = dir == 0 ? P.logdy : P.logdx;
        a.in_is_pot = (k == 0);
        a.nlines = nlines;
        a.nin = in_shape[ax];
        a.nout = out_shape[ax];
        a.yi = dir == 0 ? P.axes_y[ax] : P.axes_x[ax];
        a.xo = dir == 0 ? P.axes_x[ax] : P.axes_y[ax];
        a.inv_eps = P.inv_eps_ff[s];
        a.k2 = P.k2[s];
        a.zprev = P.zbuf[dir][k];
        a.use_prev = it > 0;
        a.zero_acc = nullptr;
        a.tc3_ok = 0;
        a.tc_err = nullptr;
        a.nbatch = 1;
        Epilogue e;
        memset(&e, 0, sizeof(e));
        e.ff = 1;
        e.eps_ff = P.eps_ff[s];
        e.inv_eps_ff = P.inv_eps_ff[s];
        if (k < d - 1) {
          e.mode = EPI_RAW;
          e.out = reinterpret_cast<double*>(P.pass[k & 1]);
        } else {
          e.mode = EPI_PROX;
          e.Fff = P.F[2 * s + dir];
          e.logp = reinterpret_cast<const double*>(dir == 0 ? P.logp : P.logq);
          e.pot = reinterpret_cast<double*>(dir == 0 ? P.U : P.V);
          e.logw = reinterpret_cast<const double*>(dir == 0 ? P.logdx : P.logdy);
          e.err = (dir == 0 && check) ? P.acc : nullptr;
        }
        const int nob = (a.nout + kOutCTA - 1) / kOutCTA;
        const int items = nlines * nob;
        for (int item = blockIdx.x; item < items; item += gridDim.x) {
          float num, den;
          grid_item_f32<kNW, 4, false>(a, e, item / nob, 0, (item % nob) * kOutCTA, sm, num, den);
          if (e.err) block_add2f<kNW * 32>(num, den, e.err);
        }
        if (!grid_barrier(P.bar, P.status)) return;
      }
      ++total;
      if (final_stage) it_final = it + 1;
      if (check) {
        if (blockIdx.x == 0 && threadIdx.x == 0) {
          volatile double* acc = P.acc;
          const double num = acc[0], den = acc[1];
          const double err = (den > 0.0) ? num / den : 0.0;
          *P.err_out = err;
          P.status[1] = (it > 0 && P.tol > 0.0 && err <= P.tol) ? 1 : 0;
          acc[0] = 0.0;
          acc[1] = 0.0;
        }
        if (!grid_barrier(P.bar, P.status)) return;
        if (*(volatile int*)(P.status + 1)) {
          stop = true;
          break;
        }
      }
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    P.status[2] = it_final;
    P.status[3] = total;
  }
}

}  // namespace

cudaError_t launch_wait_selftest(const unsigned* flag, unsigned long long limit_ns, int* status, cudaStream_t s) {
  count_launches(1);
  wait_selftest<<<1, 32, 0, s>>>(flag, limit_ns, status);
  return cudaGetLastError();
}

int grid_solve_persistent_ctas(int nin_max) {
  int nb = 0, dev = 0, sms = 0;
  const size_t smem = (size_t)nin_max * sizeof(float4);
  if (smem > 48 * 1024 &&
      smem_at_least(grid_solve_persistent, smem) != cudaSuccess)
    return 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, grid_solve_persistent, kNW * 32, smem) != cudaSuccess) return 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  return nb * sms;
}

cudaError_t launch_grid_solve_persistent(const PersistLaunch& L, int grid, cudaStream_t s) {
  PersistArgs P;
  memset(&P, 0, sizeof(P));
  P.ndim = L.ndim;
  for (int k = 0; k < UOT_MAX_DIM; ++k) {
    P.shape_x[k] = L.shape_x[k];
    P.shape_y[k] = L.shape_y[k];
    P.axes_x[k] = (const float*)L.axes_x[k];
    P.axes_y[k] = (const float*)L.axes_y[k];
    P.zbuf[0][k] = L.zbuf[0][k];
    P.zbuf[1][k] = L.zbuf[1][k];
  }
  P.U = reinterpret_cast<float2*>(L.U);
  P.V = reinterpret_cast<float2*>(L.V);
  P.logp = reinterpret_cast<const float2*>(L.logp);
  P.logq = reinterpret_cast<const float2*>(L.logq);
  P.logdx = reinterpret_cast<const float2*>(L.logdx);
  P.logdy = reinterpret_cast<const float2*>(L.logdy);
  P.pass[0] = reinterpret_cast<float2*>(L.pass[0]);
  P.pass[1] = reinterpret_cast<float2*>(L.pass[1]);
  P.nstage = L.nstage;
  P.iters_per_stage = L.iters_per_stage;
  P.max_iter = L.max_iter;
  P.check_every = L.check_every;
  P.tol = L.tol;
  P.eps_ff = L.eps_ff;
  P.inv_eps_ff = L.inv_eps_ff;
  P.k2 = L.k2;
  P.F = L.F;
  P.acc = L.acc;
  P.bar = L.bar;
  P.status = L.status;
  P.err_out = L.err_out;
  int nin_max = 1;
  for (int k = 0; k < L.ndim; ++k) nin_max = std::max(nin_max, std::max(L.shape_x[k], L.shape_y[k]));
  const size_t smem = (size_t)nin_max * sizeof(float4);
  cudaError_t e = smem_at_least(grid_solve_persistent, smem);
  if (e != cudaSuccess) return e;
  void* args[] = {&P};
  count_launches(1);
  e = cudaLaunchCooperativeKernel((const void*)grid_solve_persistent, dim3(grid), dim3(kNW * 32), args, smem, s);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// FP32 pass with float-float exponents ("precise pass").  The log-sum-exp
// tiles above stage each line value relative to the line's maximum and form
// t_j - k (x_i - y_j)^2 - m_i in FP32: a term whose value and cost are both
// large (tens to hundreds in log2 units, as with lambda >> eps) loses
// ulp(|t_j|) of its exponent, and the FP32 check stalls above 1e-6.  Here the
// staged values, the squared distance x_i - y_j (exact TwoSum), its product
// with k = log2(e)/eps and the running maximum are all float-float; only the
// final difference a_ij - m_i (small for every term that matters) is rounded
// to FP32 for the exponential.  One warp per (line, 32 R outputs), an online
// log-sum-exp per output (rescaled when a new maximum appears), the same
// float-float epilogue as the other passes.  About 30 FP32 operations per
// term: the pass the FP32 solves switch to when their check stalls, far
// cheaper than the FP64 iterations that follow it only if it stalls too.
// ---------------------------------------------------------------------------
constexpr ff kLog2eFF{1.44269502162933349609375f, 1.925963033500011e-08f};

template <int R, int WARPS>
__global__ void __launch_bounds__(WARPS * 32) grid_pass_ffp(PassArgs a, Epilogue epi) {
  extern __shared__ float4 sm_ffp[];  // [WARPS][nin] {t.hi, t.lo, y, 0}, t in log2 units
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int l = blockIdx.y * WARPS + warp;
  const int i0 = blockIdx.x * (32 * R);
  const int64_t bz = blockIdx.z;
  const int nin = a.nin, nout = a.nout, nlines = a.nlines;
  const float2* in = a.in + bz * (int64_t)nlines * nin;
  float* zprev = a.zprev ? a.zprev + bz * (int64_t)nout * nlines : nullptr;
  float num = 0.0f, den = 0.0f;
  bool owns[R];
  int64_t pt[R];
  float xr[R];
  EpiPre pre[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int i = i0 + lane + 32 * r;
    owns[r] = l < nlines && i < nout;
    pt[r] = (int64_t)i * nlines + l;
    xr[r] = a.xo[i < nout ? i : nout - 1];
    if (owns[r]) epilogue_prefetch(epi, bz, pt[r], pre[r]);
  }
  if (a.zero_acc && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < 2) a.zero_acc[2 * bz + threadIdx.x] = 0.0;
  if (l < nlines) {
    float4* line = sm_ffp + (size_t)warp * nin;
    const int64_t base = (int64_t)l * nin;
    float mx = -INFINITY;
    for (int j = lane; j < nin; j += 32) mx = fmaxf(mx, load_L_ff(a, in, base + j).hi);
    mx = warp_maxf(mx);
    if (mx == -INFINITY) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (!owns[r]) continue;
        if (zprev) zprev[pt[r]] = -INFINITY;
        float n1, d1;
        epilogue_apply(epi, bz, pt[r], ff_ninf(), pre[r], n1, d1);
        num += n1;
        den += d1;
      }
    } else {
      // staged: (L_j - mx) log2(e) in float-float; mx is any FP32 shift, added back exactly below
      for (int j = lane; j < nin; j += 32) {
        const ff v = load_L_ff(a, in, base + j);
        const ff t = (v.hi == -INFINITY) ? ff_ninf() : ff_mul(ff_add_f(v, -mx), kLog2eFF);
        line[j] = make_float4(t.hi, t.lo, a.yi[j], 0.0f);
      }
      __syncwarp();
      const ff k2 = ff_mul(ffl(a.inv_eps), kLog2eFF);
      float mh[R], ml[R], sum[R];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        mh[r] = -INFINITY;
        ml[r] = 0.0f;
        sum[r] = 0.0f;
      }
      for (int j = 0; j < nin; ++j) {
        const float4 tj = line[j];
        if (tj.x == -INFINITY) continue;  // uniform over the warp
#pragma unroll
        for (int r = 0; r < R; ++r) {
          // d = x - y exactly, d^2 and c = k2 d^2 as unnormalised float-float pairs
          const ff d = ff_two_sum(xr[r], -tj.z);
          const float p = d.hi * d.hi;
          const float pe = fmaf(d.hi, d.hi, -p) + 2.0f * d.hi * d.lo;
          const float ch = k2.hi * p;
          const float ce = fmaf(k2.hi, p, -ch) + fmaf(k2.hi, pe, k2.lo * p);
          // a = t - c
          const ff s = ff_two_sum(tj.x, -ch);
          const float al = s.lo + (tj.y - ce);
          if (mh[r] == -INFINITY) {
            mh[r] = s.hi;
            ml[r] = al;
            sum[r] = 1.0f;
            continue;
          }
          const ff q = ff_two_sum(s.hi, -mh[r]);
          const float dm = q.hi + (q.lo + (al - ml[r]));
          if (dm > 0.0f) {
            sum[r] = fmaf(sum[r], ex2_approx(-dm), 1.0f);
            mh[r] = s.hi;
            ml[r] = al;
          } else {
            sum[r] += ex2_approx(dm);
          }
        }
      }
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (!owns[r]) continue;
        ff z = ff_ninf();
        if (mh[r] != -INFINITY && sum[r] > 0.0f) {
          const ff m2 = ff_add_f(ff_fast_two_sum(mh[r], ml[r]), lg2_approx(sum[r]));  // log2 units
          z = ff_add_f(ff_mul(m2, ln2_ff()), mx);
        }
        if (zprev) zprev[pt[r]] = z.hi;
        float n1, d1;
        epilogue_apply(epi, bz, pt[r], z, pre[r], n1, d1);
        num += n1;
        den += d1;
      }
    }
  }
  if (epi.err) block_add2f<WARPS * 32>(num, den, epi.err + 2 * bz);
}

// ---------------------------------------------------------------------------
// Short lines (nin, nout <= 64, e.g. the 32- and 64-point axes of a 3-D
// colour grid): one warp per (line, batch entry), OPL = 1 or 2 outputs per
// lane, the line staged in the warp's shared memory, no combine across warps.
// Same arithmetic as grid_pass_f32 (speculative shifts with the exact
// fallback, float-float result, the same epilogue).
// ---------------------------------------------------------------------------
constexpr int kShortWarps = 8, kShortMax = 64;

// The log-sum-exp of one short line (nin <= 64) for OPL outputs per lane: v0,
// v1 the line values at lane and lane + 32 (float-float), y0, y1 their
// coordinates, xq the lane's output coordinates, zp its speculative shifts
// (natural units; used when spec).  The line is staged, shifted by its maximum
// mx, in the warp's sl[64]; the shifts are tried first and an exact max sweep
// redoes the line when any owned sum leaves [2^-90, 2^100].  Returns z = log
// sum (float-float) per output, -inf for an empty line.  Warp-collective.
template <int OPL>
__device__ __forceinline__ void short_line_lse(ff v0, ff v1, float y0, float y1, int nin, const float* xq,
                                               const float* zp, bool spec, const bool* owns, float k2,
                                               float2* sl, ff* z) {
  const int lane = threadIdx.x & 31;
  const float mx = warp_maxf(fmaxf(v0.hi, v1.hi));
#pragma unroll
  for (int q = 0; q < OPL; ++q) z[q] = ff_ninf();
  if (mx == -INFINITY) return;  // b = 0 on the whole line: every sum is empty
  auto stage = [&](ff v) { return (v.hi == -INFINITY) ? -INFINITY : ((v.hi - mx) + v.lo) * kLog2e; };
  __syncwarp();
  sl[lane] = make_float2(stage(v0), y0);
  if (lane + 32 < kShortMax) sl[lane + 32] = make_float2(stage(v1), y1);
  __syncwarp();
  const float nk2 = -k2;
  float m[OPL], S[OPL];
  bool exact = !spec;
  for (int attempt = 0; attempt < 2; ++attempt) {
#pragma unroll
    for (int q = 0; q < OPL; ++q) {
      m[q] = (zp[q] == -INFINITY) ? 0.0f : (zp[q] - mx) * kLog2e;
      S[q] = 0.0f;
    }
    if (exact) {
#pragma unroll
      for (int q = 0; q < OPL; ++q) m[q] = -INFINITY;
      for (int j = 0; j < nin; ++j) {
        const float2 v = sl[j];
#pragma unroll
        for (int q = 0; q < OPL; ++q) {
          const float d = xq[q] - v.y;
          m[q] = fmaxf(m[q], fmaf(nk2, d * d, v.x));
        }
      }
#pragma unroll
      for (int q = 0; q < OPL; ++q)
        if (m[q] == -INFINITY) m[q] = 0.0f;
    }
    for (int j = 0; j < nin; ++j) {
      const float2 v = sl[j];
#pragma unroll
      for (int q = 0; q < OPL; ++q) {
        const float d = xq[q] - v.y;
        S[q] += ex2_approx(fmaf(nk2, d * d, v.x - m[q]));
      }
    }
    bool bad = false;
#pragma unroll
    for (int q = 0; q < OPL; ++q)
      if (owns[q] && !exact) bad = bad || !(S[q] >= 0x1p-90f && S[q] <= 0x1p100f);
    if (__any_sync(0xffffffffu, bad) && !exact) {
      exact = true;
      continue;  // warp-uniform: redo with exact maxima
    }
    break;
  }
#pragma unroll
  for (int q = 0; q < OPL; ++q) {
    if (S[q] > 0.0f) {
      z[q] = pass_result(mx, m[q], S[q]);
    }
  }
}

// Short lines (nin, nout <= 64, e.g. the 32- and 64-point axes of a 3-D
// colour grid): one warp per (line, batch entry), OPL = 1 or 2 outputs per
// lane, the line staged in the warp's shared memory, no combine across warps.
// Same arithmetic as grid_pass_f32 (speculative shifts with the exact
// fallback, float-float result, the same epilogue).
template <int OPL>
__global__ void __launch_bounds__(kShortWarps * 32) grid_pass_f32_short(PassArgs a, Epilogue epi) {
  __shared__ float2 sl[kShortWarps][kShortMax];  // {t, y} of the warp's line
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t item = (int64_t)blockIdx.x * kShortWarps + warp;
  const int nin = a.nin, nout = a.nout, nlines = a.nlines;
  const bool live = item < (int64_t)nlines * a.nbatch;  // warp-uniform
  const int l = live ? (int)(item % nlines) : 0;
  const int64_t bz = live ? item / nlines : 0;
  float num = 0.0f, den = 0.0f;
  const float2* in = a.in + bz * (int64_t)nlines * nin;
  const int64_t base = (int64_t)l * nin;
  float* zprev = a.zprev ? a.zprev + bz * (int64_t)nout * nlines : nullptr;
  const bool spec = a.use_prev && zprev;
  // ---- prologue independent of the preceding kernel ----
  bool owns[OPL];
  int64_t my_pt[OPL];
  float zp[OPL], xq[OPL];
  EpiPre pre[OPL];
#pragma unroll
  for (int q = 0; q < OPL; ++q) {
    const int i = lane + 32 * q;
    owns[q] = live && i < nout;
    my_pt[q] = (int64_t)i * nlines + l;
    zp[q] = 0.0f;
    xq[q] = a.xo[i < nout ? i : nout - 1];
    if (owns[q]) {
      if (spec) zp[q] = zprev[my_pt[q]];
      epilogue_prefetch(epi, bz, my_pt[q], pre[q]);
    }
  }
  const float y0 = (lane < nin) ? a.yi[lane] : 0.0f, y1 = (lane + 32 < nin) ? a.yi[lane + 32] : 0.0f;
  pdl_wait();
  if (a.zero_acc && live && l == 0 && lane < 2) a.zero_acc[2 * bz + lane] = 0.0;
  pdl_launch_dependents();
  if (live) {
    const ff v0 = (lane < nin) ? load_L_ff(a, in, base + lane) : ff_ninf();
    const ff v1 = (lane + 32 < nin) ? load_L_ff(a, in, base + lane + 32) : ff_ninf();
    const float mx = warp_maxf(fmaxf(v0.hi, v1.hi));
    if (mx == -INFINITY) {
      // b = 0 on the whole line: every sum is empty
#pragma unroll
      for (int q = 0; q < OPL; ++q) {
        if (!owns[q]) continue;
        if (zprev) zprev[my_pt[q]] = -INFINITY;
        float n1, d1;
        epilogue_apply(epi, bz, my_pt[q], ff_ninf(), pre[q], n1, d1);
        num += n1;
        den += d1;
      }
    } else {
      auto stage = [&](ff v) { return (v.hi == -INFINITY) ? -INFINITY : ((v.hi - mx) + v.lo) * kLog2e; };
      sl[warp][lane] = make_float2(stage(v0), y0);
      if (lane + 32 < kShortMax) sl[warp][lane + 32] = make_float2(stage(v1), y1);
      __syncwarp();
      const float2* L = sl[warp];
      const float nk2 = -a.k2;
      float m[OPL], S[OPL];
      bool exact = !spec;
      for (int attempt = 0; attempt < 2; ++attempt) {
#pragma unroll
        for (int q = 0; q < OPL; ++q) {
          m[q] = (zp[q] == -INFINITY) ? 0.0f : (zp[q] - mx) * kLog2e;
          S[q] = 0.0f;
        }
        if (exact) {
#pragma unroll
          for (int q = 0; q < OPL; ++q) m[q] = -INFINITY;
          for (int j = 0; j < nin; ++j) {
            const float2 v = L[j];
#pragma unroll
            for (int q = 0; q < OPL; ++q) {
              const float d = xq[q] - v.y;
              m[q] = fmaxf(m[q], fmaf(nk2, d * d, v.x));
            }
          }
#pragma unroll
          for (int q = 0; q < OPL; ++q)
            if (m[q] == -INFINITY) m[q] = 0.0f;
        }
        for (int j = 0; j < nin; ++j) {
          const float2 v = L[j];
#pragma unroll
          for (int q = 0; q < OPL; ++q) {
            const float d = xq[q] - v.y;
            S[q] += ex2_approx(fmaf(nk2, d * d, v.x - m[q]));
          }
        }
        bool bad = false;
#pragma unroll
        for (int q = 0; q < OPL; ++q)
          if (owns[q] && !exact) bad = bad || !(S[q] >= 0x1p-90f && S[q] <= 0x1p100f);
        if (__any_sync(0xffffffffu, bad) && !exact) {
          exact = true;
          continue;  // warp-uniform: redo with exact maxima
        }
        break;
      }
#pragma unroll
      for (int q = 0; q < OPL; ++q) {
        if (!owns[q]) continue;
        ff z = ff_ninf();
        if (S[q] > 0.0f) {
          z = pass_result(mx, m[q], S[q]);
        }
        if (zprev) zprev[my_pt[q]] = z.hi;
        float n1, d1;
        epilogue_apply(epi, bz, my_pt[q], z, pre[q], n1, d1);
        num += n1;
        den += d1;
      }
    }
  }
  // the warps of a block may belong to different batch entries: one sum per warp
  if (epi.err && live) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      num += __shfl_xor_sync(0xffffffffu, num, o);
      den += __shfl_xor_sync(0xffffffffu, den, o);
    }
    if (lane == 0) {
      atomicAdd(epi.err + 2 * bz, (double)num);
      atomicAdd(epi.err + 2 * bz + 1, (double)den);
    }
  }
}

// Two consecutive short passes fused (axes ax and ax - 1 of the separable
// operator, each of at most 64 points, FP32).  A pass's line index is
// s Pn + P, with P over the axes before its own (row-major, Pn of them) and s
// over the already contracted axes after it.  Pass 1's line (s, P' n2 + j)
// writes output o at o nl1 + l1, which is element j of pass 2's line
// ((o S + s) Pc + P'): for a fixed group (P', s) the nin2 lines of pass 1 and
// the nout1 lines of pass 2 form a closed plane.  One CTA per (group, batch entry)
// computes pass 1 into shared memory (float-float, the value pass 1 would
// write), then pass 2 from it with pass 2's epilogue; the results equal the
// two separate passes bit for bit.  Saves a launch and the intermediate's
// round trip through global memory.
constexpr int kPlaneWarps = 32;  // a warp per line of each phase (two for lines of 33-64 points)

template <int OPL1, int OPL2>
__global__ void __launch_bounds__(kPlaneWarps * 32)
    grid_pass_f32_plane(PassArgs a1, PassArgs a2, int S, Epilogue epi) {
  extern __shared__ float2 inter[];  // [o1][nin2]: pass 1's results of the plane
  __shared__ float2 sl[kPlaneWarps][kShortMax];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = blockIdx.x;
  const int64_t bz = blockIdx.y;
  const int Pc = gridDim.x / S;  // prefixes over the axes before the pair
  const int sfx = g / Pc, Pp = g - sfx * Pc;
  const int nin1 = a1.nin, nout1 = a1.nout, nin2 = a2.nin, nout2 = a2.nout;
  const int64_t nl1 = a1.nlines, nl2 = a2.nlines;
  const float2* in = a1.in + bz * nl1 * nin1;
  float* zp1 = a1.zprev ? a1.zprev + bz * nl1 * nout1 : nullptr;
  float* zp2 = a2.zprev ? a2.zprev + bz * nl2 * nout2 : nullptr;
  const bool spec1 = a1.use_prev && zp1, spec2 = a2.use_prev && zp2;
  float xq1[OPL1], xq2[OPL2];
  bool own1[OPL1], own2[OPL2];
#pragma unroll
  for (int q = 0; q < OPL1; ++q) {
    const int i = lane + 32 * q;
    own1[q] = i < nout1;
    xq1[q] = a1.xo[i < nout1 ? i : nout1 - 1];
  }
#pragma unroll
  for (int q = 0; q < OPL2; ++q) {
    const int i = lane + 32 * q;
    own2[q] = i < nout2;
    xq2[q] = a2.xo[i < nout2 ? i : nout2 - 1];
  }
  const float y10 = (lane < nin1) ? a1.yi[lane] : 0.0f, y11 = (lane + 32 < nin1) ? a1.yi[lane + 32] : 0.0f;
  const float y20 = (lane < nin2) ? a2.yi[lane] : 0.0f, y21 = (lane + 32 < nin2) ? a2.yi[lane + 32] : 0.0f;
  pdl_wait();
  if (a1.zero_acc && g == 0 && threadIdx.x < 2) a1.zero_acc[2 * bz + threadIdx.x] = 0.0;
  pdl_launch_dependents();
  // ---- pass 1: the plane's nin2 lines ----
  for (int j = warp; j < nin2; j += kPlaneWarps) {
    const int64_t l1 = ((int64_t)sfx * Pc + Pp) * nin2 + j;
    const int64_t base = l1 * nin1;
    float zp[OPL1];
#pragma unroll
    for (int q = 0; q < OPL1; ++q) zp[q] = (spec1 && own1[q]) ? zp1[(int64_t)(lane + 32 * q) * nl1 + l1] : 0.0f;
    const ff v0 = (lane < nin1) ? load_L_ff(a1, in, base + lane) : ff_ninf();
    const ff v1 = (lane + 32 < nin1) ? load_L_ff(a1, in, base + lane + 32) : ff_ninf();
    ff z[OPL1];
    short_line_lse<OPL1>(v0, v1, y10, y11, nin1, xq1, zp, spec1, own1, a1.k2, sl[warp], z);
#pragma unroll
    for (int q = 0; q < OPL1; ++q) {
      if (!own1[q]) continue;
      const int i = lane + 32 * q;
      if (zp1) zp1[(int64_t)i * nl1 + l1] = z[q].hi;
      inter[i * nin2 + j] = make_float2(z[q].hi, z[q].lo);
    }
  }
  __syncthreads();
  // ---- pass 2: the plane's nout1 lines, from shared memory ----
  float num = 0.0f, den = 0.0f;
  for (int o = warp; o < nout1; o += kPlaneWarps) {
    const int64_t l2 = ((int64_t)o * S + sfx) * Pc + Pp;
    float zp[OPL2];
    EpiPre pre[OPL2];
    int64_t pt[OPL2];
#pragma unroll
    for (int q = 0; q < OPL2; ++q) {
      pt[q] = (int64_t)(lane + 32 * q) * nl2 + l2;
      zp[q] = (spec2 && own2[q]) ? zp2[pt[q]] : 0.0f;
      if (own2[q]) epilogue_prefetch(epi, bz, pt[q], pre[q]);
    }
    const ff v0 = (lane < nin2) ? ffl(inter[o * nin2 + lane]) : ff_ninf();
    const ff v1 = (lane + 32 < nin2) ? ffl(inter[o * nin2 + lane + 32]) : ff_ninf();
    ff z[OPL2];
    short_line_lse<OPL2>(v0, v1, y20, y21, nin2, xq2, zp, spec2, own2, a2.k2, sl[warp], z);
#pragma unroll
    for (int q = 0; q < OPL2; ++q) {
      if (!own2[q]) continue;
      if (zp2) zp2[pt[q]] = z[q].hi;
      float n1, d1;
      epilogue_apply(epi, bz, pt[q], z[q], pre[q], n1, d1);
      num += n1;
      den += d1;
    }
  }
  if (epi.err) block_add2f<kPlaneWarps * 32>(num, den, epi.err + 2 * bz);
}

// ---------------------------------------------------------------------------
// Tile shapes of the FP32 pass and the tuner that picks one per pass shape.
// ---------------------------------------------------------------------------
namespace {

struct TileShape {
  int nw, opl;
};
// entry 7 stands for the tensor-core pass (k_grid_tc3.cu), used where its
// block-stabilisation condition holds, entry 8 for the warp-per-line pass of
// short lines (nin, nout <= 64), entries 9-13 for the variants of the
// block-stabilised pass of uniform axes (k_grid_blk.cu); where they do not
// apply the first tile runs
constexpr TileShape kTiles[] = {{8, 4}, {4, 4}, {2, 4}, {1, 4}, {8, 2}, {4, 2}, {2, 2},
                                {0, 0}, {0, 0}, {0, 0}, {0, 0}, {0, 0}, {0, 0}, {0, 0}};
constexpr int kTc3Tile = 7;
constexpr int kShortTile = 8;
constexpr int kBlkTile0 = 9;  // + variant 0 .. grid_blk_variants() - 1
// A tile of 4 or 8 warps takes four lines (grid_pass_f32_ml) where there are lines
// enough to keep the GPU full of such CTAs.  Measured per pass, best tile of one
// line against best of four: 32 batches of 128 x 128 lines x inputs 23.3 and 18.8 us,
// of 64 x 64 6.7 and 5.8; but 224 lines of 56 3.2 and 3.5, 64 of 64 2.9 and 3.5, and in
// a solve 256 of 256 6.5 and 6.8, and a colour transfer's 2048 lines of 32 and 1024 of
// 64 8.5 and 8.7 ms: with 65536 inputs a pass is a chain of latencies, longer in the
// larger CTA.
constexpr int64_t kMlMinLines = 1024, kMlMinInputs = 131072;
constexpr size_t kMlSmemMax = 110 * 1024;
bool ml_ok(const PassArgs& a, int nbatch, int nw) {
  const int64_t lines = (int64_t)a.nlines * nbatch;
  return nw >= 4 && lines >= kMlMinLines && lines * a.nin >= kMlMinInputs && MlTile<8, 4>::smem(a.nin) <= kMlSmemMax;
}
bool is_blk(int t) { return t >= kBlkTile0 && t < kBlkTile0 + grid_blk_variants(); }
int blk_mask(const PassArgs& a) {
  int m = 0;
  for (int v = 0; v < grid_blk_variants(); ++v) m |= grid_blk_ok(a, v) ? (1 << v) : 0;
  return m;
}

bool short_ok(const PassArgs& a) { return a.nin <= kShortMax && a.nout <= kShortMax; }

cudaError_t launch_f32_short(const PassArgs& a, const Epilogue& epi, int nbatch, cudaStream_t s) {
  const int64_t items = (int64_t)a.nlines * nbatch;
  PassArgs b = a;
  b.nbatch = nbatch;
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3((unsigned)((items + kShortWarps - 1) / kShortWarps));
  cfg.blockDim = dim3(kShortWarps * 32);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (a.nout <= 32) return cudaLaunchKernelEx(&cfg, grid_pass_f32_short<1>, b, epi);
  return cudaLaunchKernelEx(&cfg, grid_pass_f32_short<2>, b, epi);
}
constexpr int kNumTiles = (int)(sizeof(kTiles) / sizeof(kTiles[0]));

template <int NW, int OPL>
cudaError_t launch_f32_tile(const PassArgs& a, const Epilogue& epi, int nbatch, cudaStream_t s) {
  dim3 grid((a.nout + 32 * OPL - 1) / (32 * OPL), a.nlines, nbatch);
  if (grid.y > 65535 || grid.z > 65535) return cudaErrorInvalidConfiguration;
  const size_t smem = (size_t)a.nin * sizeof(float4);
  if (smem > 48 * 1024) {
    cudaError_t e = smem_at_least(grid_pass_f32<NW, OPL>, smem);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = grid;
  cfg.blockDim = dim3(NW * 32);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, grid_pass_f32<NW, OPL>, a, epi);
}

template <int NW, int OPL>
cudaError_t launch_f32_ml(const PassArgs& a, const Epilogue& epi, int nbatch, cudaStream_t s) {
  typedef MlTile<NW, OPL> T;
  const dim3 grid((a.nout + T::kOut - 1) / T::kOut, (a.nlines + kMlLines - 1) / kMlLines, nbatch);
  if (grid.y > 65535 || grid.z > 65535) return cudaErrorInvalidConfiguration;
  const size_t smem = T::smem(a.nin);
  const cudaError_t e = smem_at_least(grid_pass_f32_ml<NW, OPL>, smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(grid_pass_f32_ml<NW, OPL>, grid, dim3(T::kThreads), smem, s, a, epi);
}

cudaError_t launch_f32(int t, const PassArgs& a, const Epilogue& epi, int nbatch, cudaStream_t s) {
  if (t == kTc3Tile && a.tc3_ok)
    return launch_grid_pass_tc3(a.in, a.logw, a.in_is_pot, a.nlines, a.nin, a.yi, a.nout, a.xo, a.inv_eps, a.k2,
                                nbatch, epi, s, a.tc_err, a.zero_acc);
  if (t == kShortTile && short_ok(a)) return launch_f32_short(a, epi, nbatch, s);
  if (is_blk(t) && grid_blk_ok(a, t - kBlkTile0)) return launch_grid_pass_blk(a, t - kBlkTile0, epi, nbatch, s);
  const bool ml = ml_ok(a, nbatch, kTiles[t < kNumTiles ? t : 0].nw);
  switch (t) {
    case 0: return ml ? launch_f32_ml<8, 4>(a, epi, nbatch, s) : launch_f32_tile<8, 4>(a, epi, nbatch, s);
    case 1: return ml ? launch_f32_ml<4, 4>(a, epi, nbatch, s) : launch_f32_tile<4, 4>(a, epi, nbatch, s);
    case 2: return launch_f32_tile<2, 4>(a, epi, nbatch, s);
    case 3: return launch_f32_tile<1, 4>(a, epi, nbatch, s);
    case 4: return ml ? launch_f32_ml<8, 2>(a, epi, nbatch, s) : launch_f32_tile<8, 2>(a, epi, nbatch, s);
    case 5: return ml ? launch_f32_ml<4, 2>(a, epi, nbatch, s) : launch_f32_tile<4, 2>(a, epi, nbatch, s);
    case 6: return launch_f32_tile<2, 2>(a, epi, nbatch, s);
    default: return launch_f32_tile<8, 4>(a, epi, nbatch, s);
  }
}

struct TuneKey {
  int dev, nlines, nin, nout, nbatch, tc3, blk;
  bool operator<(const TuneKey& o) const {
    if (tc3 != o.tc3) return tc3 < o.tc3;
    if (blk != o.blk) return blk < o.blk;
    if (dev != o.dev) return dev < o.dev;
    if (nlines != o.nlines) return nlines < o.nlines;
    if (nin != o.nin) return nin < o.nin;
    if (nout != o.nout) return nout < o.nout;
    return nbatch < o.nbatch;
  }
};

struct TuneEntry {
  int tile;
  float us[kNumTiles];  // measured time per launch of every tile (negative: not measured)
};

std::mutex g_tune_mu;
std::map<TuneKey, TuneEntry> g_tuned;
int g_autotune = 1;
int g_forced_tile = -1;
thread_local int g_tune_hold = 0;

// Times every tile on this pass shape.  The timed chain mimics a solve: each
// launch reads the previous launch's output (two buffers in turn, each with
// its own speculative-shift buffer), with the caller's coordinates and eps;
// the first values are finite.  The common case is timed: speculative shifts
// taken from the same buffer's previous result.
TuneEntry tune_tiles(const PassArgs& base, int nbatch, cudaStream_t s) {
  TuneEntry ent;
  ent.tile = 0;
  for (int t = 0; t < kNumTiles; ++t) ent.us[t] = -1.0f;
  // one buffer holds a pass input or output: the larger of the two shapes
  const size_t nel = (size_t)nbatch * base.nlines * (size_t)std::max(base.nin, base.nout);
  float2* buf[2] = {nullptr, nullptr};
  float* z[2] = {nullptr, nullptr};
  // the prox epilogue's arrays (potential, log density, log weight) and violation accumulators
  const size_t npt = (size_t)nbatch * base.nlines * (size_t)std::max(base.nin, base.nout);
  float2* pro[3] = {nullptr, nullptr, nullptr};
  double* acc = nullptr;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  // (a buffer is read as nlines x nin and written as nout x nlines values;
  // both fit, and every value read is finite: zeros first, results later)
  bool ok = true;
  for (int k = 0; k < 2 && ok; ++k)
    ok = cudaMallocAsync(&buf[k], nel * sizeof(float2), s) == cudaSuccess &&
         cudaMallocAsync(&z[k], nel * sizeof(float), s) == cudaSuccess &&
         cudaMemsetAsync(buf[k], 0, nel * sizeof(float2), s) == cudaSuccess;
  for (int k = 0; k < 3 && ok; ++k)
    ok = cudaMallocAsync(&pro[k], npt * sizeof(float2), s) == cudaSuccess &&
         cudaMemsetAsync(pro[k], 0, npt * sizeof(float2), s) == cudaSuccess;
  ok = ok && cudaMallocAsync(&acc, 2 * (size_t)nbatch * sizeof(double), s) == cudaSuccess &&
       cudaMemsetAsync(acc, 0, 2 * (size_t)nbatch * sizeof(double), s) == cudaSuccess;
  ok = ok && cudaEventCreate(&e0) == cudaSuccess && cudaEventCreate(&e1) == cudaSuccess;
  if (ok) {
    PassArgs a = base;
    a.logw = nullptr;
    a.in_is_pot = 0;
    a.zero_acc = nullptr;
    Epilogue e;
    memset(&e, 0, sizeof(e));
    e.mode = EPI_RAW;
    e.ff = 1;
    e.bstride = (int64_t)base.nlines * base.nout;
    // every other launch ends like a solve's last pass: the Table 1 KL row in
    // log form with the violation terms (the epilogue is part of the cost)
    const double eps = 1.0 / ((double)base.inv_eps.x + (double)base.inv_eps.y);
    Epilogue ep;
    memset(&ep, 0, sizeof(ep));
    ep.mode = EPI_PROX;
    ep.ff = 1;
    ep.eps = eps;
    ep.eps_ff = ff2(ff_make(eps));
    ep.inv_eps_ff = ff2(ff_make(1.0 / eps));
    ep.F.kind = UOT_DIV_KL;
    ep.F.lam = 0.5;
    ep.Fff.kind = UOT_DIV_KL;
    ep.Fff.zf = ff2(ff_make(0.5 / (0.5 + eps)));
    ep.Fff.lam = ff2(ff_make(0.5));
    ep.pot = reinterpret_cast<double*>(pro[0]);
    ep.logp = reinterpret_cast<const double*>(pro[1]);
    ep.logw = reinterpret_cast<const double*>(pro[2]);
    ep.err = acc;
    ep.bstride = ep.bstride_p = (int64_t)base.nlines * base.nout;
    // The chain alternates a solve's first pass (potentials in, raw
    // intermediate out) and last pass (that intermediate in, prox epilogue
    // out).  The potentials read by the first kind stay fixed (zeros), so
    // every launch sees bounded, finite data: feeding a pass's log-sums back
    // as potentials would scale them by 1/eps per step until they overflow,
    // and the timed kernels would then take their empty-line exits.
    int parity = 0;
    auto step = [&](int t, int use_prev) -> bool {
      a.use_prev = use_prev;
      parity ^= 1;
      if (parity) {
        a.in = pro[1];  // zero potentials (the prox epilogue only reads this array)
        a.in_is_pot = 1;
        a.logw = pro[2];
        a.zprev = z[0];
        e.out = reinterpret_cast<double*>(buf[0]);
        return launch_f32(t, a, e, nbatch, s) == cudaSuccess;
      }
      a.in = buf[0];
      a.in_is_pot = 0;
      a.logw = nullptr;
      a.zprev = z[1];
      return launch_f32(t, a, ep, nbatch, s) == cudaSuccess;
    };
    // Warm-up (brings the SM clock up before anything is timed; both shift
    // buffers get exact values), then rounds that visit every tile in turn; a
    // tile's time is its best round, so a clock or neighbour transient cannot
    // favour the tiles timed last.
    constexpr int kReps = 16, kRounds = 3, kWarm = 64;
    bool okt[kNumTiles];
    float tmin[kNumTiles];
    bool wok = step(0, 0) && step(0, 0);
    for (int r = 0; r < kWarm && wok; ++r) wok = step(0, 1);
    for (int t = 0; t < kNumTiles; ++t) {
      okt[t] = wok && (t != kTc3Tile || base.tc3_ok) && (t != kShortTile || short_ok(base)) &&
               (!is_blk(t) || grid_blk_ok(base, t - kBlkTile0));
      tmin[t] = 1e30f;
    }
    for (int round = 0; round < kRounds && wok; ++round) {
      for (int t = 0; t < kNumTiles; ++t) {
        if (!okt[t]) continue;
        bool tok = cudaEventRecord(e0, s) == cudaSuccess;
        for (int r = 0; r < kReps && tok; ++r) tok = step(t, 1);
        tok = tok && cudaEventRecord(e1, s) == cudaSuccess && cudaEventSynchronize(e1) == cudaSuccess;
        float ms = 0.0f;
        tok = tok && cudaEventElapsedTime(&ms, e0, e1) == cudaSuccess;
        if (!tok) {
          (void)cudaGetLastError();
          okt[t] = false;
          continue;
        }
        tmin[t] = std::min(tmin[t], ms * 1000.0f / kReps);
      }
    }
    // The block-stabilised variants are timed for the table but not chosen
    // automatically: the chain's fixed data never triggers their exact fallback,
    // so they rank a few percent ahead here while every solve measured runs them
    // slower (9.2 against 6.4 µs per 256 x 256 pass, and more iterations to tol).
    // uot_force_grid_tile still selects them.
    float best = 1e30f;
    for (int t = 0; t < kNumTiles; ++t) {
      if (!okt[t]) continue;
      ent.us[t] = tmin[t];
      if (!is_blk(t) && t != kShortTile && tmin[t] < best) {
        best = tmin[t];
        ent.tile = t;
      }
    }
    // The warp-per-line kernel has to win by 5% too: between passes of other tiles it can
    // take longer than in this chain of its own launches (20 batches of 93 x 57, 60 iterations:
    // 5.87 us here against 6.03 for the next best tile, but 2.24 against 1.94 ms in the solve).
    if (okt[kShortTile] && 1.05f * tmin[kShortTile] < best) {
      best = tmin[kShortTile];
      ent.tile = kShortTile;
    }
    // The chain above differs from a solve's (no prox epilogue, no potential
    // inputs), and tiles within a few percent of each other here can rank
    // differently there: the first tile is kept unless another one beats it by
    // more than 5%.
    if (okt[0] && tmin[0] <= 1.05f * best) ent.tile = 0;
  }
  (void)cudaGetLastError();
  for (int k = 0; k < 2; ++k) {
    if (buf[k]) cudaFreeAsync(buf[k], s);
    if (z[k]) cudaFreeAsync(z[k], s);
  }
  for (int k = 0; k < 3; ++k)
    if (pro[k]) cudaFreeAsync(pro[k], s);
  if (acc) cudaFreeAsync(acc, s);
  cudaStreamSynchronize(s);
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  (void)cudaGetLastError();
  return ent;
}

int pick_tile(const PassArgs& a, int nbatch, cudaStream_t s) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  if (g_forced_tile >= 0) return g_forced_tile;
  if (!g_autotune) return 0;
  TuneKey key;
  if (cudaGetDevice(&key.dev) != cudaSuccess) return 0;
  key.nlines = a.nlines;
  key.nin = a.nin;
  key.nout = a.nout;
  key.nbatch = nbatch;
  key.tc3 = a.tc3_ok;
  key.blk = blk_mask(a);
  auto it = g_tuned.find(key);
  if (it != g_tuned.end()) return it->second.tile;
  if (g_tune_hold) return 0;
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &st) != cudaSuccess || st != cudaStreamCaptureStatusNone) {
    (void)cudaGetLastError();
    return 0;
  }
  const TuneEntry ent = tune_tiles(a, nbatch, s);
  g_tuned[key] = ent;
  return ent.tile;
}

}  // namespace

int grid_set_autotune(int mode) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  const int prev = g_autotune;
  g_autotune = mode ? 1 : 0;
  return prev;
}

int grid_tc3_wanted() {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  if (g_tune_hold) return 0;
  return (g_forced_tile == kTc3Tile || (g_forced_tile < 0 && g_autotune)) ? 1 : 0;
}

int grid_autotune_enabled() {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  return g_autotune;
}

int grid_force_tile(int idx) {
  if (idx < -1 || idx >= kNumTiles) return -1;
  std::lock_guard<std::mutex> lk(g_tune_mu);
  g_forced_tile = idx;
  return 0;
}

int grid_tile_count() { return kNumTiles; }

void grid_tune_hold(int on) { g_tune_hold += on ? 1 : -1; }

std::string grid_tile_table() {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  std::string s;
  char buf[256];
  for (const auto& kv : g_tuned) {
    const TuneKey& k = kv.first;
    const TuneEntry& e = kv.second;
    if (e.tile == kTc3Tile)
      snprintf(buf, sizeof(buf), "dev%d lines=%d nin=%d nout=%d batch=%d -> tensor-core tc3;", k.dev, k.nlines, k.nin,
               k.nout, k.nbatch);
    else if (e.tile == kShortTile)
      snprintf(buf, sizeof(buf), "dev%d lines=%d nin=%d nout=%d batch=%d -> warp per line;", k.dev, k.nlines, k.nin,
               k.nout, k.nbatch);
    else if (is_blk(e.tile))
      snprintf(buf, sizeof(buf), "dev%d lines=%d nin=%d nout=%d batch=%d -> block-stabilised %s;", k.dev, k.nlines,
               k.nin, k.nout, k.nbatch, grid_blk_name(e.tile - kBlkTile0));
    else
      snprintf(buf, sizeof(buf), "dev%d lines=%d nin=%d nout=%d batch=%d -> warps=%d outputs/lane=%d;", k.dev,
               k.nlines, k.nin, k.nout, k.nbatch, kTiles[e.tile].nw, kTiles[e.tile].opl);
    s += buf;
    for (int t = 0; t < kNumTiles; ++t) {
      if (t == kTc3Tile)
        snprintf(buf, sizeof(buf), " tc3:%.2fus", e.us[t]);
      else if (t == kShortTile)
        snprintf(buf, sizeof(buf), " line:%.2fus", e.us[t]);
      else if (is_blk(t))
        snprintf(buf, sizeof(buf), " %s:%.2fus", grid_blk_name(t - kBlkTile0), e.us[t]);
      else
        snprintf(buf, sizeof(buf), " %dx%d:%.2fus", kTiles[t].nw, kTiles[t].opl, e.us[t]);
      s += buf;
    }
    s += "\n";
  }
  return s;
}

namespace {
std::atomic<int> g_precise_forced{0};

template <int R, int WARPS>
cudaError_t launch_ffp_shape(const PassArgs& a, const Epilogue& epi, int nbatch, cudaStream_t s) {
  const dim3 grid((a.nout + 32 * R - 1) / (32 * R), (a.nlines + WARPS - 1) / WARPS, nbatch);
  if (grid.y > 65535 || grid.z > 65535) return cudaErrorInvalidConfiguration;
  const size_t smem = (size_t)WARPS * a.nin * sizeof(float4);
  if (smem > 200 * 1024) return cudaErrorInvalidValue;
  if (smem > 48 * 1024) {
    cudaError_t e =
        smem_at_least(grid_pass_ffp<R, WARPS>, smem);
    if (e != cudaSuccess) return e;
  }
  grid_pass_ffp<R, WARPS><<<grid, WARPS * 32, smem, s>>>(a, epi);
  return cudaGetLastError();
}

// Launch shape from the work: two outputs per lane and four warps per CTA when
// there are warps enough to fill the GPU (several per SM), otherwise one
// output per lane (twice the warps) and one-warp CTAs.
cudaError_t launch_ffp(const PassArgs& a, const Epilogue& epi, int nbatch, cudaStream_t s) {
  constexpr int64_t kFill = 152 * 8;  // warps that keep every SM of a GB300 busy
  const int64_t lines = (int64_t)a.nlines * nbatch;
  const int64_t warps2 = lines * ((a.nout + 63) / 64);
  const bool r2 = warps2 >= kFill;
  if (!r2) return launch_ffp_shape<1, 1>(a, epi, nbatch, s);  // fewer than 2 kFill warps
  const bool four = warps2 >= 4 * kFill && (size_t)4 * a.nin * sizeof(float4) <= 96 * 1024;
  return four ? launch_ffp_shape<2, 4>(a, epi, nbatch, s) : launch_ffp_shape<2, 1>(a, epi, nbatch, s);
}
}  // namespace

int grid_force_precise(int on) { return g_precise_forced.exchange(on ? 1 : 0); }
int precise_forced() { return g_precise_forced.load(); }

// 1: fuse short pass pairs where they qualify; 0 (the default): separate passes.  Measured on
// the 64 x 32 x 32 colour grid: 61 ms fused against 45 ms separate per transfer (a plane per CTA
// leaves 88 of 152 SMs idle; separate passes overlap through programmatic dependent launch).
std::atomic<int> g_plane_mode{0};

int grid_fuse_short_pairs(int mode) { return g_plane_mode.exchange(mode); }

bool grid_plane_ok(int n1in, int n1out, int n2in, int n2out) {
  // a forced tile (uot_force_grid_tile) other than the short-line kernel keeps every pass on it
  return g_plane_mode.load() != 0 && (g_forced_tile < 0 || g_forced_tile == kShortTile) && n1in <= kShortMax &&
         n1out <= kShortMax && n2in <= kShortMax && n2out <= kShortMax;
}

cudaError_t launch_grid_pass_plane(const double* in, const double* logw, int in_is_pot, int64_t ngroups, int S,
                                   int nin1, const void* yi1, int nout1, const void* xo1, float* zprev1,
                                   int nin2, const void* yi2, int nout2, const void* xo2, float* zprev2,
                                   double eps, int nbatch, int use_prev, double* zero_acc, const Epilogue& epi,
                                   cudaStream_t s) {
  const int64_t Pc = ngroups / S;  // prefixes over the axes before the pair
  if (ngroups < 1 || S < 1 || ngroups % S != 0 || nbatch < 1 || nbatch > 65535 || ngroups > INT32_MAX ||
      Pc * std::max(nin2, nout1) * S > INT32_MAX)
    return cudaErrorInvalidConfiguration;
  PassArgs a1, a2;
  memset(&a1, 0, sizeof(a1));
  a1.in = reinterpret_cast<const float2*>(in);
  a1.logw = reinterpret_cast<const float2*>(logw);
  a1.in_is_pot = in_is_pot;
  a1.nlines = (int)(Pc * nin2 * S);
  a1.nin = nin1;
  a1.nout = nout1;
  a1.yi = (const float*)yi1;
  a1.xo = (const float*)xo1;
  a1.inv_eps = ff2(ff_make(1.0 / eps));
  a1.k2 = (float)((double)kLog2e / eps);
  a1.zprev = zprev1;
  a1.use_prev = use_prev;
  a1.zero_acc = zero_acc;
  a1.nbatch = nbatch;
  a2 = a1;
  a2.in = nullptr;
  a2.logw = nullptr;
  a2.in_is_pot = 0;
  a2.nlines = (int)(Pc * nout1 * S);
  a2.nin = nin2;
  a2.nout = nout2;
  a2.yi = (const float*)yi2;
  a2.xo = (const float*)xo2;
  a2.zprev = zprev2;
  a2.zero_acc = nullptr;
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3((unsigned)ngroups, (unsigned)nbatch);
  cfg.blockDim = dim3(kPlaneWarps * 32);
  cfg.dynamicSmemBytes = (size_t)nout1 * nin2 * sizeof(float2);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  auto kern = nout1 <= 32 ? (nout2 <= 32 ? grid_pass_f32_plane<1, 1> : grid_pass_f32_plane<1, 2>)
                          : (nout2 <= 32 ? grid_pass_f32_plane<2, 1> : grid_pass_f32_plane<2, 2>);
  cudaError_t e = smem_at_least(kern, cfg.dynamicSmemBytes);
  if (e != cudaSuccess) return e;
  prof_mark_begin(PROF_GRID_PASS, s);
  count_launches(1);
  if (nout1 <= 32)
    e = nout2 <= 32 ? cudaLaunchKernelEx(&cfg, grid_pass_f32_plane<1, 1>, a1, a2, S, epi)
                    : cudaLaunchKernelEx(&cfg, grid_pass_f32_plane<1, 2>, a1, a2, S, epi);
  else
    e = nout2 <= 32 ? cudaLaunchKernelEx(&cfg, grid_pass_f32_plane<2, 1>, a1, a2, S, epi)
                    : cudaLaunchKernelEx(&cfg, grid_pass_f32_plane<2, 2>, a1, a2, S, epi);
  if (e != cudaSuccess) return e;
  prof_mark_end(PROF_GRID_PASS, s);
  return cudaGetLastError();
}

cudaError_t launch_grid_pass(const double* in, const double* logw, int in_is_pot,
                             int nlines, int nin, const void* yi, int nout, const void* xo,
                             double eps, int nbatch, const Epilogue& epi, cudaStream_t s,
                             float* zprev, int use_prev, double* zero_acc, int tc3_ok, int* tc_err,
                             const BlkAxis* blk, int precise) {
  PassArgs a;
  a.in = reinterpret_cast<const float2*>(in);
  a.logw = reinterpret_cast<const float2*>(logw);
  a.in_is_pot = in_is_pot;
  a.nlines = nlines;
  a.nin = nin;
  a.nout = nout;
  a.yi = (const float*)yi;
  a.xo = (const float*)xo;
  a.inv_eps = ff2(ff_make(1.0 / eps));
  a.k2 = (float)((double)kLog2e / eps);
  a.zprev = zprev;
  a.use_prev = use_prev;
  a.zero_acc = zero_acc;
  a.tc3_ok = (tc3_ok && nin <= grid_pass_tc3_max_nin()) ? 1 : 0;
  a.tc_err = tc_err;
  a.nbatch = nbatch;
  a.blk = blk ? *blk : BlkAxis{0, 0.0f, 0.0f};
  if (precise || g_precise_forced.load()) {
    prof_mark_begin(PROF_GRID_PASS, s);
    count_launches(1);
    cudaError_t e = launch_ffp(a, epi, nbatch, s);
    if (e != cudaSuccess) return e;
    prof_mark_end(PROF_GRID_PASS, s);
    return cudaGetLastError();
  }
  const int tile = pick_tile(a, nbatch, s);
  const int fam = (is_blk(tile) && grid_blk_ok(a, tile - kBlkTile0)) ? PROF_GRID_BLK : PROF_GRID_PASS;
  prof_mark_begin(fam, s);
  count_launches(1);
  cudaError_t e = launch_f32(tile, a, epi, nbatch, s);
  if (e != cudaSuccess) return e;
  prof_mark_end(fam, s);
  return cudaGetLastError();
}

}  // namespace uot
