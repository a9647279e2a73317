// Many independent unbalanced OT problems between point clouds in one
// persistent launch (uneven sizes).
//
// Each CTA takes problems from a device work counter in a host-given order
// (largest n*m first) and runs the whole scaling iteration of that problem
// (eq. S, Sec. 3.3, log form of Sec. 4.3, eps-scaling of Sec. 4.4):
//
//   S_i = eps log sum_j exp((V_j - |x_i - y_j|^2)/eps) dy_j ;  U_i = prox_F1(S_i)
//   T_j = eps log sum_i exp((U_i - |x_i - y_j|^2)/eps) dx_i ;  V_j = prox_F2(T_j)
//
// until the marginal violation of the problem is <= tol or the iteration cap.
// There is no communication between work units except the atomic work counter,
// so no unit ever waits on another one.  A work unit is one CTA, or a cluster of
// 2, 4 or 8 CTAs that share a problem: CTA r of CL takes output blocks r, r + CL,
// ..., every CTA stages the whole input side, and a cluster barrier ends each
// half-step.  One CTA per problem is bounded by the largest problem as soon as
// its share of the work exceeds the others' (512 clouds of 64 to 2048 points in
// 2-D, 50 iterations: 28.5 ms, the time of the 2048 x 2048 problem on half an
// SM; clusters of 2: 20.9 ms, and 19.3 ms with the sweeps unrolled by 8 instead of
// 2; clusters of 4: 21.3, of 8: 27.9); the cluster size comes from a
// simulated schedule of the batch (batch_cluster).
//
// Per half-step the CTA stages the input side {t_j, y_j} in shared memory
// (the only per-problem data kept there, so several CTAs share an SM) and
// evaluates the outputs in blocks of 128 (4 per lane, two packed f32x2
// pairs).  A problem with fewer output blocks than warps splits the
// contraction index across warps and merges their partial (max, sum) pairs
// through shared memory, so small problems keep every warp busy.  Per-point
// state (potentials, last log-sums) is float-float in global memory (it stays
// in L2); the cost is recomputed on the fly from the coordinates; the
// log-sum-exp shift of every output is its value from the previous iteration
// of the same stage, with an exact fallback when a sum leaves [2^-90, 2^100].
//
// Two CTA sizes (8 or 16 warps) are compiled for each dimension; the first
// call with a given (d, largest n, largest m) times both on a sample of the
// batch and keeps the faster one.
#include <cooperative_groups.h>
#include <string.h>

#include <algorithm>
#include <cmath>
#include <functional>
#include <map>
#include <mutex>
#include <queue>
#include <string>
#include <vector>

#include "uot_internal.cuh"

namespace uot {
namespace {


constexpr int kOB = 128;  // outputs per warp block (4 per lane)

// Second staged vector of an input point: the remaining coordinates, paired.
template <int D>
struct Stage1 {
  typedef float2 T;  // {y1, y1}
};
template <>
struct Stage1<3> {
  typedef float4 T;  // {y1, y1, y2, y2}
};

template <int D>
__host__ __device__ constexpr size_t stage1_bytes() {
  return D == 1 ? 0 : sizeof(typename Stage1<D>::T);
}

template <int D, int NW>
size_t smem_bytes(int lmax) {
  return (size_t)lmax * (sizeof(float4) + stage1_bytes<D>()) + (size_t)NW * kOB * sizeof(float2);
}

template <int NT>
__device__ __forceinline__ float block_max(float v, float* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  float r = red[0];
#pragma unroll
  for (int w = 1; w < NT / 32; ++w) r = fmaxf(r, red[w]);
  return r;
}

template <int NT>
__device__ __forceinline__ float2 block_sum2(float a, float b, float* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  __syncthreads();
  if ((threadIdx.x & 31) == 0) {
    red[threadIdx.x >> 5] = a;
    red[NT / 32 + (threadIdx.x >> 5)] = b;
  }
  __syncthreads();
  float ra = 0.0f, rb = 0.0f;
#pragma unroll
  for (int w = 0; w < NT / 32; ++w) {
    ra += red[w];
    rb += red[NT / 32 + w];
  }
  return make_float2(ra, rb);
}

// Output coordinates of a lane's 4 outputs as f32x2 pairs (outputs 0,1 | 2,3).
struct XPairs {
  f2p A[3], B[3];
};

template <int D>
__device__ __forceinline__ void load_x(const float* __restrict__ xo, int nout, int base, int lane, XPairs& X,
                                       bool (&valid)[4]) {
  float xc[3][4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int i = base + lane + 32 * q;
    valid[q] = i < nout;
    const int ii = valid[q] ? i : nout - 1;
#pragma unroll
    for (int k = 0; k < 3; ++k) xc[k][q] = (k < D) ? xo[(int64_t)ii * D + k] : 0.0f;
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    X.A[k] = pk(xc[k][0], xc[k][1]);
    X.B[k] = pk(xc[k][2], xc[k][3]);
  }
}

// Squared distances of the pairs A, B to staged point j, times -k2, plus Tm.
template <int D>
__device__ __forceinline__ void term_exponents(const float4* st0, const typename Stage1<D>::T* st1, int j,
                                               const XPairs& X, f2p nk2, f2p MA, f2p MB, f2p& EA, f2p& EB) {
  const float4 s0 = st0[j];
  const f2p T = pk(s0.x, s0.y), Y0 = pk(s0.z, s0.w);
  f2p DA = sub2(X.A[0], Y0), DB = sub2(X.B[0], Y0);
  f2p QA = mul2(DA, DA), QB = mul2(DB, DB);
  if constexpr (D >= 2) {
    const auto s1 = st1[j];
    const f2p Y1 = pk(s1.x, s1.y);
    DA = sub2(X.A[1], Y1);
    DB = sub2(X.B[1], Y1);
    QA = fma2(DA, DA, QA);
    QB = fma2(DB, DB, QB);
    if constexpr (D == 3) {
      const f2p Y2 = pk(s1.z, s1.w);
      DA = sub2(X.A[2], Y2);
      DB = sub2(X.B[2], Y2);
      QA = fma2(DA, DA, QA);
      QB = fma2(DB, DB, QB);
    }
  }
  EA = fma2(nk2, QA, sub2(T, MA));
  EB = fma2(nk2, QB, sub2(T, MB));
}

// body(j) for j0 <= j < j1, eight at a time and the rest in pairs: problems of 64 points leave a
// warp four inputs, which a loop unrolled by eight alone takes one by one.
template <typename F>
__device__ __forceinline__ void for_inputs(int j0, int j1, F&& body) {
  int j = j0;
#pragma unroll 1
  for (; j + 8 <= j1; j += 8) {
#pragma unroll
    for (int u = 0; u < 8; ++u) body(j + u);
  }
#pragma unroll 1
  for (; j + 2 <= j1; j += 2) {
    body(j);
    body(j + 1);
  }
  if (j < j1) body(j);
}

// Log2-sum-exp of a lane's 4 outputs over staged inputs [j0, j1): with
// `exact` the per-output maxima are computed first (returned in mq), else
// the shifts in mq are used.  Returns the shifted sums in sq.
template <int D>
__device__ __forceinline__ void sweep(const float4* st0, const typename Stage1<D>::T* st1, int j0, int j1,
                                      const XPairs& X, f2p nk2, bool exact, float (&mq)[4], float (&sq)[4]) {
  const f2p zero2 = pk(0.0f, 0.0f);
  if (exact) {
    float m4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
    for_inputs(j0, j1, [&](int j) {
      f2p EA, EB;
      term_exponents<D>(st0, st1, j, X, nk2, zero2, zero2, EA, EB);
      const float2 A = upk(EA), B = upk(EB);
      m4[0] = fmaxf(m4[0], A.x);
      m4[1] = fmaxf(m4[1], A.y);
      m4[2] = fmaxf(m4[2], B.x);
      m4[3] = fmaxf(m4[3], B.y);
    });
#pragma unroll
    for (int q = 0; q < 4; ++q) mq[q] = m4[q];
  }
  const f2p MA = pk(mq[0] == -INFINITY ? 0.0f : mq[0], mq[1] == -INFINITY ? 0.0f : mq[1]);
  const f2p MB = pk(mq[2] == -INFINITY ? 0.0f : mq[2], mq[3] == -INFINITY ? 0.0f : mq[3]);
  f2p SA = zero2, SB = zero2;
  for_inputs(j0, j1, [&](int j) {
    f2p EA, EB;
    term_exponents<D>(st0, st1, j, X, nk2, MA, MB, EA, EB);
    const float2 A = upk(EA), B = upk(EB);
    SA = add2(SA, pk(ex2_approx(A.x), ex2_approx(A.y)));
    SB = add2(SB, pk(ex2_approx(B.x), ex2_approx(B.y)));
  });
  const float2 a = upk(SA), b = upk(SB);
  sq[0] = a.x;
  sq[1] = a.y;
  sq[2] = b.x;
  sq[3] = b.y;
}

// Operands of one half-step: outputs on one side of the current problem,
// inputs on the other.
struct Half {
  int nin, nout;
  const float* xo;      // [nout][D] output coordinates
  const float* yi;      // [nin][D] input coordinates
  const float2* Win;    // [nin] input potential (float-float)
  const float2* lwin;   // [nin] log weights of the inputs
  float2* Wout;         // [nout] output potential (read: old value, written: new)
  const float2* lpout;  // [nout] log densities of the outputs
  const float2* lwout;  // [nout] log weights of the outputs
  float* zprev;         // [nout] last log-sums (shift of the next half-step)
  bool use_prev, check;
  DivFF F;
  float2 eps_ff, inv_eps_ff;
  float k2;
};

// Result of one output: log-sum z = mx + ln2 (Mo + log2 So), prox update and
// violation terms.
__device__ __forceinline__ void output_epilogue(const Half& h, int i, float Mo, float So, float mx, float& num,
                                                float& den) {
  ff z = ff_ninf();
  if (Mo != -INFINITY && So > 0.0f) z = pass_result(mx, Mo, So);
  h.zprev[i] = z.hi;
  const ff eps = ffl(h.eps_ff);
  ff S = ffn_mul(z, eps);
  if (z.hi == -INFINITY) S = ff_ninf();
  const ff Un = prox_update_ff(h.F, ffl(h.lpout[i]), S, eps);
  if (h.check) {
    float va, vb;
    violation_terms_ff(ffl(h.Wout[i]), Un, S, ffl(h.lwout[i]), ffl(h.inv_eps_ff), va, vb);
    num += va;
    den += vb;
  }
  h.Wout[i] = ff2(Un);
}

// CTA `rank` of the CL that share the problem computes output blocks rank,
// rank + CL, ...; its local block b is the problem's block rank + CL b.
template <int D, int NW>
__device__ void half_step(const Half& h, int rank, int CL, float4* st0, typename Stage1<D>::T* st1, float2* part,
                          float* red, float& num, float& den) {
  constexpr int NT = NW * 32;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nin = h.nin, nout = h.nout;
  // ---- input line L_j = W_j/eps + log w_j (float-float), staged relative to its maximum ----
  float mx = -INFINITY;
  for (int j = tid; j < nin; j += NT) {
    const ff L = line_value_ff(ffl(h.Win[j]), ffl(h.inv_eps_ff), ffl(h.lwin[j]));
    st0[j] = make_float4(L.hi, L.lo, 0.0f, 0.0f);  // rewritten below by the same thread
    mx = fmaxf(mx, L.hi);
  }
  mx = block_max<NT>(mx, red);
  if (mx == -INFINITY) {
    // b = 0 everywhere: every sum is empty
    for (int i = tid; i < nout; i += NT)
      if (CL == 1 || (i / kOB) % CL == rank) output_epilogue(h, i, -INFINITY, 0.0f, 0.0f, num, den);
    __syncthreads();
    return;
  }
  for (int j = tid; j < nin; j += NT) {
    const float4 v = st0[j];
    const float t = (v.x == -INFINITY) ? -INFINITY : ((v.x - mx) + v.y) * kLog2e;
    const float c0 = h.yi[(int64_t)j * D];
    st0[j] = make_float4(t, t, c0, c0);
    if constexpr (D == 2) {
      const float c1 = h.yi[(int64_t)j * D + 1];
      st1[j] = make_float2(c1, c1);
    }
    if constexpr (D == 3) {
      const float c1 = h.yi[(int64_t)j * D + 1], c2 = h.yi[(int64_t)j * D + 2];
      st1[j] = make_float4(c1, c1, c2, c2);
    }
  }
  __syncthreads();

  const f2p nk2 = pk(-h.k2, -h.k2);
  const int nblk = ((nout + kOB - 1) / kOB - rank + CL - 1) / CL;  // this CTA's blocks
  if (nblk < 1) {
    __syncthreads();
    return;
  }
  const int split = nblk >= NW ? 1 : NW / nblk;
  if (split == 1) {
    // one warp per block of 128 outputs, the whole contraction each
    for (int b = warp; b < nblk; b += NW) {
      const int base = (rank + CL * b) * kOB;
      XPairs X;
      bool valid[4];
      load_x<D>(h.xo, nout, base, lane, X, valid);
      float mq[4], sq[4];
      bool exact = !h.use_prev;
      if (!exact) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float zp = valid[q] ? h.zprev[base + lane + 32 * q] : mx;
          mq[q] = (zp == -INFINITY) ? 0.0f : (zp - mx) * kLog2e;
        }
      }
      for (int attempt = 0; attempt < 2; ++attempt) {
        sweep<D>(st0, st1, 0, nin, X, nk2, exact, mq, sq);
        bool bad = false;
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (valid[q] && !exact && !(sq[q] >= 0x1p-90f && sq[q] <= 0x1p100f)) bad = true;
        if (__any_sync(0xffffffffu, bad)) {
          exact = true;  // warp-uniform retry with exact maxima
          continue;
        }
        break;
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (valid[q]) output_epilogue(h, base + lane + 32 * q, mq[q], mq[q] == -INFINITY ? 0.0f : sq[q], mx, num, den);
    }
    __syncthreads();
    return;
  }

  // fewer blocks than warps: `split` warps share each block's contraction
  const bool active = warp < nblk * split;
  const int b = warp % nblk, r = warp / nblk;
  const int J = (nin + split - 1) / split;
  const int j0 = min(nin, r * J), j1 = min(nin, j0 + J);
  const int base = (rank + CL * b) * kOB;
  XPairs X;
  bool valid[4];
  load_x<D>(h.xo, nout, base, lane, X, valid);
  float shift[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float zp = (h.use_prev && valid[q]) ? h.zprev[base + lane + 32 * q] : mx;
    shift[q] = (zp == -INFINITY) ? 0.0f : (zp - mx) * kLog2e;
  }
  constexpr int OWN = (NW * kOB + NT - 1) / NT;  // combined outputs per thread (4)
  float Mo[OWN], So[OWN];
  bool exact = !h.use_prev;
  for (int attempt = 0; attempt < 2; ++attempt) {
    if (active) {
      float mq[4], sq[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) mq[q] = shift[q];
      sweep<D>(st0, st1, j0, j1, X, nk2, exact, mq, sq);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const bool empty = mq[q] == -INFINITY;
        part[warp * kOB + lane + 32 * q] = make_float2(empty ? 0.0f : mq[q], empty ? 0.0f : sq[q]);
      }
    }
    __syncthreads();
    bool bad = false;
#pragma unroll
    for (int u = 0; u < OWN; ++u) {
      const int o = tid + u * NT;  // output o of the CTA's nblk*128
      const int bo = o / kOB, oo = o % kOB;
      Mo[u] = -INFINITY;
      So[u] = 0.0f;
      if (bo < nblk && (rank + CL * bo) * kOB + oo < nout) {
        for (int rr = 0; rr < split; ++rr) {
          const float2 pr = part[(rr * nblk + bo) * kOB + oo];
          if (pr.y > 0.0f) Mo[u] = fmaxf(Mo[u], pr.x);
        }
        if (Mo[u] != -INFINITY) {
          for (int rr = 0; rr < split; ++rr) {
            const float2 pr = part[(rr * nblk + bo) * kOB + oo];
            if (pr.y > 0.0f) So[u] += pr.y * ex2_approx(pr.x - Mo[u]);
          }
        }
        if (!exact && !(So[u] >= 0x1p-90f && So[u] <= 0x1p100f)) bad = true;
      }
    }
    const int any_bad = __syncthreads_or(bad ? 1 : 0);
    if (any_bad && !exact) {
      exact = true;  // block-uniform retry with exact maxima
      continue;
    }
    break;
  }
#pragma unroll
  for (int u = 0; u < OWN; ++u) {
    const int o = tid + u * NT;
    const int i = (rank + CL * (o / kOB)) * kOB + o % kOB;
    if (o < nblk * kOB && i < nout) output_epilogue(h, i, Mo[u], So[u], mx, num, den);
  }
  __syncthreads();
}

// log sum_i e^{lw_i + lp_i - W_i / lam} over one side of the CTA's problem
// (entries with lp_i = -inf or W_i = -inf take no part); every thread gets
// the result.  Shifts in FP64, exponentials of shifted differences in FP32.
template <int NW>
__device__ double block_side_lse(const float2* W, const float2* lp, const float2* lw, int len, double inv_lam,
                                 double* red) {
  constexpr int NT = NW * 32;
  double mx = -kInf, sm = 0.0;
  for (int i = threadIdx.x; i < len; i += NT) {
    const float2 l = lp[i], w = W[i];
    if (l.x == -INFINITY || w.x == -INFINITY) continue;
    const float2 g = lw[i];
    const double t = ((double)g.x + (double)g.y) + ((double)l.x + (double)l.y) - ((double)w.x + (double)w.y) * inv_lam;
    if (t > mx) {
      sm = sm * (double)expf((float)(mx - t)) + 1.0;
      mx = t;
    } else {
      sm += (double)expf((float)(t - mx));
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    double m2 = __shfl_down_sync(0xffffffffu, mx, o);
    double s2 = __shfl_down_sync(0xffffffffu, sm, o);
    if (m2 > mx) {
      const double tm = mx, ts = sm;
      mx = m2;
      sm = s2;
      m2 = tm;
      s2 = ts;
    }
    if (m2 != -kInf) sm += s2 * (double)expf((float)(m2 - mx));
  }
  __syncthreads();  // red is free
  if ((threadIdx.x & 31) == 0) {
    red[threadIdx.x >> 5] = mx;
    red[NW + (threadIdx.x >> 5)] = sm;
  }
  __syncthreads();
  double M = -kInf, S = 0.0;
  for (int w = 0; w < NW; ++w) M = fmax(M, red[w]);
  if (M == -kInf) return -kInf;
  for (int w = 0; w < NW; ++w)
    if (red[w] != -kInf) S += red[NW + w] * (double)expf((float)(red[w] - M));
  return M + log(S);
}

// Barrier of the CTAs that share a problem; orders their global writes too.
template <bool kCl>
__device__ __forceinline__ void unit_sync() {
  if constexpr (kCl) cooperative_groups::this_cluster().sync();
  else __syncthreads();
}

// Translation step (uot_opts.translate; not in the paper: the translation-
// invariant formulation of Sejourne, Vialard, Peyre 2022): U += c, V -= c with
// c = lam1 lam2 / (lam1 + lam2) (log A - log B), the exact maximum of the dual
// along that direction for KL penalties; A = sum dx p e^{-U/lam1}, B = sum dy
// q e^{-V/lam2}.  The plan is unchanged.
template <int NW, bool kCl>
__device__ void translate_problem(int rank, int CL, float2* U, float2* V, const float2* lpU, const float2* lwU, const float2* lpV,
                                  const float2* lwV, int n, int m, double2 lam, double* red) {
  constexpr int NT = NW * 32;
  const double la = block_side_lse<NW>(U, lpU, lwU, n, 1.0 / lam.x, red);
  const double lb = block_side_lse<NW>(V, lpV, lwV, m, 1.0 / lam.y, red);
  const double c = (la != -kInf && lb != -kInf) ? lam.x * lam.y / (lam.x + lam.y) * (la - lb) : 0.0;
  const ff cp = ff_make(c), cn = ff_make(-c);
  unit_sync<kCl>();  // every CTA of the unit has summed the old U and V
  for (int i = threadIdx.x + rank * NT; i < n; i += NT * CL) {
    const float2 u = U[i];
    if (!isinf(u.x)) U[i] = ff2(ff_add(ffl(u), cp));
  }
  for (int j = threadIdx.x + rank * NT; j < m; j += NT * CL) {
    const float2 v = V[j];
    if (!isinf(v.x)) V[j] = ff2(ff_add(ffl(v), cn));
  }
  unit_sync<kCl>();
}

template <int D, int NW, bool kCl>
__global__ void __launch_bounds__(NW * 32, NW == 8 ? 3 : 2) batch_solve(BatchArgs a) {
  constexpr int NT = NW * 32;
  typedef typename Stage1<D>::T S1;
  extern __shared__ float4 smem4[];
  __shared__ float red[2 * NW];
  __shared__ int s_prob;
  __shared__ int s_stop;
  __shared__ double tr_red[2 * NW];
  __shared__ float2 csum;  // this CTA's violation sums, read by its cluster
  const int tid = threadIdx.x;
  int rank = 0, CL = 1;
  if constexpr (kCl) {
    rank = (int)cooperative_groups::this_cluster().block_rank();
    CL = (int)cooperative_groups::this_cluster().num_blocks();
  }
  const int lmax = a.nmax > a.mmax ? a.nmax : a.mmax;
  float4* st0 = smem4;
  S1* st1 = reinterpret_cast<S1*>(st0 + lmax);
  float2* part = reinterpret_cast<float2*>(reinterpret_cast<char*>(st0 + lmax) + (size_t)lmax * stage1_bytes<D>());
  // Shared memory of another CTA may be written once that CTA is known to run.
  if constexpr (kCl) unit_sync<kCl>();
  for (;;) {
    if (tid == 0 && rank == 0) {
      const int t = atomicAdd(a.next, 1);
      s_prob = (t < a.nprob) ? a.order[t] : -1;
      if constexpr (kCl)
        for (int r = 1; r < CL; ++r) *cooperative_groups::this_cluster().map_shared_rank(&s_prob, r) = s_prob;
    }
    unit_sync<kCl>();
    const int k = s_prob;
    if (k < 0) break;
    const int n = a.n[k], m = a.m[k];
    const int64_t xo = a.xoff[k], yo = a.yoff[k];
    const float* xk = a.x + xo * D;
    const float* yk = a.y + yo * D;
    float2* U = a.Uff + xo;
    float2* V = a.Vff + yo;
    for (int i = tid + rank * NT; i < n; i += NT * CL) U[i] = make_float2(0.0f, 0.0f);
    for (int j = tid + rank * NT; j < m; j += NT * CL) V[j] = make_float2(0.0f, 0.0f);
    unit_sync<kCl>();
    int it_final = 0;
    float err = INFINITY;
    Half h1, h2;
    h1.nin = m;
    h1.nout = n;
    h1.xo = xk;
    h1.yi = yk;
    h1.Win = V;
    h1.lwin = a.logdy + yo;
    h1.Wout = U;
    h1.lpout = a.logp + xo;
    h1.lwout = a.logdx + xo;
    h1.zprev = a.zU + xo;
    h2.nin = n;
    h2.nout = m;
    h2.xo = yk;
    h2.yi = xk;
    h2.Win = U;
    h2.lwin = a.logdx + xo;
    h2.Wout = V;
    h2.lpout = a.logq + yo;
    h2.lwout = a.logdy + yo;
    h2.zprev = a.zV + yo;
    h2.check = false;
    for (int s = 0; s <= a.nstage; ++s) {
      const int iters = (s < a.nstage) ? a.iters_per_stage : a.max_iter;
      h1.F = a.divs[((int64_t)s * a.ndiv + k) * 2];
      h2.F = a.divs[((int64_t)s * a.ndiv + k) * 2 + 1];
      h1.eps_ff = h2.eps_ff = a.eps_ff[s];
      h1.inv_eps_ff = h2.inv_eps_ff = a.inv_eps_ff[s];
      h1.k2 = h2.k2 = a.k2[s];
      for (int it = 0; it < iters; ++it) {
        const bool final_stage = (s == a.nstage);
        const bool check = final_stage && (((it + 1) % a.check_every == 0) || it == iters - 1);
        h1.use_prev = h2.use_prev = it > 0;
        h1.check = check;
        float num = 0.0f, den = 0.0f;
        half_step<D, NW>(h1, rank, CL, st0, st1, part, red, num, den);
        if (kCl) unit_sync<kCl>();
        float dn = 0.0f, dd = 0.0f;
        half_step<D, NW>(h2, rank, CL, st0, st1, part, red, dn, dd);
        if (kCl) unit_sync<kCl>();
        if (a.translate && (final_stage ? check : (it + 1) % a.check_every == 0))
          translate_problem<NW, kCl>(rank, CL, U, V, a.logp + xo, a.logdx + xo, a.logq + yo, a.logdy + yo, n, m, a.lam[k],
                                tr_red);
        if (final_stage) it_final = it + 1;
        if (check) {
          float2 tot = block_sum2<NT>(num, den, red);
          if constexpr (kCl) {  // the CTAs' sums, added in rank order by every CTA
            if (tid == 0) csum = tot;
            unit_sync<kCl>();
            tot = make_float2(0.0f, 0.0f);
            for (int r = 0; r < CL; ++r) {
              const float2 c = *cooperative_groups::this_cluster().map_shared_rank(&csum, r);
              tot.x += c.x;
              tot.y += c.y;
            }
            unit_sync<kCl>();  // csum may be written again
          }
          err = (tot.y > 0.0f) ? tot.x / tot.y : 0.0f;
          if (tid == 0) s_stop = (it > 0 && a.tol > 0.0f && err <= a.tol) ? 1 : 0;
          __syncthreads();
          if (s_stop) break;
        }
      }
    }
    for (int i = tid + rank * NT; i < n; i += NT * CL) {
      const float2 u = U[i];
      if (a.Uout64)
        a.Uout64[xo + i] = (u.x == -INFINITY) ? -kInf : (double)u.x + (double)u.y;
      else
        a.Uout[xo + i] = (u.x == -INFINITY) ? u.x : u.x + u.y;
    }
    for (int j = tid + rank * NT; j < m; j += NT * CL) {
      const float2 v = V[j];
      if (a.Vout64)
        a.Vout64[yo + j] = (v.x == -INFINITY) ? -kInf : (double)v.x + (double)v.y;
      else
        a.Vout[yo + j] = (v.x == -INFINITY) ? v.x : v.x + v.y;
    }
    if (tid == 0 && rank == 0) {
      a.iters_out[k] = it_final;
      a.err_out[k] = err;
    }
    unit_sync<kCl>();  // s_prob has been read by every thread
  }
}

// ---- variants: (dimension, warps per CTA) ----
constexpr int kVariantWarps[2] = {8, 16};

template <int D, int NW>
cudaError_t launch_variant(const BatchArgs& a, int grid, cudaStream_t s) {
  const int lmax = std::max(a.nmax, a.mmax);
  const size_t smem = smem_bytes<D, NW>(lmax);
  cudaError_t e = smem_at_least(batch_solve<D, NW, false>, smem);
  if (e != cudaSuccess) return e;
  batch_solve<D, NW, false><<<grid, NW * 32, smem, s>>>(a);
  return cudaGetLastError();
}

template <int D, int NW>
int ctas_variant(int nmax, int mmax) {
  const size_t smem = smem_bytes<D, NW>(std::max(nmax, mmax));
  int nb = 0;
  if (smem_at_least(batch_solve<D, NW, false>, smem) !=
      cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, batch_solve<D, NW, false>, NW * 32, smem) != cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  return nb;
}

cudaError_t launch_any(const BatchArgs& a, int variant, int grid, cudaStream_t s) {
  switch (a.d * 2 + variant) {
    case 2: return launch_variant<1, 8>(a, grid, s);
    case 3: return launch_variant<1, 16>(a, grid, s);
    case 4: return launch_variant<2, 8>(a, grid, s);
    case 5: return launch_variant<2, 16>(a, grid, s);
    case 6: return launch_variant<3, 8>(a, grid, s);
    case 7: return launch_variant<3, 16>(a, grid, s);
    default: return cudaErrorInvalidValue;
  }
}

int ctas_any(int d, int variant, int nmax, int mmax) {
  switch (d * 2 + variant) {
    case 2: return ctas_variant<1, 8>(nmax, mmax);
    case 3: return ctas_variant<1, 16>(nmax, mmax);
    case 4: return ctas_variant<2, 8>(nmax, mmax);
    case 5: return ctas_variant<2, 16>(nmax, mmax);
    case 6: return ctas_variant<3, 8>(nmax, mmax);
    case 7: return ctas_variant<3, 16>(nmax, mmax);
    default: return 0;
  }
}

struct BKey {
  int dev, d, nmax, mmax;
  bool operator<(const BKey& o) const {
    if (dev != o.dev) return dev < o.dev;
    if (d != o.d) return d < o.d;
    if (nmax != o.nmax) return nmax < o.nmax;
    return mmax < o.mmax;
  }
};
struct BEntry {
  int variant;
  float ms[2];
  int sample;
};
std::mutex g_bmu;
std::map<BKey, BEntry> g_btuned;
int g_bforced = -1;  // forced variant, -1: tuned
int g_cforced = 0;   // forced CTAs per problem, 0: estimated

// ---- clusters ----

// Launch configuration of clusters of CL 16-warp CTAs, and how many clusters
// the device holds at once (0: not available).
constexpr int kClWarps = 16;
template <int D>
int cluster_config(int CL, int lmax, cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, cudaStream_t s) {
  const size_t smem = smem_bytes<D, kClWarps>(lmax);
  int n = 0;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3(CL);
  cfg.blockDim = dim3(kClWarps * 32);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CL;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (smem_at_least(batch_solve<D, kClWarps, true>, smem) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&n, batch_solve<D, kClWarps, true>, &cfg) != cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  return n;
}

int cluster_count(int d, int CL, int lmax) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  return d == 1 ? cluster_config<1>(CL, lmax, cfg, attr, nullptr)
         : d == 2 ? cluster_config<2>(CL, lmax, cfg, attr, nullptr)
                  : cluster_config<3>(CL, lmax, cfg, attr, nullptr);
}

template <int D>
cudaError_t launch_cluster(const BatchArgs& a, int CL, cudaStream_t s) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  const int n = cluster_config<D>(CL, std::max(a.nmax, a.mmax), cfg, attr, s);
  if (n < 1) return cudaErrorInvalidConfiguration;
  cfg.gridDim = dim3((unsigned)(CL * std::min(n, a.nprob)));
  return cudaLaunchKernelEx(&cfg, batch_solve<D, kClWarps, true>, a);
}

// Cycles of the two half-steps of a problem on a cluster of CL CTAs: `pipe`, the sweeps, takes
// `shared` times as long where a second CTA shares the SM, `wait` (staging, barriers, merge, epilogue)
// does not.  From the time per half-step of equal 2-D problems, one and two CTAs per SM: 300
// points 6.7 and 11.8 us on one CTA, 6.2 and 9.6 on two; 1000 points 37.1 and 70.5, 21.1 and
// 38.5 (1.95 times the sweeps), eight 8.6 and 13.7 (1.75); 512 points 14.0 us, 16.1 in 3-D.
struct BatchCost {
  double pipe, wait, shared;
};
BatchCost problem_cost(int d, int n, int m, int CL) {
  BatchCost c{0.0, 0.0, CL > 4 ? 1.75 : 1.95};
  for (int h = 0; h < 2; ++h) {
    const int nout = h ? m : n, nin = h ? n : m;
    const int loc = ((nout + kOB - 1) / kOB + CL - 1) / CL;
    const int split = loc >= kClWarps ? 1 : kClWarps / loc;
    const int on_pipe = (loc * split + 3) / 4;  // sweeps on the fullest of the SM's four partitions
    c.pipe += on_pipe * std::ceil((double)nin / split) * (18.5 + 8.25 * d) + 2000.0;
    c.wait += 2500.0 + 3.0 * nin + (CL > 1 ? 2000.0 : 0.0);
  }
  return c;
}

// Time at which the last problem ends: queue order, `groups` sets of SMs that hold up to
// `slots` (1 or 2) problems each, the next problem into the slot that becomes free; two problems
// of a group take turns on its pipes.  Where the first problems fill more than a slot per
// group, neighbours in the queue share one (300 clouds of 64 to 2048 points last as long as the
// largest two together).
double batch_end(const std::vector<BatchCost>& jobs, int groups, int slots) {
  struct Group {
    int job[2] = {-1, -1};
    double left[2] = {0.0, 0.0};  // fraction of the job
    double at = 0.0, next = 0.0;
  };
  std::vector<Group> g(groups);
  typedef std::pair<double, int> Event;
  std::priority_queue<Event, std::vector<Event>, std::greater<Event>> events;
  const int njobs = (int)jobs.size();
  int queued = 0;
  double end = 0.0;
  auto duration = [&](const Group& q, int u) {
    const BatchCost& c = jobs[q.job[u]];
    return (q.job[0] >= 0 && q.job[1] >= 0 ? c.shared : 1.0) * c.pipe + c.wait;
  };
  auto plan = [&](int i) {
    Group& q = g[i];
    q.next = kInf;
    for (int u = 0; u < 2; ++u)
      if (q.job[u] >= 0) q.next = std::min(q.next, q.at + q.left[u] * duration(q, u));
    if (q.next < kInf) events.push(Event(q.next, i));
  };
  const int pairs = std::max(0, std::min(njobs, groups * slots) - groups);
  for (int i = 0; i < groups; ++i)
    for (int u = 0; u < (i < pairs ? 2 : 1) && queued < njobs; ++u) {
      g[i].job[u] = queued++;
      g[i].left[u] = 1.0;
    }
  for (int i = 0; i < groups; ++i) plan(i);
  while (!events.empty()) {
    const Event e = events.top();
    events.pop();
    Group& q = g[e.second];
    double todo[2], time[2];
    for (int u = 0; u < 2; ++u) {
      time[u] = q.job[u] >= 0 ? duration(q, u) : 0.0;
      todo[u] = q.job[u] >= 0 ? q.left[u] * time[u] : kInf;
    }
    const double step = std::min(todo[0], todo[1]);  // (not from the clock: its rounding could end no job)
    q.at = end = e.first;
    for (int u = 0; u < 2; ++u) {
      if (q.job[u] < 0) continue;
      if (todo[u] > step * (1.0 + 1e-9)) {
        q.left[u] -= step / time[u];
        continue;
      }
      q.job[u] = queued < njobs ? queued++ : -1;
      q.left[u] = 1.0;
    }
    plan(e.second);
  }
  return end;
}

// Times both CTA sizes on a sample of the batch: every (nprob/S)-th problem
// of the size-ordered queue, six iterations at the first eps, no tolerance
// stop.  S = 8 problems per SM, so that the queue matters: with two per SM every problem starts
// at once, the largest sets the time, and 8 warps were taken for half of the batches where 16 are
// 2 to 25% faster (1000 clouds of 64 to 2048 points, 3-D: 36.0 against 28.7 ms) and 16 where 8
// are 10% faster (4096 of 200 to 300).  The sample's outputs land in the caller's output and state buffers,
// which the full solve overwrites afterwards.
BEntry tune_batch(const BatchArgs& full, const int* h_order, cudaStream_t s) {
  BEntry ent;
  ent.variant = 0;
  ent.ms[0] = ent.ms[1] = -1.0f;
  const int sms = sm_count();
  const int S = std::min(full.nprob, std::max(1, 8 * sms));
  ent.sample = S;
  std::vector<int> samp(S);
  for (int t = 0; t < S; ++t) samp[t] = h_order[(int64_t)t * full.nprob / S];
  int* d_samp = nullptr;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  bool ok = cudaMallocAsync(&d_samp, S * sizeof(int), s) == cudaSuccess &&
            cudaMemcpyAsync(d_samp, samp.data(), S * sizeof(int), cudaMemcpyHostToDevice, s) == cudaSuccess &&
            cudaEventCreate(&e0) == cudaSuccess && cudaEventCreate(&e1) == cudaSuccess;
  if (ok) {
    BatchArgs a = full;
    a.nprob = S;
    a.order = d_samp;
    a.nstage = 0;
    a.max_iter = 6;
    a.tol = 0.0f;
    a.check_every = 1 << 30;
    a.translate = 0;
    float best = 1e30f;
    for (int v = 0; v < 2; ++v) {
      const int per = ctas_any(a.d, v, a.nmax, a.mmax);
      if (per < 1) continue;
      const int grid = std::min(S, per * sms);
      float tmin = 1e30f;
      bool vok = true;
      for (int rep = 0; rep < 3 && vok; ++rep) {  // the first run warms up
        vok = cudaMemsetAsync(a.next, 0, sizeof(int), s) == cudaSuccess && cudaEventRecord(e0, s) == cudaSuccess &&
              launch_any(a, v, grid, s) == cudaSuccess && cudaEventRecord(e1, s) == cudaSuccess &&
              cudaEventSynchronize(e1) == cudaSuccess;
        float ms = 0.0f;
        vok = vok && cudaEventElapsedTime(&ms, e0, e1) == cudaSuccess;
        if (vok && rep > 0) tmin = std::min(tmin, ms);
      }
      if (!vok) {
        (void)cudaGetLastError();
        continue;
      }
      ent.ms[v] = tmin;
      if (tmin < best) {
        best = tmin;
        ent.variant = v;
      }
    }
    // the 8-warp CTA stays unless the other is more than 3% faster
    if (ent.ms[0] > 0.0f && ent.ms[0] <= 1.03f * best) ent.variant = 0;
  }
  (void)cudaGetLastError();
  if (d_samp) cudaFreeAsync(d_samp, s);
  cudaStreamSynchronize(s);
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  (void)cudaGetLastError();
  return ent;
}

}  // namespace

int batch_force_warps(int warps) {
  std::lock_guard<std::mutex> lk(g_bmu);
  if (warps == 0) {
    g_bforced = -1;
    return 0;
  }
  for (int v = 0; v < 2; ++v) {
    if (kVariantWarps[v] == warps) {
      g_bforced = v;
      return 0;
    }
  }
  return -1;
}

int batch_force_cluster(int ctas) {
  if (ctas != 0 && ctas != 1 && ctas != 2 && ctas != 4 && ctas != 8) return -1;
  std::lock_guard<std::mutex> lk(g_bmu);
  g_cforced = ctas;
  return 0;
}

int batch_pick_variant(const BatchArgs& a, const int* h_order, cudaStream_t s) {
  std::lock_guard<std::mutex> lk(g_bmu);
  if (g_bforced >= 0) return g_bforced;
  BKey key;
  if (cudaGetDevice(&key.dev) != cudaSuccess) return 0;
  key.d = a.d;
  key.nmax = a.nmax;
  key.mmax = a.mmax;
  auto it = g_btuned.find(key);
  if (it != g_btuned.end()) return it->second.variant;
  if (!grid_autotune_enabled()) return 0;
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &st) != cudaSuccess || st != cudaStreamCaptureStatusNone) {
    (void)cudaGetLastError();
    return 0;
  }
  const BEntry ent = tune_batch(a, h_order, s);
  g_btuned[key] = ent;
  return ent.variant;
}

std::string batch_tune_table() {
  std::lock_guard<std::mutex> lk(g_bmu);
  std::string s;
  char buf[256];
  for (const auto& kv : g_btuned) {
    snprintf(buf, sizeof(buf), "dev%d batch d=%d nmax=%d mmax=%d sample=%d -> warps=%d; 8:%.3fms 16:%.3fms\n",
             kv.first.dev, kv.first.d, kv.first.nmax, kv.first.mmax, kv.second.sample,
             kVariantWarps[kv.second.variant], kv.second.ms[0], kv.second.ms[1]);
    s += buf;
  }
  return s;
}

// CTAs per problem: the cluster size whose schedule ends earliest (batch_end), the smaller one
// within 3%, and none of more CTAs than the largest side has output blocks.  One CTA where no
// problem is larger than a fourth of an SM's average load: clusters could shorten such a batch
// by little.  A first form of the estimate counted every CTA as sharing its SM and took two CTAs
// for 152 problems of 300 points, 1.60 ms where one CTA takes 1.31.
int batch_cluster(int d, int nmax, int mmax, const int* n, const int* m, const int* order, int nprob) {
  {
    std::lock_guard<std::mutex> lk(g_bmu);
    if (g_cforced > 0) return g_cforced;
    if (g_bforced >= 0) return 1;
  }
  const int sms = sm_count(), slots = std::min(2, ctas_any(d, 1, nmax, mmax));
  if (slots < 1 || sms < 1) return 1;
  std::vector<BatchCost> jobs(nprob);
  int best = 1;
  double best_t = 0.0;
  for (int CL : {1, 2, 4, 8}) {
    if (CL > (std::max(nmax, mmax) + kOB - 1) / kOB) break;
    const int groups = CL == 1 ? sms : cluster_count(d, CL, std::max(nmax, mmax)) / slots;
    if (groups < 1) continue;
    double sum = 0.0, most = 0.0;
    for (int t = 0; t < nprob; ++t) {
      const int k = order[t];
      jobs[t] = problem_cost(d, n[k], m[k], CL);
      sum += jobs[t].pipe;
      most = std::max(most, jobs[t].pipe);
    }
    if (CL == 1 && most <= sum / sms / 4.0) return 1;
    const double end = batch_end(jobs, groups, slots);
    if (CL == 1 || end < 0.97 * best_t) {
      best_t = end;
      best = CL;
    }
  }
  return best;
}

cudaError_t launch_batch_cluster(const BatchArgs& a, int CL, cudaStream_t s) {
  count_launches(1);
  return a.d == 1 ? launch_cluster<1>(a, CL, s) : a.d == 2 ? launch_cluster<2>(a, CL, s) : launch_cluster<3>(a, CL, s);
}

int batch_ctas_per_sm(int d, int variant, int nmax, int mmax) { return ctas_any(d, variant, nmax, mmax); }

cudaError_t launch_batch(const BatchArgs& a, int variant, int grid, cudaStream_t s) {
  count_launches(1);
  return launch_any(a, variant, grid, s);
}

}  // namespace uot
