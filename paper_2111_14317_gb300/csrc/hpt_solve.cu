// Consolidated Euler+Newton solve (Section 6, eq. (11), affine form) and the
// per-path step control, plus the small kernels around them (state init,
// active count, Newton polish at t = 1, implicit-function adjoint).
//
// The scratch holds D_z H = H_y diag(y) (z = log y).  H_y d = r is solved as
// D_z H w = r, d = diag(y) w: the diag(1/y) scaling of op. 3 of Algorithm 2
// costs n products per path here instead of n^2 in the evaluation.
//
// Three solves.  FP64 (step, polish, adjoint, re-solve): LU in shared memory,
// hpt_lu64.cuh.  FP32, n <= 16: Gauss-Jordan with the rows in registers
// (gj_path).  FP32, n > 16 (group_solve): a group of G lanes owns one path and
// every lane holds R rows of [D_z H | -H_tau | -H] in registers (rows lane,
// lane + G, ...), n <= G R.  The rows are equilibrated by exact powers of two,
// then Gaussian elimination with partial pivoting runs over a run-time column
// loop.  Rows are "shifted": after column j is eliminated every live row moves
// one register to the left, so the current column is always register 0 and the
// loop body uses static register indices only.  The pivot (largest |.|^2; ties
// to the lowest row, as LAPACK's getrf) comes from one packed integer max per
// butterfly level; its owner writes the pivot row, relative to column j, into
// row j of the group's shared-memory factor U, from where every lane reads it.
// Back substitution works column by column on U.  Two right-hand sides
// [-H_tau, -H] give the Euler direction dE and the Newton direction dN from one
// factorisation, in every form.
#include <math.h>

#include <algorithm>

#include "hpt_cx.cuh"
#include "hpt_fx.cuh"
#include "hpt_internal.h"
#include "hpt_lu64.cuh"

namespace hpt {
namespace {

// Pivot key: |a|^2 with the low five mantissa bits replaced
// by (31 - row), so that one integer max picks the largest magnitude, ties to
// the lowest row.  Rows already used as pivots get key 0.
__device__ __forceinline__ unsigned pivot_key(float f, bool used, int row) {
  if (used) return 0u;
  if (!(f == f)) f = 0.f;   // NaN rows stay eligible; the pivot test flags them
  return (__float_as_uint(f) & ~31u) | (unsigned)(31 - row);
}

// Shared memory of one group: U (NC rows of LD complex; LD even keeps rows
// 16-byte aligned, LD - 1 odd keeps the column reads of the back substitution
// on distinct banks) then the column scales (NC reals), padded so that
// consecutive groups start 8 banks apart.
template <int NC>
struct GroupSmem {
  static constexpr int LD = NC + 4;
  static constexpr int raw_words = NC * LD * 2 + NC;
  static constexpr int words = (raw_words + 31) / 32 * 32 + 8;
  static constexpr int bytes = words * 4;
};

constexpr int kSolveThreads = 128;

// Rows of one path for a group: lane l holds rows l + G s, s < R, as
// a[s][0..NC) plus the two right-hand sides.
template <int G, int R>
struct PathRows {
  static constexpr int NC = G * R;
  cx<float> a[R][NC];
  cx<float> bE[R], bN[R];
};


// Loads the rows of [D_z H | -H_tau | -H] of one path; returns whether every
// entry is finite (group-uniform).
template <int G, int R>
__device__ __forceinline__ bool load_rows(int n, int nmax, const void* ext, int64_t q, bool valid,
                                          PathRows<G, R>& P) {
  constexpr int NC = G * R;
  const int lane = threadIdx.x & (G - 1);
  float chk = 0.f;
#pragma unroll
  for (int s = 0; s < R; ++s) {
    const int r = lane + G * s;
    const bool have = valid && r < n;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      P.a[s][c] = mk<float>(0, 0);
      if (have && c < n) {
        P.a[s][c] = ld<float>(ext, ext_index(q, r, c, nmax));
        chk += t_abs(P.a[s][c].x) + t_abs(P.a[s][c].y);
      }
    }
    P.bE[s] = mk<float>(0, 0);
    P.bN[s] = mk<float>(0, 0);
    if (have) {
      const cx<float> ht = ld<float>(ext, ext_index(q, r, n, nmax));
      const cx<float> h = ld<float>(ext, ext_index(q, r, n + 1, nmax));
      P.bE[s] = mk<float>(-ht.x, -ht.y);
      P.bN[s] = mk<float>(-h.x, -h.y);
      chk += t_abs(P.bE[s].x) + t_abs(P.bE[s].y) + t_abs(P.bN[s].x) + t_abs(P.bN[s].y);
    }
  }
  // a sum of magnitudes is finite iff every entry is
  const unsigned ball = __ballot_sync(0xffffffffu, isfinite(chk));
  const unsigned seg = group_mask<G>();
  return (ball & seg) == seg;
}

// 32-lane groups (one path per warp) would load every entry of the
// position-interleaved scratch from its own 32-byte sector.  Instead the
// block's four paths (consecutive positions q0..q0+3 of one tile, so one n)
// are staged cooperatively: four threads read the same entry of the four
// paths, one sector, and write it to the path's group region in shared memory
// as rows of kStageLD entries (odd, so the row reads below hit distinct
// banks).  Only paths with act set are read.  Call with every thread of the
// block between two block barriers.
constexpr int kStageLD = 35;
__device__ __forceinline__ void stage_block_rows(int n, int nmax, const void* __restrict__ ext, int64_t q0, bool act,
                                                 unsigned char* smem, int region_bytes) {
  if (!act) return;   // act: path (threadIdx.x & 3) of the block is to be solved
  const int i = threadIdx.x & 3;
  float2* region = (float2*)(smem + i * region_bytes);
  const int np2 = n + 2, total = n * np2;
  for (int e = threadIdx.x >> 2; e < total; e += 32) {
    const int k = e / np2, u = e - k * np2;
    region[k * kStageLD + u] = ((const float2*)ext)[ext_index(q0 + i, k, u, nmax)];
  }
}

// load_rows for a 32-lane group from its staged region (lane r = row r).
__device__ __forceinline__ bool load_rows_staged(int n, const unsigned char* region, bool valid, PathRows<32, 1>& P) {
  const float2* rg = (const float2*)region;
  const int r = threadIdx.x & 31;
  const bool have = valid && r < n;
  float chk = 0.f;
#pragma unroll
  for (int c = 0; c < 32; ++c) {
    P.a[0][c] = mk<float>(0, 0);
    if (have && c < n) {
      const float2 v = rg[r * kStageLD + c];
      P.a[0][c] = mk<float>(v.x, v.y);
      chk += t_abs(P.a[0][c].x) + t_abs(P.a[0][c].y);
    }
  }
  P.bE[0] = mk<float>(0, 0);
  P.bN[0] = mk<float>(0, 0);
  if (have) {
    const float2 ht = rg[r * kStageLD + n], h = rg[r * kStageLD + n + 1];
    P.bE[0] = mk<float>(-ht.x, -ht.y);
    P.bN[0] = mk<float>(-h.x, -h.y);
    chk += t_abs(P.bE[0].x) + t_abs(P.bE[0].y) + t_abs(P.bN[0].x) + t_abs(P.bN[0].y);
  }
  __syncwarp();   // every row is in registers before the solve writes U over the region
  return __all_sync(0xffffffffu, isfinite(chk));
}

// Solves the path held in P (n <= G R) with equilibration and partial
// pivoting.  Returns false (group-uniform) when a pivot is zero or not
// finite; cond receives max |u_jj| / min |u_jj|.  On return lane l holds
// solution components l + G s in xE[s], xN[s].  sm is the group's shared
// memory (GroupSmem).
template <int G, int R>
__device__ __forceinline__ bool group_solve(int n, PathRows<G, R>& P, cx<float> (&xE)[R], cx<float> (&xN)[R],
                                            float& cond, unsigned char* sm) {
  constexpr int NC = G * R, LD = GroupSmem<NC>::LD;
  cx<float>* U = (cx<float>*)sm;
  float* dcol = (float*)(sm + NC * LD * sizeof(cx<float>));
  const int lane = threadIdx.x & (G - 1);

  // equilibration: rows, then columns, by exact powers of two
#pragma unroll
  for (int s = 0; s < R; ++s) {
    float m = 0.f;
#pragma unroll
    for (int c = 0; c < NC; ++c) m = t_max(m, cmag(P.a[s][c]));
    const float dr = pow2_inv(m);
#pragma unroll
    for (int c = 0; c < NC; ++c) P.a[s][c] = cscale(P.a[s][c], dr);
    P.bE[s] = cscale(P.bE[s], dr);
    P.bN[s] = cscale(P.bN[s], dr);
  }
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    if (c < n) {
      float m = 0.f;
#pragma unroll
      for (int s = 0; s < R; ++s) m = t_max(m, cmag(P.a[s][c]));
#pragma unroll
      for (int o = G / 2; o > 0; o >>= 1) m = t_max(m, __shfl_xor_sync(0xffffffffu, m, o, G));
      const float d = pow2_inv(m);
#pragma unroll
      for (int s = 0; s < R; ++s) P.a[s][c] = cscale(P.a[s][c], d);
      if (lane == 0) dcol[c] = d;
    }
  }

  bool used[R];
#pragma unroll
  for (int s = 0; s < R; ++s) used[s] = lane + G * s >= n;
  bool ok = true;
  float pmax = 0, pmin = 0;   // extreme |u_jj|^2
#pragma unroll 1
  for (int j = 0; j < n; ++j) {
    unsigned key = 0u;
#pragma unroll
    for (int s = 0; s < R; ++s) key = max(key, pivot_key(abs2(P.a[s][0]), used[s], lane + G * s));
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) key = max(key, __shfl_xor_sync(0xffffffffu, key, o, G));
    const int br = 31 - (int)(key & 31u);
    if (lane == (br & (G - 1))) {
      // the owner's slot chosen entry by entry (a per-slot conditional store
      // would be turned into a dynamically indexed, local-memory row)
      const int bs = br / G;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        cx<float> v = P.a[0][c];
#pragma unroll
        for (int s = 1; s < R; ++s) v = (bs == s) ? P.a[s][c] : v;
        U[j * LD + c] = v;
      }
      cx<float> e = P.bE[0], f = P.bN[0];
#pragma unroll
      for (int s = 1; s < R; ++s) {
        e = (bs == s) ? P.bE[s] : e;
        f = (bs == s) ? P.bN[s] : f;
      }
      U[j * LD + NC] = e;
      U[j * LD + NC + 1] = f;
#pragma unroll
      for (int s = 0; s < R; ++s) used[s] = used[s] || (bs == s);
    }
    __syncwarp();
    const cx<float> pj = U[j * LD];
    const float p2 = abs2(pj);
    if (!(p2 > 0.f) || !isfinite(p2)) ok = false;
    pmax = j == 0 ? p2 : t_max(pmax, p2);
    pmin = j == 0 ? p2 : t_min(pmin, p2);
    const float rp = t_rcp(p2);   // one reciprocal per pivot, shared by all rows
    // multipliers; rows already used get 0, so the unpredicated update below
    // only shifts them (their values are no longer read)
    cx<float> l[R];
#pragma unroll
    for (int s = 0; s < R; ++s) l[s] = used[s] ? mk<float>(0, 0) : cmul_conj_scale(P.a[s][0], pj, rp);
    // shifted update: a[c-1] = a[c] - l u_{j, j+c} over the live width, in
    // chunks of four columns behind one warp-uniform branch each (the
    // columns of the last chunk beyond the live width are updated too; they
    // are never read again)
    const int lim = n - 1 - j;
#pragma unroll
    for (int c0 = 1; c0 < NC; c0 += 4) {
      if (c0 <= lim) {
#pragma unroll
        for (int c = c0; c < c0 + 4; ++c) {
          if (c < NC) {
            const cx<float> u = U[j * LD + c];
#pragma unroll
            for (int s = 0; s < R; ++s) P.a[s][c - 1] = csub_mul(P.a[s][c], l[s], u);
          }
        }
      }
    }
    const cx<float> uE = U[j * LD + NC], uN = U[j * LD + NC + 1];
#pragma unroll
    for (int s = 0; s < R; ++s) {
      P.bE[s] = csub_mul(P.bE[s], l[s], uE);
      P.bN[s] = csub_mul(P.bN[s], l[s], uN);
    }
  }
  __syncwarp();
  // back substitution on U (row i holds u_{i, i+c} at c, then the two
  // right-hand sides); lane l carries the right-hand sides of rows l + G s
  cx<float> rE[R], rN[R];
#pragma unroll
  for (int s = 0; s < R; ++s) {
    const int i = lane + G * s;
    rE[s] = i < n ? U[i * LD + NC] : mk<float>(0, 0);
    rN[s] = i < n ? U[i * LD + NC + 1] : mk<float>(0, 0);
    xE[s] = mk<float>(0, 0);
    xN[s] = mk<float>(0, 0);
  }
#pragma unroll 1
  for (int j = n - 1; j >= 0; --j) {
    const cx<float> ujj = U[j * LD];
    const int js = j / G;
    cx<float> vE = rE[0], vN = rN[0];
#pragma unroll
    for (int s = 1; s < R; ++s)
      if (s == js) { vE = rE[s]; vN = rN[s]; }
    vE = shfl<float, G>(vE, j & (G - 1));
    vN = shfl<float, G>(vN, j & (G - 1));
    const float ru = t_rcp(abs2(ujj));
    const cx<float> xe = cmul_conj_scale(vE, ujj, ru), xn = cmul_conj_scale(vN, ujj, ru);
#pragma unroll
    for (int s = 0; s < R; ++s) {
      const int i = lane + G * s;
      if (i == j) { xE[s] = xe; xN[s] = xn; }
      if (i < j) {
        const cx<float> u = U[i * LD + (j - i)];
        rE[s] = csub_mul(rE[s], u, xe);
        rN[s] = csub_mul(rN[s], u, xn);
      }
    }
  }
#pragma unroll
  for (int s = 0; s < R; ++s) {
    const int i = lane + G * s;
    if (i < n) {
      const float d = dcol[i];
      xE[s] = cscale(xE[s], d);
      xN[s] = cscale(xN[s], d);
    }
  }
  __syncwarp();   // the group's shared memory is reused by its next solve
  cond = pmin > 0.f ? t_sqrt(pmax / pmin) : INFINITY;
  return ok;
}

// Step control of one path (all lanes of its group), given the directions:
// accept/reject, then the next prediction (Euler, or with prm.predictor = 1
// and two accepted points the cubic Hermite interpolant through them; the
// point being replaced by an accept is kept in the state's *_prev arrays).
// TS is the state precision; lane l handles the variables l + G s.
// The state a step reads, loaded ahead of the solve so that its loads are in
// flight together with the Jacobian's (the Hermite predictor's extra fields
// are read only when used).
template <typename TS, int R>
struct StepState {
  cx<TS> y[R], yacc[R], dEacc[R];
  double tau, dtau, tauacc;
  int32_t steps, accepts, rejects, streak;
};

template <typename TS, int G, int R>
__device__ __forceinline__ void load_step_state(int n, int64_t path, size_t vbase, const hpt_paths& S,
                                                StepState<TS, R>& Q) {
  const int lane = threadIdx.x & (G - 1);
#pragma unroll
  for (int s = 0; s < R; ++s) {
    const int j = lane + G * s;
    const bool mine = j < n;
    const size_t vi = vbase + j;
    Q.y[s] = mine ? ld<TS>(S.y, vi) : mk<TS>(0, 0);
    Q.yacc[s] = mine ? ld<TS>(S.y_acc, vi) : mk<TS>(0, 0);
    Q.dEacc[s] = mine ? ld<TS>(S.dE_acc, vi) : mk<TS>(0, 0);
  }
  Q.tau = S.tau[path];
  Q.dtau = S.dtau[path];
  Q.tauacc = S.tau_acc[path];
  Q.steps = S.steps[path];
  Q.accepts = S.accepts[path];
  Q.rejects = S.rejects[path];
  Q.streak = S.streak[path];
}

// Largest modulus over a group's entries: the largest square first (bit
// patterns of non-negative doubles compare as integers) and one square root,
// since each hypot costs some 25 instructions of the FP64 pipe; squares
// outside [1e-280, 1e280] take the hypots.  NaN entries are the caller's to
// find.
template <int G, int R>
__device__ __forceinline__ double group_max_abs(const cx<double> (&v)[R], int n, unsigned gmask) {
  const int lane = threadIdx.x & (G - 1);
  unsigned long long m2 = 0;
#pragma unroll
  for (int s = 0; s < R; ++s)
    if (lane + G * s < n) m2 = max(m2, (unsigned long long)__double_as_longlong(abs2(v[s])));
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) m2 = max(m2, __shfl_xor_sync(gmask, m2, o, G));
  const double sq = __longlong_as_double((long long)m2);
  if (m2 == 0 || (sq > 1e-280 && sq < 1e280)) return sqrt(sq);
  double m = 0.0;
#pragma unroll
  for (int s = 0; s < R; ++s)
    if (lane + G * s < n) m = fmax(m, cabs_t(v[s]));
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(gmask, m, o, G));
  return m;
}

// Whether a modulus lies outside (1/bound, bound) (or is NaN); FP64 by
// squares where these cannot leave the range.
template <typename TS>
__device__ __forceinline__ bool outside_bound(cx<TS> v, double bound) {
  if constexpr (sizeof(TS) == 8) {
    if (bound < 1e140) {
      const double m2 = abs2(v), b2 = bound * bound;
      return !(m2 < b2) || !(m2 * b2 > 1.0);
    }
  }
  const TS m = cabs_t(v);
  return !(m < (TS)bound) || !(m > (TS)(1.0 / bound));
}

template <typename TS, int G, int R>
__device__ __forceinline__ void update_path(int n, int64_t path, size_t vbase, int32_t status, bool ok,
                                            const cx<TS> (&wE)[R], const cx<TS> (&wN)[R], const hpt_paths& S,
                                            const hpt_params& prm, const StepState<TS, R>& Q) {
  const int lane = threadIdx.x & (G - 1);
  const unsigned gmask = group_mask<G>();
  cx<TS> y[R], yacc[R], dEacc[R], xE[R], xN[R];
  bool solfin = true;
  TS ny = TS(0), nd = TS(0);
#pragma unroll
  for (int s = 0; s < R; ++s) {
    const int j = lane + G * s;
    const bool mine = j < n;
    y[s] = Q.y[s];
    yacc[s] = Q.yacc[s];
    dEacc[s] = Q.dEacc[s];
    // the scratch holds D_z H = H_y diag(y): the solve gave diag(1/y) times
    // the directions
    xE[s] = cmul(y[s], wE[s]);
    xN[s] = cmul(y[s], wN[s]);
    if (mine) {
      solfin = solfin && finite(xE[s]) && finite(xN[s]);
      if constexpr (sizeof(TS) == 4) {
        ny = t_max(ny, cabs_t(y[s]));
        nd = t_max(nd, cabs_t(xN[s]));
      }
    }
  }
  solfin = (__ballot_sync(gmask, solfin) & gmask) == gmask;
  if constexpr (sizeof(TS) == 4) {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
      ny = t_max(ny, __shfl_xor_sync(gmask, ny, o, G));
      nd = t_max(nd, __shfl_xor_sync(gmask, nd, o, G));
    }
  } else {
    ny = group_max_abs<G, R>(y, n, gmask);
    nd = group_max_abs<G, R>(xN, n, gmask);
  }
  const bool bad = !(ok && solfin);
  double tau = Q.tau, dtau = Q.dtau, tauacc = Q.tauacc;
  int32_t steps = Q.steps + 1, accepts = Q.accepts, rejects = Q.rejects, streak = Q.streak;
  const TS err = nd / t_max(TS(1), ny);
  const bool accept = !bad && err <= (TS)prm.tol_accept;
  const bool herm = prm.predictor == 1;
  bool predict = true, keep_prev = false, retry = false;
  cx<TS> yp[R], dp[R];   // the accepted point before the last one (Hermite predictor)
  double taup = 0.0;
  if (accept) {
    keep_prev = herm && accepts >= 1;
#pragma unroll
    for (int s = 0; s < R; ++s) {
      yp[s] = yacc[s];
      dp[s] = dEacc[s];
      yacc[s] = mk<TS>(y[s].x + xN[s].x, y[s].y + xN[s].y);
      dEacc[s] = xE[s];
    }
    taup = tauacc;
    tauacc = tau;
    accepts += 1;
    streak += 1;
    if (tauacc == 0.0) {
      status = HPT_PATH_CONVERGED;
      predict = false;
    } else {
      bool div = false;
#pragma unroll
      for (int s = 0; s < R; ++s) {
        if (lane + G * s < n) div = div || outside_bound<TS>(yacc[s], prm.div_bound);
      }
      div = (__ballot_sync(gmask, div) & gmask) != 0u;
      if (div) {
        status = HPT_PATH_DIVERGED;
        predict = false;
      } else if (streak >= prm.grow_after) {
        dtau = fmin(dtau * prm.grow, prm.dtau_max);
        streak = 0;
      }
    }
  } else {
    rejects += 1;
    streak = 0;
    if (accepts == 0) {
      predict = false;
      if (bad) {
        status = HPT_PATH_SINGULAR;
      } else {
#pragma unroll
        for (int s = 0; s < R; ++s) {
          y[s] = mk<TS>(y[s].x + xN[s].x, y[s].y + xN[s].y);
          yacc[s] = y[s];
        }
        if (steps >= prm.max_steps) status = HPT_PATH_MAX_STEPS;
      }
    } else {
      // a rejected cubic prediction is retried with Euler at the same step
      // size; a rejected Euler prediction shrinks the step
      retry = herm && S.hermite[path] != 0;
      if (!retry) {
        dtau *= prm.shrink;
        if (dtau < prm.dtau_min) {
          status = HPT_PATH_UNDERFLOW;
          predict = false;
        }
      }
    }
  }
  if (predict) {
    const double h = fmin(dtau, -tauacc);
    bool cubic = false;
    if (herm && !retry && accepts >= 2) {
      if (!keep_prev) {   // a rejected step: the previous point from the state
#pragma unroll
        for (int s = 0; s < R; ++s) {
          const bool mine = lane + G * s < n;
          yp[s] = mine ? ld<TS>(S.y_prev, vbase + lane + G * s) : mk<TS>(0, 0);
          dp[s] = mine ? ld<TS>(S.dE_prev, vbase + lane + G * s) : mk<TS>(0, 0);
        }
        taup = S.tau_prev[path];
      }
      cubic = tauacc - taup > 0.0;
    }
    if (cubic) {
      // cubic Hermite through (taup, yp, dp) and (tauacc, yacc, dEacc) at tauacc + h
      const double d = tauacc - taup, u = 1.0 + h / d, u2 = u * u, u3 = u2 * u;
      const TS h00 = (TS)(2 * u3 - 3 * u2 + 1), h10 = (TS)((u3 - 2 * u2 + u) * d);
      const TS h01 = (TS)(-2 * u3 + 3 * u2), h11 = (TS)((u3 - u2) * d);
#pragma unroll
      for (int s = 0; s < R; ++s)
        y[s] = mk<TS>(h00 * yp[s].x + h10 * dp[s].x + h01 * yacc[s].x + h11 * dEacc[s].x,
                      h00 * yp[s].y + h10 * dp[s].y + h01 * yacc[s].y + h11 * dEacc[s].y);
    } else {
#pragma unroll
      for (int s = 0; s < R; ++s) y[s] = mk<TS>(yacc[s].x + (TS)h * dEacc[s].x, yacc[s].y + (TS)h * dEacc[s].y);
    }
    tau = tauacc + h;
    if (steps >= prm.max_steps) status = HPT_PATH_MAX_STEPS;
    if (herm && lane == 0) S.hermite[path] = cubic ? 1 : 0;
  }
#pragma unroll
  for (int s = 0; s < R; ++s) {
    const int j = lane + G * s;
    if (j < n) {
      const size_t vi = vbase + j;
      st<TS>(S.y, vi, y[s]);
      st<TS>(S.y_acc, vi, yacc[s]);
      st<TS>(S.dE_acc, vi, dEacc[s]);
      if (keep_prev) {
        st<TS>(S.y_prev, vi, yp[s]);
        st<TS>(S.dE_prev, vi, dp[s]);
      }
    }
  }
  if (keep_prev && lane == 0) S.tau_prev[path] = taup;
  if (lane == 0) {
    S.tau[path] = tau;
    S.dtau[path] = dtau;
    S.tau_acc[path] = tauacc;
    S.status[path] = status;
    S.steps[path] = steps;
    S.accepts[path] = accepts;
    S.rejects[path] = rejects;
    S.streak[path] = streak;
  }
}

template <typename TS, int G, int R>
__device__ __forceinline__ void update_path(int n, int64_t path, size_t vbase, int32_t status, bool ok,
                                            const cx<TS> (&wE)[R], const cx<TS> (&wN)[R], const hpt_paths& S,
                                            const hpt_params& prm) {
  StepState<TS, R> Q;
  load_step_state<TS, G, R>(n, path, vbase, S, Q);
  update_path<TS, G, R>(n, path, vbase, status, ok, wE, wN, S, prm, Q);
}

__device__ __forceinline__ int64_t pm_path(const PathMap& m, int64_t q) { return m.list ? m.list[q] : q; }
__device__ __forceinline__ int pm_n(const PathMap& m, int64_t q, int n) {
  return m.sys_n ? m.sys_n[m.tile_sys[q >> 7]] : n;
}
__device__ __forceinline__ size_t pm_vbase(const PathMap& m, int64_t path, int n) {
  return m.vofs ? (size_t)m.vofs[path] : (size_t)path * n;
}
__device__ __forceinline__ int64_t pm_count(const PathMap& m, int64_t p) { return m.npos ? (int64_t)*m.npos : p; }
__device__ __forceinline__ int64_t pm_begin(const PathMap& m) { return m.pos_begin ? (int64_t)*m.pos_begin : 0; }

// FP64 re-solve of the paths that a warp's FP32 solves flagged (pivot ratio
// above prm.cond_max): same FP32 Jacobian, FP64 factorisation, then the step
// control in the FP32 state, in the warp's own shared memory.  Flagged paths
// are rare; a launch of their own, with its list and counter to clear, cost
// every step 6 us whether there was one or not (250 paths, n = 14: 28.7 ->
// 22.6 us a step; 65,536 paths, n = 16: 212 -> 206 us).
// resolve_round: the first 32 / GS flagged groups of m (a bit for each group's
// first lane), GS lanes each; W holds 32 / GS times lu64_entries +
// lu64_col_entries of n; n <= GS RS.
template <int GS, int RS>
__device__ __noinline__ void resolve_round(unsigned m, int n, int nmax, int64_t q, int64_t path, size_t vbase,
                                           const float2* __restrict__ ext, const hpt_paths& S, const hpt_params& prm,
                                           double2* W) {
  constexpr int K = 32 / GS;
  const int l = threadIdx.x & (GS - 1), g = (threadIdx.x & 31) / GS;
  double2* A = W + g * lu64_entries(n);
  int* colx = (int*)(W + K * lu64_entries(n)) + g * 4 * lu64_col_entries(n);
#pragma unroll
  for (int k = 0; k + 1 < K; ++k)
    if (k < g) m &= m - 1;
  const bool act = m != 0;
  const int src = act ? __ffs(m) - 1 : 0;
  const int64_t qs = __shfl_sync(0xffffffffu, q, src), ps = __shfl_sync(0xffffffffu, path, src);
  const size_t vs = __shfl_sync(0xffffffffu, (unsigned long long)vbase, src);
  __syncwarp();   // the warp's shared memory is free
  const int np2 = n + 2;
  for (int e = l; act && e < n * np2; e += GS) {
    const int k = e / np2, u = e - k * np2;
    const float2 v = ext[ext_index(qs, k, u, nmax)];
    A[e] = make_double2((double)v.x, (double)v.y);
  }
  __syncwarp();
  const bool ok = lu64_solve<GS>(n, A, colx, -1);
  if (act) {   // group-uniform; only group-masked shuffles
    cx<float> fE[RS], fN[RS];
#pragma unroll
    for (int s = 0; s < RS; ++s) {
      const int c = l + GS * s;
      fE[s] = fN[s] = mk<float>(0.f, 0.f);
      if (c < n) {
        const cx<double> e = lu64_x(n, A, colx, c, 0), f = lu64_x(n, A, colx, c, 1);
        fE[s] = mk<float>((float)e.x, (float)e.y);
        fN[s] = mk<float>((float)f.x, (float)f.y);
      }
    }
    update_path<float, GS, RS>(n, ps, vs, HPT_PATH_ACTIVE, ok, fE, fN, S, prm);
  }
  __syncwarp();
}
// The flagged paths of a warp, a single one with all 32 lanes, more of them 32
// / GS at a time: their chains of dependent steps, which bound it, run side by
// side.  us a step with every path flagged, for a launch of its own, one after
// another in the warp, and so: n = 8, 128 paths 54, 81, 35; n = 16, 128 paths
// 165, 178, 117, 65,536 paths 4,172, 2,426, 1,646; many systems, n = 20 and 24,
// 128 paths 214, 263, 200 and 263, 347, 269 (a single path at n = 24: 121).
// Call with the warp converged; flag and the path's data are uniform in the
// groups of G lanes.
template <int GS, int RS>
__device__ __noinline__ void resolve_flagged(int G, bool flag, int n, int nmax, int64_t q, int64_t path, size_t vbase,
                                             const float2* __restrict__ ext, const hpt_paths& S,
                                             const hpt_params& prm, double2* W) {
  unsigned m = __ballot_sync(0xffffffffu, flag && (threadIdx.x & (G - 1)) == 0);
  while (m) {
    if (GS == 32 || (m & (m - 1)) == 0) {
      resolve_round<32, 1>(m, n, nmax, q, path, vbase, ext, S, prm, W);
      m &= m - 1;
    } else {
      resolve_round<GS, RS>(m, n, nmax, q, path, vbase, ext, S, prm, W);
#pragma unroll
      for (int k = 0; k < 32 / GS; ++k) m &= m - 1;
    }
  }
}
// Lanes per re-solved path and unknowns per lane, by the FP32 solve's shape: 8
// (four paths at once) for n <= 8, 16 for n <= 24, 32 where a warp has one path.
template <int G, int R>
struct Resolve {
  static constexpr int GS = G == 32 ? 32 : (R == 1 ? 8 : 16), RS = G * R <= GS ? 1 : 2;
};
// Whether the warp has a flagged path at all (the usual answer is no).
__device__ __forceinline__ bool any_flagged(bool flag) { return __any_sync(0xffffffffu, flag); }
// Shared memory of one warp of a solve kernel: its groups' regions, or the
// FP64 matrices of the paths re-solved at once, whichever is larger.
template <int G, int R>
__host__ __device__ constexpr int warp_smem(int groups_bytes, int n) {
  const int mats = 32 / Resolve<G, R>::GS * (lu64_entries(n) + lu64_col_entries(n)) * 16;
  return groups_bytes > mats ? groups_bytes : mats;
}

// One FP32 Euler-Newton step per ACTIVE path: consolidated solve, then the
// step control.  Solves whose pivot ratio (after equilibration) exceeds
// prm.cond_max are not applied but solved again in FP64 (resolve_flagged).
// One system, n > 16: a warp per path, a grid that covers every path once;
// ws: bytes of shared memory per warp.
__global__ void __launch_bounds__(kSolveThreads)
solve_update_kernel(int n, int64_t p, const float2* __restrict__ ext, const __grid_constant__ hpt_paths S,
                    const __grid_constant__ hpt_params prm, int ws) {
  extern __shared__ __align__(16) unsigned char smem[];
  grid_wait();
  const int64_t path = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32;
  const int32_t status = path < p ? S.status[path] : -1;
  const bool valid = status == HPT_PATH_ACTIVE;
  unsigned char* sm = smem + (threadIdx.x / 32) * ws;
  const int64_t q0 = (int64_t)blockIdx.x * (kSolveThreads / 32);
  const int64_t qi = q0 + (threadIdx.x & 3);
  stage_block_rows(n, n, ext, q0, qi < p && S.status[qi] == HPT_PATH_ACTIVE, smem, ws);
  __syncthreads();
  if (!valid) return;   // warp-uniform
  const size_t vbase = (size_t)path * n;
  PathRows<32, 1> P;
  const bool fin = load_rows_staged(n, sm, valid, P);
  cx<float> xE[1], xN[1];
  float cond;
  const bool ok = group_solve<32, 1>(n, P, xE, xN, cond, sm) && fin;
  if (ok && !(cond <= (float)prm.cond_max))
    resolve_flagged<32, 1>(32, true, n, n, path, path, vbase, ext, S, prm, (double2*)sm);
  else
    update_path<float, 32, 1>(n, path, vbase, status, ok, xE, xN, S, prm);
}

// FP32 step of one system with n <= G R by Gauss-Jordan elimination.  A
// G-lane group owns one path as in group_solve: lane l holds rows l + G s,
// s < R, of [D_z H | -H_tau | -H] in registers, here as packed FP32 pairs
// (rows >= n are zero).  After the exact power-of-two row and column
// equilibration of group_solve (the column magnitudes go through shared
// memory, one reduction per column instead of a butterfly per column), each
// column is eliminated from every other row, the rows already used as pivots
// included: group_solve updates those rows too, with zero multipliers, so
// the elimination costs the same and no back substitution follows.  At the
// end row i holds only its pivot u_i and its two right-hand sides, and the
// unknowns of the column it pivoted are b_i / u_i.  The pivot of a column is
// the one of group_solve (largest |.|^2 among the unused rows, ties to the
// lowest row), so the pivots, the condition proxy and the FP64 re-solve
// list are those of the LU form.  Each entry of the pivot row reaches the
// group by a shuffle from its owner (every lane selects the pivot's slot, the
// same in the whole group): no shared-memory round trip, and no per-entry
// packing by the owner alone, which cost 25 of 140 us.  A row's update
// a - l u is two paired FMAs with u and u swapped.  Rows are shifted as in
// group_solve (column j is always register 0).
template <int NC>
struct GjSmem {
  union {
    float cm[NC][NC + 4];       // the rows' entry magnitudes, read back by column
    struct {
      float4 x[NC];             // the solutions by column: (xE.re, xE.im, xN.re, xN.im)
    } e;
  } u;
  float dcol[NC];               // the column scales
};
// Per-group stride in words, = G (mod 32): the column reads of cm by the
// groups of a warp fall on distinct banks.
template <int G, int NC>
struct GjLayout {
  static constexpr int raw = (int)(sizeof(GjSmem<NC>) / 4);
  static constexpr int words = (raw - G + 31) / 32 * 32 + G;
  static constexpr int bytes = words * 4;
};

__device__ __forceinline__ float cmag2(uint64_t v) {
  const float2 f = upk2(v);
  return fmaxf(fabsf(f.x), fabsf(f.y));
}

// One path (position q of the scratch, laid out for nmax variables) for
// every lane of its group; call with the whole warp converged.  Returns with
// the state updated, or true (group-uniform): to be solved again in FP64.
// smem is the group's.
template <int G, int R>
__device__ __forceinline__ bool gj_path(int n, int nmax, int64_t q, int64_t path, size_t vbase, int32_t status,
                                        const float2* __restrict__ ext, const hpt_paths& S, const hpt_params& prm,
                                        unsigned char* smem) {
  constexpr int NC = G * R;
  const int lane = threadIdx.x & (G - 1);
  const bool valid = status == HPT_PATH_ACTIVE;
  GjSmem<NC>& sh = *(GjSmem<NC>*)smem;
  const unsigned gmask = group_mask<G>();

  // rows lane + G s and their right-hand sides
  uint64_t a[R][NC], bE[R], bN[R];
  float chk = 0.f;
#pragma unroll
  for (int s = 0; s < R; ++s) {
    const int r = lane + G * s;
    const bool have = valid && r < n;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      float2 v = make_float2(0.f, 0.f);
      if (have && c < n) v = ext[ext_index(q, r, c, nmax)];
      a[s][c] = pk2(v.x, v.y);
      chk += fabsf(v.x) + fabsf(v.y);
    }
    float2 ht = make_float2(0.f, 0.f), h = make_float2(0.f, 0.f);
    if (have) {
      ht = ext[ext_index(q, r, n, nmax)];
      h = ext[ext_index(q, r, n + 1, nmax)];
    }
    bE[s] = pk2(-ht.x, -ht.y);
    bN[s] = pk2(-h.x, -h.y);
    chk += fabsf(ht.x) + fabsf(ht.y) + fabsf(h.x) + fabsf(h.y);
  }
  // a sum of magnitudes is finite iff every entry is
  const bool fin = (__ballot_sync(0xffffffffu, isfinite(chk)) & gmask) == gmask;

  // equilibration: each row, then the columns, by exact powers of two
#pragma unroll
  for (int s = 0; s < R; ++s) {
    float m = 0.f;
#pragma unroll
    for (int c = 0; c < NC; ++c) m = fmaxf(m, cmag2(a[s][c]));
    const float dr = pow2_inv(m);
    const uint64_t DR = pk2(dr, dr);
#pragma unroll
    for (int c = 0; c < NC; ++c) a[s][c] = mul_x2(a[s][c], DR);
    bE[s] = mul_x2(bE[s], DR);
    bN[s] = mul_x2(bN[s], DR);
#pragma unroll
    for (int c = 0; c < NC; c += 4)
      *(float4*)&sh.u.cm[lane + G * s][c] =
          make_float4(cmag2(a[s][c]), cmag2(a[s][c + 1]), cmag2(a[s][c + 2]), cmag2(a[s][c + 3]));
  }
  __syncwarp();
  float dc[R];   // the scales of columns lane + G s
#pragma unroll
  for (int s = 0; s < R; ++s) {
    float mc = 0.f;
#pragma unroll
    for (int r = 0; r < NC; ++r) mc = fmaxf(mc, sh.u.cm[r][lane + G * s]);
    dc[s] = pow2_inv(mc);   // 1 for a zero column
    sh.dcol[lane + G * s] = dc[s];
  }
  __syncwarp();   // every column magnitude read before the pivot rows reuse the space
#pragma unroll
  for (int c = 0; c < NC; c += 4) {
    const float4 d = *(const float4*)&sh.dcol[c];
    const uint64_t D0 = pk2(d.x, d.x), D1 = pk2(d.y, d.y), D2 = pk2(d.z, d.z), D3 = pk2(d.w, d.w);
#pragma unroll
    for (int s = 0; s < R; ++s) {
      a[s][c] = mul_x2(a[s][c], D0);
      a[s][c + 1] = mul_x2(a[s][c + 1], D1);
      a[s][c + 2] = mul_x2(a[s][c + 2], D2);
      a[s][c + 3] = mul_x2(a[s][c + 3], D3);
    }
  }

  // elimination
  bool used[R];
  int step[R];
  uint64_t piv[R];
#pragma unroll
  for (int s = 0; s < R; ++s) {
    used[s] = lane + G * s >= n;
    step[s] = 0;
    piv[s] = pk2(1.f, 0.f);
  }
  bool ok = true;
  float pmax = 0.f, pmin = 0.f;   // extreme |u_jj|^2
#pragma unroll 1
  for (int j = 0; j < n; ++j) {
    unsigned key = 0u;
#pragma unroll
    for (int s = 0; s < R; ++s) {
      const float2 v = upk2(a[s][0]);
      key = max(key, pivot_key(v.x * v.x + v.y * v.y, used[s], lane + G * s));
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) key = max(key, __shfl_xor_sync(0xffffffffu, key, o, G));
    const int br = 31 - (int)(key & 31u);
    const int bs = br / G;
    const bool owner = lane == (br & (G - 1));
    const int lim = n - 1 - j;   // live registers 1..lim
    // the pivot row by shuffles from its owner: every lane picks slot bs
    // (uniform in the group) and reads the owner's copy
    const int ol = br & (G - 1);
    auto pick_bcast = [&](const uint64_t* col) -> uint64_t {   // col[s] for s < R
      uint64_t v = col[0];
#pragma unroll
      for (int s = 1; s < R; ++s) v = bs == s ? col[s] : v;
      return __shfl_sync(0xffffffffu, v, ol, G);
    };
    if (owner) {
#pragma unroll
      for (int s = 0; s < R; ++s) {
        if (bs == s) {
          used[s] = true;
          step[s] = j;
          piv[s] = a[s][0];
        }
      }
    }
    uint64_t col0[R];
#pragma unroll
    for (int s = 0; s < R; ++s) col0[s] = a[s][0];
    const float2 pv = upk2(pick_bcast(col0));
    const float p2 = pv.x * pv.x + pv.y * pv.y;
    if (!(p2 > 0.f) || !isfinite(p2)) ok = false;
    pmax = j == 0 ? p2 : fmaxf(pmax, p2);
    pmin = j == 0 ? p2 : fminf(pmin, p2);
    const float rp = t_rcp(p2);   // one reciprocal per pivot, shared by all rows
    // multipliers a_s0 / pivot; the pivot row itself keeps its values
    uint64_t NL[R], LS[R];
#pragma unroll
    for (int s = 0; s < R; ++s) {
      const float2 v = upk2(a[s][0]);
      float lr = (v.x * pv.x + v.y * pv.y) * rp, li = (v.y * pv.x - v.x * pv.y) * rp;
      if (owner && bs == s) {
        lr = 0.f;
        li = 0.f;
      }
      NL[s] = pk2(-lr, -lr);
      LS[s] = pk2(li, -li);
    }
    // shifted update a[c-1] = a[c] - l u over the live width, in chunks of
    // four columns behind one warp-uniform branch each (the columns of the
    // last chunk beyond the live width are never read again)
#pragma unroll
    for (int c0 = 1; c0 < NC; c0 += 4) {
      if (c0 <= lim) {
#pragma unroll
        for (int c = c0; c < c0 + 4 && c < NC; ++c) {
          uint64_t colc[R];
#pragma unroll
          for (int s = 0; s < R; ++s) colc[s] = a[s][c];
          const uint64_t U = pick_bcast(colc);
          const float2 uf = upk2(U);
          const uint64_t US = pk2(uf.y, uf.x);
#pragma unroll
          for (int s = 0; s < R; ++s) a[s][c - 1] = fma_x2(LS[s], US, fma_x2(NL[s], U, a[s][c]));
        }
      }
    }
    {
      const uint64_t U = pick_bcast(bE), V = pick_bcast(bN);
      const float2 uf = upk2(U), vf = upk2(V);
      const uint64_t US = pk2(uf.y, uf.x), VS = pk2(vf.y, vf.x);
#pragma unroll
      for (int s = 0; s < R; ++s) {
        bE[s] = fma_x2(LS[s], US, fma_x2(NL[s], U, bE[s]));
        bN[s] = fma_x2(LS[s], VS, fma_x2(NL[s], V, bN[s]));
      }
    }
  }
  // row i < n now holds its pivot and right-hand sides: the unknowns of the
  // column it pivoted, put in column order through shared memory
#pragma unroll
  for (int s = 0; s < R; ++s) {
    if (lane + G * s < n) {
      const float2 u = upk2(piv[s]), e = upk2(bE[s]), f = upk2(bN[s]);
      const float ru = t_rcp(u.x * u.x + u.y * u.y);
      sh.u.e.x[step[s]] = make_float4((e.x * u.x + e.y * u.y) * ru, (e.y * u.x - e.x * u.y) * ru,
                                      (f.x * u.x + f.y * u.y) * ru, (f.y * u.x - f.x * u.y) * ru);
    }
  }
  __syncwarp();
  cx<float> wE[R], wN[R];
#pragma unroll
  for (int s = 0; s < R; ++s) {
    wE[s] = mk<float>(0.f, 0.f);
    wN[s] = mk<float>(0.f, 0.f);
    if (lane + G * s < n) {
      const float4 v = sh.u.e.x[lane + G * s];
      wE[s] = mk<float>(v.x * dc[s], v.y * dc[s]);
      wN[s] = mk<float>(v.z * dc[s], v.w * dc[s]);
    }
  }
  const float cond = pmin > 0.f ? sqrtf(pmax / pmin) : INFINITY;
  ok = ok && fin;
  __syncwarp();   // the group's shared memory is reused by its next path
  if (!valid) return false;   // group-uniform; only group-masked shuffles below
  if (ok && !(cond <= (float)prm.cond_max)) return true;
  update_path<float, G, R>(n, path, vbase, status, ok, wE, wN, S, prm);
  return false;
}
// Bytes of a warp's groups.
template <int G, int R>
__host__ __device__ constexpr int gj_groups_bytes() { return (32 / G) * GjLayout<G, G * R>::bytes; }

template <int G, int R>
__global__ void __launch_bounds__(kSolveThreads, R == 1 ? 6 : 4)
gj_update_kernel(int n, int64_t p, const float2* __restrict__ ext, const __grid_constant__ hpt_paths S,
                 const __grid_constant__ hpt_params prm, int ws) {
  extern __shared__ __align__(16) unsigned char smem[];
  grid_wait();
  const int64_t path = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
  const int32_t status = path < p ? S.status[path] : -1;
  if (!__any_sync(0xffffffffu, status == HPT_PATH_ACTIVE)) return;   // warp-uniform exit
  unsigned char* wsm = smem + (threadIdx.x / 32) * ws;
  const bool again = gj_path<G, R>(n, n, path, path, (size_t)path * n, status, ext, S, prm,
                                   wsm + ((threadIdx.x & 31) / G) * GjLayout<G, G * R>::bytes);
  if (any_flagged(again))
    resolve_flagged<Resolve<G, R>::GS, Resolve<G, R>::RS>(G, again, n, n, path, path, (size_t)path * n, ext, S, prm,
                                                          (double2*)wsm);
}

// The same over a position map (many systems), persistent as
// solve_update_map_kernel: a warp's 32/G consecutive positions lie in one
// 128-position tile, so n is warp-uniform.
template <int G, int R>
__global__ void __launch_bounds__(kSolveThreads, R == 1 ? 6 : 4)
gj_update_map_kernel(int n0, int64_t p, const float2* __restrict__ ext, const __grid_constant__ hpt_paths S,
                     const __grid_constant__ hpt_params prm, PathMap pm, int ws) {
  extern __shared__ __align__(16) unsigned char smem[];
  grid_wait();
  unsigned char* wsm = smem + (threadIdx.x / 32) * ws;
  constexpr int per_warp = 32 / G;
  const int64_t warp_id = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32;
  const int64_t nwarps = (int64_t)gridDim.x * blockDim.x / 32;
  const int g = (threadIdx.x & 31) / G;
  const int64_t npos = pm_count(pm, p);
  for (int64_t base = pm_begin(pm) + warp_id * per_warp; base < npos; base += nwarps * per_warp) {
    const int64_t q = base + g;
    const int n = pm_n(pm, base, n0);
    const int64_t path = q < npos ? pm_path(pm, q) : -1;
    const int32_t status = path >= 0 ? S.status[path] : -1;
    if (!__any_sync(0xffffffffu, status == HPT_PATH_ACTIVE)) continue;   // warp-uniform skip
    const size_t vbase = status == HPT_PATH_ACTIVE ? pm_vbase(pm, path, n) : 0;
    const bool again = gj_path<G, R>(n, pm.nmax, q, path, vbase, status, ext, S, prm, wsm + g * GjLayout<G, G * R>::bytes);
    if (any_flagged(again))
      resolve_flagged<Resolve<G, R>::GS, Resolve<G, R>::RS>(G, again, n, pm.nmax, q, path, vbase, ext, S, prm,
                                                            (double2*)wsm);
  }
}

// The same over a position map (many systems).  Persistent: the warps loop
// over the positions of [*pos_begin, *npos) (32/G consecutive positions per
// warp, always inside one 128-position tile, so n is warp-uniform).
template <int G, int R>
__global__ void __launch_bounds__(kSolveThreads)
solve_update_map_kernel(int n0, int64_t p, const float2* __restrict__ ext, const __grid_constant__ hpt_paths S,
                        const __grid_constant__ hpt_params prm, PathMap pm, int ws) {
  extern __shared__ __align__(16) unsigned char smem[];
  grid_wait();
  constexpr int per_warp = 32 / G;
  const int64_t warp_id = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32;
  const int64_t nwarps = (int64_t)gridDim.x * blockDim.x / 32;
  const int g = (threadIdx.x & 31) / G;
  unsigned char* wsm = smem + (threadIdx.x / 32) * ws;
  unsigned char* sm = wsm + g * GroupSmem<G * R>::bytes;
  const int64_t npos = pm_count(pm, p);
  const int nmax = pm.nmax;
  // with 32-lane groups the block's four warps take consecutive positions of
  // one tile and run the same number of iterations (npos is a multiple of
  // 128), so the staging barriers below are reached by the whole block
  for (int64_t base = pm_begin(pm) + warp_id * per_warp; base < npos; base += nwarps * per_warp) {
    const int64_t q = base + g;
    const int n = pm_n(pm, base, n0);
    const int64_t path = q < npos ? pm_path(pm, q) : -1;
    const int32_t status = path >= 0 ? S.status[path] : -1;
    const bool valid = status == HPT_PATH_ACTIVE;
    if (G == 32) {
      const int64_t q0 = base - (threadIdx.x >> 5);
      const int64_t pi = pm_path(pm, q0 + (threadIdx.x & 3));
      __syncthreads();   // the previous iteration's solves are done with the regions
      stage_block_rows(n, nmax, ext, q0, pi >= 0 && S.status[pi] == HPT_PATH_ACTIVE, smem, ws);
      __syncthreads();
    }
    if (!__any_sync(0xffffffffu, valid)) continue;   // warp-uniform skip
    const size_t vbase = valid ? pm_vbase(pm, path, n) : 0;
    PathRows<G, R> P;
    bool fin;
    if constexpr (G == 32) fin = load_rows_staged(n, sm, valid, P);
    else fin = load_rows<G, R>(n, nmax, ext, q, valid, P);
    cx<float> xE[R], xN[R];
    float cond;
    const bool ok = group_solve<G, R>(n, P, xE, xN, cond, sm) && fin;
    const bool again = valid && ok && !(cond <= (float)prm.cond_max);
    if (valid && !again) update_path<float, G, R>(n, path, vbase, status, ok, xE, xN, S, prm);   // group-uniform
    __syncwarp();
    if (any_flagged(again))
      resolve_flagged<Resolve<G, R>::GS, Resolve<G, R>::RS>(G, again, n, nmax, q, path, vbase, ext, S, prm,
                                                            (double2*)wsm);
    __syncwarp();
  }
}

// One FP64 Euler-Newton step per ACTIVE path: consolidated solve in shared
// memory (lu64_solve), then the step control.  128 / G consecutive paths per
// block.
template <int G, int R>
__global__ void __launch_bounds__(kLuThreads)
step_fp64_kernel(int n, int64_t p, const double2* __restrict__ ext, hpt_paths S, hpt_params prm) {
  extern __shared__ __align__(16) unsigned char smem[];
  grid_wait();
  constexpr int P = lu64_paths<G>();
  const int lane = threadIdx.x & (G - 1), g = threadIdx.x / G;
  const int64_t q0 = (int64_t)blockIdx.x * P;
  const int stride = lu64_entries(n), cstride = 4 * lu64_col_entries(n);
  double2* mats = (double2*)smem;
  {
    const int i = threadIdx.x % P;
    const int64_t qi = q0 + i;
    lu64_stage<G>(n, n, n, ext, qi, qi < p && S.status[qi] == HPT_PATH_ACTIVE, mats + i * stride, false);
  }
  const int64_t path = q0 + g;
  const int32_t status = path < p ? S.status[path] : -1;
  const bool valid = status == HPT_PATH_ACTIVE;
  __syncthreads();
  if (!__any_sync(0xffffffffu, valid)) return;   // warp-uniform exit
  double2* A = mats + g * stride;
  int* colx = (int*)(mats + P * stride) + g * cstride;
  const bool ok = lu64_solve<G>(n, A, colx, -1);
  if (!valid) return;   // group-uniform; only group-masked shuffles below
  cx<double> xE[R], xN[R];
#pragma unroll
  for (int s = 0; s < R; ++s) {
    const int c = lane + G * s;
    xE[s] = c < n ? lu64_x(n, A, colx, c, 0) : mk<double>(0, 0);
    xN[s] = c < n ? lu64_x(n, A, colx, c, 1) : mk<double>(0, 0);
  }
  update_path<double, G, R>(n, path, (size_t)path * n, status, ok, xE, xN, S, prm);
}

// Newton polish update at t = 1 (FP64): x += dN until the error left is below
// tol: |dN|/max(1,|x|) <= tol, or, once the corrections shrink quadratically,
// the error after this update, about r_k^3 / r_{k-1}^2 for the relative
// corrections r of the last two iterations (last[] keeps r_{k-1}; 0: none).
// MAP: positions [*pm.pos_begin, *pm.npos) of a position map (a block's
// positions lie in one tile, so n is block-uniform); otherwise the p paths of
// one system.
template <int G, int R, bool MAP>
__global__ void __launch_bounds__(kLuThreads)
newton_kernel(int n0, int64_t p, const double2* __restrict__ ext, double2* __restrict__ x,
              int32_t* __restrict__ done, float* __restrict__ last, double tol, PathMap pm) {
  extern __shared__ __align__(16) unsigned char smem[];
  grid_wait();
  constexpr int P = lu64_paths<G>();
  const int lane = threadIdx.x & (G - 1), g = threadIdx.x / G;
  const int64_t q0 = (int64_t)blockIdx.x * P + (MAP ? (int64_t)*pm.pos_begin : 0);
  const int64_t end = MAP ? (int64_t)*pm.npos : p;
  if (q0 >= end) return;
  const int n = MAP ? pm.sys_n[pm.tile_sys[q0 >> 7]] : n0;
  const int stride = lu64_entries(n), cstride = 4 * lu64_col_entries(n);
  double2* mats = (double2*)smem;
  {
    const int i = threadIdx.x % P;
    const int64_t qi = q0 + i, pi = qi < end ? (MAP ? pm.list[qi] : qi) : -1;
    lu64_stage<G>(n, n, MAP ? pm.nmax : n, ext, qi, pi >= 0 && done[pi] == 0, mats + i * stride, false);
  }
  const int64_t q = q0 + g;
  const int64_t path = q < end ? (MAP ? pm.list[q] : q) : -1;
  const bool valid = path >= 0 && done[path] == 0;
  __syncthreads();
  if (!__any_sync(0xffffffffu, valid)) return;
  double2* A = mats + g * stride;
  int* colx = (int*)(mats + P * stride) + g * cstride;
  const bool ok = lu64_solve<G>(n, A, colx, -1);
  if (!valid) return;
  const size_t vbase = MAP ? (size_t)pm.vofs[path] : (size_t)path * n;
  const unsigned gmask = group_mask<G>();
  bool sfin = true;
  cx<double> y[R], xN[R];
#pragma unroll
  for (int s = 0; s < R; ++s) {
    const int j = lane + G * s;
    y[s] = xN[s] = mk<double>(0, 0);
    if (j < n) {
      y[s] = ld<double>(x, vbase + j);
      xN[s] = cmul(y[s], lu64_x(n, A, colx, j, 1));   // D_z H in the scratch: the correction is x * w
      sfin = sfin && finite(xN[s]);
      y[s] = mk<double>(y[s].x + xN[s].x, y[s].y + xN[s].y);
    }
  }
  sfin = (__ballot_sync(gmask, sfin) & gmask) == gmask;
  if (!(ok && sfin)) {
    if (lane == 0) done[path] = 2;
    return;
  }
  const double ny = group_max_abs<G, R>(y, n, gmask), nd = group_max_abs<G, R>(xN, n, gmask);
#pragma unroll
  for (int s = 0; s < R; ++s) {
    const int j = lane + G * s;
    if (j < n) st<double>(x, vbase + j, y[s]);
  }
  if (lane == 0) {
    const double r = nd / fmax(1.0, ny), rp = (double)last[path];
    const bool settled = rp > 0.0 && r <= 0.1 * rp && r * r * r <= tol * rp * rp;
    if (r <= tol || settled) done[path] = 1;
    last[path] = (float)r;
  }
}

// Adjoint, part 1: per solution, lambda from J^H lambda = gx (J from the
// extended Jacobian at t = 1), then contrib[q][i] = -lambda_k conj(x^{a_i})
// for every monomial i of equation k.  The monomials of a solution are dealt
// to its G lanes (consecutive contributions, whole sectors) and come from the
// fixed-point logarithm and exponential (hpt_fx.cuh), which leave the FP64
// pipe four operations a monomial; systems beyond their range (no mono)
// take exp of <a, log x> in FP64.
template <int G, int R>
__global__ void __launch_bounds__(kLuThreads)
adjoint_kernel(Fp64Sys sys, int64_t p, int M, const double2* __restrict__ ext, const double2* __restrict__ x,
               const double2* __restrict__ gx, double2* __restrict__ contrib) {
  extern __shared__ __align__(16) unsigned char smem[];
  grid_wait();
  constexpr int P = lu64_paths<G>();
  __shared__ ulonglong2 zsh[P][G * R];
  __shared__ float lfs[P][G * R];
  __shared__ int64_t exp1[64], exp2[64], cs1[64][2], cs2[64][2];   // looked up per lane: L1 would serve a sector a lane
  if (threadIdx.x < 64) {
    const fx::Tables& T = fx::tables();
    const int i = threadIdx.x;
    exp1[i] = T.exp1[i];
    exp2[i] = T.exp2[i];
    cs1[i][0] = T.cs1[i][0];
    cs1[i][1] = T.cs1[i][1];
    cs2[i][0] = T.cs2[i][0];
    cs2[i][1] = T.cs2[i][1];
  }
  const int n = sys.n;
  const int lane = threadIdx.x & (G - 1), g = threadIdx.x / G;
  const int64_t q0 = (int64_t)blockIdx.x * P;
  const int stride = lu64_entries(n), cstride = 4 * lu64_col_entries(n);
  double2* mats = (double2*)smem;
  {
    const int i = threadIdx.x % P;
    lu64_stage<G>(n, n, n, ext, q0 + i, q0 + i < p, mats + i * stride, true);
  }
  const int64_t path = q0 + g;
  const bool valid = path < p;
  double2* A = mats + g * stride;
  int* colx = (int*)(mats + P * stride) + g * cstride;
  // D_z H = H_y diag(x) in the scratch: H_y^H lambda = g becomes
  // (D_z H)^H lambda = conj(x) g
#pragma unroll
  for (int s = 0; s < R; ++s) {
    const int r = lane + G * s;
    if (valid && r < n) {
      const double2 v = x[(size_t)path * n + r], w = gx[(size_t)path * n + r];
      const cx<double> b = cmul(mk<double>(v.x, -v.y), mk<double>(w.x, w.y));
      A[r * (n + 2) + n] = make_double2(b.x, b.y);
      A[r * (n + 2) + n + 1] = make_double2(0.0, 0.0);
      if (sys.mono) {
        fx::Log lg;
        fx::log_of(v.x, v.y, lg);
        zsh[g][r] = make_ulonglong2((unsigned long long)lg.l, lg.turn);
        lfs[g][r] = lg.lf;
      } else {
        zsh[g][r] = make_ulonglong2((unsigned long long)__double_as_longlong(log(hypot(v.x, v.y))),
                                    (unsigned long long)__double_as_longlong(atan2(v.y, v.x)));
      }
    }
  }
  __syncthreads();
  if (!__any_sync(0xffffffffu, valid)) return;
  const bool ok = lu64_solve<G>(n, A, colx, 1);
  if (!valid) return;
  for (int k = 0, i = lane; i < M; i += G) {
    while (i >= sys.off[k] + sys.msz[k]) ++k;
    double mr, mi;
    if (sys.mono) {
      const FxMono m = sys.mono[i];
      fx::Sum w{0, 0, 0.f};
      for (int t = 0; t < m.nnz; ++t) {
        const int a = sys.ent[m.ent + t].a, j = sys.ent[m.ent + t].j;
        const ulonglong2 z = zsh[g][j];
        fx::add_power(w, a, z.x, z.y, lfs[g][j]);
      }
      if (fx::exp_in_range(w.f)) fx::exp_in((int64_t)w.w, w.turn, w.f, exp1, exp2, cs1, cs2, mr, mi);
      else fx::exp_of((int64_t)w.w, w.turn, w.f, exp1, exp2, cs1, cs2, mr, mi);
    } else {
      const double* ai = sys.ahat + (size_t)i * (n + 1);
      double wr = 0.0, wi = 0.0;
      for (int j = 0; j < n; ++j) {
        wr = fma(ai[j], __longlong_as_double((long long)zsh[g][j].x), wr);
        wi = fma(ai[j], __longlong_as_double((long long)zsh[g][j].y), wi);
      }
      sincos(wi, &mi, &mr);
      const double m = exp(wr);
      mr *= m;
      mi *= m;
    }
    // -lambda_k conj(x^a)
    const cx<double> lam = lu64_x(n, A, colx, k, 0);
    double2 v = make_double2(-(lam.x * mr + lam.y * mi), lam.x * mi - lam.y * mr);
    if (!ok) v = make_double2(NAN, NAN);
    contrib[(size_t)path * M + i] = v;
  }
}

// Adjoint, part 2: gc[i] += sum over the chunk's solutions of contrib[q][i],
// in a fixed order (the same bits on every run).  First pass: block (cb, r)
// takes 32 consecutive columns and the rows r, r + kAdjRowBlocks, .., its 32
// warps each a strided subset (a warp reads 32 consecutive columns of one
// row: coalesced) and then a tree over the warps; second pass: a tree over the
// kAdjRowBlocks partial sums.  What bounds it is the latency of dependent FP64
// additions (4,096 x 96 contributions: 16.6 us for the two passes, 18.6 with
// chains of 64).
constexpr int kAdjRowBlocks = 16;

__device__ __forceinline__ double2 add2(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }

__global__ void __launch_bounds__(1024) sum_columns_part_kernel(int64_t p, int M, const double2* __restrict__ contrib,
                                                                 double2* __restrict__ part) {
  __shared__ double2 red[32][33];
  grid_wait();
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + tx;
  double2 acc = make_double2(0.0, 0.0);
  if (i < M) {
#pragma unroll 8
    for (int64_t q = (int64_t)blockIdx.y + (int64_t)kAdjRowBlocks * ty; q < p; q += (int64_t)kAdjRowBlocks * 32)
      acc = add2(acc, contrib[(size_t)q * M + i]);
  }
  red[ty][tx] = acc;
  __syncthreads();
  // the tree: column ty's 32 sums, one per lane
  double2 v = red[tx][ty];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    v = add2(v, make_double2(__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o)));
  const int col = blockIdx.x * 32 + ty;
  if (tx == 0 && col < M) part[(size_t)blockIdx.y * M + col] = v;
}

__global__ void sum_columns_kernel(int M, const double2* __restrict__ part, double2* __restrict__ gc) {
  grid_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= M) return;
  double2 v[kAdjRowBlocks];
#pragma unroll
  for (int r = 0; r < kAdjRowBlocks; ++r) v[r] = part[(size_t)r * M + i];
#pragma unroll
  for (int o = kAdjRowBlocks / 2; o > 0; o >>= 1)
#pragma unroll
    for (int r = 0; r < o; ++r) v[r] = add2(v[r], v[r + o]);
  gc[i] = add2(gc[i], v[0]);   // chunks of solutions are added in order
}

template <typename T>
__global__ void paths_init_kernel(int n, int64_t p, const double2* __restrict__ y0, double tau0,
                                  double dtau0, hpt_paths S) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < p * n) {
    const double2 v = y0[i];
    cx<T> c = mk<T>((T)v.x, (T)v.y);
    st<T>(S.y, i, c);
    st<T>(S.y_acc, i, c);
    st<T>(S.dE_acc, i, mk<T>(0, 0));
    if (S.y_prev) {
      st<T>(S.y_prev, i, mk<T>(0, 0));
      st<T>(S.dE_prev, i, mk<T>(0, 0));
    }
  }
  if (i < p) {
    if (S.tau_prev) S.tau_prev[i] = tau0;
    if (S.hermite) S.hermite[i] = 0;
    S.tau[i] = tau0;
    S.tau_acc[i] = tau0;
    S.dtau[i] = dtau0;
    S.status[i] = HPT_PATH_ACTIVE;
    S.steps[i] = 0;
    S.accepts[i] = 0;
    S.rejects[i] = 0;
    S.streak[i] = 0;
  }
}

__global__ void count_active_kernel(int64_t p, const int32_t* __restrict__ status, int32_t* count) {
  int c = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < p;
       i += (int64_t)gridDim.x * blockDim.x)
    c += status[i] == HPT_PATH_ACTIVE;
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(count, c);
}

template <typename T>
__global__ void finish_track_kernel(int n, int64_t p, hpt_paths S, double2* __restrict__ x,
                                    int32_t* __restrict__ status_out, int32_t* __restrict__ steps_out,
                                    int32_t* __restrict__ done) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < p * n) {
    cx<T> v = ld<T>(S.y_acc, i);
    x[i] = make_double2((double)v.x, (double)v.y);
  }
  if (i < p) {
    const int32_t s = S.status[i];
    if (status_out) status_out[i] = s;
    if (steps_out) steps_out[i] = S.steps[i];
    done[i] = s == HPT_PATH_CONVERGED ? 0 : 3;
  }
}

__global__ void init_done_kernel(int64_t p, const int32_t* __restrict__ status, int32_t* done) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < p) done[i] = (!status || status[i] == HPT_PATH_CONVERGED) ? 0 : 3;
}

inline unsigned blocks_for(int64_t threads, int bs) { return (unsigned)((threads + bs - 1) / bs); }

// Lane-group shape for n: (G, R) = (8, 1) for n <= 8, (8, 2) for n <= 16,
// (32, 1) for n <= 32.
inline int shape_of(int n) { return n <= 8 ? 0 : (n <= 16 ? 1 : 2); }

// Persistent grids: enough blocks to cover the positions once, capped at a
// few waves of resident blocks (the kernels loop over positions).
inline unsigned solve_grid(int64_t p, int G) {
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 1;
  }
  const int64_t need = std::max<int64_t>(1, (p * G + kSolveThreads - 1) / kSolveThreads);
  return (unsigned)std::min<int64_t>(need, (int64_t)sms * 32);
}

template <int G, int R>
cudaError_t launch_solve_map(const StepArgs& a, cudaStream_t st) {
  PathMap pm = a.map;
  if (!pm.nmax) pm.nmax = a.n;
  constexpr int groups = (32 / G) * GroupSmem<G * R>::bytes;
  const int ws = warp_smem<G, R>(groups, std::min(pm.nmax, G * R)), smem = (kSolveThreads / 32) * ws;
  cudaError_t e = allow_smem<(kSolveThreads / 32) * warp_smem<G, R>(groups, G * R)>(solve_update_map_kernel<G, R>, smem);
  if (e != cudaSuccess) return e;
  return launch_chained(solve_update_map_kernel<G, R>, solve_grid(a.p, G), kSolveThreads, smem, st, pm.chained, a.n, a.p,
                        (const float2*)a.ext, a.st, a.prm, pm, ws);
}

// FP32 Gauss-Jordan solve + update (n <= 16: (G, R) = (8, 1) or (8, 2)), one
// system or a position map.
template <int G, int R>
cudaError_t launch_gj(const StepArgs& a, cudaStream_t st) {
  constexpr int groups = gj_groups_bytes<G, R>(), most = (kSolveThreads / 32) * warp_smem<G, R>(groups, G * R);
  PathMap pm = a.map;
  if (!pm.nmax) pm.nmax = a.n;
  const int ws = warp_smem<G, R>(groups, std::min(pm.nmax, G * R)), smem = (kSolveThreads / 32) * ws;
  if (!a.map.list) {
    cudaError_t e = allow_smem<most>(gj_update_kernel<G, R>, smem);
    if (e != cudaSuccess) return e;
    return launch_chained(gj_update_kernel<G, R>, blocks_for(a.p * G, kSolveThreads), kSolveThreads, smem, st, true, a.n,
                          a.p, (const float2*)a.ext, a.st, a.prm, ws);
  }
  cudaError_t e = allow_smem<most>(gj_update_map_kernel<G, R>, smem);
  if (e != cudaSuccess) return e;
  return launch_chained(gj_update_map_kernel<G, R>, solve_grid(a.p, G), kSolveThreads, smem, st, pm.chained, a.n, a.p,
                        (const float2*)a.ext, a.st, a.prm, pm, ws);
}

template <int G, int R>
cudaError_t launch_step64_shape(const StepArgs& a, cudaStream_t st) {
  const int smem = lu64_smem<G>(a.n);
  cudaError_t e = allow_smem<lu64_smem<G>(G * R)>(step_fp64_kernel<G, R>, smem);
  if (e != cudaSuccess) return e;
  return launch_chained(step_fp64_kernel<G, R>, blocks_for(a.p, lu64_paths<G>()), kLuThreads, smem, st, true, a.n, a.p,
                        (const double2*)a.ext, a.st, a.prm);
}

template <int G, int R>
cudaError_t launch_newton_shape(int n, int64_t p, const void* ext, void* x, int32_t* done, float* last,
                                double tol, const PathMap* pm, cudaStream_t st) {
  const int smem = lu64_smem<G>(n);   // map: n bounds the range's systems
  cudaError_t e = pm ? allow_smem<lu64_smem<G>(G * R)>(newton_kernel<G, R, true>, smem)
                     : allow_smem<lu64_smem<G>(G * R)>(newton_kernel<G, R, false>, smem);
  if (e != cudaSuccess) return e;
  const unsigned nb = blocks_for(p, lu64_paths<G>());
  return pm ? launch_chained(newton_kernel<G, R, true>, nb, kLuThreads, smem, st, true, n, p, (const double2*)ext,
                             (double2*)x, done, last, tol, *pm)
            : launch_chained(newton_kernel<G, R, false>, nb, kLuThreads, smem, st, true, n, p, (const double2*)ext,
                             (double2*)x, done, last, tol, PathMap());
}

cudaError_t launch_newton(int n, int64_t p, const void* ext, void* x, int32_t* done, float* last, double tol,
                          const PathMap* pm, cudaStream_t st) {
  const int sh = lu_shape(n, p);
  return sh == 0 ? launch_newton_shape<8, 1>(n, p, ext, x, done, last, tol, pm, st)
       : sh == 1 ? launch_newton_shape<8, 2>(n, p, ext, x, done, last, tol, pm, st)
       : sh == 2 ? launch_newton_shape<16, 2>(n, p, ext, x, done, last, tol, pm, st)
       : sh == 3 ? launch_newton_shape<32, 1>(n, p, ext, x, done, last, tol, pm, st)
                 : launch_newton_shape<16, 1>(n, p, ext, x, done, last, tol, pm, st);
}

template <int G, int R>
cudaError_t launch_adjoint_shape(hpt_system s, int64_t p, const void* ext, const void* x, const void* gx,
                                 void* contrib, cudaStream_t st) {
  const int smem = lu64_smem<G>(s->n);
  cudaError_t e = allow_smem<lu64_smem<G>(G * R)>(adjoint_kernel<G, R>, smem);
  if (e != cudaSuccess) return e;
  return launch_chained(adjoint_kernel<G, R>, blocks_for(p, lu64_paths<G>()), kLuThreads, smem, st, true, fp64_sys_of(s), p,
                        s->M, (const double2*)ext, (const double2*)x, (const double2*)gx, (double2*)contrib);
}

}  // namespace

cudaError_t launch_solve_update(hpt_system s, const StepArgs& a, cudaStream_t st) {
  if (a.p <= 0) return cudaSuccess;
  cudaError_t e;
  if (s->prec == HPT_FP64) {
    int pi = prof_begin(s, "solve_update_fp64", st);
    const int sh = lu_shape(a.n, a.p);
    e = sh == 0 ? launch_step64_shape<8, 1>(a, st)
      : sh == 1 ? launch_step64_shape<8, 2>(a, st)
      : sh == 2 ? launch_step64_shape<16, 2>(a, st)
      : sh == 3 ? launch_step64_shape<32, 1>(a, st)
                : launch_step64_shape<16, 1>(a, st);
    prof_end(s, pi, st);
    return e;
  }
  const int shape = shape_of(a.n);
  int pi;
  if (shape <= 1) {   // n <= 16: Gauss-Jordan
    pi = prof_begin(s, "solve_gj_fp32", st);
    e = shape == 0 ? launch_gj<8, 1>(a, st) : launch_gj<8, 2>(a, st);
  } else {
    pi = prof_begin(s, "solve_update_fp32", st);
    const int ws = warp_smem<32, 1>(GroupSmem<32>::bytes, a.n), smem = (kSolveThreads / 32) * ws;
    e = allow_smem<(kSolveThreads / 32) * warp_smem<32, 1>(GroupSmem<32>::bytes, kMaxN)>(solve_update_kernel, smem);
    if (e != cudaSuccess) return e;
    e = launch_chained(solve_update_kernel, blocks_for(a.p, kSolveThreads / 32), kSolveThreads, smem, st, true, a.n, a.p,
                       (const float2*)a.ext, a.st, a.prm, ws);
  }
  prof_end(s, pi, st);
  return e;
}

cudaError_t launch_newton_map(int nbound, int64_t cap, const void* ext, void* x, int32_t* done, float* last,
                              double tol, const PathMap& pm, cudaStream_t st) {
  if (cap <= 0) return cudaSuccess;
  if (!pm.list || !pm.tile_sys || !pm.sys_n || !pm.vofs || !pm.npos || !pm.pos_begin) return cudaErrorInvalidValue;
  return launch_newton(nbound, cap, ext, x, done, last, tol, &pm, st);
}

cudaError_t launch_solve_fp32_shape(int shape, const StepArgs& a, cudaStream_t st) {
  if (a.p <= 0) return cudaSuccess;
  return shape == 0 ? launch_gj<8, 1>(a, st)
       : shape == 1 ? launch_gj<8, 2>(a, st)
       : shape == kShape8x3 ? launch_solve_map<8, 3>(a, st)
                            : launch_solve_map<32, 1>(a, st);
}

cudaError_t launch_newton_update(hpt_system s, int64_t p, const void* ext, void* x, int32_t* done,
                                 float* last, double tol, cudaStream_t st) {
  if (p <= 0) return cudaSuccess;
  int pi = prof_begin(s, "newton_fp64", st);
  cudaError_t e = launch_newton(s->n, p, ext, x, done, last, tol, nullptr, st);
  prof_end(s, pi, st);
  return e;
}

size_t adjoint_part_bytes(int M) { return (size_t)kAdjRowBlocks * M * 16; }

cudaError_t launch_adjoint(hpt_system s, int64_t p, const void* ext, const void* x, const void* gx,
                           void* partial, void* part, void* gc, cudaStream_t st) {
  if (p <= 0) return cudaSuccess;
  const int shape = lu_shape(s->n, p);
  int pi = prof_begin(s, "adjoint_fp64", st);
  cudaError_t e = shape == 0 ? launch_adjoint_shape<8, 1>(s, p, ext, x, gx, partial, st)
                : shape == 1 ? launch_adjoint_shape<8, 2>(s, p, ext, x, gx, partial, st)
                : shape == 2 ? launch_adjoint_shape<16, 2>(s, p, ext, x, gx, partial, st)
                : shape == 3 ? launch_adjoint_shape<32, 1>(s, p, ext, x, gx, partial, st)
                             : launch_adjoint_shape<16, 1>(s, p, ext, x, gx, partial, st);
  prof_end(s, pi, st);
  if (e != cudaSuccess) return e;
  pi = prof_begin(s, "adjoint_sum", st);
  e = launch_chained(sum_columns_part_kernel, dim3((unsigned)((s->M + 31) / 32), kAdjRowBlocks), 1024, 0, st, true, p, s->M,
                     (const double2*)partial, (double2*)part);
  if (e == cudaSuccess)
    e = launch_chained(sum_columns_kernel, blocks_for(s->M, 32), 32, 0, st, true, s->M, (const double2*)part, (double2*)gc);
  prof_end(s, pi, st);
  return e;
}

cudaError_t launch_paths_init(hpt_system s, int64_t p, const void* y0, double tau0,
                              const hpt_params& prm, const hpt_paths& S, cudaStream_t st) {
  if (p <= 0) return cudaSuccess;
  const unsigned nb = blocks_for(p * s->n, 256);
  if (s->prec == HPT_FP64)
    paths_init_kernel<double><<<nb, 256, 0, st>>>(s->n, p, (const double2*)y0, tau0, prm.dtau_init, S);
  else
    paths_init_kernel<float><<<nb, 256, 0, st>>>(s->n, p, (const double2*)y0, tau0, prm.dtau_init, S);
  return cudaGetLastError();
}

cudaError_t launch_count_active(int64_t p, const int32_t* status, int32_t* count, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(count, 0, sizeof(int32_t), st);
  if (e != cudaSuccess || p <= 0) return e;
  unsigned nb = blocks_for(p, 256);
  if (nb > 1024) nb = 1024;
  count_active_kernel<<<nb, 256, 0, st>>>(p, status, count);
  return cudaGetLastError();
}

cudaError_t launch_finish_track(hpt_system s, int64_t p, const hpt_paths& S, void* x_out,
                                int32_t* status_out, int32_t* steps_out, int32_t* done,
                                cudaStream_t st) {
  if (p <= 0) return cudaSuccess;
  const unsigned nb = blocks_for(p * s->n, 256);
  if (s->prec == HPT_FP64)
    finish_track_kernel<double><<<nb, 256, 0, st>>>(s->n, p, S, (double2*)x_out, status_out, steps_out, done);
  else
    finish_track_kernel<float><<<nb, 256, 0, st>>>(s->n, p, S, (double2*)x_out, status_out, steps_out, done);
  return cudaGetLastError();
}

cudaError_t launch_init_done(int64_t p, const int32_t* status, int32_t* done, cudaStream_t st) {
  if (p <= 0) return cudaSuccess;
  init_done_kernel<<<blocks_for(p, 256), 256, 0, st>>>(p, status, done);
  return cudaGetLastError();
}

}  // namespace hpt
