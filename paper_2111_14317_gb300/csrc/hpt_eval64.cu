// FP64 evaluation of the homotopy and its extended Jacobian (Algorithm 2,
// Section 5) on the CUDA cores.
//
// For every point: z = log y (eq. (6)); for every monomial W = <z, a> +
// tau e/D (one row of Z A, eq. (7)); E = exp(W); the extended Jacobian row of
// equation k is sum_i E_i B_k[:, i] = [D_z h_k | D_tau h_k | h_k] (eq. (8) and
// the extended-Jacobian identity), and D_y h_k = D_z h_k diag(e^{-z}).
//
// The same kernels serve the projective form (Section 2.2): n equations in nv
// = n + 1 homogeneous coordinates, exponents (a, deg_k - 1^T a); the extended
// Jacobian row is then [D_z h_k (nv entries) | D_tau h_k | h_k].
//
// Two kernels.  eval_fx_kernel is the one that runs: it keeps the FP64 pipe
// (two lanes a clock per SM) for the sums that need it, 2 nnz + 4 operations
// per monomial with nnz nonzero exponents, and does the rest in integers.
// eval_fp64_kernel takes the systems whose exponents are beyond the fixed
// point's range (kFxSum, kFxTexp).
#include <math.h>

#include <algorithm>

#include "hpt_fx.cuh"
#include "hpt_internal.h"

namespace hpt {
namespace {

// Mapping of eval_fp64_kernel: a block owns 32 points (one per lane) and its
// four warps take the equations k = warp, warp + 4, ...; all lanes of a warp
// read the same monomial constants (broadcast), z is staged in shared memory
// transposed so that lane q reads column q without bank conflicts.
// MAP: 32 consecutive positions of a position map per block (inside one
// 128-position tile, so one system: S from the per-system table); otherwise
// positions are the paths of the single system S.  NMAX bounds the variables.
template <int NMAX, bool MAP>
__global__ void __launch_bounds__(128)
eval_fp64_kernel(Fp64Sys S, int64_t p, const double2* __restrict__ y, const double* __restrict__ tin,
                 int tau_is_t, double2* __restrict__ ext, double2* __restrict__ oH, double2* __restrict__ oHy,
                 double2* __restrict__ oHt, PathMap pm, const Fp64Sys* __restrict__ tab) {
  __shared__ double2 zs[NMAX][32];
  __shared__ double2 iys[NMAX][32];
  __shared__ double taus[32];
  __shared__ double tinv[32];
  __shared__ int64_t spath[32];
  int64_t base = (int64_t)blockIdx.x * 32;
  int nmax = S.nv;
  if (MAP) {
    base += *pm.pos_begin;
    if (base >= *pm.npos) return;
    S = tab[pm.tile_sys[base >> 7]];
    nmax = pm.nmax;
  }
  const int n = S.n, nv = S.nv;
  const int32_t* __restrict__ msz = S.msz;
  const int32_t* __restrict__ off = S.off;
  const double* __restrict__ ahat = S.ahat;
  const double2* __restrict__ bcol = S.b;
  if (threadIdx.x < 32) {
    const int64_t q = base + threadIdx.x;
    spath[threadIdx.x] = MAP ? pm.list[q] : (q < p ? q : -1);
  }
  __syncthreads();

  // op. 1 of Algorithm 2: Z <- log Y (principal branch), and 1/y for the
  // final diag(e^{-z}) scaling.
  for (int idx = threadIdx.x; idx < 32 * nv; idx += blockDim.x) {
    const int q = idx / nv, j = idx - q * nv;
    const int64_t path = spath[q];
    double2 v = make_double2(1.0, 0.0);
    if (path >= 0) v = y[(MAP ? (size_t)pm.vofs[path] : (size_t)path * nv) + j];
    const double r2 = v.x * v.x + v.y * v.y;
    zs[j][q] = make_double2(log(hypot(v.x, v.y)), atan2(v.y, v.x));
    iys[j][q] = make_double2(v.x / r2, -v.y / r2);
  }
  if (threadIdx.x < 32) {
    const int64_t path = spath[threadIdx.x];
    double tv = (path >= 0 && tin) ? tin[path] : (tau_is_t ? 1.0 : 0.0);   // no tin: t = 1
    double tau = tau_is_t ? log(tv) : tv;
    taus[threadIdx.x] = tau;
    tinv[threadIdx.x] = tau_is_t ? 1.0 / tv : exp(-tau);
  }
  __syncthreads();

  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t path = spath[lane];
  const int64_t pos = base + lane;
  const double tau = taus[lane];
  const int np2 = nv + 2;
  for (int k = warp; k < n; k += 4) {
    double2 accJ[NMAX];
#pragma unroll
    for (int u = 0; u < NMAX; ++u) accJ[u] = make_double2(0.0, 0.0);
    double2 accT = make_double2(0.0, 0.0), accH = make_double2(0.0, 0.0);
    const int i0 = off[k], i1 = off[k] + msz[k];
    for (int i = i0; i < i1; ++i) {
      // op. 2 of Algorithm 2, one monomial: W = [z, tau] . A[:, i]
      const double* a = ahat + (size_t)i * (nv + 1);
      double wr = a[nv] * tau, wi = 0.0;
#pragma unroll
      for (int j = 0; j < NMAX; ++j) {
        if (j < nv) {
          const double aj = a[j];
          const double2 z = zs[j][lane];
          wr = fma(aj, z.x, wr);
          wi = fma(aj, z.y, wi);
        }
      }
      double sn, cs;
      sincos(wi, &sn, &cs);
      const double mag = exp(wr);
      const double er = mag * cs, ei = mag * sn;
      // ... times B_k[:, i] (complex), accumulated over the equation's monomials
      const double2* bb = bcol + (size_t)i * np2;
#pragma unroll
      for (int u = 0; u < NMAX; ++u) {
        if (u < nv) {
          const double2 c = bb[u];
          accJ[u].x = fma(er, c.x, fma(-ei, c.y, accJ[u].x));
          accJ[u].y = fma(er, c.y, fma(ei, c.x, accJ[u].y));
        }
      }
      const double2 ct = bb[nv], ch = bb[nv + 1];
      accT.x = fma(er, ct.x, fma(-ei, ct.y, accT.x));
      accT.y = fma(er, ct.y, fma(ei, ct.x, accT.y));
      accH.x = fma(er, ch.x, fma(-ei, ch.y, accH.x));
      accH.y = fma(er, ch.y, fma(ei, ch.x, accH.y));
    }
    if (path < 0) continue;
    // the step scratch keeps D_z h_k: op. 3 of Algorithm 2 (the diag(e^{-z})
    // scaling) is applied by the solve to its n-vector solutions instead of
    // to the n x n block here
    if (ext) {
#pragma unroll
      for (int u = 0; u < NMAX; ++u)
        if (u < nv) ext[ext_index(pos, k, u, nmax)] = accJ[u];
      ext[ext_index(pos, k, nv, nmax)] = accT;
      ext[ext_index(pos, k, nv + 1, nmax)] = accH;
    }
    // op. 3 of Algorithm 2 for the caller's H_y: D_y h_k = D_z h_k diag(e^{-z})
    if (oHy) {
      double2* row = oHy + ((size_t)path * n + k) * nv;
#pragma unroll
      for (int u = 0; u < NMAX; ++u) {
        if (u < nv) {
          const double2 iy = iys[u][lane];
          row[u] = make_double2(accJ[u].x * iy.x - accJ[u].y * iy.y, accJ[u].x * iy.y + accJ[u].y * iy.x);
        }
      }
    }
    if (oH) oH[(size_t)path * n + k] = accH;
    if (oHt) {
      const double ti = tinv[lane];   // dH/dt = (dH/dtau) / t
      oHt[(size_t)path * n + k] = make_double2(accT.x * ti, accT.y * ti);
    }
  }
}

// One monomial of the fixed-point evaluation.  op. 2 of Algorithm 2: W = log c
// + [z, tau] . A[:, i] ..
__device__ __forceinline__ fx::Sum fx_begin(const FxMono& m, const fx::Wide& tw, float tf) {
  fx::Sum s{(uint64_t)m.lc, m.turn, fmaf(m.ef, tf, m.lcf)};
  if (m.e) s.w += fx::times((int64_t)m.e, tw);
  return s;
}
__device__ __forceinline__ void fx_add(const FxEnt& e, const ulonglong2* zl, const float* ll, fx::Sum& s) {
  const ulonglong2 z = zl[e.j * 32];
  fx::add_power(s, e.a, z.x, z.y, ll[e.j * 32]);
}
// The FP32 sum of a monomial at a point with coordinates 0 or infinite (mask;
// their log2|y| is -inf or +inf in ll), or with tau infinite: -inf (the
// monomial is 0), or NaN where the product is not defined: a factor infinite,
// 0 times infinity, or such a coordinate (or t) to the power 0, as
// exp(<a, log y>) has it.
__device__ __noinline__ float fx_special(const FxMono* __restrict__ mono, const FxEnt* __restrict__ en, uint32_t mask,
                                         float tf, const float* ll) {
  const FxMono m = *mono;
  float f = m.e ? m.ef * tf : tf - tf;
  f += m.lcf;
  for (int t = 0; t < m.nnz; ++t) {
    const FxEnt x = en[t];
    f += (float)x.a * ll[x.j * 32];
    mask &= ~(1u << x.j);
  }
  return mask ? __int_as_float(0x7fffffff) : f;
}
// .. and its value times (a, e/D, 1), accumulated over the equation's
// monomials.
__device__ __forceinline__ void fx_accumulate(const FxMono& m, const FxEnt* __restrict__ en, double er, double ei,
                                              double2* acc, double2& accT, double2& accH) {
  accH.x += er;
  accH.y += ei;
  if (m.e) {
    accT.x = fma(m.eD, er, accT.x);
    accT.y = fma(m.eD, ei, accT.y);
  }
  int t = 0;
  for (; t + 4 <= m.nnz; t += 4) {
    double2 v[4];
    FxEnt x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) x[u] = en[t + u];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = acc[x[u].j * 32];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      v[u].x = fma(x[u].ad, er, v[u].x);
      v[u].y = fma(x[u].ad, ei, v[u].y);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) acc[x[u].j * 32] = v[u];   // the entries of a monomial are distinct
  }
  for (; t < m.nnz; ++t) {
    const FxEnt x = en[t];
    double2 v = acc[x.j * 32];
    v.x = fma(x.ad, er, v.x);
    v.y = fma(x.ad, ei, v.y);
    acc[x.j * 32] = v;
  }
}

// The fixed-point evaluation.  A block of four warps owns 32 points, one per
// lane; warp w takes the equations 4 g + w of its group g = blockIdx.y (groups
// share a tile's points, so that few tiles still fill the chip).
//
// What bounds it: the FP64 pipe.  Per monomial the exponent sum is integer
// (log2|y| and the phase in fixed point, the t-part as e times a 128-bit
// tau log2(e)/D), the coefficient enters the sum as its own logarithm, exp2
// and sincos are integer too, and FP64 only adds a_j T to the entries with
// a_j != 0, e/D T to D_tau h and T to h.  The accumulators of D_z h live in
// shared memory, since the entry is known at run time only; the nonzeros of a
// monomial are taken four at a time to cover the round trip.  The dense form
// (eval_fp64_kernel: FP64 dot products, exp, sincos, complex B columns over
// all variables) issues about 10 nv + 70 FP64 instructions a monomial.
template <bool MAP>
__global__ void __launch_bounds__(128)
eval_fx_kernel(Fp64Sys S, int64_t p, const double2* __restrict__ y, const double* __restrict__ tin, int tau_is_t,
               double2* __restrict__ ext, double2* __restrict__ oH, double2* __restrict__ oHy,
               double2* __restrict__ oHt, PathMap pm, const Fp64Sys* __restrict__ tab, int nvs) {
  extern __shared__ __align__(16) unsigned char smem[];
  // [log coordinates: nvs x 32 (l, turn)][accumulators: 4 x nvs x 32][1/y: nvs x 32, for H_y only]
  // [log2|y| in FP32: nvs x 32]
  ulonglong2* zs = (ulonglong2*)smem;
  double2* accs = (double2*)(zs + nvs * 32);
  double2* iys = accs + 4 * nvs * 32;
  float* lfs = (float*)(iys + (oHy ? nvs * 32 : 0));
  __shared__ int64_t exp1[64], exp2[64], cs1[64][2], cs2[64][2];
  __shared__ uint64_t tau_hi[32], tau_lo[32];
  __shared__ float tau_f[32], tau_inf[32];   // NaN in tau_f sends a point's monomials to fx_special
  __shared__ uint32_t special[32];           // coordinates 0 or infinite
  __shared__ double tinv[32];
  __shared__ int64_t spath[32];
  grid_wait();
  int64_t base = (int64_t)blockIdx.x * 32;
  int nmax = S.nv;
  if (MAP) {
    base += *pm.pos_begin;
    if (base >= *pm.npos) return;
    S = tab[pm.tile_sys[base >> 7]];
    nmax = pm.nmax;
  }
  const int n = S.n, nv = S.nv;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x < 32) {
    const int64_t q = base + threadIdx.x;
    const int64_t path = MAP ? pm.list[q] : (q < p ? q : -1);
    spath[threadIdx.x] = path;
    const double tv = (path >= 0 && tin) ? tin[path] : (tau_is_t ? 1.0 : 0.0);   // no tin: t = 1
    const double tau = !tin ? 0.0 : (tau_is_t ? log(tv) : tv);
    const bool fin = isfinite(tau);
    fx::Wide w{0, 0};
    float tf = 0.f;
    if (tin && fin) {
      const double td = S.D == 1.0 ? tau : tau / S.D;
      w = fx::log2e_times(td);
      tf = (float)fmin(fmax(td, -1e30), 1e30) * 1.44269504f;   // finite, so that e = 0 takes nothing of it
    }
    tau_hi[threadIdx.x] = w.hi;
    tau_lo[threadIdx.x] = w.lo;
    tau_f[threadIdx.x] = fin ? tf : __int_as_float(0x7fffffff);
    tau_inf[threadIdx.x] = fin ? tf : (float)tau;
    special[threadIdx.x] = 0;
    if (oHt) tinv[threadIdx.x] = 1.0 / tv;   // user layout: t is given
  }
  if (threadIdx.x >= 64) {   // the last two warps stage the tables
    const int i = threadIdx.x - 64;
    const fx::Tables& T = fx::tables();
    exp1[i] = T.exp1[i];
    exp2[i] = T.exp2[i];
    cs1[i][0] = T.cs1[i][0];
    cs1[i][1] = T.cs1[i][1];
    cs2[i][0] = T.cs2[i][0];
    cs2[i][1] = T.cs2[i][1];
  }
  __syncthreads();

  // op. 1 of Algorithm 2: Z <- log Y, and 1/y for the final diag(e^{-z})
  // scaling.  A coordinate without a logarithm: 0 and infinity are fx_special's
  // (its sums are -inf or NaN), NaN makes the whole point NaN.
  for (int idx = threadIdx.x; idx < 32 * nv; idx += 128) {
    const int q = idx / nv, j = idx - q * nv;
    const int64_t path = spath[q];
    double2 v = make_double2(1.0, 0.0);
    if (path >= 0) v = y[(MAP ? (size_t)pm.vofs[path] : (size_t)path * nv) + j];
    fx::Log lg;
    if (!fx::log_of(v.x, v.y, lg)) {
      tau_f[q] = __int_as_float(0x7fffffff);
      lg.lf = v.x != v.x || v.y != v.y ? __int_as_float(0x7fffffff) : (v.x == 0.0 && v.y == 0.0 ? -INFINITY : INFINITY);
      atomicOr(&special[q], 1u << j);
    }
    zs[j * 32 + q] = make_ulonglong2((unsigned long long)lg.l, lg.turn);
    lfs[j * 32 + q] = lg.lf;
    if (oHy) {
      const double r2 = v.x * v.x + v.y * v.y;
      iys[j * 32 + q] = make_double2(v.x / r2, -v.y / r2);
    }
  }
  __syncthreads();

  const int64_t path = spath[lane];
  const int64_t pos = base + lane;
  const fx::Wide tw{tau_hi[lane], tau_lo[lane]};
  const float tf = tau_f[lane];
  double2* acc = accs + (size_t)warp * nvs * 32 + lane;
  const ulonglong2* zl = zs + lane;
  const float* ll = lfs + lane;
  for (int k = blockIdx.y * 4 + warp; k < n; k += 4 * gridDim.y) {
    for (int u = 0; u < nv; ++u) acc[u * 32] = make_double2(0.0, 0.0);
    double2 accT = make_double2(0.0, 0.0), accH = make_double2(0.0, 0.0);
    const int i0 = S.off[k], i1 = i0 + S.msz[k];
    // two monomials at a time: their integer chains interleave (1.075 -> 1.048 ms
    // at the size above, 43 -> 39 us at n = 24, 1,000 points)
    for (int i = i0; i < i1; i += 2) {
      const int two = i + 1 < i1;   // the last one of an odd support stands in for its partner
      const FxMono m0 = S.mono[i], m1 = S.mono[i + two];
      const FxEnt* __restrict__ e0 = S.ent + m0.ent;
      const FxEnt* __restrict__ e1 = S.ent + m1.ent;
      fx::Sum s0 = fx_begin(m0, tw, tf), s1 = fx_begin(m1, tw, tf);
      const int both = min(m0.nnz, m1.nnz);
      int t = 0;
#pragma unroll 4
      for (; t < both; ++t) {
        fx_add(e0[t], zl, ll, s0);
        fx_add(e1[t], zl, ll, s1);
      }
      for (int u = t; u < m0.nnz; ++u) fx_add(e0[u], zl, ll, s0);
      for (int u = t; u < m1.nnz; ++u) fx_add(e1[u], zl, ll, s1);
      double er0, ei0, er1, ei1;
      if (fx::exp_in_range(s0.f) && fx::exp_in_range(s1.f)) {
        fx::exp_in((int64_t)s0.w, s0.turn, s0.f, exp1, exp2, cs1, cs2, er0, ei0);
        fx::exp_in((int64_t)s1.w, s1.turn, s1.f, exp1, exp2, cs1, cs2, er1, ei1);
      } else {
        if (tf != tf) {
          s0.f = fx_special(S.mono + i, e0, special[lane], tau_inf[lane], ll);
          s1.f = fx_special(S.mono + i + two, e1, special[lane], tau_inf[lane], ll);
        }
        fx::exp_of((int64_t)s0.w, s0.turn, s0.f, exp1, exp2, cs1, cs2, er0, ei0);
        fx::exp_of((int64_t)s1.w, s1.turn, s1.f, exp1, exp2, cs1, cs2, er1, ei1);
      }
      fx_accumulate(m0, e0, er0, ei0, acc, accT, accH);
      if (two) fx_accumulate(m1, e1, er1, ei1, acc, accT, accH);
    }
    if (path < 0) continue;
    // a row whose sum is not finite (a point without a logarithm, a monomial
    // past the range) is NaN in every entry
    const bool bad = !(isfinite(accH.x) && isfinite(accH.y));
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    // the step scratch keeps D_z h_k: op. 3 of Algorithm 2 (the diag(e^{-z})
    // scaling) is applied by the solve to its n-vector solutions instead of
    // to the n x n block here
    if (ext) {
      for (int u = 0; u < nv; ++u) ext[ext_index(pos, k, u, nmax)] = bad ? make_double2(nan, nan) : acc[u * 32];
      ext[ext_index(pos, k, nv, nmax)] = bad ? make_double2(nan, nan) : accT;
      ext[ext_index(pos, k, nv + 1, nmax)] = accH;
    }
    // op. 3 of Algorithm 2 for the caller's H_y: D_y h_k = D_z h_k diag(e^{-z})
    if (oHy) {
      double2* row = oHy + ((size_t)path * n + k) * nv;
      for (int u = 0; u < nv; ++u) {
        const double2 iy = iys[u * 32 + lane], v = acc[u * 32];
        row[u] = bad ? make_double2(nan, nan) : make_double2(v.x * iy.x - v.y * iy.y, v.x * iy.y + v.y * iy.x);
      }
    }
    if (oH) oH[(size_t)path * n + k] = accH;
    if (oHt) {
      const double ti = tinv[lane];   // dH/dt = (dH/dtau) / t
      oHt[(size_t)path * n + k] = bad ? make_double2(nan, nan) : make_double2(accT.x * ti, accT.y * ti);
    }
  }
}

constexpr int fx_smem(int nvs, bool hy) { return nvs * 32 * (16 + 4 * 16 + (hy ? 16 : 0) + 4); }

// Equation groups per tile: a block takes as many rounds of four equations as
// still leave kFxBlocks blocks (the logarithms of a tile's points are taken
// once per block).
constexpr int64_t kFxBlocks = 152 * 4 * 6;
int fx_groups(int64_t tiles, int n) {
  const int64_t n4 = (n + 3) / 4;
  const int64_t rounds = std::max<int64_t>(1, std::min<int64_t>(n4, n4 * tiles / kFxBlocks));
  return (int)((n4 + rounds - 1) / rounds);
}

template <bool MAP>
cudaError_t launch_fx(const Fp64Sys& f, int nvs, int neq, int64_t p, const double2* y, const double* tau, int tau_is_t,
                      double2* ext, double2* H, double2* Hy, double2* Ht, const PathMap& pm, const Fp64Sys* tab,
                      cudaStream_t st) {
  const int64_t tiles = (p + 31) / 32;
  if (tiles > 0x7fffffff) return cudaErrorInvalidValue;
  const int smem = fx_smem(nvs, Hy != nullptr);
  const cudaError_t e = allow_smem<fx_smem(kMaxN, true)>(eval_fx_kernel<MAP>, smem);
  if (e != cudaSuccess) return e;
  return launch_chained(eval_fx_kernel<MAP>, dim3((unsigned)tiles, (unsigned)fx_groups(tiles, neq)), 128, smem, st,
                        ext != nullptr, f, p, y, tau, tau_is_t, ext, H, Hy, Ht, pm, tab, nvs);
}

}  // namespace

Fp64Sys fp64_sys_of(const hpt_system s) {
  Fp64Sys f;
  f.n = s->n;
  f.nv = s->nv;
  f.msz = s->d_msz;
  f.off = s->d_off;
  f.ahat = s->d_ahat;
  f.b = (const double2*)s->d_b;
  f.mono = s->d_mono;
  f.ent = s->d_ent;
  f.D = (double)s->D;
  return f;
}

cudaError_t launch_eval_fp64(hpt_system s, int64_t p, const void* y, const double* tau,
                             int tau_is_t, const EvalOut& out, cudaStream_t st) {
  if (p <= 0) return cudaSuccess;
  const int64_t blocks = (p + 31) / 32;
  if (blocks > 0x7fffffff) return cudaErrorInvalidValue;
  int pi = prof_begin(s, "eval_fp64", st);
  const double2* yy = (const double2*)y;
  double2* ext = (double2*)out.ext;
  double2* H = (double2*)out.H;
  double2* Hy = (double2*)out.Hy;
  double2* Ht = (double2*)out.Ht;
  const Fp64Sys f = fp64_sys_of(s);
  const PathMap none;
  if (s->d_mono) {
    const cudaError_t e = launch_fx<false>(f, s->nv, s->n, p, yy, tau, tau_is_t, ext, H, Hy, Ht, none, nullptr, st);
    prof_end(s, pi, st);
    return e;
  }
  if (s->nv <= 8)
    eval_fp64_kernel<8, false><<<(unsigned)blocks, 128, 0, st>>>(f, p, yy, tau, tau_is_t, ext, H, Hy, Ht, none, nullptr);
  else if (s->nv <= 16)
    eval_fp64_kernel<16, false><<<(unsigned)blocks, 128, 0, st>>>(f, p, yy, tau, tau_is_t, ext, H, Hy, Ht, none, nullptr);
  else if (s->nv <= 24)
    eval_fp64_kernel<24, false><<<(unsigned)blocks, 128, 0, st>>>(f, p, yy, tau, tau_is_t, ext, H, Hy, Ht, none, nullptr);
  else
    eval_fp64_kernel<32, false><<<(unsigned)blocks, 128, 0, st>>>(f, p, yy, tau, tau_is_t, ext, H, Hy, Ht, none, nullptr);
  prof_end(s, pi, st);
  return cudaGetLastError();
}

cudaError_t launch_eval_fp64_map(int shape, const Fp64Sys* tab, bool fixed, int64_t cap, const void* y, const double* tau,
                                 const PathMap& pm, void* ext, cudaStream_t st) {
  if (cap <= 0) return cudaSuccess;
  if (!pm.list || !pm.tile_sys || !pm.vofs || !pm.npos || !pm.pos_begin || !tab) return cudaErrorInvalidValue;
  const int64_t blocks = (cap + 31) / 32;
  if (blocks > 0x7fffffff) return cudaErrorInvalidValue;
  const Fp64Sys f{};
  const double2* yy = (const double2*)y;
  double2* e = (double2*)ext;
  if (fixed) {
    const int nvs = shape == 0 ? 8 : (shape == 1 ? 16 : (shape == kEval24 ? 24 : kMaxN));
    return launch_fx<true>(f, nvs, nvs, cap, yy, tau, 0, e, nullptr, nullptr, nullptr, pm, tab, st);
  }
  if (shape == 0)
    eval_fp64_kernel<8, true><<<(unsigned)blocks, 128, 0, st>>>(f, cap, yy, tau, 0, e, nullptr, nullptr, nullptr, pm, tab);
  else if (shape == 1)
    eval_fp64_kernel<16, true><<<(unsigned)blocks, 128, 0, st>>>(f, cap, yy, tau, 0, e, nullptr, nullptr, nullptr, pm, tab);
  else if (shape == kEval24)
    eval_fp64_kernel<24, true><<<(unsigned)blocks, 128, 0, st>>>(f, cap, yy, tau, 0, e, nullptr, nullptr, nullptr, pm, tab);
  else
    eval_fp64_kernel<32, true><<<(unsigned)blocks, 128, 0, st>>>(f, cap, yy, tau, 0, e, nullptr, nullptr, nullptr, pm, tab);
  return cudaGetLastError();
}

}  // namespace hpt
