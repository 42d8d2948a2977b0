// FP64 solve of one path's consolidated system in shared memory, for the FP64
// step (affine and projective), the directions, the polish, the adjoint and the
// mixed step's re-solves.  Internal to libhpt.
//
// What bounds an FP64 solve on sm_103a is the FP64 pipe, two lanes a clock
// per SM: one warp-wide FP64 instruction takes as long as 64 issue slots,
// whether its lanes carry live matrix entries or not.  So the layout serves
// one aim, that every lane of every FP64 instruction does needed work: the
// matrix sits in shared memory, and each elimination step deals the live
// entries (rows below the pivot x columns right of it and the right-hand
// sides) one by one to the group's G lanes.  With rows in registers (one or
// two a lane) the finished rows and the rounded-up widths were updated too,
// 2.2 times the operations.  Everything else runs in integers: finiteness,
// the power-of-two equilibration (exponent fields), the pivot search (FP32
// magnitudes from the bit pattern).  The arithmetic of an entry does not
// depend on G, so every G gives the same bits.
// Measured, n = 16, 65,536 paths (8 lanes each): 3.4 -> 1.30 ms for solve and
// step control (needed FP64 operations alone: 0.95 ms); n = 24, 1,000 paths
// (32 lanes each): 275 -> 110 us a step.
#pragma once

#include "hpt_cx.cuh"
#include "hpt_internal.h"

namespace hpt {
namespace {

constexpr int kLuThreads = 128;

// Entries of one path's region: n rows of n + 2, padded to an odd count so
// that the staging stores of eight neighbouring paths fall on distinct banks;
// then the column exponents (n ints).
__host__ __device__ constexpr int lu64_entries(int n) { return (n * (n + 2)) | 1; }
__host__ __device__ constexpr int lu64_col_entries(int n) { return (n + 3) / 4; }   // ints, in double2 units
template <int G>
__host__ __device__ constexpr int lu64_paths() { return kLuThreads / G; }
template <int G>
constexpr int lu64_smem(int n) { return lu64_paths<G>() * (lu64_entries(n) + lu64_col_entries(n)) * 16; }

__device__ __forceinline__ int exp_field(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }
// v 2^k, in integers; operands and results below the normal range (and
// overflows) go to the library's, zeros, infinities and NaN stay.
__device__ __noinline__ double scale_far(double v, int k) { return scalbn(v, k); }
__device__ __forceinline__ double scale_exp(double v, int k) {
  const int hi = __double2hiint(v), lo = __double2loint(v), e = (hi >> 20) & 0x7ff;
  const bool in = (unsigned)(e - 1) < 0x7feu && (unsigned)(e + k - 1) < 0x7feu;
  if (!in && e != 0x7ff && ((hi << 1) | lo) != 0) return scale_far(v, k);   // seldom, so no branch for the zeros
  return __hiloint2double(hi + (in ? (int)((unsigned)k << 20) : 0), lo);
}
// FP32 copy by bit pattern (truncated; 0 below FP32's range, infinity above).
__device__ __forceinline__ float trunc_f32(double v) {
  const int hi = __double2hiint(v), e = (hi >> 20) & 0x7ff;
  if (e < 897) return 0.f;
  if (e > 1150) return __int_as_float(0x7f800000);
  return __int_as_float(((e - 896) << 23) | ((hi & 0xfffff) << 3) | (int)((unsigned)__double2loint(v) >> 29));
}
// 1/v for a normal v (and a normal 1/v): the hardware's approximation, whose
// relative error squares in each of the two Newton steps (from about 2^-20 to
// 2^-40 and below 2^-75), so that only the last fma's rounding is left.
__device__ __forceinline__ double rcp_newton(double v) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(v));
  r = fma(r, fma(-v, r, 1.0), r);
  return fma(r, fma(-v, r, 1.0), r);
}

// Stages the block's paths: thread t reads the entries t / P, t / P + G, ..
// of path t % P (P = 128 / G paths, consecutive positions from q0), so that P
// threads read consecutive addresses of the position-interleaved scratch.
// conj: the entry (k, u < n) goes to row u, column k, conjugated (the adjoint
// system); the right-hand sides are then the caller's.  rows < n: the
// projective system's equations (its last row is the caller's).
template <int G>
__device__ __forceinline__ void lu64_stage(int rows, int n, int nmax, const double2* __restrict__ ext, int64_t q, bool act,
                                           double2* region, bool conj) {
  if (!act) return;
  const int np2 = n + 2, e0 = threadIdx.x / lu64_paths<G>();
  const double2* src = ext + (size_t)(q >> 7) * (size_t)(nmax * (nmax + 2)) * 128 + (size_t)(q & 127);
  if (nmax == n && !conj) {
    const int total = rows * np2;
#pragma unroll 6
    for (int e = e0; e < total; e += G) region[e] = src[(size_t)e * 128];
    return;
  }
  const int w = conj ? n : np2;
  for (int e = e0; e < rows * w; e += G) {
    const int k = e / w, u = e - k * w;
    const double2 v = src[((size_t)k * (nmax + 2) + u) * 128];
    if (conj) region[u * np2 + k] = make_double2(v.x, -v.y);
    else region[k * np2 + u] = v;
  }
}

// Solves region [A | b0 | b1] (rows of n + 2) in place by LU with partial
// pivoting; the columns n, n + 1 then hold the solutions.  sign -1 solves for
// -b.  Returns false (group-uniform) when an entry is not finite or a pivot is
// zero or not finite.  Call with the warp converged and the same n for all
// its groups.
template <int G>
__device__ __forceinline__ bool lu64_solve(int n, double2* A, int* colx, int sign) {
  const int lane = threadIdx.x & (G - 1), LD = n + 2;
  constexpr int R = 32 / G;   // columns (or rows) a lane owns in the equilibration, n <= 32
  // exponents: each row's largest, then each column's largest after the row
  // scaling (the row's entries become < 1, the columns' likewise)
  int colmax[R], bad = 0;
#pragma unroll
  for (int t = 0; t < R; ++t) colmax[t] = 0;
  for (int r = 0; r < n; ++r) {
    int ex[R], m = 0;
#pragma unroll
    for (int t = 0; t < R; ++t) {
      ex[t] = 0;
      const int c = lane + G * t;
      if (c < n) {
        const double2 v = A[r * LD + c];
        ex[t] = max(exp_field(v.x), exp_field(v.y));
      }
      m = max(m, ex[t]);
    }
    if (lane < 2) {
      const double2 v = A[r * LD + n + lane];
      bad |= max(exp_field(v.x), exp_field(v.y)) == 0x7ff;
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o, G));
    bad |= m == 0x7ff;
    const int kr = m == 0 ? 0 : 1022 - m;
#pragma unroll
    for (int t = 0; t < R; ++t) {
      const int c = lane + G * t;
      if (c < n) {
        const double2 v = A[r * LD + c];
        const double x = scale_exp(v.x, kr), y = scale_exp(v.y, kr);
        colmax[t] = max(colmax[t], max(exp_field(x), exp_field(y)));
        A[r * LD + c] = make_double2(x, y);
      }
    }
    if (lane < 2) {
      const double2 v = A[r * LD + n + lane];
      const double x = scale_exp(v.x, kr), y = scale_exp(v.y, kr);
      A[r * LD + n + lane] = sign < 0 ? make_double2(-x, -y) : make_double2(x, y);
    }
  }
  const bool fin = (__ballot_sync(0xffffffffu, bad) & group_mask<G>()) == 0;
#pragma unroll
  for (int t = 0; t < R; ++t) {
    const int c = lane + G * t;
    if (c < n) {
      const int kc = colmax[t] == 0 ? 0 : 1022 - colmax[t];
      colx[c] = kc;
      for (int r = 0; r < n; ++r) {
        const double2 v = A[r * LD + c];
        A[r * LD + c] = make_double2(scale_exp(v.x, kc), scale_exp(v.y, kc));
      }
    }
  }
  __syncwarp();
  bool ok = fin;
  for (int j = 0; j < n; ++j) {
    // pivot: largest |.|^2 of the column's live rows, ties to the upper row
    unsigned key = 0u;
    for (int i = j + lane; i < n; i += G) {
      const double2 v = A[i * LD + j];
      const float x = trunc_f32(v.x), y = trunc_f32(v.y);
      key = max(key, (__float_as_uint(x * x + y * y) & ~31u) | (unsigned)(31 - i));
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) key = max(key, __shfl_xor_sync(0xffffffffu, key, o, G));
    const int br = 31 - (int)(key & 31u);
    if (br != j) {
      for (int c = j + lane; c < LD; c += G) {
        const double2 u = A[j * LD + c], v = A[br * LD + c];
        A[j * LD + c] = v;
        A[br * LD + c] = u;
      }
    }
    __syncwarp();
    const double2 pj = A[j * LD + j];
    const double p2 = pj.x * pj.x + pj.y * pj.y;
    double rp = rcp_newton(p2);
    if (exp_field(p2) == 0 || exp_field(p2) == 0x7ff) {   // seldom: the reciprocal by division while it is finite
      rp = 1.0 / p2;
      if (!(p2 > 0.0) || exp_field(p2) == 0x7ff || exp_field(rp) == 0x7ff) ok = false;
    }
    const double2 inv = make_double2(pj.x * rp, -pj.y * rp);
    for (int i = j + 1 + lane; i < n; i += G) {
      const double2 v = A[i * LD + j];
      A[i * LD + j] = make_double2(fma(v.x, inv.x, -(v.y * inv.y)), fma(v.x, inv.y, v.y * inv.x));
    }
    __syncwarp();
    if (lane == 0) A[j * LD + j] = inv;   // read again by the back substitution only
    // the live block, dealt entry by entry, four in flight
    const unsigned w = (unsigned)(LD - 1 - j), total = w * (unsigned)(n - 1 - j);
    const unsigned magic = 0xffffffffu / w + 1u;   // e / w for e < 2^16
    double2* B = A + (j + 1) * LD + j + 1;
    const double2* Urow = A + j * LD + j + 1;
    unsigned e = lane;
    for (; e + 3 * G < total; e += 4 * G) {
      double2 a[4], l[4], u[4];
      unsigned at[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const unsigned r = __umulhi(e + t * G, magic), c = e + t * G - r * w;
        at[t] = r * LD + c;
        a[t] = B[at[t]];
        l[t] = B[(int)(r * LD) - 1];
        u[t] = Urow[c];
      }
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        a[t].x = fma(l[t].y, u[t].y, fma(-l[t].x, u[t].x, a[t].x));
        a[t].y = fma(-l[t].y, u[t].x, fma(-l[t].x, u[t].y, a[t].y));
      }
#pragma unroll
      for (int t = 0; t < 4; ++t) B[at[t]] = a[t];
    }
    for (; e < total; e += G) {
      const unsigned r = __umulhi(e, magic), c = e - r * w;
      double2 a = B[r * LD + c];
      const double2 l = B[(int)(r * LD) - 1], u = Urow[c];
      a.x = fma(l.y, u.y, fma(-l.x, u.x, a.x));
      a.y = fma(-l.y, u.x, fma(-l.x, u.y, a.y));
      B[r * LD + c] = a;
    }
    __syncwarp();
  }
  // back substitution, column by column; even lanes take the first
  // right-hand side, odd lanes the second
  const int rhs = n + (lane & 1);
  for (int j = n - 1; j >= 0; --j) {
    const double2 inv = A[j * LD + j], b = A[j * LD + rhs];
    const double2 x = make_double2(fma(b.x, inv.x, -(b.y * inv.y)), fma(b.x, inv.y, b.y * inv.x));
    for (int i = lane >> 1; i < j; i += G / 2) {
      const double2 u = A[i * LD + j];
      double2 v = A[i * LD + rhs];
      v.x = fma(u.y, x.y, fma(-u.x, x.x, v.x));
      v.y = fma(-u.y, x.x, fma(-u.x, x.y, v.y));
      A[i * LD + rhs] = v;
    }
    __syncwarp();
    if (lane < 2) A[j * LD + rhs] = x;
  }
  __syncwarp();
  return ok;
}

// The unknown c of right-hand side b, with the column scale undone.
__device__ __forceinline__ cx<double> lu64_x(int n, const double2* A, const int* colx, int c, int b) {
  const double2 v = A[c * (n + 2) + n + b];
  const int k = colx[c];
  return mk<double>(scale_exp(v.x, k), scale_exp(v.y, k));
}

// The FP64 solves, lanes per path: 8 for n <= 16 and 16 for n <= 32 where the
// paths fill the chip with kLuWarps warps; otherwise 16 (n <= 16) or 32, the
// fewest that do, or 32.  More lanes make a path's chain shorter and leave
// more of them without an entry (n = 8: 75 FP64 instructions a path with 8
// lanes, 116 with 16, 200 with 32); below kLuWarps the chain counts (adjoint, n
// = 8, 4,096 solutions: kernel 70 us with 32 lanes, 63 with 8, 61 with 16).
// For n > 16 the line lies at four fifths of that, 1,946 paths (32 and 16
// lanes, 1,500 | 1,946 paths: step at n = 24 150, 162 | 195, 162 us at 2,300;
// whole calls at n = 18, directions 130, 132 | 155, 134, projective directions
// 140, 141 | 168, 142, polish 148, 147 | 173, 149, adjoint 144, 153 | 169, 153;
// at n = 24, 186, 202 | 232, 204; 200, 216 | 251, 216; 203, 216 | 250, 219;
// 202, 223 | 248, 225).  The 16-lane blocks take twice the shared memory, and
// past one wave of them (2,432 paths at n = 24, 1,216 at n = 31) 32 lanes are
// faster again for a while (3,000 paths, directions at n = 24 366 and 292, at n
// = 31 643 and 552): one line for all n is kept.
// Shapes: 0 (8, 1), 1 (8, 2), 2 (16, 2), 3 (32, 1), 4 (16, 1), (lanes, unknowns
// per lane).  Every shape gives the same bits.
constexpr int64_t kLuWarps = 152 * 4 * 2;
inline int lu_shape(int n, int64_t p) {
  auto fills = [p](int G) { return p * G >= 32 * kLuWarps; };
  if (n > 16) return p * 16 >= 32 * (kLuWarps * 4 / 5) ? 2 : 3;
  return fills(8) ? (n <= 8 ? 0 : 1) : (fills(16) ? 4 : 3);
}

}  // namespace
}  // namespace hpt
