// Start points on the device: the |det V| solutions of the binomial start
// system of a pairs cell (Section 2: H(y, t = 0) = 0 keeps the cell's two
// monomials per equation), enumerated from the host's exact setup
// (binomial_setup: Hermite diagonal, adj V modulo |det V|).  Solution
// `first + q` has the mixed-radix digits k (last coordinate fastest); the
// phase of its coordinate r is sum_j k_j adjm_rj / D modulo 1.
//
// What bounds it: integer issue slots (the 16 bytes written per coordinate
// take 60 us of the 370 that 1,048,576 x 24 coordinates take; one thread per solution
// with FP64 sincos, exp and a 128-bit remainder per product: 2,500 us).
// adjm_rj / D enters as a 128-bit fraction, so that a phase is a sum of 64 x
// 128-bit products modulo 2^128 (within n 2^62 / 2^128 revolution), the
// modulus |y_r| is the same for every solution and comes from the host, cos
// and sin are fixed point (hpt_fx.cuh), and the otherwise idle FP64 pipe turns
// them into doubles and multiplies by |y_r|.  A block writes the coordinates
// of its solutions in address order.
#include <math.h>

#include "hpt_fx.cuh"
#include "hpt_internal.h"

namespace hpt {
namespace {

constexpr int kStartThreads = 256;
constexpr int kStartTile = kStartThreads;   // solutions per block: a thread finds one's digits

// Digits with radix 1 are always 0 and left out: nj radices, the fastest
// first.
struct StartDev {
  int32_t n, nj;
  uint64_t h[kMaxN];
  uint64_t turn0[kMaxN];          // arg of the first solution's coordinate, Q64 revolutions
  double mag[kMaxN];              // |y_r|
  uint64_t F[2 * kMaxN * kMaxN];  // adjm / D as 128-bit fractions (hi, lo), nj rows of n
};

// v 2^-62, rounded once, on the FP64 pipe: the halves of v are the low words of
// 2^22 + 2 + hi 2^-30 and 2^-10 + lo 2^-62.
__device__ __forceinline__ double q62_to_double(int64_t v) {
  const double hi = __hiloint2double(0x41500000, (int)((uint32_t)(v >> 32) ^ 0x80000000u));
  const double lo = __hiloint2double(0x3f500000, (int)(uint32_t)v);
  return (hi - 4194306.0009765625) + lo;
}

__global__ void __launch_bounds__(kStartThreads)
start_points_kernel(const __grid_constant__ StartDev S, int64_t first, int64_t count, double2* __restrict__ y0) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int64_t cs1[64][2], cs2[64][2];
  const int n = S.n, nj = S.nj, t = threadIdx.x;
  ulonglong2* F = (ulonglong2*)smem;                 // [nj][n]
  uint64_t* digit = (uint64_t*)(F + nj * n);         // [nj][kStartTile]
  const int64_t q0 = (int64_t)blockIdx.x * kStartTile;
  for (int i = t; i < nj * n; i += kStartThreads) F[i] = make_ulonglong2(S.F[2 * i], S.F[2 * i + 1]);
  if (t < 64) {
    const fx::Tables& T = fx::tables();
    cs1[t][0] = T.cs1[t][0];
    cs1[t][1] = T.cs1[t][1];
    cs2[t][0] = T.cs2[t][0];
    cs2[t][1] = T.cs2[t][1];
  }
  uint64_t idx = (uint64_t)(first + q0 + t);
  for (int j = 0; j < nj; ++j) {
    const uint64_t d = idx / S.h[j];
    digit[j * kStartTile + t] = idx - d * S.h[j];
    idx = d;
  }
  __syncthreads();
  const int64_t left = count - q0;
  const unsigned total = (unsigned)(left < kStartTile ? left : kStartTile) * n;
  const unsigned magic = 0xffffffffu / (unsigned)n + 1u;   // e / n for e < 2^16 (n = 1: wraps to 0)
  double2* out = y0 + (size_t)q0 * n;
  for (unsigned e = t; e < total; e += kStartThreads) {
    const unsigned q = n == 1 ? e : __umulhi(e, magic), r = e - q * n;
    uint64_t hi = 0, lo = 0;
    for (int j = 0; j < nj; ++j) {
      const uint64_t k = digit[j * kStartTile + q];
      const ulonglong2 f = F[j * n + r];
      const uint64_t pl = k * f.y;
      hi += k * f.x + __umul64hi(k, f.y);
      lo += pl;
      hi += lo < pl ? 1 : 0;
    }
    int64_t c, s;
    // rounded: the truncated fractions of a whole number of quarter turns lie
    // just below it
    fx::cossin(S.turn0[r] + hi + (lo >> 63), cs1, cs2, c, s);
    const double m = S.mag[r];
    out[e] = make_double2(m * q62_to_double(c), m * q62_to_double(s));
  }
}

StartDev device_consts(const StartConsts& S) {
  StartDev d;
  d.n = S.n;
  d.nj = 0;
  for (int j = S.n - 1; j >= 0; --j) {
    if (S.h[j] == 1) continue;
    d.h[d.nj] = (uint64_t)S.h[j];
    for (int r = 0; r < S.n; ++r) {
      const unsigned __int128 a = (unsigned __int128)S.adjm[r * S.n + j] << 64;
      const unsigned __int128 b = (a % S.D) << 64;
      d.F[2 * (d.nj * S.n + r)] = (uint64_t)(a / S.D);
      d.F[2 * (d.nj * S.n + r) + 1] = (uint64_t)(b / S.D);
    }
    ++d.nj;
  }
  for (int r = 0; r < S.n; ++r) {
    const long double turn = (long double)S.zi0[r] / 6.283185307179586476925286766559L;
    d.turn0[r] = (uint64_t)((turn - floorl(turn)) * 9223372036854775808.0L) << 1;
    d.mag[r] = exp(S.zr0[r]);
  }
  return d;
}

}  // namespace
}  // namespace hpt

using namespace hpt;

extern "C" hpt_status hpt_binomial_start_device(int32_t n, const int32_t* msz, const int32_t* exps,
                                                const double* coeffs, const int32_t* pairs, int64_t first,
                                                int64_t count, void* y0_dev, int64_t* total, void* stream) {
  StartConsts S;
  hpt_status rc = binomial_setup(n, msz, exps, coeffs, pairs, first, count, y0_dev != nullptr, S, total);
  if (rc) return rc;
  if (count == 0) return HPT_OK;
  const int64_t blocks = (count + kStartTile - 1) / kStartTile;
  if (blocks > 0x7fffffff) { set_error("count too large"); return HPT_ERANGE; }
  const StartDev d = device_consts(S);
  const int smem = d.nj * (d.n * 16 + kStartTile * 8);
  cudaError_t e = allow_smem<kMaxN * (kMaxN * 16 + kStartTile * 8)>(start_points_kernel, smem);
  if (e == cudaSuccess) {
    start_points_kernel<<<(unsigned)blocks, kStartThreads, smem, (cudaStream_t)stream>>>(d, first, count,
                                                                                        (double2*)y0_dev);
    e = cudaGetLastError();
  }
  return e == cudaSuccess ? HPT_OK : cuda_fail(e, "start point launch");
}
