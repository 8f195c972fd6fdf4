// diag_inv.cuh -- inverse of one lower-triangular diagonal block in binary64.
#pragma once
#include <cstdint>

constexpr int kInvThreads = 256;

// A CTA of kInvThreads inverts the kb x kb (kb <= 64) lower-triangular block at P
// (column-major, leading dimension ld): thread group g (four lanes) solves
// L x = e_g by substitution, lane q holding rows q + 4 mm in x[mm]: column g of
// the inverse. Lk: 64 x 65 and rinv: 64 doubles of shared memory.
__device__ __forceinline__ void inv64_columns(const double* __restrict__ P, int64_t ld, int kb, double* Lk, double* rinv,
                                              double (&x)[16]) {
  const int tid = threadIdx.x;
  for (int e = tid; e < 64 * 64; e += kInvThreads) {
    const int rr = e & 63, cc = e >> 6;   // consecutive threads read consecutive rows of a column
    Lk[rr + cc * 65] = (rr < kb && cc <= rr) ? P[rr + (int64_t)cc * ld] : 0.0;
  }
  __syncthreads();
  if (tid < 64) rinv[tid] = tid < kb ? 1.0 / Lk[tid * 66] : 0.0;
  __syncthreads();
  const int g = tid >> 2, q = tid & 3;
#pragma unroll
  for (int mm = 0; mm < 16; ++mm) x[mm] = (q + 4 * mm == g) ? 1.0 : 0.0;
  // only the first kb steps and the warps holding columns g < kb do work (a
  // ragged block of a small supernode is often much narrower than 64)
  if ((tid >> 5) * 8 < kb) {
#pragma unroll
    for (int jm = 0; jm < 16; ++jm) {
      if (jm * 4 >= kb) break;   // uniform across the CTA
#pragma unroll
      for (int jq = 0; jq < 4; ++jq) {
        const int jj = jm * 4 + jq;
        const double xj = __shfl_sync(0xffffffffu, x[jm] * rinv[jj], jq, 4);
        if (q == jq) x[jm] = xj;
#pragma unroll
        for (int mm = jm; mm < 16; ++mm) {
          const int c = q + 4 * mm;
          if (c > jj && 4 * mm < kb) x[mm] = fma(-xj, Lk[c + jj * 65], x[mm]);
        }
      }
    }
  }
}
