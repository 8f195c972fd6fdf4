// split_op.cuh -- splitting of strided binary64 operands into the slices of
// split_gemm.cuh (the selected inverse's products, the solves' panel products).
#pragma once
#include "split_gemm.cuh"

// K may be rebalanced: with ksgn = +-1 the entries (i, k) are taken times
// 2^(ksgn x_k), x_k = kexps[kx + k], one operand of a product with +1 and the
// other with -1, x_k the row exponent of row k of L. A product whose K index
// carries a scaling of the system (A -> D A D, D diagonal: L_RJ^T x_R, Z_RR U,
// U^T Z_RJ) then has the same slices for every D of powers of two; with one
// exponent a row alone the entries of small d_k would fall below the last slice.
// ksgn = 0 with kx >= 0: the operand's own row exponents are kept at kexps[kx].
struct SplitOp {          // operand rows (i, k) at p[i rs + k ks], i < rows, k < K
  const double* p;
  int64_t rs, ks;
  int64_t off, exp0;      // first slice row and first exponent in the workspace
  int64_t kx;             // first exponent of K, or -1
  int32_t rows, K, prows; // prows: rows per slice, whole tiles
  int16_t mode;           // 0 general, 1 zero for k > i, 2 symmetric (k <= i stored), 3 zero for i > k
  int16_t ksgn;
};
struct SplitTask {
  int32_t op, r0;   // first of split_rows(K) rows
};
__device__ __forceinline__ double split_el(const SplitOp& o, int i, int k) {
  if (i >= o.rows || k >= o.K) return 0.0;
  if (o.mode == 2) return k <= i ? o.p[i * o.rs + k * o.ks] : o.p[k * o.rs + i * o.ks];
  if ((o.mode == 1 && k > i) || (o.mode == 3 && i > k)) return 0.0;
  return o.p[i * o.rs + k * o.ks];
}

// Exponent of K entry k as stored: a row exponent; 0 for rows with an infinity or a NaN.
__device__ __forceinline__ int32_t k_exponent(int32_t e) { return e == sg::kExpNaN ? 0 : e; }

// Order-preserving key of |x| 2^x_k's exponent (0: x = 0), and the row exponent
// from the largest key of a row.
__device__ __forceinline__ uint32_t exponent_key(double x, int32_t xk) {
  const uint32_t hi = (uint32_t)__double2hiint(x) & 0x7fffffffu;
  const int E = (int)(hi >> 20);
  if (E == 0x7ff) return 0xffffffffu;
  return (hi | (uint32_t)__double2loint(x)) ? (uint32_t)((E > 1 ? E : 1) + xk + (1 << 20)) : 0u;
}
__device__ __forceinline__ int32_t key_exponent(uint32_t key) {
  return key == 0xffffffffu ? sg::kExpNaN : (key ? (int32_t)key - (1 << 20) - 1021 : sg::kExpMin);
}

// 16 to 64 rows of an operand: a thread takes 8 consecutive columns of a row a
// step, with the lanes along whichever index is contiguous (a symmetric operand
// changes at the diagonal). Two passes, the second from L2.
constexpr int kSplitOpThreads = sg::kSplitThreads;
static __global__ void __launch_bounds__(kSplitOpThreads)
k_split_op(const SplitOp* __restrict__ ops, const SplitTask* __restrict__ tasks, unsigned char* __restrict__ slab,
           int32_t* __restrict__ exps, int32_t* __restrict__ kexps) {
  __shared__ uint32_t hmax[64];
  const SplitTask t = tasks[blockIdx.x];
  const SplitOp o = ops[t.op];
  const int tid = threadIdx.x;
  const int rsh = sg::split_rows_log2(o.K), R = 1 << rsh, csh = sg::kSplitThreadsLog2 - rsh;
  const int step = 8 << csh;   // columns a step
  if (tid < 64) hmax[tid] = 0;
  __syncthreads();
  const int32_t* kx = o.ksgn ? kexps + o.kx : nullptr;
  auto scale = [&](int k) { return kx && k < o.K ? o.ksgn * k_exponent(kx[k]) : 0; };
  const bool kc = o.ks == 1 && o.rs != 1;
  // (row, first column) of the thread in the step at column k0
  auto place = [&](int k0, int& r, int& c) {
    const bool kfast = o.mode == 2 ? (k0 >= t.r0 + R ? o.rs == 1 : kc) : kc;
    r = kfast ? (tid >> csh) : (tid & (R - 1));
    c = 8 * (kfast ? (tid & ((1 << csh) - 1)) : (tid >> rsh));
  };
#pragma unroll 2
  for (int k0 = 0; k0 < o.K; k0 += step) {
    int r, c;
    place(k0, r, c);
    uint32_t m = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) m = max(m, exponent_key(split_el(o, t.r0 + r, k0 + c + i), scale(k0 + c + i)));
    if (m) atomicMax(&hmax[r], m);
  }
  __syncthreads();
  if (tid < R) {
    const int32_t e = key_exponent(hmax[tid]);
    exps[o.exp0 + t.r0 + tid] = e;
    if (o.ksgn == 0 && o.kx >= 0 && t.r0 + tid < o.rows) kexps[o.kx + t.r0 + tid] = e;
  }
  const int kend = (o.K + 31) / 32 * 32;
  for (int k0 = 0; k0 < kend; k0 += step) {
    int r, c;
    place(k0, r, c);
    if (k0 + c >= kend) continue;
    const int32_t e = key_exponent(hmax[r]);
    double y[8];
    int32_t ee[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      y[i] = e == sg::kExpNaN ? 0.0 : split_el(o, t.r0 + r, k0 + c + i);
      ee[i] = e - scale(k0 + c + i);
    }
    uint4 w[sg::kSlices];
    sg::digits8(y, ee, w);
    const int kb = (k0 + c) >> 5;
    unsigned char* out = slab + (o.off + (int64_t)kb * sg::kSlices * o.prows) * 64 +
                         sg::chunk_offset(t.r0 + r, (c >> 3) & 3);
#pragma unroll
    for (int q = 0; q < sg::kSlices; ++q) *reinterpret_cast<uint4*>(out + (int64_t)q * o.prows * 64) = w[q];
  }
}
