// split_gemm.cu -- the binary64 factor's updates on the tensor cores
// (split_gemm.cuh): operand splitting, the panel's trailing update, the update
// matrices U_J = L_RJ L_RJ^T and the RLB form of the latter.
//
// Kernels
//   k_sg_split_rows   the off-diagonal rows L_RJ, one exponent per row over all
//                     of J's columns (the SYRK's operands)
//   k_sg_trailing     C -= A B^T on the panel, K = one 64-column block (its
//                     operands come from k_trsm, one exponent per row of the block)
//   k_sg_syrk         U_J tiles, any K; RLB: subtracted from the ancestors
#include "device.h"
#include "mixed.h"
#include "split_gemm.cuh"

namespace {

using sg::kSplitThreads;

__device__ __forceinline__ uint32_t abs_high(double x) { return (uint32_t)__double2hiint(x) & 0x7fffffffu; }

// 16 to 64 off-diagonal rows of J (split_rows_log2) and all its columns: a first
// pass over the entries for the rows' exponents, a second (from L2) for the
// digits; a thread takes 8 columns of a row a step, the lanes along the rows.
__global__ void __launch_bounds__(kSplitThreads)
k_sg_split_rows(const SnodeDev* __restrict__ sn, const SplitDev* __restrict__ sd, const TileTask* __restrict__ tasks,
                const double* __restrict__ L, unsigned char* __restrict__ slab, int32_t* __restrict__ exps) {
  __shared__ uint32_t hmax[64];
  const TileTask t = tasks[blockIdx.x];
  const SnodeDev d = sn[t.J];
  const SplitDev z = sd[t.J];
  const int b = d.len - d.s;
  const int rsh = sg::split_rows_log2(d.s), R = 1 << rsh, step = 8 << (sg::kSplitThreadsLog2 - rsh);
  const int r = threadIdx.x & (R - 1), c0 = 8 * (threadIdx.x >> rsh);
  const int row = t.r0 + r;
  const bool in = row < b;
  const double* G = L + d.loff + d.s + row;
  if (threadIdx.x < 64) hmax[threadIdx.x] = 0;
  __syncthreads();
  uint32_t m = 0;
#pragma unroll 2
  for (int k0 = c0; k0 < d.s; k0 += step) {
#pragma unroll
    for (int i = 0; i < 8; ++i) m = max(m, in && k0 + i < d.s ? abs_high(G[(int64_t)(k0 + i) * d.ld]) : 0u);
  }
  if (m) atomicMax(&hmax[r], m);
  __syncthreads();
  const int32_t e = sg::row_exponent(hmax[r]);
  if (threadIdx.x < R) exps[z.srow0 + row] = e;
  for (int k0 = c0; k0 < z.sblk * sg::kBlockK; k0 += step) {
    double y[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) y[i] = (in && k0 + i < d.s && e != sg::kExpNaN) ? G[(int64_t)(k0 + i) * d.ld] : 0.0;
    uint4 w[sg::kSlices];
    sg::digits8(y, e, w);
    unsigned char* out = slab + (z.soff + (int64_t)(k0 / sg::kBlockK) * sg::kSlices * z.srows) * 64 +
                         sg::chunk_offset(row, (k0 >> 3) & 3);
#pragma unroll
    for (int q = 0; q < sg::kSlices; ++q) *reinterpret_cast<uint4*>(out + (int64_t)q * z.srows * 64) = w[q];
  }
}

__device__ __forceinline__ uint32_t smem_base(const unsigned char* p) { return (tc::smem_u32(p) + 1023u) & ~1023u; }

// Trailing update of the panel: tiles of 64 columns and 128 (or only 64) rows,
// K = 64, one chunk per tile. The thread's entries of C are loaded before the wait for the products.
__global__ void __launch_bounds__(sg::kThreads, 1)
k_sg_trailing(const SnodeDev* __restrict__ sn, const SplitDev* __restrict__ sd, const TileTask* __restrict__ tasks,
              const unsigned char* __restrict__ slab, const int32_t* __restrict__ exps,
              double* __restrict__ L, sg::Waits waits) {
  extern __shared__ unsigned char sg_smem[];
  __shared__ __align__(8) sg::Shared S;
  const uint32_t base = smem_base(sg_smem);
  const uint32_t tmem = sg::setup(S);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  auto next = [&](int i, sg::Tile& t) {   // one tile a CTA
    if (i > 0) return false;
    const TileTask k = tasks[blockIdx.x];
    const SplitDev z = sd[k.J];
    t.a = {slab + z.toff * 64, exps + z.trow0, z.trows, k.r0};
    t.b = {slab + z.toff * 64, exps + z.trow0, z.trows, k.c0};
    t.nblk = 2;
    return true;
  };
  if (warp == sg::kEpiWarps) {
    if (lane == 0) sg::copy_loop(S, base, next, waits);
  } else if (warp == sg::kEpiWarps + 1) {
    if (lane == 0) sg::mma_loop(S, base, tmem, next, waits);
  } else {
    sg::Tile t;
    next(0, t);
    const TileTask k = tasks[blockIdx.x];
    const SnodeDev d = sn[k.J];
    const int r = k.r0 + sg::epi_row(), c0 = k.c0 + sg::epi_col();
    // the thread's columns c0 .. c0 + n - 1 (on or below the diagonal)
    const int n = r < min(d.len, k.r0 + k.k0) ? min(sg::kCols, min(d.s, r + 1) - c0) : 0;
    const int32_t ea = n > 0 ? t.a.exps[r] : 0;
    double* C = L + d.loff + r + (int64_t)c0 * d.ld;
    double cv[sg::kCols];
#pragma unroll
    for (int c = 0; c < sg::kCols; ++c) cv[c] = c < n ? C[(int64_t)c * d.ld] : 0.0;
    long long hi[sg::kCols], lo[sg::kCols];
#pragma unroll
    for (int c = 0; c < sg::kCols; ++c) hi[c] = lo[c] = 0;
    if (sg::drain(S, tmem, 0, hi, lo, waits)) {
#pragma unroll
      for (int c = 0; c < sg::kCols; ++c)
        if (c < n) C[(int64_t)c * d.ld] = cv[c] - sg::combine(hi[c], lo[c], ea, t.b.exps[c0 + c]);
    }
  }
  __syncwarp();
  sg::teardown(S, tmem);
}

// Position of global row `key` in the sorted row structure rk[0, len).
__device__ __forceinline__ int row_pos(const int32_t* __restrict__ rk, int len, int32_t key) {
  int lo = 0, hi = len;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (rk[mid] < key) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// U_J tiles (lower triangle), K = all of J's columns in chunks of 64 whose
// integer sums stay in registers. RLB: the tile is subtracted from the
// ancestors' panels pair by pair (see k_syrk_rlb), a thread per row of the tile.
template <bool RLB>
__global__ void __launch_bounds__(sg::kThreads, 1)
k_sg_syrk(const SnodeDev* __restrict__ sn, const SplitDev* __restrict__ sd, const TileTask* __restrict__ tasks,
          int ntasks, const unsigned char* __restrict__ slab, const int32_t* __restrict__ exps,
          double* __restrict__ U, const int4* __restrict__ pairs, const int32_t* __restrict__ pbeg,
          const int32_t* __restrict__ rows, double* __restrict__ L, sg::Waits waits) {
  extern __shared__ unsigned char sg_smem[];
  __shared__ __align__(8) sg::Shared S;
  const uint32_t base = smem_base(sg_smem);
  const uint32_t tmem = sg::setup(S);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  auto next = [&](int i, sg::Tile& t) {
    const int64_t q = blockIdx.x + (int64_t)i * gridDim.x;
    if (q >= ntasks) return false;
    const TileTask k = tasks[q];
    const SplitDev z = sd[k.J];
    t.a = {slab + z.soff * 64, exps + z.srow0, z.srows, k.r0};
    t.b = {slab + z.soff * 64, exps + z.srow0, z.srows, k.c0};
    t.nblk = z.sblk;
    return true;
  };
  if (warp == sg::kEpiWarps) {
    if (lane == 0) sg::copy_loop(S, base, next, waits);
  } else if (warp == sg::kEpiWarps + 1) {
    if (lane == 0) sg::mma_loop(S, base, tmem, next, waits);
  } else {
    sg::Tile t;
    int chunk = 0;
    bool ok = true;
    for (int i = 0; ok && next(i, t); ++i) {
      const TileTask k = tasks[blockIdx.x + (int64_t)i * gridDim.x];
      const SnodeDev d = sn[k.J];
      const int b = d.len - d.s;
      const int r = k.r0 + sg::epi_row(), c0 = k.c0 + sg::epi_col();
      // the thread's columns c0 .. c0 + n - 1 (on or below the diagonal)
      const int n = r < b ? min(sg::kCols, r + 1 - c0) : 0;
      const int32_t ea = n > 0 ? t.a.exps[r] : 0;
      long long hi[sg::kCols], lo[sg::kCols];
#pragma unroll
      for (int c = 0; c < sg::kCols; ++c) hi[c] = lo[c] = 0;
      for (int k0 = 0; ok && k0 < t.nblk; k0 += sg::kStagesPerChunk) ok = sg::drain(S, tmem, chunk++, hi, lo, waits);
      if (!ok) break;
      if constexpr (!RLB) {
        double* C = U + d.uoff + r + (int64_t)c0 * b;
#pragma unroll
        for (int c = 0; c < sg::kCols; ++c)
          if (c < n) C[(int64_t)c * b] = sg::combine(hi[c], lo[c], ea, t.b.exps[c0 + c]);
      } else {
        const int32_t* rj = rows + d.roff + d.s;
        double v[sg::kCols];
#pragma unroll
        for (int c = 0; c < sg::kCols; ++c) v[c] = c < n ? sg::combine(hi[c], lo[c], ea, t.b.exps[c0 + c]) : 0.0;
        for (int p = pbeg[k.J]; n > 0 && p < pbeg[k.J + 1]; ++p) {
          const int4 pr = pairs[p];   // (K, first column, end column, -)
          if (pr.z <= c0) continue;
          if (pr.y >= c0 + n) break;
          const SnodeDev dk = sn[pr.x];
          if (r < pr.y) break;        // the pair's rows start at its first column
          double* T = L + dk.loff + row_pos(rows + dk.roff, dk.len, rj[r]);
#pragma unroll
          for (int c = 0; c < sg::kCols; ++c) {
            const int cg = c0 + c;
            if (c < n && cg >= pr.y && cg < pr.z) atomicAdd(T + (int64_t)(rj[cg] - dk.f) * dk.ld, -v[c]);
          }
        }
      }
    }
  }
  __syncwarp();
  sg::teardown(S, tmem);
}

}  // namespace

namespace {

struct SgBuffer { void** p; int64_t bytes; };

std::vector<SgBuffer> sg_buffers(chol_handle* h) {
  DeviceState* D = h->dev;
  return {{(void**)&D->sg_slab, h->split_slab_rows * 64},
          {(void**)&D->sg_exps, h->split_exps * 4},
          {(void**)&D->sgt_slab[0], h->split_trows * 64},
          {(void**)&D->sgt_slab[1], h->split_trows * 64},
          {(void**)&D->sgt_slab[2], h->split_trows * 64},
          {(void**)&D->sgt_exps[0], h->split_texps * 4},
          {(void**)&D->sgt_exps[1], h->split_texps * 4},
          {(void**)&D->sgt_exps[2], h->split_texps * 4},
          {(void**)&D->sg_dev, (int64_t)(sizeof(SplitDev) * h->split.size())},
          {(void**)&D->sg_split, (int64_t)(sizeof(TileTask) * h->split_tasks.size())},
          {(void**)&D->sg_syrk, (int64_t)(sizeof(TileTask) * h->sgs_tasks.size())},
          {(void**)&D->sg_trail, (int64_t)(sizeof(TileTask) * h->sgt_tasks.size())}};
}

}  // namespace

int32_t chol_tc_products(const chol_handle* h) {
  const DeviceState* D = h->dev;
  if (!D) return 0;
  const bool factor = D->sg_ready == 1;
  return (factor ? 1 : 0) | (factor && D->vs_ready == 1 ? 2 : 0) | (chol_adjoint_split(h) ? 4 : 0);
}

// Gives the workspaces back; later factorizations run on the binary64 pipe.
void chol_sg_release(chol_handle* h) {
  DeviceState* D = h->dev;
  D->sg_ready = -1;
  for (const SgBuffer& a : sg_buffers(h))
    if (*a.p) {
      cudaFree(*a.p);   // waits for the work that uses it
      *a.p = nullptr;
      D->bytes -= a.bytes;
    }
}

// Workspaces and plan of the tensor-core updates, created by the first
// factorization. D->sg_ready: 1 = in use, -1 = not: a handle with a memory cap,
// or a device without the room, keeps the binary64 pipe's kernels, which need
// no slices. (A later allocation that finds no room gets these back first, see
// chol_dalloc.)
int chol_sg_ensure(chol_handle* h) {
  DeviceState* D = h->dev;
  if (D->sg_ready) return CHOL_OK;
  D->sg_ready = -1;
  if ((h->split_tasks.empty() && h->sgt_tasks.empty()) || h->opt.device_mem_cap > 0) return CHOL_OK;
  for (const SgBuffer& a : sg_buffers(h))
    if (chol_dalloc(h, a.p, (size_t)a.bytes)) {
      chol_sg_release(h);
      return CHOL_OK;
    }
  CHOL_CUDA_TRY(cudaMemcpy(D->sg_dev, h->split.data(), sizeof(SplitDev) * h->split.size(), cudaMemcpyHostToDevice));
  auto up = [](TileTask* dst, const std::vector<TileTask>& v) {
    return v.empty() ? cudaSuccess : cudaMemcpy(dst, v.data(), sizeof(TileTask) * v.size(), cudaMemcpyHostToDevice);
  };
  CHOL_CUDA_TRY(up(D->sg_split, h->split_tasks));
  CHOL_CUDA_TRY(up(D->sg_syrk, h->sgs_tasks));
  CHOL_CUDA_TRY(up(D->sg_trail, h->sgt_tasks));
  CHOL_CUDA_TRY(cudaStreamSynchronize(cudaStreamLegacy));   // non-blocking streams do not wait for the copies
  const void* kernels[] = {(const void*)k_sg_trailing, (const void*)k_sg_syrk<false>, (const void*)k_sg_syrk<true>};
  for (const void* k : kernels)
    CHOL_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, sg::kSmemBytes));
  D->sg_ready = 1;
  return CHOL_OK;
}

// n > 0 trailing tiles from the slices in buffer `buf` (written by k_trsm).
void chol_sg_trailing(chol_handle* h, const TileTask* tasks, int n, int buf, cudaStream_t st) {
  DeviceState* D = h->dev;
  const sg::Waits waits{D->sg_err, chol_test_wait(h, kTestWaitFactor)};
  k_sg_trailing<<<n, sg::kThreads, sg::kSmemBytes, st>>>(D->sn, D->sg_dev, tasks, D->sgt_slab[buf], D->sgt_exps[buf], D->L,
                                                         waits);
}

// U_J of every blocked supernode of a level (RLB: subtracted from the ancestors).
void chol_sg_syrk(chol_handle* h, const LevelPlan& P, cudaStream_t st) {
  DeviceState* D = h->dev;
  k_sg_split_rows<<<P.sgr_n, kSplitThreads, 0, st>>>(D->sn, D->sg_dev, D->sg_split + P.sgr_b, D->L, D->sg_slab,
                                                     D->sg_exps);
  const int grid = std::min(P.sgs_n, D->sms);
  const sg::Waits waits{D->sg_err, chol_test_wait(h, kTestWaitFactor)};
  if (h->opt.update_mode == CHOL_UPDATE_RLB)
    k_sg_syrk<true><<<grid, sg::kThreads, sg::kSmemBytes, st>>>(D->sn, D->sg_dev, D->sg_syrk + P.sgs_b, P.sgs_n, D->sg_slab,
                                                                D->sg_exps, nullptr, D->rlb_pairs, D->rlb_pbeg, D->rows,
                                                                D->L, waits);
  else
    k_sg_syrk<false><<<grid, sg::kThreads, sg::kSmemBytes, st>>>(D->sn, D->sg_dev, D->sg_syrk + P.sgs_b, P.sgs_n,
                                                                 D->sg_slab, D->sg_exps, D->U, nullptr, nullptr, nullptr,
                                                                 nullptr, waits);
}
