// solve_split.cu -- the solves' panel products with several right-hand sides on
// the tensor cores (split_gemm.cuh): W_J = L_RJ Y_J going forward and
// Y_J -= L_RJ^T X_R going backward, X_R gathered from the ancestors' rows.
//
// Per level: the panels' off-diagonal blocks are split into slices (rows of
// L_RJ forward, its columns backward, one exponent a row of the operand), the
// right-hand sides likewise, and tiles of 128 rows and 16 right-hand sides run
// over K in parts of at least 256 where a level has few tiles, the parts' sums
// added in part order by the last part to arrive. The splitting reads 8 and the
// tiles read 14 bytes an entry whatever the number of right-hand sides, where
// the FP64 pipe, two FMAs a cycle and SM, needs half a cycle for each. 3D 48^3 with
// 16 right-hand sides: the products of a solve 4.9 -> 2.9 ms; of that, 1.2 ms
// splitting (two passes over a row, latency at the 50 to 1,000 CTAs of a level),
// 1.1 ms tiles, 0.3 ms right-hand sides.
#include "device.h"
#include "split_op.cuh"

namespace {

constexpr int kN = 16;                    // right-hand sides of a tile
using Cfg = sg::Cfg<kN>;

// Right-hand side blockIdx.y of J: forward y_J, backward x_R gathered. A thread
// takes 8 consecutive entries of every 1024 (one warp a right-hand side, 256, took
// 50 us at 3,000 rows).
constexpr int kRhsThreads = 128;
template <bool TRANS>
__global__ void __launch_bounds__(kRhsThreads)
k_vs_rhs(const SnodeDev* __restrict__ sn, const SolveSplitDev* __restrict__ vd, const int32_t* __restrict__ list,
         const int32_t* __restrict__ rows, const double* __restrict__ Y, int n, const int32_t* __restrict__ lexps,
         unsigned char* __restrict__ slab, int32_t* __restrict__ exps) {
  __shared__ uint32_t key;
  const int r = blockIdx.y;
  const int J = list[blockIdx.x];
  const SnodeDev d = sn[J];
  const SolveSplitDev z = vd[J];
  const int K = TRANS ? d.len - d.s : d.s;
  const int32_t* rj = rows + d.roff + d.s;
  const double* y = Y + (TRANS ? 0 : d.f) + (int64_t)r * n;
  auto at = [&](int k) { return k < K ? (TRANS ? y[rj[k]] : y[k]) : 0.0; };
  // backward: times the exponents of the rows of L_RJ, which L_RJ^T is divided by
  auto scale = [&](int k) { return TRANS && k < K ? k_exponent(lexps[z.fexp + k]) : 0; };
  if (threadIdx.x == 0) key = 0;
  __syncthreads();
  uint32_t m = 0;
  for (int k0 = 8 * threadIdx.x; k0 < K; k0 += 8 * kRhsThreads) {
#pragma unroll
    for (int i = 0; i < 8; ++i) m = max(m, exponent_key(at(k0 + i), scale(k0 + i)));
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0 && m) atomicMax(&key, m);
  __syncthreads();
  const int32_t e = key_exponent(key);
  if (threadIdx.x == 0) exps[z.rexp + r] = e;
  const int kend = (K + 31) / 32 * 32;
  for (int k0 = 8 * threadIdx.x; k0 < kend; k0 += 8 * kRhsThreads) {
    double v[8];
    int32_t ee[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      v[i] = e == sg::kExpNaN ? 0.0 : at(k0 + i);
      ee[i] = e - scale(k0 + i);
    }
    uint4 w[sg::kSlices];
    sg::digits8(v, ee, w);
    unsigned char* out = slab + (z.roff + (int64_t)(k0 >> 5) * sg::kSlices * kN) * 64 + sg::chunk_offset(r, (k0 >> 3) & 3);
#pragma unroll
    for (int q = 0; q < sg::kSlices; ++q) *reinterpret_cast<uint4*>(out + (int64_t)q * kN * 64) = w[q];
  }
}

template <bool TRANS>
__global__ void __launch_bounds__(Cfg::kThreads, 1)
k_vs_tile(const SnodeDev* __restrict__ sn, const SolveSplitDev* __restrict__ vd, const SolveTile* __restrict__ tiles,
          int ntiles, const unsigned char* __restrict__ lslab, const int32_t* __restrict__ lexps,
          const unsigned char* __restrict__ rslab, const int32_t* __restrict__ rexps, double* __restrict__ Y,
          double* __restrict__ W, int n, int nr, double* __restrict__ part, int* __restrict__ cnt, sg::Waits waits) {
  extern __shared__ unsigned char sg_smem[];
  __shared__ __align__(8) sg::Shared S;
  __shared__ int s_last;
  const uint32_t base = (tc::smem_u32(sg_smem) + 1023u) & ~1023u;
  const uint32_t tmem = sg::setup<kN>(S);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  auto next = [&](int i, sg::Tile& t) {
    const int64_t q = blockIdx.x + (int64_t)i * gridDim.x;
    if (q >= ntiles) return false;
    const SolveTile k = tiles[q];
    const SolveSplitDev z = vd[k.J];
    const int64_t rows = TRANS ? z.brows : z.frows;
    const int64_t off = TRANS ? z.boff : z.foff;
    t.a = {lslab + (off + (int64_t)k.kb0 * sg::kSlices * rows) * 64, lexps + (TRANS ? z.bexp : z.fexp), rows, k.r0};
    t.b = {rslab + (z.roff + (int64_t)k.kb0 * sg::kSlices * kN) * 64, rexps + z.rexp, kN, 0};
    t.nblk = k.kb1 - k.kb0;
    return true;
  };
  if (warp == Cfg::kEpiWarps) {
    if (lane == 0) sg::copy_loop<kN>(S, base, next, waits);
  } else if (warp == Cfg::kEpiWarps + 1) {
    if (lane == 0) sg::mma_loop<kN>(S, base, tmem, next, waits);
  } else {
    sg::Tile t;
    int chunk = 0;
    bool ok = true;
    for (int i = 0; ok && next(i, t); ++i) {
      const SolveTile k = tiles[blockIdx.x + (int64_t)i * gridDim.x];
      const SnodeDev d = sn[k.J];
      const int M = TRANS ? d.s : d.len - d.s;
      const int r = k.r0 + sg::epi_row();
      const bool in = r < M;
      const int32_t ea = in ? t.a.exps[r] : 0;
      long long hi[sg::kCols], lo[sg::kCols];
#pragma unroll
      for (int c = 0; c < sg::kCols; ++c) hi[c] = lo[c] = 0;
      for (int k0 = 0; ok && k0 < t.nblk; k0 += sg::kStagesPerChunk) ok = sg::drain<kN>(S, tmem, chunk++, hi, lo, waits);
      // one verdict for the four warps, which meet at barriers below: a warp whose wait
      // gave up and one whose wait was met just after it leave together
      ok = sg::epi_vote<kN>(ok);
      if (!ok) break;
      double v[sg::kCols];
#pragma unroll
      for (int c = 0; c < sg::kCols; ++c) v[c] = in && c < nr ? sg::combine(hi[c], lo[c], ea, t.b.exps[c]) : 0.0;
      bool write = in;
      if (k.parts > 1) {
        double* mine = part + (int64_t)(k.slot + k.part) * (kN * sg::kM) + sg::epi_row();
#pragma unroll
        for (int c = 0; c < sg::kCols; ++c) mine[c * sg::kM] = v[c];
        __threadfence();
        asm volatile("bar.sync 1, 128;" ::: "memory");
        if (threadIdx.x == 0) {
          s_last = atomicAdd(cnt + k.slot, 1) == k.parts - 1;
          if (s_last) cnt[k.slot] = 0;   // for the next level or solve
        }
        asm volatile("bar.sync 1, 128;" ::: "memory");
        write = in && s_last;
        if (write) {
          __threadfence();
          const double* p0 = part + (int64_t)k.slot * (kN * sg::kM) + sg::epi_row();
          // columns inside parts: 32 loads in flight, where a column's parts one
          // after another took 40 us for 15 of them
#pragma unroll
          for (int c = 0; c < sg::kCols; ++c) v[c] = 0.0;
#pragma unroll 2
          for (int q = 0; q < k.parts; ++q)
#pragma unroll
            for (int c = 0; c < sg::kCols; ++c) v[c] += __ldcg(p0 + (int64_t)q * (kN * sg::kM) + c * sg::kM);
        }
        asm volatile("bar.sync 1, 128;" ::: "memory");   // s_last is read
      }
      if (write) {
        if constexpr (TRANS) {
          double* y = Y + d.f + r;
#pragma unroll
          for (int c = 0; c < sg::kCols; ++c)
            if (c < nr) y[(int64_t)c * n] -= v[c];
        } else {
          double* w = W + d.wpre * nr + r;
#pragma unroll
          for (int c = 0; c < sg::kCols; ++c)
            if (c < nr) w[(int64_t)c * M] = v[c];
        }
      }
    }
  }
  __syncwarp();
  sg::teardown<kN>(S, tmem);
}

struct VsBuffer { void** p; int64_t bytes; };
std::vector<VsBuffer> vs_buffers(const chol_handle* h) {
  DeviceState* D = h->dev;
  return {{(void**)&D->vs_slab, h->vs_slab_rows * 64},
          {(void**)&D->vs_exps, h->vs_exps * 4},
          {(void**)&D->vs_rslab, h->vs_rslab_rows * 64},
          {(void**)&D->vs_rexps, h->vs_rexps * 4},
          {(void**)&D->vs_part, h->vs_slots * (int64_t)(sizeof(double) * kN * sg::kM)},
          {(void**)&D->vs_cnt, h->vs_slots * 4},
          {(void**)&D->vs_dev, (int64_t)(sizeof(SolveSplitDev) * h->vs_dev.size())},
          {(void**)&D->vs_ops, (int64_t)(sizeof(SplitOp) * 2 * h->vs_list.size())},
          {(void**)&D->vs_list, (int64_t)(4 * h->vs_list.size())},
          {(void**)&D->vs_tasks, (int64_t)(sizeof(SplitTask) * h->vs_tasks.size())},
          {(void**)&D->vs_tiles, (int64_t)(sizeof(SolveTile) * h->vs_tiles.size())}};
}

}  // namespace

void chol_vs_release(chol_handle* h) {
  DeviceState* D = h->dev;
  D->vs_ready = -1;
  for (const VsBuffer& b : vs_buffers(h))
    if (*b.p) {
      cudaFree(*b.p);   // waits for the work that uses it
      *b.p = nullptr;
      D->bytes -= b.bytes;
    }
}

// Creates the plan and its workspaces: while the caller's stream is being captured
// too, so that whether a solve takes the tensor cores does not depend on what was
// called before it. For that the thread's captures do not restrict the calls made
// here (relaxed mode), none of them goes to the stream under capture or to the
// legacy stream, and what they do is done once, not at the replays.
static int vs_create(chol_handle* h) {
  DeviceState* D = h->dev;
  const cudaStream_t ps = D->lstream;
  // the panel operands of both directions
  std::vector<SplitOp> ops;
  ops.reserve(2 * h->vs_list.size());
  for (int32_t J : h->vs_list) {
    const SnodeDev& d = h->snodes[J];
    const SolveSplitDev& z = h->vs_dev[J];
    const double* p = D->L + d.loff + d.s;
    ops.push_back({p, 1, d.ld, z.foff, z.fexp, -1, d.len - d.s, d.s, z.frows, 0, 0});
    ops.push_back({p, d.ld, 1, z.boff, z.bexp, z.fexp, d.s, d.len - d.s, z.brows, 0, -1});
  }
  bool ok = true;
  for (const VsBuffer& b : vs_buffers(h)) {
    if (b.bytes == 0) continue;
    ok = ok && cudaMalloc(b.p, (size_t)b.bytes) == cudaSuccess;
    if (!ok) {
      *b.p = nullptr;
      break;
    }
    D->bytes += b.bytes;
  }
  auto up = [&](void* dst, const void* src, size_t bytes) {
    ok = ok && cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, ps) == cudaSuccess;
  };
  if (ok) {
    up(D->vs_dev, h->vs_dev.data(), sizeof(SolveSplitDev) * h->vs_dev.size());
    up(D->vs_ops, ops.data(), sizeof(SplitOp) * ops.size());
    up(D->vs_list, h->vs_list.data(), 4 * h->vs_list.size());
    up(D->vs_tasks, h->vs_tasks.data(), sizeof(SplitTask) * h->vs_tasks.size());
    up(D->vs_tiles, h->vs_tiles.data(), sizeof(SolveTile) * h->vs_tiles.size());
  }
  ok = ok && (h->vs_slots == 0 || cudaMemsetAsync(D->vs_cnt, 0, h->vs_slots * 4, ps) == cudaSuccess) &&
       cudaStreamSynchronize(ps) == cudaSuccess &&
       cudaFuncSetAttribute(k_vs_tile<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::kSmemBytes) == cudaSuccess &&
       cudaFuncSetAttribute(k_vs_tile<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::kSmemBytes) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    chol_vs_release(h);
    return -1;
  }
  return D->vs_ready = 1;
}

// Plan and workspaces, created by the first solve that can use them. Handles
// without the factor's slices (a memory cap, a device without room) go without,
// and a later allocation that finds no room gets these back first, unless a
// captured solve holds their addresses.
int chol_vs_ensure(chol_handle* h, cudaStream_t st) {
  DeviceState* D = h->dev;
  if (D->vs_ready == -1 || D->sg_ready != 1 || h->vs_list.empty()) return -1;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cap) != cudaSuccess) {
    cudaGetLastError();
    return -1;
  }
  if (D->vs_ready == 0) {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    if (cudaThreadExchangeStreamCaptureMode(&mode) != cudaSuccess) {
      cudaGetLastError();
      return -1;
    }
    vs_create(h);
    cudaThreadExchangeStreamCaptureMode(&mode);
  }
  if (D->vs_ready == 1 && cap != cudaStreamCaptureStatusNone) D->vs_pinned = true;
  return D->vs_ready;
}

// The level's panel products of one direction for nr <= 16 right-hand sides.
void chol_vs_products(chol_handle* h, const LevelPlan& P, bool trans, double* Y, double* W, int nr, cudaStream_t st) {
  DeviceState* D = h->dev;
  const int n = h->n, t = trans ? 1 : 0;
  k_split_op<<<P.vs_task_n[t], kSplitOpThreads, 0, st>>>((const SplitOp*)D->vs_ops, (const SplitTask*)D->vs_tasks + P.vs_task_b[t],
                                                         D->vs_slab, D->vs_exps, D->vs_exps);
  const SolveTile* tiles = D->vs_tiles + P.vs_tile_b[t];
  const int nt = P.vs_tile_n[t], grid = std::min(nt, D->sms);
  const sg::Waits waits{D->sg_err, chol_test_wait(h, kTestWaitSolve)};
  if (trans) {
    k_vs_rhs<true><<<dim3(P.vs_n, nr), kRhsThreads, 0, st>>>(D->sn, D->vs_dev, D->vs_list + P.vs_b, D->rows, Y, n, D->vs_exps,
                                               D->vs_rslab, D->vs_rexps);
    k_vs_tile<true><<<grid, Cfg::kThreads, Cfg::kSmemBytes, st>>>(D->sn, D->vs_dev, tiles, nt, D->vs_slab, D->vs_exps,
                                                                  D->vs_rslab, D->vs_rexps, Y, W, n, nr, D->vs_part,
                                                                  D->vs_cnt, waits);
  } else {
    k_vs_rhs<false><<<dim3(P.vs_n, nr), kRhsThreads, 0, st>>>(D->sn, D->vs_dev, D->vs_list + P.vs_b, D->rows, Y, n, D->vs_exps,
                                                D->vs_rslab, D->vs_rexps);
    k_vs_tile<false><<<grid, Cfg::kThreads, Cfg::kSmemBytes, st>>>(D->sn, D->vs_dev, tiles, nt, D->vs_slab, D->vs_exps,
                                                                   D->vs_rslab, D->vs_rexps, Y, W, n, nr, D->vs_part,
                                                                   D->vs_cnt, waits);
  }
}
