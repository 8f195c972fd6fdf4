// adjoint.cu -- selected inverse and gradients of x = A^{-1} b and log det A.
//
// The loss l = sum_k w_k^T x_k + alpha log det A, with X = A^{-1} B, has
//   dl/dB = Xbar = A^{-1} W          (two triangular solves with the factor)
//   dl/dA = -Xbar X^T + alpha A^{-1}
// and, for the stored lower entries (a_ij and a_ji move together):
//   g_ii = G_ii,  g_ij = G_ij + G_ji (i > j).
// Only the entries of A^{-1} on the pattern of A are needed. They come from
// the selected inverse Z = (P A P^T)^{-1} on the pattern of L. Z is computed
// supernode by supernode from the root down, with dense blocks:
//   T    = L_JJ^{-1}
//   Uhat = L_RJ T
//   Z_RJ = -Z_RR Uhat          (Z_RR gathered from the ancestors by the factor's
//                               assembly tasks in reverse)
//   Z_JJ = T^T T - Uhat^T Z_RJ
// Z is stored in the layout of the factor's panels (binary64, column-major).
#include <algorithm>
#include <cstring>
#include <vector>

#include "device.h"
#include "mixed.h"
#include "split_op.cuh"
#include "diag_inv.cuh"

namespace {

constexpr int kGT = 256;
constexpr int kGTile = 64;

// Generic strided binary64 GEMM tile: C = beta C + alpha A B over a 64 x 64
// tile. A(i,k) = A[i*ar + k*ac], B(k,j) = B[k*br + j*bc], C(i,j) = C[i*cr + j*cc].
// amode: 0 general, 1 A lower triangular (A(i,k) = 0 for k > i), 2 A symmetric
// stored in its lower triangle. bmode: 0 general, 1 B lower triangular
// (B(k,j) = 0 for j > k). lower_c: write only i >= j.
struct GenGemm {
  const double* A;
  int64_t ar, ac;
  const double* B;
  int64_t br, bc;
  double* C;
  int64_t cr, cc;
  int M, N, K;
  double alpha, beta;
  int amode, bmode, lower_c;
  int ksplit, kchunk;   // K split over ksplit CTAs of kchunk (a multiple of 16) each
  int64_t part;         // split: first partial tile of this product in the workspace
};

// Grouped form: one CTA per (descriptor, tile i, tile j) entry of a task list,
// so the GEMMs of every supernode of a level run in one launch.
struct GemmTile {
  int32_t desc, ti, tj, kc;   // product, output tile, K chunk
};

__device__ __forceinline__ void gen_gemm_tile(const GenGemm& g, int i0, int j0, int kc, double* __restrict__ part_ws,
                                              int64_t tile_idx) {
  constexpr int KC = 16;
  __shared__ double As[KC][kGTile + 1];
  __shared__ double Bs[KC][kGTile + 1];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  int kbeg = 0, kend = g.K;
  if (g.amode == 1) kend = min(kend, i0 + kGTile);
  if (g.bmode == 1) kbeg = (j0 / KC) * KC;
  if (g.ksplit > 1) {
    kbeg = max(kbeg, kc * g.kchunk);
    kend = min(kend, (kc + 1) * g.kchunk);
  }
  double acc[4][4] = {};
  // the thread -> element map of each operand follows its contiguous index
  const bool bkf = g.br == 1 && g.bc != 1;
  for (int k = kbeg; k < kend; k += KC) {
    // symmetric A: the chunk reads its stored transpose wholly above the diagonal
    const bool akf = g.amode == 2 ? (k >= i0 + kGTile ? g.ar == 1 : (g.ac == 1 && g.ar != 1))
                                  : (g.ac == 1 && g.ar != 1);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int idx = tid + kGT * q;
      {
        const int kk = akf ? (idx & 15) : (idx >> 6), r = akf ? (idx >> 4) : (idx & 63);
        const int kg = k + kk, ia = i0 + r;
        double av = 0.0;
        if (kg < kend && ia < g.M) {
          if (g.amode == 0 || (g.amode == 1 && kg <= ia)) av = g.A[ia * g.ar + kg * g.ac];
          else if (g.amode == 2) av = kg <= ia ? g.A[ia * g.ar + kg * g.ac] : g.A[kg * g.ar + ia * g.ac];
        }
        As[kk][r] = av;
      }
      {
        const int kk = bkf ? (idx & 15) : (idx >> 6), r = bkf ? (idx >> 4) : (idx & 63);
        const int kg = k + kk, jb = j0 + r;
        double bv = 0.0;
        if (kg < kend && jb < g.N && (g.bmode == 0 || jb <= kg)) bv = g.B[kg * g.br + jb * g.bc];
        Bs[kk][r] = bv;
      }
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < KC; ++kk) {
      double a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
  if (g.ksplit > 1) {
    // partial tile (row-major 64 x 64), summed by k_gen_reduce
    double* pp = part_ws + g.part + (tile_idx * g.ksplit + kc) * (kGTile * kGTile);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) pp[(ty + 16 * i) * kGTile + tx + 16 * j] = acc[i][j];
    return;
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int r = i0 + ty + 16 * i, c = j0 + tx + 16 * j;
      if (r < g.M && c < g.N && (!g.lower_c || r >= c)) {
        double* p = g.C + r * g.cr + c * g.cc;
        *p = (g.beta == 0.0 ? 0.0 : g.beta * *p) + g.alpha * acc[i][j];
      }
    }
}

__global__ void __launch_bounds__(kGT, 3)
k_gen_gemm_grouped(const GenGemm* __restrict__ descs, const GemmTile* __restrict__ tiles,
                   double* __restrict__ part_ws) {
  const GemmTile t = tiles[blockIdx.x];
  const GenGemm g = descs[t.desc];
  const int64_t ntj = (g.N + kGTile - 1) / kGTile;
  gen_gemm_tile(g, t.ti * kGTile, t.tj * kGTile, t.kc, part_ws, t.ti * ntj + t.tj);
}

// Split products: C = beta C + alpha sum_kc partial(kc), the partials added in
// chunk order (deterministic); one CTA per output tile.
__global__ void __launch_bounds__(kGT)
k_gen_reduce(const GenGemm* __restrict__ descs, const GemmTile* __restrict__ tiles,
             const double* __restrict__ part_ws) {
  const GemmTile t = tiles[blockIdx.x];
  const GenGemm g = descs[t.desc];
  const int64_t ntj = (g.N + kGTile - 1) / kGTile;
  const double* pp = part_ws + g.part + (t.ti * ntj + t.tj) * g.ksplit * (kGTile * kGTile);
  for (int e = threadIdx.x; e < kGTile * kGTile; e += kGT) {
    const int r = t.ti * kGTile + e / kGTile, c = t.tj * kGTile + e % kGTile;
    if (r >= g.M || c >= g.N || (g.lower_c && r < c)) continue;
    double acc = 0.0;
    for (int kc = 0; kc < g.ksplit; ++kc) acc += pp[(int64_t)kc * (kGTile * kGTile) + e];
    double* p = g.C + r * g.cr + c * g.cc;
    *p = (g.beta == 0.0 ? 0.0 : g.beta * *p) + g.alpha * acc;
  }
}

// ---------------------------------------------------------------------------
// The same grouped products on the tensor cores (split_gemm.cuh): first every
// operand of the group is split (rows of A, columns of B; one exponent a row),
// then the 128 x 64 tiles run. The FP64 pipe kept the tiles above at 97% of its
// 2 FMAs per cycle and SM on busy SMs; they remain for handles with a memory
// cap and devices without room for the slices.
struct SplitTile {
  int32_t desc, i0, j0, kb0, kb1, pad;   // product, tile origin, range of 32-column K blocks
};

// Tiles of the group's products: operand 2 desc is A, 2 desc + 1 is B.
__global__ void __launch_bounds__(sg::kThreads, 1)
k_split_gemm(const GenGemm* __restrict__ descs, const SplitOp* __restrict__ ops, const SplitTile* __restrict__ tiles,
             int ntiles, const unsigned char* __restrict__ slab, const int32_t* __restrict__ exps, sg::Waits waits) {
  extern __shared__ unsigned char sg_smem[];
  __shared__ __align__(8) sg::Shared S;
  const uint32_t base = (tc::smem_u32(sg_smem) + 1023u) & ~1023u;
  const uint32_t tmem = sg::setup(S);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  auto next = [&](int i, sg::Tile& t) {
    const int64_t q = blockIdx.x + (int64_t)i * gridDim.x;
    if (q >= ntiles) return false;
    const SplitTile k = tiles[q];
    const SplitOp a = ops[2 * k.desc], b = ops[2 * k.desc + 1];
    t.a = {slab + (a.off + (int64_t)k.kb0 * sg::kSlices * a.prows) * 64, exps + a.exp0, a.prows, k.i0};
    t.b = {slab + (b.off + (int64_t)k.kb0 * sg::kSlices * b.prows) * 64, exps + b.exp0, b.prows, k.j0};
    t.nblk = k.kb1 - k.kb0;
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
      const SplitTile k = tiles[blockIdx.x + (int64_t)i * gridDim.x];
      const GenGemm g = descs[k.desc];
      const int r = k.i0 + sg::epi_row(), c0 = k.j0 + sg::epi_col();
      const int n = r < g.M ? min(sg::kCols, (g.lower_c ? min(g.N, r + 1) : g.N) - c0) : 0;
      const int32_t ea = n > 0 ? t.a.exps[r] : 0;
      long long hi[sg::kCols], lo[sg::kCols];
#pragma unroll
      for (int c = 0; c < sg::kCols; ++c) hi[c] = lo[c] = 0;
      for (int k0 = 0; ok && k0 < t.nblk; k0 += sg::kStagesPerChunk) ok = sg::drain(S, tmem, chunk++, hi, lo, waits);
      if (!ok) break;
      double* C = g.C + r * g.cr + c0 * g.cc;
#pragma unroll
      for (int c = 0; c < sg::kCols; ++c)
        if (c < n) {
          double* p = C + c * g.cc;
          const double v = g.alpha * sg::combine(hi[c], lo[c], ea, t.b.exps[c0 + c]);
          *p = g.beta == 0.0 ? v : g.beta * *p + v;
        }
    }
  }
  __syncwarp();
  sg::teardown(S, tmem);
}

struct InvTask {
  const double* src;
  int64_t lds;
  double* dst;
  int64_t ldt;
  const double* inv;   // the factor's inverse of the block (64 x 64, leading dimension 64), or null
  int32_t kb, pad;
};

// Inverses of kb x kb (kb <= 64) lower-triangular blocks into T: a copy where the
// factor has formed the inverse for the triangle solves, else by substitution.
__global__ void __launch_bounds__(kInvThreads)
k_inv64_grouped(const InvTask* __restrict__ tasks) {
  __shared__ double Lk[64 * 65], rinv[64];
  const InvTask t = tasks[blockIdx.x];
  const int tid = threadIdx.x;
  if (t.inv) {
    for (int e = tid; e < 64 * t.kb; e += kInvThreads) {
      const int r = e & 63, c = e >> 6;
      if (r < t.kb) t.dst[r + c * t.ldt] = t.inv[r + 64 * c];
    }
    return;
  }
  double x[16];
  inv64_columns(t.src, t.lds, t.kb, Lk, rinv, x);
#pragma unroll
  for (int mm = 0; mm < 16; ++mm) {
    const int c = (tid & 3) + 4 * mm, g = tid >> 2;
    if (c < t.kb && g < t.kb) t.dst[c + g * t.ldt] = x[mm];
  }
}

// Longest supernode structure the selected inverse takes (else CHOL_ENOTSUP).
constexpr int kSelinvMaxLen = 200 * 1024 / 4 - 512;

// g[t] = -(xbar_r . x_c + [r != c] xbar_c . x_r) + alpha (1 + [r != c]) Z(entry t)
__global__ void k_adj_grad(const int32_t* __restrict__ rowind, const int32_t* __restrict__ colidx,
                           const int64_t* __restrict__ amap, const double* __restrict__ Z, double alpha,
                           const double* __restrict__ Xb, const double* __restrict__ X, int n, int nrhs, int64_t nnz,
                           double* __restrict__ g) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nnz; t += (int64_t)gridDim.x * blockDim.x) {
    const int r = rowind[t], c = colidx[t];
    double s = 0.0;
    for (int k = 0; k < nrhs; ++k) s = fma(Xb[r + (int64_t)k * n], X[c + (int64_t)k * n], s);
    if (r != c)
      for (int k = 0; k < nrhs; ++k) s = fma(Xb[c + (int64_t)k * n], X[r + (int64_t)k * n], s);
    double v = -s;
    if (Z) v += alpha * (r != c ? 2.0 : 1.0) * Z[amap[t]];
    g[t] = v;
  }
}

__global__ void k_take(const double* __restrict__ Z, const int64_t* __restrict__ map, int64_t m,
                       double* __restrict__ out) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < m; t += (int64_t)gridDim.x * blockDim.x)
    out[t] = Z[map[t]];
}

inline unsigned grid1d(int64_t n, int threads) {
  int64_t g = (n + threads - 1) / threads;
  if (g > 152 * 32) g = 152 * 32;
  return (unsigned)(g > 0 ? g : 1);
}

GenGemm mk(const double* A, int64_t ar, int64_t ac, const double* B, int64_t br, int64_t bc, double* C, int64_t cr,
           int64_t cc, int M, int N, int K, double alpha, double beta, int amode = 0, int bmode = 0, int lower = 0) {
  GenGemm g;
  g.A = A; g.ar = ar; g.ac = ac; g.B = B; g.br = br; g.bc = bc; g.C = C; g.cr = cr; g.cc = cc;
  g.M = M; g.N = N; g.K = K; g.alpha = alpha; g.beta = beta; g.amode = amode; g.bmode = bmode; g.lower_c = lower;
  g.ksplit = 1; g.kchunk = K; g.part = 0;
  return g;
}

template <class T>
int upload_v(chol_handle* h, T** dst, const std::vector<T>& v) {
  if (v.empty()) { *dst = nullptr; return CHOL_OK; }
  int rc = chol_dalloc(h, (void**)dst, v.size() * sizeof(T));
  if (rc) return rc;
  CHOL_CUDA_TRY(cudaMemcpy(*dst, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice));
  return CHOL_OK;
}

int ensure_adjoint(chol_handle* h) {
  DeviceState* D = h->dev;
  if (D->Zp && D->a_col && D->a_row) return CHOL_OK;   // an earlier call may have found room for some of them only
  int rc;
  if (!D->Zp &&
      (rc = chol_dalloc(h, (void**)&D->Zp, sizeof(double) * (size_t)std::max<int64_t>(h->panel_doubles, 1))))
    return rc;
  // column index of every stored entry of A (original ordering)
  std::vector<int32_t> colidx(h->nnz_a), rowidx(h->nnz_a);
  for (int32_t c = 0; c < h->n; ++c)
    for (int64_t t = h->a_colptr[c]; t < h->a_colptr[c + 1]; ++t) colidx[t] = c;
  if (!D->a_col && (rc = upload_v(h, &D->a_col, colidx))) return rc;
  if (!D->a_row && (rc = upload_v(h, &D->a_row, h->a_rowind))) return rc;
  return CHOL_OK;
}

// Level plan of the selected inverse (built once, on first use).
// Products launched together: their tiles (incl. K chunks) and, for the split
// ones, the output tiles of the reduction.
struct Group {
  int32_t tb = 0, tn = 0, rb = 0, rn = 0;
  int32_t sb = 0, sn = 0, gb = 0, gn = 0;   // tensor cores: split tasks, tiles
  double flops = 0.0;
};
struct SiStep {
  int32_t inv_b, inv_n;
  Group g1, g2;
  double flops;                         // algorithmic flops of the step
};
struct SiLevel {
  int64_t t_doubles;                    // T workspace of the level (zeroed first)
  std::vector<SiStep> steps;            // the L_JJ^{-1} recurrence, batched
  Group uh, zrj, zjj1, zjj2;
  int32_t level;                        // of the factor's schedule (its assembly tasks gather Z_RR)
  double gemm_flops;                    // Uhat, Z_RJ and Z_JJ products
};

// Algorithmic flops of a descriptor: 2 M N K, halved for a triangular operand
// and for a triangular output.
double gemm_flops(const GenGemm& g) {
  double f = 2.0 * g.M * (double)g.N * g.K;
  if (g.amode == 1 || g.bmode == 1) f *= 0.5;
  if (g.lower_c) f *= 0.5;
  return f;
}

struct SiPlan {
  std::vector<SiLevel> levels;
  std::vector<GenGemm> descs;
  std::vector<GemmTile> tiles, rtiles;
  std::vector<InvTask> invs;
  int64_t part_max = 0;                 // partial-tile workspace (doubles)
  // tensor cores: two operands per product, tasks, and the workspace of the largest group
  std::vector<SplitOp> ops;
  std::vector<SplitTask> stasks;
  std::vector<SplitTile> stiles;
  int64_t slab_rows = 0, nexps = 0, nkexps = 0;
  bool sg = false;
  bool pinned = false;   // a captured selected inverse holds the plan's addresses
  SplitOp* d_ops = nullptr;
  int32_t* d_kexps = nullptr;
  SplitTask* d_stasks = nullptr;
  SplitTile* d_stiles = nullptr;
  unsigned char* d_slab = nullptr;
  int32_t* d_exps = nullptr;
  GenGemm* d_descs = nullptr;
  GemmTile* d_tiles = nullptr;
  GemmTile* d_rtiles = nullptr;
  InvTask* d_invs = nullptr;
  double* d_part = nullptr;
};

// Emit the tiles of products launched together. Products with K > 256 may be
// split over K chunks (of at least 128): each chunk writes a partial tile to
// the workspace and a second launch adds them in chunk order. The split factor
// is chosen per group for the fill of whole waves of resident CTAs (tiles of
// unequal cost counted alike): a small group is spread over the SMs, and a
// group of, say, 384 tiles on 456 CTA slots, which would leave some SMs idle
// for a third of the launch, becomes 7 x 384 = 5.9 waves. Only groups below
// two waves are split, and a split must gain at least 8% of fill to pay for
// its partial tiles.
constexpr int kGenCtasPerSm = 3;   // __launch_bounds__ of k_gen_gemm_grouped
// kx: place of x_k of each product (SplitOp), or empty; ksgn: A's sign, 0: A's row
// exponents are the x_k of products to come.
Group emit_group(SiPlan& pl, const std::vector<GenGemm>& gs, int sms, const std::vector<int64_t>& kx = {},
                 int16_t ksgn = 0) {
  Group gr;
  gr.tb = (int32_t)pl.tiles.size();
  gr.rb = (int32_t)pl.rtiles.size();
  auto out_tiles = [](const GenGemm& g) {
    int64_t n = 0;
    for (int ti = 0; ti * kGTile < g.M; ++ti)
      for (int tj = 0; tj * kGTile < g.N; ++tj)
        if (!g.lower_c || ti * kGTile + kGTile - 1 >= tj * kGTile) ++n;
    return n;
  };
  const int64_t slots = (int64_t)kGenCtasPerSm * sms;
  auto split_of = [](const GenGemm& g, int ks) {
    return g.K > 256 ? (int)std::min<int64_t>(ks, (g.K + 127) / 128) : 1;
  };
  auto fill = [&](int ks) {
    int64_t t = 0;
    for (const GenGemm& g : gs)
      if (g.M > 0 && g.N > 0) t += out_tiles(g) * split_of(g, ks);
    return t == 0 ? 1.0 : (double)t / ((double)((t + slots - 1) / slots) * (double)slots);
  };
  int64_t nt = 0;
  for (const GenGemm& g : gs)
    if (g.M > 0 && g.N > 0) nt += out_tiles(g);
  int ksel = 1;
  double best = fill(1);
  const double base = best;
  // from two waves on, tiles of unequal cost already even out the tail
  for (int ks = 2; ks <= 32 && nt < 2 * slots; ++ks) {
    const double f = fill(ks);
    if (f > best + 0.02) { best = f; ksel = ks; }
  }
  if (best < base + 0.08) ksel = 1;
  int64_t part = 0;
  gr.sb = (int32_t)pl.stasks.size();
  gr.gb = (int32_t)pl.stiles.size();
  int64_t srow = 0, sexp = 0;
  for (size_t gi = 0; gi < gs.size(); ++gi) {
    GenGemm g = gs[gi];
    if (g.M <= 0 || g.N <= 0) continue;
    {
      const int32_t d = (int32_t)pl.descs.size();
      auto operand = [&](const double* p, int64_t rs, int64_t ks, int rows, int16_t mode, int extra, int16_t ksgn,
                         bool has_kx) {
        SplitOp o{p, rs, ks, srow, sexp, has_kx && !kx.empty() ? kx[gi] : -1, rows, g.K, (rows + 63) / 64 * 64 + extra, mode, ksgn};
        for (int r0 = 0; r0 < rows; r0 += 1 << SPLIT_ROWS_LOG2(g.K)) pl.stasks.push_back({(int32_t)pl.ops.size(), r0});
        pl.ops.push_back(o);
        srow += (int64_t)((g.K + 31) / 32) * sg::kSlices * o.prows;
        sexp += o.prows;
      };
      operand(g.A, g.ar, g.ac, g.M, (int16_t)g.amode, 64, ksgn, true);               // a 128-row tile may end 64 rows past
      operand(g.B, g.bc, g.br, g.N, g.bmode == 1 ? 3 : 0, 0, (int16_t)-ksgn, ksgn != 0);   // rows: B's columns
      for (int j0 = 0; j0 < g.N; j0 += sg::kN)
        for (int i0 = 0; i0 < g.M; i0 += sg::kM) {
          if (g.lower_c && i0 + sg::kM - 1 < j0) continue;
          const int kend = g.amode == 1 ? std::min(g.K, i0 + sg::kM) : g.K;
          const int kb0 = g.bmode == 1 ? j0 / sg::kBlockK : 0, kb1 = (kend + sg::kBlockK - 1) / sg::kBlockK;
          pl.stiles.push_back({d, i0, j0, std::min(kb0, kb1 - 1), kb1, 0});
        }
    }
    gr.flops += gemm_flops(g);
    int ks = split_of(g, ksel);
    if (ks > 1) {
      g.kchunk = (((g.K + ks - 1) / ks) + 15) / 16 * 16;
      ks = (g.K + g.kchunk - 1) / g.kchunk;
    }
    g.ksplit = ks;
    if (ks == 1) g.kchunk = g.K;
    g.part = part;
    const int32_t d = (int32_t)pl.descs.size();
    pl.descs.push_back(g);
    const int ntj = (g.N + kGTile - 1) / kGTile;
    for (int ti = 0; ti * kGTile < g.M; ++ti)
      for (int tj = 0; tj < ntj; ++tj) {
        if (g.lower_c && ti * kGTile + kGTile - 1 < tj * kGTile) continue;
        for (int kc = 0; kc < ks; ++kc) pl.tiles.push_back({d, ti, tj, kc});
        if (ks > 1) pl.rtiles.push_back({d, ti, tj, 0});
      }
    if (ks > 1) part += (int64_t)((g.M + kGTile - 1) / kGTile) * ntj * ks * kGTile * kGTile;
  }
  // long sums first, so that the last tiles of the launch are short ones
  std::stable_sort(pl.stiles.begin() + gr.gb, pl.stiles.end(),
                   [](const SplitTile& x, const SplitTile& y) { return x.kb1 - x.kb0 > y.kb1 - y.kb0; });
  gr.sn = (int32_t)pl.stasks.size() - gr.sb;
  gr.gn = (int32_t)pl.stiles.size() - gr.gb;
  pl.slab_rows = std::max(pl.slab_rows, srow);
  pl.nexps = std::max(pl.nexps, sexp);
  gr.tn = (int32_t)pl.tiles.size() - gr.tb;
  gr.rn = (int32_t)pl.rtiles.size() - gr.rb;
  pl.part_max = std::max(pl.part_max, part);
  return gr;
}

template <class T>
void si_drop(chol_handle* h, T** p, int64_t bytes) {
  if (*p) {
    cudaFree(*p);   // waits for the work that uses it
    h->dev->bytes -= bytes;
  }
  *p = nullptr;
}

void free_si_split(chol_handle* h, SiPlan* pl) {
  auto drop = [&](auto** p, int64_t bytes) { si_drop(h, p, bytes); };
  drop(&pl->d_ops, (int64_t)(sizeof(SplitOp) * pl->ops.size()));
  drop(&pl->d_stasks, (int64_t)(sizeof(SplitTask) * pl->stasks.size()));
  drop(&pl->d_stiles, (int64_t)(sizeof(SplitTile) * pl->stiles.size()));
  drop(&pl->d_slab, pl->slab_rows * 64);
  drop(&pl->d_exps, (int64_t)(sizeof(int32_t) * pl->nexps));
  drop(&pl->d_kexps, (int64_t)(sizeof(int32_t) * std::max<int64_t>(pl->nkexps, 1)));
}

void free_si_plan(chol_handle* h, SiPlan* pl) {
  free_si_split(h, pl);
  si_drop(h, &pl->d_descs, (int64_t)(sizeof(GenGemm) * pl->descs.size()));
  si_drop(h, &pl->d_tiles, (int64_t)(sizeof(GemmTile) * pl->tiles.size()));
  si_drop(h, &pl->d_rtiles, (int64_t)(sizeof(GemmTile) * pl->rtiles.size()));
  si_drop(h, &pl->d_invs, (int64_t)(sizeof(InvTask) * pl->invs.size()));
  si_drop(h, &pl->d_part, (int64_t)sizeof(double) * pl->part_max);
  delete pl;
}

int build_si_plan(chol_handle* h) {
  DeviceState* D = h->dev;
  if (D->si_plan) return CHOL_OK;
  SiPlan* pl = new SiPlan();
  auto fail = [&](int rc) {
    free_si_plan(h, pl);
    return rc;
  };
  const double* L = D->L;
  // Z_RR of a level lives in the update workspace, at U_J's place; an RLB
  // handle has none, so it gets its own
  if (h->update_doubles < h->update_doubles_rl && !D->zrr_ws) {
    const int rz = chol_dalloc(h, (void**)&D->zrr_ws, sizeof(double) * (size_t)h->update_doubles_rl);
    if (rz) return fail(rz);
  }
  double* ZRR = D->zrr_ws ? D->zrr_ws : D->U;
  double* Z = D->Zp;
  int64_t tmax = 0, hmax = 0, wmax = 0;
  // per-level offsets of T (s^2), Uhat (b s) and W (s^2 / 2)
  std::vector<int64_t> toff(h->ns), hoff(h->ns), woff(h->ns);
  for (const LevelPlan& P : h->levels) {
    int64_t t = 0, u = 0, w = 0;
    for (int32_t q = 0; q < P.snode_n; ++q) {
      const int32_t J = h->level_snodes[P.snode_b + q];
      const SnodeDev& d = h->snodes[J];
      toff[J] = t; hoff[J] = u; woff[J] = w;
      t += (int64_t)d.s * d.s;
      u += (int64_t)(d.len - d.s) * d.s;
      w += ((int64_t)d.s * d.s + 1) / 2;   // B A^{-1} of one doubling step: at most s^2 / 2
    }
    tmax = std::max(tmax, t); hmax = std::max(hmax, u); wmax = std::max(wmax, w);
  }
  int rc;
  auto work = [&](double** p, int64_t n) {   // kept by a build that found no room further on
    return *p ? CHOL_OK : chol_dalloc(h, (void**)p, sizeof(double) * (size_t)std::max<int64_t>(n, 1));
  };
  if ((rc = work(&D->Tw, tmax)) || (rc = work(&D->Uh, hmax)) || (rc = work(&D->Ww, wmax))) return fail(rc);
  std::vector<int32_t> fbase(h->ns, -1);   // first block of J in the solve's inverses
  for (const TriItemHost& q : h->tri_items) fbase[q.J] = q.fbase;
  for (int lv = h->nlevels - 1; lv >= 0; --lv) {
    const LevelPlan& P = h->levels[lv];
    SiLevel sl{};
    sl.level = lv;
    std::vector<int32_t> Js(h->level_snodes.begin() + P.snode_b, h->level_snodes.begin() + P.snode_b + P.snode_n);
    int maxnbk = 0;
    int64_t tl = 0;
    for (int32_t J : Js) {
      maxnbk = std::max(maxnbk, (h->snodes[J].s + 63) / 64);
      tl += (int64_t)h->snodes[J].s * h->snodes[J].s;
    }
    sl.t_doubles = tl;
    // T = L_JJ^{-1} by recursive doubling: first every 64 x 64 diagonal block
    // is inverted (all at once), then blocks of size bs = 64, 128, ... are
    // combined pairwise, [A 0; B C]^{-1} = [A^{-1} 0; -C^{-1} B A^{-1} C^{-1}],
    // W = B A^{-1} then the off-diagonal block = -C^{-1} W, every pair of every
    // supernode of the level in one launch per product
    {
      SiStep st{};
      st.inv_b = (int32_t)pl->invs.size();
      for (int32_t J : Js) {
        const SnodeDev& d = h->snodes[J];
        double* T = D->Tw + toff[J];
        for (int k0 = 0; k0 < d.s; k0 += 64) {
          const int kb = std::min(64, d.s - k0);
          const double* inv = fbase[J] < 0 ? nullptr : (const double*)D->dinv + (int64_t)(fbase[J] + k0 / 64) * 4096;
          pl->invs.push_back({L + d.loff + k0 + (int64_t)k0 * d.ld, d.ld, T + k0 + (int64_t)k0 * d.s, d.s, inv, kb, 0});
          st.flops += (double)kb * kb * kb / 3.0;
        }
      }
      st.inv_n = (int32_t)pl->invs.size() - st.inv_b;
      sl.steps.push_back(st);
    }
    for (int bs = 64; bs < maxnbk * 64; bs *= 2) {
      SiStep st{};
      st.inv_b = (int32_t)pl->invs.size();
      std::vector<GenGemm> g1s, g2s;
      std::vector<int64_t> kx;
      int64_t xoff = 0;
      for (int32_t J : Js) {
        const SnodeDev& d = h->snodes[J];
        double* T = D->Tw + toff[J];
        double* Wp = D->Ww + woff[J];
        for (int i0 = 0; i0 + bs < d.s; i0 += 2 * bs) {
          const int c0 = i0 + bs, mc = std::min(c0 + bs, d.s) - c0;
          g1s.push_back(mk(L + d.loff + c0 + (int64_t)i0 * d.ld, 1, d.ld, T + i0 + (int64_t)i0 * d.s, 1, d.s, Wp, 1, mc,
                           mc, bs, bs, 1.0, 0.0, 0, 1, 0));
          g2s.push_back(mk(T + c0 + (int64_t)c0 * d.s, 1, d.s, Wp, 1, mc, T + c0 + (int64_t)i0 * d.s, 1, d.s, mc, bs, mc,
                           -1.0, 0.0, 1, 0, 0));
          kx.push_back(xoff);
          xoff += mc;
          Wp += (int64_t)mc * bs;
        }
      }
      pl->nkexps = std::max(pl->nkexps, xoff);
      st.g1 = emit_group(*pl, g1s, D->sms, kx, 0);
      st.g2 = emit_group(*pl, g2s, D->sms, kx, 1);
      st.flops = st.g1.flops + st.g2.flops;
      sl.steps.push_back(st);
    }
    // Uhat = L_RJ T
    std::vector<GenGemm> gs;
    std::vector<int64_t> kx;   // row exponents of L_RJ
    int64_t xoff = 0;
    for (int32_t J : Js) {
      const SnodeDev& d = h->snodes[J];
      const int b = d.len - d.s;
      if (b > 0) {
        gs.push_back(mk(L + d.loff + d.s, 1, d.ld, D->Tw + toff[J], 1, d.s, D->Uh + hoff[J], 1, b, b, d.s, d.s, 1.0,
                        0.0, 0, 1, 0));
        kx.push_back(xoff);
        xoff += b;
      }
    }
    pl->nkexps = std::max(pl->nkexps, xoff);
    sl.uh = emit_group(*pl, gs, D->sms, kx, 0);
    // Z_RJ = -Z_RR Uhat  (Z_RR at U_J's place in the update workspace)
    gs.clear();
    for (int32_t J : Js) {
      const SnodeDev& d = h->snodes[J];
      const int b = d.len - d.s;
      if (b > 0)
        gs.push_back(mk(ZRR + d.uoff, 1, b, D->Uh + hoff[J], 1, b, Z + d.loff + d.s, 1, d.ld, b, d.s, b, -1.0, 0.0, 2,
                        0, 0));
    }
    sl.zrj = emit_group(*pl, gs, D->sms, kx, 1);
    // Z_JJ = T^T T, then -= Uhat^T Z_RJ
    gs.clear();
    for (int32_t J : Js) {
      const SnodeDev& d = h->snodes[J];
      double* T = D->Tw + toff[J];
      gs.push_back(mk(T, d.s, 1, T, 1, d.s, Z + d.loff, 1, d.ld, d.s, d.s, d.s, 1.0, 0.0, 0, 0, 1));
    }
    sl.zjj1 = emit_group(*pl, gs, D->sms);
    gs.clear();
    for (int32_t J : Js) {
      const SnodeDev& d = h->snodes[J];
      const int b = d.len - d.s;
      if (b > 0)
        gs.push_back(mk(D->Uh + hoff[J], b, 1, Z + d.loff + d.s, 1, d.ld, Z + d.loff, 1, d.ld, d.s, d.s, b, -1.0, 1.0, 0,
                        0, 1));
    }
    sl.zjj2 = emit_group(*pl, gs, D->sms, kx, -1);
    sl.gemm_flops = sl.uh.flops + sl.zrj.flops + sl.zjj1.flops + sl.zjj2.flops;
    pl->levels.push_back(std::move(sl));
  }
  auto up = [&](auto** dst, const auto& v) -> int {
    if (v.empty()) return CHOL_OK;
    int r = chol_dalloc(h, (void**)dst, v.size() * sizeof(v[0]));
    if (r) return r;
    CHOL_CUDA_TRY(cudaMemcpy(*dst, v.data(), v.size() * sizeof(v[0]), cudaMemcpyHostToDevice));
    return CHOL_OK;
  };
  if ((rc = up(&pl->d_descs, pl->descs))) return fail(rc);
  // the tensor-core form where its slices find room (as for the factor's updates)
  if (h->opt.device_mem_cap == 0 && D->sg_ready == 1 && !pl->stiles.empty()) {
    pl->sg = up(&pl->d_ops, pl->ops) == CHOL_OK && up(&pl->d_stasks, pl->stasks) == CHOL_OK &&
             up(&pl->d_stiles, pl->stiles) == CHOL_OK &&
             chol_dalloc(h, (void**)&pl->d_slab, (size_t)pl->slab_rows * 64) == CHOL_OK &&
             chol_dalloc(h, (void**)&pl->d_kexps, sizeof(int32_t) * (size_t)std::max<int64_t>(pl->nkexps, 1)) == CHOL_OK &&
             chol_dalloc(h, (void**)&pl->d_exps, sizeof(int32_t) * (size_t)pl->nexps) == CHOL_OK &&
             cudaFuncSetAttribute(k_split_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, sg::kSmemBytes) ==
                 cudaSuccess;
    if (!pl->sg) free_si_split(h, pl);
  }
  if (!pl->sg) {
    if ((rc = up(&pl->d_tiles, pl->tiles))) return fail(rc);
    if ((rc = up(&pl->d_rtiles, pl->rtiles))) return fail(rc);
    if (pl->part_max > 0 && (rc = chol_dalloc(h, (void**)&pl->d_part, sizeof(double) * (size_t)pl->part_max)))
      return fail(rc);
  }
  if ((rc = up(&pl->d_invs, pl->invs))) return fail(rc);
  if (cudaStreamSynchronize(cudaStreamLegacy) != cudaSuccess) return fail(CHOL_ECUDA);   // the copies
  D->si_plan = pl;
  return CHOL_OK;
}

// Selected inverse into D->Zp (once per factorization), level by level from the
// root, every supernode of a level at once.
int selinv(chol_handle* h, cudaStream_t st) {
  // a captured call computes whether Z is there or not: its replays may follow another factor
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  CHOL_CUDA_TRY(cudaStreamIsCapturing(st, &cap));
  const bool capturing = cap != cudaStreamCaptureStatusNone;
  if (h->selinv_valid && !capturing) return CHOL_OK;
  if (h->max_len > kSelinvMaxLen) return CHOL_ENOTSUP;
  int rc = ensure_adjoint(h);
  if (rc) return rc;
  if ((rc = build_si_plan(h))) return rc;
  DeviceState* D = h->dev;
  SiPlan* pl = (SiPlan*)D->si_plan;
  if (capturing) pl->pinned = true;
  auto launch = [&](const Group& gr) {
    if (pl->sg) {
      if (gr.gn == 0) return;
      k_split_op<<<gr.sn, kSplitOpThreads, 0, st>>>(pl->d_ops, pl->d_stasks + gr.sb, pl->d_slab, pl->d_exps, pl->d_kexps);
      k_split_gemm<<<std::min(gr.gn, D->sms), sg::kThreads, sg::kSmemBytes, st>>>(
          pl->d_descs, pl->d_ops, pl->d_stiles + gr.gb, gr.gn, pl->d_slab, pl->d_exps,
          sg::Waits{D->sg_err, chol_test_wait(h, kTestWaitSelinv)});
      return;
    }
    if (gr.tn > 0) k_gen_gemm_grouped<<<gr.tn, kGT, 0, st>>>(pl->d_descs, pl->d_tiles + gr.tb, pl->d_part);
    if (gr.rn > 0) k_gen_reduce<<<gr.rn, kGT, 0, st>>>(pl->d_descs, pl->d_rtiles + gr.rb, pl->d_part);
  };
  auto nl = [&](const Group& gr) { return pl->sg ? 2 * (gr.gn > 0) : (gr.tn > 0) + (gr.rn > 0); };
  for (const SiLevel& sl : pl->levels) {
    CHOL_CUDA_TRY(cudaMemsetAsync(D->Tw, 0, sizeof(double) * (size_t)sl.t_doubles, st));
    for (const SiStep& q : sl.steps) {
      KScope ks(h, CHOL_K_SELINV_INV, st, q.flops, 0.0);
      ks.launches((q.inv_n > 0) + nl(q.g1) + nl(q.g2));
      if (q.inv_n > 0) k_inv64_grouped<<<q.inv_n, kInvThreads, 0, st>>>(pl->d_invs + q.inv_b);
      launch(q.g1);
      launch(q.g2);
    }
    if (const LevelPlan& P = h->levels[sl.level]; P.asm_n + P.asmw_n > 0) {
      KScope ks(h, CHOL_K_SELINV_GATHER, st, 0.0, 16.0 * P.asm_entries);
      const AsmSplit a = asm_split(P, D->sms);
      ks.launches((a.ctas > 0) + (a.warps > 0));
      chol_gather_zrr(h, P, D->Zp, D->zrr_ws ? D->zrr_ws : D->U, st);
    }
    {
      KScope ks(h, CHOL_K_SELINV_GEMM, st, sl.gemm_flops, 0.0);
      ks.launches(nl(sl.uh) + nl(sl.zrj) + nl(sl.zjj1) + nl(sl.zjj2));
      launch(sl.uh);
      launch(sl.zrj);
      launch(sl.zjj1);
      launch(sl.zjj2);
    }
  }
  CHOL_CUDA_TRY(cudaGetLastError());
  if (!capturing) h->selinv_valid = true;
  return CHOL_OK;
}

}  // namespace

void chol_adjoint_free(chol_handle* h) {
  DeviceState* D = h->dev;
  if (!D || !D->si_plan) return;
  free_si_plan(h, (SiPlan*)D->si_plan);
  D->si_plan = nullptr;
}

bool chol_adjoint_split(const chol_handle* h) {
  const SiPlan* pl = (const SiPlan*)h->dev->si_plan;
  return pl && pl->sg;
}

// Gives back a plan that holds slices (the next call builds one without them).
bool chol_adjoint_release(chol_handle* h) {
  const SiPlan* pl = (const SiPlan*)h->dev->si_plan;
  if (!pl || !pl->sg || pl->pinned) return false;
  chol_adjoint_free(h);
  return true;
}

extern "C" int chol_selected_inverse(chol_handle* h, double* zvals, void* stream) {
  NvtxRange nvtx_range("chol_selected_inverse");
  if (!h) return -1;
  if (!zvals && h->nnz_a > 0) return -2;
  if (int rc_state = chol_factored_here(h)) return rc_state;
  if (h->opt.precision != CHOL_PREC_FP64) return CHOL_ENOTSUP;
  cudaStream_t st = (cudaStream_t)stream;
  int rc = selinv(h, st);
  if (rc) return rc;
  DeviceState* D = h->dev;
  if (h->nnz_a > 0) k_take<<<grid1d(h->nnz_a, 256), 256, 0, st>>>(D->Zp, D->amap, h->nnz_a, zvals);
  CHOL_CUDA_TRY(cudaGetLastError());
  return CHOL_OK;
}

extern "C" int chol_adjoint(chol_handle* h, const double* w, const double* x, int32_t nrhs, double logdet_weight,
                            double* bbar, double* grad, void* stream) {
  NvtxRange nvtx_range("chol_adjoint");
  if (!h) return -1;
  if (!w && nrhs > 0) return -2;
  if (!x && nrhs > 0) return -3;
  if (nrhs < 0) return -4;
  if (!grad && h->nnz_a > 0) return -7;
  if (int rc_state = chol_factored_here(h)) return rc_state;
  if (h->opt.precision != CHOL_PREC_FP64) return CHOL_ENOTSUP;
  cudaStream_t st = (cudaStream_t)stream;
  int rc = ensure_adjoint(h);
  if (rc) return rc;
  DeviceState* D = h->dev;
  double* xb = bbar;
  if (nrhs > 0) {
    if (!xb) {
      if (D->adj_cap < nrhs) {
        if (D->adj_xb) cudaFree(D->adj_xb);
        D->adj_xb = nullptr;
        if ((rc = chol_dalloc(h, (void**)&D->adj_xb, sizeof(double) * (size_t)h->n * nrhs))) return rc;
        D->adj_cap = nrhs;
      }
      xb = D->adj_xb;
    }
    // Xbar = A^{-1} W
    CHOL_CUDA_TRY(cudaMemcpyAsync(xb, w, sizeof(double) * (size_t)h->n * nrhs, cudaMemcpyDeviceToDevice, st));
    if ((rc = chol_solve(h, xb, nrhs, (void*)st))) return rc;
  }
  if (logdet_weight != 0.0 && (rc = selinv(h, st))) return rc;
  if (h->nnz_a > 0) {
    KScope ks(h, CHOL_K_ADJOINT, st, 4.0 * nrhs * (double)h->nnz_a, 0.0);
    k_adj_grad<<<grid1d(h->nnz_a, 256), 256, 0, st>>>(D->a_row, D->a_col, D->amap,
                                                      logdet_weight != 0.0 ? D->Zp : nullptr, logdet_weight, xb, x,
                                                      h->n, nrhs, h->nnz_a, grad);
  }
  CHOL_CUDA_TRY(cudaGetLastError());
  return CHOL_OK;
}
