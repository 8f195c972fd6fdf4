// split_gemm.cuh -- binary64 products on the bf16 tensor cores.
//
// The binary64 pipe of this part retires two FMAs per cycle and SM, the tensor
// cores about 4,096 bf16 multiply-adds, so a binary64 product D = A B^T is
// computed from exact pieces (the error-free splitting of Ozaki, Ogita, Oishi
// and Rump, "Error-free transformations of matrix multiplication by using fast
// routines of matrix multiplication", Numer. Algorithms 59, 2012):
// - each row of an operand gets one exponent e with |x| 2^-e < 1/2 for its
//   entries, and every entry becomes the integer Y = round(x 2^(63 - e)),
//   written with kSlices = 7 signed base-512 digits, Y = sum_i d_i 512^(6 - i),
//   d_i in [-256, 256]. A digit is exact in bf16.
// - the product of slices i and j has weight 2^(ea + eb - 9 (i + j + 2)). The
//   slice products of one order i + j = q <= 6 share one binary32 accumulator
//   over kChunkK = 64 columns. Its integers stay at most (q + 1) 64 2^16: exact
//   for the orders 0..3 whatever the digits; the orders 4..6 (weights of 2^-54
//   and less) pass 2^24 only if almost all their digits are extreme and agree
//   in sign (digits in general position give about 2^19), and then lose their
//   last bit. Orders above 6 (2^-81 times 2^16 K at most) are left out.
// - the seven sums are added as integers, rounded once to binary64 and scaled.
// So an entry's error is its one rounding plus about sqrt(K) 2^-62, at most about
// K 2^-60 (equal entries), times the product of the two rows' largest entries.
// Normwise that is less than the error of K binary64 FMAs (K 2^-53), and it does
// not change when rows are scaled by powers of two (nor does the result, but for
// last bits where the rows' exponents add to more than 900). It is not relative to the sum's
// own terms, as the FMAs' is: an entry below 2^-10 of its row's largest keeps fewer
// than 53 bits and one below 2^-63 none, so where every large entry of one row
// meets a small one of the other (graded rows), the result has fewer correct
// bits than FMAs give it (chol_options.fp64_products).
// (Digits of base 256 with the same orders,
// 2^-57, were measured too: on the irregular 36^3 Laplacian, whose solution
// hangs on small entries of L, x was 4 times further off than with FMAs.)
// The summation order is fixed, so results are reproducible bit for bit. A row
// that holds an infinity or a NaN gives NaN in its row of the product.
//
// Slices are stored in the layout the tensor cores read from shared memory:
// per 32-column block of K, per slice, rows of 32 bf16 (64 bytes) with the
// 64-byte swizzle (16-byte chunk c of row r at chunk c ^ ((r >> 1) & 3)), so a
// 128-row operand slice is one contiguous 8 KiB copy without a tensor map.
#pragma once
#include <cuda_bf16.h>

#include <climits>
#include <cstdint>

#include "internal.h"
#include "tc_gemm.cuh"

namespace sg {

constexpr int kSlices = kSplitSlices;
constexpr int kM = 128, kN = 64;          // output tile (kN: of the updates; Cfg<N>)
constexpr int kBlockK = 32;               // K of one stage
constexpr int kDigit = 9;                 // bits of a digit
constexpr int kChunkK = 64;               // K per accumulator chunk (see above)
constexpr int kStagesPerChunk = kChunkK / kBlockK;
constexpr int kABytes = kM * 64;          // one slice of an operand stage
constexpr int kCols = 16;                 // columns of an epilogue thread
// A kernel with tiles of N columns: 64 (updates, one stage of 86 KB) or 16 (the
// products with right-hand sides, 64 KB).
template <int N>
struct Cfg {
  static constexpr int kBBytes = N * 64;
  static constexpr int kStageBytes = kSlices * (kABytes + kBBytes);
  static constexpr int kStages = N == 64 ? 2 : 3;
  static constexpr int kSmemBytes = kStages * kStageBytes + 1024;
  static constexpr int kEpiWarps = 4 * (N / kCols);   // 16 or 4: the epilogue is integer work with short chains
  static constexpr int kThreads = 32 * (kEpiWarps + 2);   // epilogue, copy and MMA warps
  static constexpr int kTmemCols = N == 64 ? 512 : 128;   // 7 accumulators of N columns
  static constexpr uint32_t kIdesc =
      (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(kM >> 4) << 24);
};
constexpr int kEpiWarps = Cfg<kN>::kEpiWarps, kThreads = Cfg<kN>::kThreads, kSmemBytes = Cfg<kN>::kSmemBytes;

// Operand splitting: 512 threads take R rows, 8 columns a thread, so that an
// operand of few rows and many columns still gives enough CTAs and loads in
// flight (64 rows and 64 columns a step took 31 us where this takes 13).
constexpr int kSplitThreadsLog2 = 9, kSplitThreads = 1 << kSplitThreadsLog2;
__device__ __forceinline__ int split_rows_log2(int K) { return SPLIT_ROWS_LOG2(K); }

constexpr int32_t kExpNaN = INT_MIN;      // exponent of a row with an infinity or a NaN
constexpr int32_t kExpMin = -1020;        // rows of zeros and subnormals

// Row exponent from the largest high word (sign cleared) of a row's entries.
__device__ __forceinline__ int32_t row_exponent(uint32_t hi_max) {
  const int E = (int)(hi_max >> 20);
  if (E == 0x7ff) return kExpNaN;
  return (E > 1 ? E : 1) - 1021;          // |x| < 2^(E - 1022), so |x| 2^-e < 1/2
}

// round(x 2^(63 - e)), |.| <= 2^62, for an entry of a row with exponent e.
__device__ __forceinline__ long long fixed_point(double x, int32_t e) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)(u >> 52) & 0x7ff;
  unsigned long long m = u & 0xfffffffffffffull;
  if (ex) m |= 1ull << 52;
  const int sh = e + 1021 - (ex ? ex : 1);          // E - ex >= 0: Y = m 2^(9 - sh), rounded
  m <<= 9;
  if (sh > 0) m = sh < 63 ? (m + (1ull << (sh - 1))) >> sh : 0;
  return (u >> 63) ? -(long long)m : (long long)m;
}

// binary32 bits of a small integer (exact; the low 16 bits of the result are 0
// for |d| <= 256 and its high 16 bits are the bf16 value)
__device__ __forceinline__ uint32_t digit_bits(int d) {
  return __float_as_uint(__int_as_float(0x4B400000 + d) - 12582912.0f);
}

// The digits of eight consecutive entries of a row (e: exponent of each): out[i] =
// the 16 bytes (8 bf16) of slice i.
__device__ __forceinline__ void digits8(const double (&x)[8], const int32_t (&e)[8], uint4 (&out)[kSlices]) {
  uint32_t w[kSlices][4];
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    long long y0 = fixed_point(x[2 * p], e[2 * p]), y1 = fixed_point(x[2 * p + 1], e[2 * p + 1]);
#pragma unroll
    for (int i = kSlices - 1; i >= 0; --i) {
      // the low digit, sign-extended (the one left last is the top digit)
      const int d0 = i ? (int)((uint32_t)y0 << (32 - kDigit)) >> (32 - kDigit) : (int)y0;
      const int d1 = i ? (int)((uint32_t)y1 << (32 - kDigit)) >> (32 - kDigit) : (int)y1;
      w[i][p] = __byte_perm(digit_bits(d0), digit_bits(d1), 0x7632);
      y0 = (y0 - d0) >> kDigit;
      y1 = (y1 - d1) >> kDigit;
    }
  }
#pragma unroll
  for (int i = 0; i < kSlices; ++i) out[i] = make_uint4(w[i][0], w[i][1], w[i][2], w[i][3]);
}

__device__ __forceinline__ void digits8(const double (&x)[8], int32_t e, uint4 (&out)[kSlices]) {
  const int32_t ee[8] = {e, e, e, e, e, e, e, e};
  digits8(x, ee, out);
}

// Byte offset of the 16-byte chunk c (0..3) of row r inside one slice.
__device__ __forceinline__ int64_t chunk_offset(int r, int c) {
  return (int64_t)r * 64 + ((c ^ ((r >> 1) & 3)) << 4);
}

// m 2^e as binary64, m rounded to nearest even (once).
__device__ __forceinline__ double scaled_int(long long m, int e) {
  if (m == 0) return 0.0;
  unsigned long long u = m < 0 ? (unsigned long long)(-m) : (unsigned long long)m;
  const int lz = __clzll((long long)u);
  u <<= lz;                                         // value = u 2^(e - lz), bit 63 set
  const int E = 63 + 1023 + e - lz;                 // biased exponent
  unsigned long long mant = u >> 11;
  const uint32_t rem = (uint32_t)u & 0x7ff;
  mant += (rem > 0x400u || (rem == 0x400u && (mant & 1))) ? 1u : 0u;
  if (E >= 1 && E <= 2045) {
    const unsigned long long b = ((unsigned long long)(E - 1) << 52) + mant;   // mant carries the implicit bit
    return __longlong_as_double((long long)(b | (m < 0 ? 1ull << 63 : 0ull)));
  }
  return ldexp((double)m, e);
}

// The sum hi 2^-45 + lo 2^-72 times 2^(ea + eb) (hi, lo: the integer sums of
// the orders 0..3 and 4..6), rounded to binary64: hi takes lo's carry, the
// magnitude is normalised with two funnel shifts and rounded at bit 53, and the
// exponent is put together: about 35 integer instructions and no binary64 ones. Sums below 2^-45 and exponents
// near the limits (zero rows, NaN) take scaled_int.
__device__ __forceinline__ double combine(long long hi, long long lo, int32_t ea, int32_t eb) {
  constexpr int kLow = 3 * kDigit;
  const int e = ea + eb;
  hi += lo >> kLow;
  const uint32_t low = (uint32_t)lo & ((1u << kLow) - 1);
  const uint32_t sgn = (uint32_t)(hi >> 63);
  // the magnitude's three words: complement, plus one at the lowest bit
  const uint32_t one = sgn & (1u << (32 - kLow));
  uint32_t w0 = ((low << (32 - kLow)) ^ (sgn << (32 - kLow))) + one;
  const unsigned long long w = ((unsigned long long)hi ^ (unsigned long long)(hi >> 63)) + (w0 < one ? 1u : 0u);
  uint32_t w2 = (uint32_t)(w >> 32), w1 = (uint32_t)w;
  if ((uint32_t)(e + 900) <= 1800u && ea != kExpNaN && eb != kExpNaN && (w2 | w1)) {
    int E = 1023 + 18 - 1 + e;                     // biased exponent of bit 63 of hi, less the implicit bit's one
    if (w2 == 0) { w2 = w1; w1 = w0; w0 = 0; E -= 32; }
    const int lz = __clz((int)w2);
    const uint32_t u1 = __funnelshift_l(w1, w2, lz), u0 = __funnelshift_l(w0, w1, lz);
    // the top 53 bits, rounded (bit 52 is the implicit one and adds to the exponent field)
    const unsigned long long m =
        (((unsigned long long)u1 << 32 | u0) >> 11) + ((u0 >> 10) & 1u) + ((unsigned long long)(uint32_t)(E - lz) << 52);
    return __longlong_as_double((long long)(m | (unsigned long long)(sgn & 0x80000000u) << 32));
  }
  if (ea == kExpNaN || eb == kExpNaN) return __longlong_as_double(0x7ff8000000000000ll);
  const int q = max(0, kLow + 1 - __clzll(hi ^ (hi >> 63)));   // low bits that do not fit beside hi
  const long long m = (long long)(((unsigned long long)hi << (kLow - q)) | (low >> q));
  return scaled_int(m, e - 8 * kDigit + q);
}

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// K-major operand, 64-byte swizzle, rows of 64 bytes, 8-row groups 512 bytes apart.
__device__ __forceinline__ uint64_t sw64_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(512 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)4 << 61;
  return d;
}

// Bounded wait that also gives up when another role of the CTA has.
__device__ __forceinline__ bool wait_or_abort(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  const long long t0 = clock64();
  for (uint32_t it = 0;; ++it) {
    if (tc::mbar_try_wait(bar, parity)) return true;
    if ((it & 63) == 63) {
      if (*abort_flag) return false;
      if (clock64() - t0 > (1ll << 31)) return false;
    }
  }
}

// One operand: slices of `rows` rows (K blocks of 32: [block][slice][rows][32]),
// the tile's first row, and the rows' exponents.
struct Operand {
  const unsigned char* slab;
  const int32_t* exps;
  int64_t rows;
  int row0;
};

struct Tile {
  Operand a, b;
  int nblk;      // K blocks
};

// Where a wait that gave up is recorded. fail (testing the failure path only,
// else -1): the epilogue warp whose waits count as run out at once.
struct Waits {
  int* err;
  int fail;
};

// Shared state of the CTA.
constexpr int kMaxStages = 3;
struct Shared {
  // accumulators change hands in two groups: orders 0..3 and 4..6
  uint64_t full[kMaxStages], empty[kMaxStages], acc_full[2], acc_empty[2], done;
  uint32_t tmem;
  int abort_flag, issued;
};

template <int N = kN>
__device__ __forceinline__ uint32_t setup(Shared& S) {
  const int warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    for (int s = 0; s < Cfg<N>::kStages; ++s) {
      tc::mbar_init(tc::smem_u32(&S.full[s]), 1);
      tc::mbar_init(tc::smem_u32(&S.empty[s]), 1);
    }
    for (int q = 0; q < 2; ++q) {
      tc::mbar_init(tc::smem_u32(&S.acc_full[q]), 1);
      tc::mbar_init(tc::smem_u32(&S.acc_empty[q]), Cfg<N>::kEpiWarps);
    }
    tc::mbar_init(tc::smem_u32(&S.done), 1);
    S.abort_flag = 0;
    S.issued = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(&S.tmem)),
                 "r"(Cfg<N>::kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  return S.tmem;
}

// Ends the CTA: waits (bounded) for the last copy issued into each stage and for the
// MMAs already issued; then frees the tensor memory. The copies are waited for
// whether a wait has given up or not: one that gives up later, after the copy
// thread has got here, may leave copies that no MMA has waited for.
template <int N = kN>
__device__ __forceinline__ void teardown(Shared& S, uint32_t tmem) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int never = 0;
  if (warp == Cfg<N>::kEpiWarps && lane == 0) {
    for (int s = 0; s < Cfg<N>::kStages && s < S.issued; ++s)
      wait_or_abort(tc::smem_u32(&S.full[s]), (uint32_t)(((S.issued - 1 - s) / Cfg<N>::kStages) & 1), &never);
  }
  if (warp == Cfg<N>::kEpiWarps + 1 && lane == 0) {
    tc::mma_commit(tc::smem_u32(&S.done));
    wait_or_abort(tc::smem_u32(&S.done), 0, &never);
  }
  __syncwarp();
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(Cfg<N>::kTmemCols) : "memory");
}

// The copy thread's loop over the CTA's tiles: `next(i, tile)` gives the i-th tile.
template <int N = kN, class Next>
__device__ __forceinline__ void copy_loop(Shared& S, uint32_t base, Next next, Waits w) {
  int it = 0;
  Tile t;
  for (int i = 0; next(i, t); ++i) {
    for (int k = 0; k < t.nblk; ++k, ++it) {
      const int s = it % Cfg<N>::kStages, round = it / Cfg<N>::kStages;
      if (round > 0 && !wait_or_abort(tc::smem_u32(&S.empty[s]), (uint32_t)((round - 1) & 1), &S.abort_flag)) {
        atomicExch(w.err, tc::kErrTimeoutEmpty);
        *(volatile int*)&S.abort_flag = 1;
        S.issued = it;
        return;
      }
      const uint32_t fb = tc::smem_u32(&S.full[s]);
      tc::mbar_expect_tx(fb, (uint32_t)Cfg<N>::kStageBytes);
      const uint32_t a0 = base + s * Cfg<N>::kStageBytes, b0 = a0 + kSlices * kABytes;
      const unsigned char* pa = t.a.slab + ((int64_t)k * kSlices * t.a.rows + t.a.row0) * 64;
      const unsigned char* pb = t.b.slab + ((int64_t)k * kSlices * t.b.rows + t.b.row0) * 64;
#pragma unroll
      for (int q = 0; q < kSlices; ++q) {
        bulk_load(a0 + q * kABytes, pa + (int64_t)q * t.a.rows * 64, kABytes, fb);
        bulk_load(b0 + q * Cfg<N>::kBBytes, pb + (int64_t)q * t.b.rows * 64, Cfg<N>::kBBytes, fb);
      }
    }
  }
  S.issued = it;
}

// The products of the orders [Q0, Q1) of one K block; `first`: the accumulators
// start here. Unrolled: the descriptors become additions of constants, and the
// issue keeps up with the 48 cycles that a 128 x 64 x 16 product takes (operand
// reads); in a loop over the slice pairs it took 112.
template <int N, int Q0, int Q1>
__device__ __forceinline__ void mma_orders(uint32_t tmem, uint64_t ad, uint64_t bd, bool first) {
#pragma unroll
  for (int q = Q0; q < Q1; ++q) {
    const uint32_t d = tmem + (uint32_t)(q * N);
#pragma unroll
    for (int a = 0; a <= q; ++a) {
      const uint64_t da = ad + (uint64_t)(a * (kABytes >> 4)), db = bd + (uint64_t)((q - a) * (Cfg<N>::kBBytes >> 4));
      tc::mma<1>(d, da, db, Cfg<N>::kIdesc, (first && a == 0) ? 0u : 1u);
      tc::mma<1>(d, da + 2, db + 2, Cfg<N>::kIdesc, 1u);
    }
  }
}

// The MMA thread's loop: per K block the 28 slice products of the orders 0..6;
// a group of orders is handed to the epilogue at the end of each chunk of
// kChunkK and taken back before its next use, so the epilogue reads one group
// while the other's products run.
template <int N = kN, class Next>
__device__ __forceinline__ void mma_loop(Shared& S, uint32_t base, uint32_t tmem, Next next, Waits w) {
  int it = 0, chunk = 0;
  Tile t;
  auto give_up = [&](int code) {
    atomicExch(w.err, code);
    *(volatile int*)&S.abort_flag = 1;
  };
  for (int i = 0; next(i, t); ++i) {
    for (int k = 0; k < t.nblk; ++k, ++it) {
      const int s = it % Cfg<N>::kStages, round = it / Cfg<N>::kStages;
      if (!wait_or_abort(tc::smem_u32(&S.full[s]), (uint32_t)(round & 1), &S.abort_flag)) {
        give_up(tc::kErrTimeoutFull);
        return;
      }
      const uint32_t a0 = base + s * Cfg<N>::kStageBytes;
      const uint64_t ad = sw64_desc(a0), bd = sw64_desc(a0 + kSlices * kABytes);
      const bool first = k % kStagesPerChunk == 0;
      const bool last = k % kStagesPerChunk == kStagesPerChunk - 1 || k == t.nblk - 1;
      const bool take = first && chunk > 0;
      const uint32_t par = (uint32_t)((chunk - 1) & 1);
      if (take && !wait_or_abort(tc::smem_u32(&S.acc_empty[0]), par, &S.abort_flag)) {
        give_up(tc::kErrTimeoutAccum);
        return;
      }
      tc::fence_after();
      mma_orders<N, 0, 4>(tmem, ad, bd, first);
      if (last) tc::mma_commit(tc::smem_u32(&S.acc_full[0]));
      if (take && !wait_or_abort(tc::smem_u32(&S.acc_empty[1]), par, &S.abort_flag)) {
        give_up(tc::kErrTimeoutAccum);
        return;
      }
      tc::fence_after();
      mma_orders<N, 4, kSlices>(tmem, ad, bd, first);
      if (last) tc::mma_commit(tc::smem_u32(&S.acc_full[1]));
      tc::mma_commit(tc::smem_u32(&S.empty[s]));
      if (last) ++chunk;
    }
  }
}

// A whole epilogue warp waits for group g of the chunk (uniform over the warp; other
// warps may see the same wait met, so a barrier among them needs epi_vote first).
__device__ __forceinline__ bool epi_wait(Shared& S, int g, int chunk, Waits w) {
  const bool ok = (int)(threadIdx.x >> 5) != w.fail &&
                  wait_or_abort(tc::smem_u32(&S.acc_full[g]), (uint32_t)(chunk & 1), &S.abort_flag);
  if (__all_sync(0xffffffffu, ok)) return true;
  atomicExch(w.err, tc::kErrTimeoutAccum);
  *(volatile int*)&S.abort_flag = 1;
  return false;
}

// True in every epilogue warp if `ok` is true in all of them: a barrier (named
// barrier 1) that each of them passes once a tile, whether its waits were met or not.
template <int N = kN>
__device__ __forceinline__ bool epi_vote(bool ok) {
  int all;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.b32 p, %1, 0;\n bar.red.and.pred q, 1, %2, p;\n selp.s32 %0, 1, 0, q;\n}\n"
      : "=r"(all)
      : "r"((int)ok), "n"(32 * Cfg<N>::kEpiWarps)
      : "memory");
  return all != 0;
}

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}

// The tile rows and columns of an epilogue thread: row (its tensor memory lane)
// 32 (warp mod 4) + lane, columns [16 (warp / 4), ... + 16).
__device__ __forceinline__ int epi_row() { return (int)(threadIdx.x & 127); }
__device__ __forceinline__ int epi_col() { return (int)(threadIdx.x >> 7) * kCols; }

// Adds one chunk's sums of the thread's 16 entries to hi (orders 0..3) and lo
// (orders 4..6) and gives the accumulators back. False if a wait gave up.
template <int N = kN>
__device__ __forceinline__ bool drain(Shared& S, uint32_t tmem, int chunk, long long (&hi)[kCols],
                                      long long (&lo)[kCols], Waits w) {
  const uint32_t t0 = tmem + ((uint32_t)((threadIdx.x >> 5) & 3) << 21) + (uint32_t)epi_col();
  if (!epi_wait(S, 0, chunk, w)) return false;
  tc::fence_after();
#pragma unroll
  for (int c = 0; c < kCols; c += 4) {
    uint32_t r[4][4];
#pragma unroll
    for (int q = 0; q < 4; ++q) tmem_ld4(t0 + (uint32_t)(q * N + c), r[q]);
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int q = 0; q < 4; ++q)
        hi[c + i] += (long long)__float2int_rn(__uint_as_float(r[q][i])) * (1 << (kDigit * (3 - q)));
  }
  tc::fence_before();
  __syncwarp();
  if ((threadIdx.x & 31) == 0) mbar_arrive(tc::smem_u32(&S.acc_empty[0]));
  if (!epi_wait(S, 1, chunk, w)) return false;
  tc::fence_after();
#pragma unroll
  for (int c = 0; c < kCols; c += 4) {
    uint32_t r[3][4];
#pragma unroll
    for (int q = 0; q < 3; ++q) tmem_ld4(t0 + (uint32_t)((q + 4) * N + c), r[q]);
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int q = 0; q < 3; ++q)
        lo[c + i] += (long long)__float2int_rn(__uint_as_float(r[q][i])) * (1 << (kDigit * (2 - q)));
  }
  tc::fence_before();
  __syncwarp();
  if ((threadIdx.x & 31) == 0) mbar_arrive(tc::smem_u32(&S.acc_empty[1]));
  return true;
}

}  // namespace sg
