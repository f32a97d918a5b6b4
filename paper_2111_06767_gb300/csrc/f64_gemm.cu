// FP64 subdomain-inverse GEMM on the tensor cores: exact products of 7-bit digits (the splitting of
// Ozaki, Ogita, Oishi & Rump, Numer. Algorithms 59, 2012, with digits of a fixed width).
//
// du_S = A_S^-1 r_S of an FP64 domain is bound by GB300's FP64 pipe (1.2 TFLOP/s) on CUDA cores. Here
// both operands are written as sums of S digits, a = 2^e sum_i d_i 2^(-6-7i) with integers
// |d_i| <= 64 and one power of two 2^e per row of the inverse and per column of r_S: 7 S bits below the
// row's or column's largest magnitude. Digits are exact in BF16, a product of two is at most 2^12, and
// the sums of one level l = i + j (at most 14 pairs) over at most 256 terms stay within 2^24, so that the
// FP32 accumulators of tcgen05 hold every level exactly. After each 256 terms the levels 0 .. S - 1 leave
// tensor memory as integers and are added into three 64-bit integers per output; pairs with i + j >= S lie at
// 2^(-7 S) of row times column maximum and below, and the one rounding to FP64 is at the very end.
//
// S = 12, 13 or 14 per level, the fewest that hold every entry of the level's inverses with all its 53 bits: the
// entries of one row span 2^20 to 2^25 at N = 4, 2^34 at N = 8 (overlap 2), up to 2^42 for wide overlaps and thin
// elements. A level whose rows span more than 14 digits hold (2^44) keeps the CUDA-core product. So |A_ik| >= 2^(53 -
// 7 S) max_k |A_ik|, and the error of every component, whatever r_S holds, is of the order of 2^-53 |A| |r_S|, as for
// FP64 sums, and not only its norm. Largest error relative to |A| |r_S| before the final rounding, overlap 2, N = 4, 6, 8: 13
// digits 6e-25 for a rough r_S, 4e-23 over 12 decades, 3e-18 for one point (FP64 sums in order: 2.5e-15, 3.9e-15 and
// 1e-16); 8 digits with levels 0..8 had 1.8e-15, 6e-14 and 3e-8.
//
// Work split: a CTA computes 128 rows x nc columns (nc = 16 or 32, so that the columns of a class
// carry little padding). The digits of X lie one slice after another, so the slices of nc columns
// are one N = S nc operand: digit i of the inverse multiplies slices 0 .. S - 1 - i in one sweep and
// lands on levels i .. S - 1, contiguous in tensor memory (S nc <= 448 columns). A warp streams the inverse's
// digit tiles (128 x 64, 16 KB) through a 7-stage TMA ring and X's chunk (S x nc x 64) through a double
// buffer, a warp issues the MMAs, eight warps drain the levels. K may be split over a cluster; the
// integer partial sums are added through distributed shared memory, so the result does not depend on
// the split.
//
// What bounds it: the chain inside a CTA. S digit tiles a chunk go through the ring and the MMAs in series, the MMAs wait
// for the drain of all levels every 256 terms, and a cluster's CTAs for each other: at 8^3 elements, N = 8 (13 digits,
// split 4, 760 CTAs) the tensor pipe is 36 % busy (43 % on the busiest SM), L2 19 %, DRAM 25 % from cold caches; unsplit
// (190 CTAs on 152 SMs) 46 % with 81 % on the busiest and 230 us. 8^3, N = 8: 187 us a launch against 1450 us on the CUDA
// cores; 6 x 8 x 4, N = 5: 26 and 4 us of slicing against 111. With 8 digits, in tiles of up to 48 columns, these took 93
// and 20 us: the price of every component's accuracy. Tiles ordered longest first: 185 us, no change.
#include <mutex>
#include <set>

#include "internal.h"
#include "pdl.cuh"
#include "tcgen05.cuh"

namespace dg {

namespace {

constexpr int BM = 128;         // rows of a tile
constexpr int BK = 64;          // K of a chunk: 128 bytes of BF16
constexpr int SEG = 4;          // chunks between drains: 256 terms
constexpr int MAXC = 32;        // columns of a tile, at most
constexpr int A_STAGES = 7, A_BYTES = BM * BK * 2;
constexpr int DRAIN = 256;      // threads of the draining warps
constexpr int THREADS = DRAIN + 64;

// S digits, and so S levels i + j = 0 .. S - 1
template <int S>
struct Digits {
  static constexpr int BITS = 7 * S - 1;  // of a digit string: |x| 2^(BITS - e) < 2^BITS
  static constexpr int B_BYTES = S * MAXC * BK * 2;
  static constexpr int SMEM_BYTES = 2 * B_BYTES + A_STAGES * A_BYTES + 1024 + 512;
  static_assert(S >= 10 && S <= 14, "three groups of levels, of five, five and at least one");
  static_assert(SMEM_BYTES <= 227 * 1024, "shared memory per CTA");
  static_assert(2 * MAXC * BM * 8 <= 2 * B_BYTES, "split-K partial sums fit in the idle X buffers");
  static_assert(S * BK * SEG * 4096 <= 1 << 24, "a level's sum is exact in FP32");
  static_assert(S * MAXC <= 512, "levels fit in tensor memory");
};
// FP32 accumulate, BF16 x BF16, both K-major, M = 128; N is added per instruction
constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BM >> 4) << 24);

__device__ __forceinline__ void mma_bf16(uint32_t tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred P1;\n\t"
      "setp.ne.b32 P1, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, P1;\n\t}" ::"r"(tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}

// Eight columns of one level, as integers.
__device__ __forceinline__ void tmem_ld8(uint32_t a, int (&d)[8]) {
  float v[8];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
      : "r"(a)
      : "memory");
#pragma unroll
  for (int j = 0; j < 8; ++j) d[j] = __float2int_rn(v[j]);
}

// The same of two levels `step` columns apart, joined: 128 times the first plus the second (level l is at most
// (l + 1) 2^20, so that fits in 32 bits up to l = 13).
__device__ __forceinline__ void tmem_ld8x2(uint32_t a, uint32_t step, int (&d)[8]) {
  float v[2][8];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%16];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8, %9, %10, %11, %12, %13, %14, %15}, [%17];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=f"(v[0][0]), "=f"(v[0][1]), "=f"(v[0][2]), "=f"(v[0][3]), "=f"(v[0][4]), "=f"(v[0][5]), "=f"(v[0][6]),
        "=f"(v[0][7]), "=f"(v[1][0]), "=f"(v[1][1]), "=f"(v[1][2]), "=f"(v[1][3]), "=f"(v[1][4]), "=f"(v[1][5]),
        "=f"(v[1][6]), "=f"(v[1][7])
      : "r"(a), "r"(a + step)
      : "memory");
#pragma unroll
  for (int j = 0; j < 8; ++j) d[j] = __float2int_rn(v[0][j]) * 128 + __float2int_rn(v[1][j]);
}

// COUNT <= 5 levels from the one at a on, in units of the last, added to sum.
template <int COUNT>
__device__ __forceinline__ void add_levels(uint32_t a, uint32_t step, int64_t (&sum)[8]) {
  int d[8];
  if constexpr (COUNT == 1) {
    tmem_ld8(a, d);
#pragma unroll
    for (int j = 0; j < 8; ++j) sum[j] += d[j];
  } else {
    constexpr int REST = COUNT - 2;
    tmem_ld8x2(a, step, d);
#pragma unroll
    for (int j = 0; j < 8; ++j) sum[j] += (int64_t)d[j] * (1 << 7 * REST);
    if constexpr (REST > 0) add_levels<REST>(a + 2 * step, step, sum);
  }
}

__device__ __forceinline__ int64_t ld_cluster_s64(uint32_t addr) {
  int64_t v;
  asm volatile("ld.shared::cluster.s64 %0, [%1];" : "=l"(v) : "r"(addr));
  return v;
}

// V 2^(e - 5 - 7 S) as a double, V the levels in units of the last (e: the operands' exponents), rounded to nearest, in integer arithmetic (one conversion and
// one multiplication per output on the FP64 pipe would cost more than the products of a small level).
template <int S>
__device__ __forceinline__ double combine(__int128 V, int e) {
  if (V == 0) return 0.0;
  const bool neg = V < 0;
  unsigned __int128 w = neg ? -(unsigned __int128)V : (unsigned __int128)V;
  int p = 127;  // place of the leading bit
  if ((uint64_t)(w >> 64) == 0) {
    w <<= 64;
    p -= 64;
  }
  const int s = __clzll((long long)(uint64_t)(w >> 64));
  const uint64_t t = (uint64_t)((w << s) >> 64);
  const int ex = 1023 + p - s - 5 - 7 * S + e;  // biased exponent of the leading bit
  const uint64_t m = (t >> 11) + ((t >> 10) & 1);
  double v;
  if (ex > 0 && ex < 2046) v = __longlong_as_double((long long)(((uint64_t)(ex - 1) << 52) + m));
  else v = ldexp((double)m, ex - 1023 - 52);
  return neg ? -v : v;
}

constexpr int kNonFinite = 1 << 20;  // scale exponent of a row or column with a NaN or an infinity

template <int S, int SPLIT>
__global__ void __launch_bounds__(THREADS, 1)
    f64_gemm_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB16,
                    const __grid_constant__ CUtensorMap mapB32, const int* __restrict__ row_exp,
                    const int* __restrict__ col_exp, double* __restrict__ Y, int ld, const int4* __restrict__ tiles,
                    const int* __restrict__ kchunks, int* __restrict__ err) {
  constexpr int B_BYTES = Digits<S>::B_BYTES;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  unsigned char* sB = smem;
  unsigned char* sA = smem + 2 * B_BYTES;
  uint64_t* bars = (uint64_t*)(sA + A_STAGES * A_BYTES);
  // a_full[7], a_empty[7], b_full[2], b_empty[2], levels ready, levels drained
  const uint32_t a_full = smem_u32(bars), a_empty = a_full + 8 * A_STAGES, b_full = a_empty + 8 * A_STAGES,
                 b_empty = b_full + 16, b_acc = b_empty + 16, b_drained = b_acc + 8;
  uint32_t* tmem_slot = (uint32_t*)(bars + 2 * A_STAGES + 6);
  int* s_count = (int*)(tmem_slot + 1);  // A tiles issued, A tiles seen, X chunks issued, X chunks seen

  const int rank = SPLIT > 1 ? (int)cluster_rank() : 0;
  const int4 tile = tiles[blockIdx.x / SPLIT];
  const int cls = tile.x & 0xFFFF, wc = (tile.x >> 24) & 3, nc = 16 * (wc + 1);
  const int row0 = tile.y, col0 = tile.z, ncol = min(tile.w, nc);
  const bool zero = (tile.x >> 30) & 1;  // rows only in the slots of missing neighbours: zeros
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nk64 = (ld + BK - 1) / BK;
  const int* kl = kchunks + (size_t)cls * (nk64 + 1);
  const int nk_all = zero ? 0 : kl[0];
  const int kc0 = rank * nk_all / SPLIT, nk = (rank + 1) * nk_all / SPLIT - kc0;
  kl += 1 + kc0;
  const uint32_t tmem_cols = nc == 16 ? 256 : 512;  // a power of two, at least S nc

  if (threadIdx.x == 0) {
    for (int i = 0; i < 4; ++i) s_count[i] = 0;
    for (int i = 0; i < A_STAGES; ++i) {
      mbar_init(a_full + 8 * i, 1);
      mbar_init(a_empty + 8 * i, 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(b_full + 8 * i, 1);
      mbar_init(b_empty + 8 * i, 1);
    }
    mbar_init(b_acc, 1);
    mbar_init(b_drained, DRAIN);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 9) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  // the inverse's first tiles, which nothing writes, overlap the previous kernel
  pdl_launch_dependents();
  const int ahead = min(A_STAGES, nk * S);
  if (warp == 8 && lane == 0) {
    for (int q = 0; q < ahead; ++q) {
      mbar_expect_tx(a_full + 8 * q, A_BYTES);
      tma_load_3d(smem_u32(sA + q * A_BYTES), &mapA, a_full + 8 * q, kl[q / S] * BK, row0, cls * S + q % S);
    }
    s_count[0] = ahead;
  }
  pdl_wait();

  bool ok = true;
  // this thread's row, columns half (nc / 2) + 8 g + j: levels 0-4, 5-9 and 10.. in units of the last of each
  int64_t H[2][8], M[2][8], L[2][8];
  if (warp == 8) {
    if (lane == 0) {
      const CUtensorMap* mapB = wc == 0 ? &mapB16 : &mapB32;
      for (int kc = 0; kc < nk && ok; ++kc) {
        const int bs = kc & 1, k0 = kl[kc] * BK;
        if (kc >= 2 && !(ok = mbar_wait(b_empty + 8 * bs, ((kc >> 1) - 1) & 1, err))) break;
        mbar_expect_tx(b_full + 8 * bs, (uint32_t)(S * nc * BK * 2));
        tma_load_3d(smem_u32(sB + bs * B_BYTES), mapB, b_full + 8 * bs, k0, col0, 0);
        s_count[2] = kc + 1;
        for (int i = 0; i < S; ++i) {
          const int q = kc * S + i, st = q % A_STAGES;
          if (q < ahead) continue;
          if (!(ok = mbar_wait(a_empty + 8 * st, ((q / A_STAGES) - 1) & 1, err))) break;
          mbar_expect_tx(a_full + 8 * st, A_BYTES);
          tma_load_3d(smem_u32(sA + st * A_BYTES), &mapA, a_full + 8 * st, k0, row0, cls * S + i);
          s_count[0] = q + 1;
        }
      }
    }
  } else if (warp == 9) {
    if (lane == 0) {
      for (int kc = 0; kc < nk && ok; ++kc) {
        const int bs = kc & 1, in_seg = kc % SEG;
        // the levels of the previous 256 terms have left tensor memory
        if (kc > 0 && in_seg == 0) ok = mbar_wait(b_drained, (kc / SEG - 1) & 1, err);
        ok = ok && mbar_wait(b_full + 8 * bs, (kc >> 1) & 1, err);
        if (!ok) break;
        s_count[3] = kc + 1;
        const uint32_t b0 = smem_u32(sB + bs * B_BYTES);
        for (int i = 0; i < S; ++i) {
          const int q = kc * S + i, st = q % A_STAGES;
          if (!(ok = mbar_wait(a_full + 8 * st, (q / A_STAGES) & 1, err))) break;
          s_count[1] = q + 1;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t a0 = smem_u32(sA + st * A_BYTES);
          const int ntot = (S - i) * nc;  // rows of the slices 0 .. S - 1 - i
          for (int n0 = 0; n0 < ntot; n0 += 256) {
            const int n = min(256, ntot - n0);
            const uint32_t idesc = IDESC | ((uint32_t)(n >> 3) << 17);
#pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk)  // the first digit's first products overwrite every level
              mma_bf16(tmem + i * nc + n0, smem_desc(a0 + 32 * kk), smem_desc(b0 + n0 * 128 + 32 * kk), idesc,
                       !(in_seg == 0 && i == 0 && kk == 0));
          }
          mma_commit(a_empty + 8 * st);
        }
        if (!ok) break;
        mma_commit(b_empty + 8 * bs);
        if (in_seg == SEG - 1 || kc == nk - 1) mma_commit(b_acc);
      }
      if (!ok) mma_commit(b_acc);
    }
  } else {
#pragma unroll
    for (int g = 0; g < 2; ++g)
#pragma unroll
      for (int j = 0; j < 8; ++j) H[g][j] = M[g][j] = L[g][j] = 0;
    const int half = warp >> 2, ng = nc / 16;  // this half's groups of 8 columns
    const uint32_t t0 = tmem + ((uint32_t)((warp & 3) * 32) << 16) + half * (nc / 2);
    for (int seg = 0; seg * SEG < nk; ++seg) {
      ok = __all_sync(0xffffffffu, mbar_wait(b_acc, seg & 1, err));
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
      for (int g = 0; g < 2; ++g) {
        if (g >= ng) break;
        const uint32_t a = t0 + g * 8;
        add_levels<5>(a, nc, H[g]);
        add_levels<5>(a + 5 * nc, nc, M[g]);
        add_levels<S - 10>(a + 10 * nc, nc, L[g]);
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      mbar_arrive(b_drained);
    }
  }
  __syncwarp();

  const int r_local = (warp & 3) * 32 + lane, row = row0 + r_local;
  auto sum = [&](int g, int j) { return ((__int128)H[g][j] << 7 * (S - 5)) + ((__int128)M[g][j] << 7 * (S - 10)) + L[g][j]; };
  auto output = [&](__int128 v, int er, int c) {
    const int ec = col_exp[col0 + c];
    if (zero) return 0.0;
    return ec == kNonFinite || er == kNonFinite ? __longlong_as_double(0x7FF8000000000000ll) : combine<S>(v, er + ec);
  };
  if constexpr (SPLIT == 1) {
    if (warp < 8 && row < ld) {
      const int er = row_exp[(size_t)cls * ld + row];
      const int c0 = (warp >> 2) * (nc / 2);
#pragma unroll
      for (int g = 0; g < 2; ++g) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int c = c0 + g * 8 + j;
          if (g * 16 >= nc || c >= ncol) continue;
          Y[(size_t)(col0 + c) * ld + row] = output(sum(g, j), er, c);
        }
      }
    }
  } else {
    // partial sums [low, high 64 bits][column][row] in the X buffers (every copy into them has been consumed)
    int64_t* part = reinterpret_cast<int64_t*>(smem);
    __syncthreads();
    if (warp < 8) {
      const int c0 = (warp >> 2) * (nc / 2);
#pragma unroll
      for (int g = 0; g < 2; ++g) {
        if (g * 16 >= nc) break;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const __int128 v = sum(g, j);
          part[(c0 + g * 8 + j) * BM + r_local] = (int64_t)v;
          part[(nc + c0 + g * 8 + j) * BM + r_local] = (int64_t)(v >> 64);
        }
      }
    }
    cluster_sync();
    if (warp < 8 && row < ld) {
      const int er = row_exp[(size_t)cls * ld + row];
      const int per = nc / SPLIT;
      const uint32_t base = smem_u32(part);
      for (int c = rank * per + (warp >> 2); c < (rank + 1) * per; c += 2) {
        __int128 v = 0;
#pragma unroll
        for (int p = 0; p < SPLIT; ++p) {
          const uint32_t peer = map_peer(base, (uint32_t)p);
          v += (__int128)(uint64_t)ld_cluster_s64(peer + (uint32_t)((c * BM + r_local) * 8));
          v += (__int128)ld_cluster_s64(peer + (uint32_t)(((nc + c) * BM + r_local) * 8)) << 64;
        }
        if (c < ncol) Y[(size_t)(col0 + c) * ld + row] = output(v, er, c);
      }
    }
    cluster_sync();  // no CTA leaves while a peer still reads its partial sums
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  const int bad = __syncthreads_or(!ok);
  if (bad && threadIdx.x == 0) {
    // a wait gave up: let the copies already issued land (bounded) before the CTA exits
    for (int q = s_count[1]; q < s_count[0]; ++q) mbar_wait(a_full + 8 * (q % A_STAGES), (q / A_STAGES) & 1, err);
    for (int q = s_count[3]; q < s_count[2]; ++q) mbar_wait(b_full + 8 * (q & 1), (q >> 1) & 1, err);
  }
  __syncthreads();
  if (warp == 9)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols) : "memory");
}

// Exponents h_k that equilibrate a class inverse: 2^h_k is the square root of its diagonal, so that the
// columns of the inverse (divided by 2^h_k) and the entries of r_S (times 2^h_k) of face and interior
// points, which differ by the penalty's factor of about 10^3, share one range of digits. Exact: powers
// of two. Without it the error of a smoothing step on 8^3 elements at N = 8 was 2.4 times the CUDA-core
// product's.
__global__ void equilibrate_kernel(const double* __restrict__ inv, int ld, int* __restrict__ hexp) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= ld) return;
  const double a = inv[((int64_t)blockIdx.y * ld + k) * ld + k];
  const int ex = (int)((uint64_t)__double_as_longlong(a) >> 52) & 0x7FF;
  // floor(log2(a) / 2); padding rows (zero diagonal) need none
  hexp[(int64_t)blockIdx.y * ld + k] = ex > 0 && ex < 0x7FF ? (ex - 1023) >> 1 : 0;
}

// Biased exponent of v 2^shift; subnormal values count as exponent 1, zero as kNone.
constexpr int kNone = -4096;
__device__ __forceinline__ int exponent_of(int64_t v, int shift) {
  const int xe = (int)((uint64_t)v >> 52) & 0x7FF;
  return (v << 1) == 0 ? kNone : (xe == 0x7FF ? kNonFinite : max(xe, 1) + shift);
}

// *range = the largest difference between the exponents of two entries (not zero, finite) of one row of the inverses,
// scaled as slice_kernel takes them (grid: rows x classes). *range starts at 0.
__global__ void __launch_bounds__(256) range_kernel(const double* __restrict__ src, int ld, double alpha,
                                                    const int* __restrict__ hexp, int* __restrict__ range) {
  const int* h = hexp + (int64_t)blockIdx.y * ld;
  const double* x = src + ((int64_t)blockIdx.y * ld + blockIdx.x) * ld;
  __shared__ int s_hi, s_lo;
  if (threadIdx.x == 0) {
    s_hi = kNone;
    s_lo = kNonFinite;
  }
  __syncthreads();
  int hi = kNone, lo = kNonFinite;
  for (int k = threadIdx.x; k < ld; k += 256) {
    const int e = exponent_of(__double_as_longlong(alpha * x[k]), -h[k]);
    if (e == kNone || e >= kNonFinite) continue;
    hi = max(hi, e);
    lo = min(lo, e);
  }
  atomicMax(&s_hi, hi);
  atomicMin(&s_lo, lo);
  __syncthreads();
  if (threadIdx.x == 0 && s_hi > s_lo) atomicMax(range, s_hi - s_lo);
}

// Digits of `rows` rows of ld doubles per group (grid: rows x groups) into BF16 slices
// dst[group][digit][row][ld], and the row's exponent e, every |x| < 2^e. Values are taken times
// 2^(sign h_k), h of the row's class (class_of[row], or the group), and times alpha (the inverses, once
// at set-up). A row with a NaN or an infinity gets the exponent kNonFinite, which the product hands on
// as NaN: for r_S to the whole column, for an inverse to the row of every column of its class. Integer arithmetic: the FP64 pipe would take ten times as long.
template <int S, bool ALPHA>
__global__ void __launch_bounds__(256) slice_kernel(const double* __restrict__ src, int ld, double alpha, int sign,
                                                    const int* __restrict__ hexp, const int* __restrict__ class_of,
                                                    uint16_t* __restrict__ dst, int* __restrict__ row_exp) {
  __shared__ int s_max[8];
  const int rows = gridDim.x, r = blockIdx.x;
  const int64_t row = (int64_t)blockIdx.y * rows + r;
  pdl_launch_dependents();
  const int2* h = reinterpret_cast<const int2*>(hexp + (int64_t)(class_of ? class_of[row] : blockIdx.y) * ld);
  pdl_wait();
  const double2* x = reinterpret_cast<const double2*>(src + row * ld);
  auto load = [&](int q) {
    double2 v = x[q];
    if constexpr (ALPHA) v = make_double2(alpha * v.x, alpha * v.y);
    return make_longlong2(__double_as_longlong(v.x), __double_as_longlong(v.y));
  };
  int ex = kNone;  // the largest exponent
  for (int q = threadIdx.x; q < ld / 2; q += 256) {
    const longlong2 v = load(q);
    const int2 hh = h[q];
    ex = max(ex, max(exponent_of(v.x, sign * hh.x), exponent_of(v.y, sign * hh.y)));
  }
  ex = __reduce_max_sync(0xffffffffu, ex);
  if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = ex;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < 8; ++w) ex = max(ex, s_max[w]);
  const bool finite = ex < kNonFinite;
  const int e = ex == kNone || !finite ? 0 : ex - 1022;
  if (threadIdx.x == 0) row_exp[row] = finite ? e : kNonFinite;
  uint16_t* out = dst + ((int64_t)blockIdx.y * S * rows + r) * ld;
  const int64_t stride = (int64_t)rows * ld;
  for (int q = threadIdx.x; q < ld / 2; q += 256) {
    const longlong2 v2 = load(q);
    const int2 hh = h[q];
    const int64_t v[2] = {v2.x, v2.y};
    const int shift[2] = {sign * hh.x, sign * hh.y};
    unsigned pack[S];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int xe = (int)((uint64_t)v[c] >> 52) & 0x7FF;
      uint64_t m = (uint64_t)v[c] & 0xFFFFFFFFFFFFFull;
      if (xe) m |= 0x10000000000000ull;
      const int sh = max(xe, 1) + shift[c] - (1075 - Digits<S>::BITS) - e;  // |x| 2^(BITS - e) = m 2^sh
      unsigned __int128 a = 0;
      if (sh >= 0) a = (unsigned __int128)m << sh;
      else if (sh > -64) a = (m + (1ull << (-sh - 1))) >> -sh;
      if (!finite || m == 0) a = 0;
      __int128 t = v[c] < 0 ? -(__int128)a : (__int128)a;
#pragma unroll
      for (int i = S - 1; i >= 0; --i) {
        const int d = i > 0 ? (int)(((unsigned)t + 64) & 127) - 64 : (int)t;
        t = (t - d) >> 7;
        const unsigned b = __float_as_uint((float)d) >> 16;  // exact in BF16
        pack[i] = c ? pack[i] | (b << 16) : b;
      }
    }
#pragma unroll
    for (int i = 0; i < S; ++i) *reinterpret_cast<unsigned*>(out + i * stride + 2 * q) = pack[i];
  }
}

CUtensorMap slice_map(const uint16_t* base, uint64_t ld, uint64_t rows, uint64_t slices, uint32_t box_rows,
                      uint32_t box_slices) {
  CUtensorMap m;
  auto fn = tensor_map_encoder();
  if (!fn) fail(DG_ERR_CUDA, "cuTensorMapEncodeTiled is unavailable");
  const cuuint64_t dims[3] = {ld, rows, slices}, strides[2] = {ld * 2, ld * rows * 2};
  const cuuint32_t box[3] = {BK, box_rows, box_slices}, one[3] = {1, 1, 1};
  const CUresult r = fn(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, (void*)base, dims, strides, box, one,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) fail(DG_ERR_CUDA, "cuTensorMapEncodeTiled failed: " + std::to_string((int)r));
  return m;
}

template <int S>
void set_attributes() {
  static std::mutex mu;
  static std::set<int> done;
  int dev = 0;
  DG_CUDA(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lk(mu);
  if (done.count(dev)) return;
  for (auto k : {f64_gemm_kernel<S, 1>, f64_gemm_kernel<S, 2>, f64_gemm_kernel<S, 4>, f64_gemm_kernel<S, 8>})
    DG_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, Digits<S>::SMEM_BYTES));
  done.insert(dev);
}

template <int S>
void launch_gemm(const F64Maps& maps, const int* inv_exp, const int* x_exp, double* Y, int ld, const int4* d_tiles,
                 int n_tiles, const int* d_kchunks, int* err, cudaStream_t s, int split) {
  set_attributes<S>();
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_tiles * split);
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = Digits<S>::SMEM_BYTES;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = split;
  at[1].val.clusterDim.y = 1;
  at[1].val.clusterDim.z = 1;
  const bool pdl = pdl_enabled();
  cfg.attrs = pdl ? at : at + 1;
  cfg.numAttrs = (pdl ? 1 : 0) + (split == 1 ? 0 : 1);
  auto k = split == 1 ? f64_gemm_kernel<S, 1>
                      : (split == 2 ? f64_gemm_kernel<S, 2> : (split == 4 ? f64_gemm_kernel<S, 4> : f64_gemm_kernel<S, 8>));
  DG_CUDA(cudaLaunchKernelEx(&cfg, k, maps.a, maps.x[0], maps.x[1], inv_exp, x_exp, Y, ld, d_tiles, d_kchunks, err));
  DG_LAUNCHED(1);
}

template <int S>
void launch_inverse_digits(const double* inv, double alpha, int n_classes, int ld, const int* hexp, uint16_t* dst,
                           int* row_exp, cudaStream_t s) {
  slice_kernel<S, true><<<dim3(ld, n_classes), 256, 0, s>>>(inv, ld, alpha, -1, hexp, nullptr, dst, row_exp);
}

template <int S>
void launch_column_digits(const double* X, int n_cols, int ld, const int* hexp, const int* class_of_col, uint16_t* dst,
                          int* col_exp, cudaStream_t s) {
  launch_pdl(slice_kernel<S, false>, dim3(n_cols), dim3(256), 0, s, X, ld, 1.0, 1, hexp, class_of_col, dst, col_exp);
}

}  // namespace

int f64_default_split(int n_tiles, int ld) {
  int split = 1;
  while (split < 8 && n_tiles * split * 2 <= 152 && (ld + BK - 1) / BK / (split * 2) >= 1) split *= 2;
  return split;
}

int f64_digits_for(int range) {
  for (int S : {12, 13, 14})
    if (range <= 7 * S - 54) return S;
  return 0;
}

void launch_f64_equilibrate(const double* inv, double alpha, int n_classes, int ld, int* hexp, int* range,
                            cudaStream_t s) {
  if (n_classes == 0) return;
  DG_REQUIRE(ld % 32 == 0 && n_classes <= 65535, "digit slices need a 32-aligned stride");
  equilibrate_kernel<<<dim3((ld + 127) / 128, n_classes), 128, 0, s>>>(inv, ld, hexp);
  DG_CUDA(cudaMemsetAsync(range, 0, sizeof(int), s));
  range_kernel<<<dim3(ld, n_classes), 256, 0, s>>>(inv, ld, alpha, hexp, range);
  DG_LAUNCHED(2);
}

void launch_f64_inverse_digits(int digits, const double* inv, double alpha, int n_classes, int ld, const int* hexp,
                               uint16_t* dst, int* row_exp, cudaStream_t s) {
  if (n_classes == 0) return;
  if (digits == 12) launch_inverse_digits<12>(inv, alpha, n_classes, ld, hexp, dst, row_exp, s);
  else if (digits == 13) launch_inverse_digits<13>(inv, alpha, n_classes, ld, hexp, dst, row_exp, s);
  else launch_inverse_digits<14>(inv, alpha, n_classes, ld, hexp, dst, row_exp, s);
  DG_LAUNCHED(1);
}

void launch_f64_column_digits(int digits, const double* X, int n_cols, int ld, const int* hexp, const int* class_of_col,
                              uint16_t* dst, int* col_exp, cudaStream_t s) {
  if (n_cols == 0) return;
  if (digits == 12) launch_column_digits<12>(X, n_cols, ld, hexp, class_of_col, dst, col_exp, s);
  else if (digits == 13) launch_column_digits<13>(X, n_cols, ld, hexp, class_of_col, dst, col_exp, s);
  else launch_column_digits<14>(X, n_cols, ld, hexp, class_of_col, dst, col_exp, s);
  DG_LAUNCHED(1);
}

void make_f64_maps(F64Maps& m, int digits, const uint16_t* inv, int n_classes, const uint16_t* X, int n_cols, int ld) {
  m.a = slice_map(inv, ld, ld, (uint64_t)n_classes * digits, BM, 1);
  for (int w = 0; w < 2; ++w) m.x[w] = slice_map(X, ld, n_cols, digits, 16 * (w + 1), digits);
}

void launch_f64_gemm(int digits, const F64Maps& maps, const int* inv_exp, const int* x_exp, double* Y, int ld,
                     const int4* d_tiles, int n_tiles, const int* d_kchunks, int* err, cudaStream_t s, int split) {
  if (n_tiles == 0) return;
  if (split == 0) split = f64_default_split(n_tiles, ld);
  DG_REQUIRE(split == 1 || split == 2 || split == 4 || split == 8, "GEMM split must be 1, 2, 4 or 8");
  auto run = digits == 12 ? launch_gemm<12> : (digits == 13 ? launch_gemm<13> : launch_gemm<14>);
  run(maps, inv_exp, x_exp, Y, ld, d_tiles, n_tiles, d_kchunks, err, s, split);
}

}  // namespace dg
