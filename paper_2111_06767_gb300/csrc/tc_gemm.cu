// Subdomain-inverse GEMM on the 5th-generation tensor cores (tcgen05, TF32 inputs, FP32 accumulate).
//
// du_S = A_S^-1 r_S for all subdomains of a class (Sec. III.E, explicit-inverse solver) is the one
// dense contraction of the method: Y[:, cols] = Inv_c (ld x ld, row-major) * X[:, cols] with every
// subdomain column of X contiguous. Both operands are K-major, so each CTA computes a 128 x nc output
// tile: TMA streams 128 x 32 tiles of Inv_c and nc x 32 tiles of X (128-byte swizzle) into a
// shared-memory ring, one elected thread issues tcgen05.mma (M = 128, N = nc, K = 8 per instruction)
// accumulating in tensor memory, and the four warps read the accumulator back with tcgen05.ld and store
// it column-contiguously. Only the K chunks that meet a slot of the subdomain present in the class are
// streamed (the slots of missing neighbours have zero coupling), and tiles whose rows lie only in such
// slots write zeros without a K loop. When the tiles alone cannot fill the GPU, the K range is split
// across a cluster of 2, 4 or 8 CTAs and the partial tiles are summed through distributed shared memory
// in a fixed order. Every wait is bounded: on timeout the CTA raises an error flag, drains and frees its
// tensor memory.
//
// What bounds it: the chunks' way through an SM's shared memory. A CTA alone moves one 24 KB chunk in 0.22
// us without the MMAs and in 0.31 us with them, whatever the ring's depth, and a launch without its K loop
// takes 1.7 us (one CTA per tile) to 3.6 us (clusters of 8). So the tile follows the class: nc is the number
// of its subdomains in equal parts, rounded up to 16, 32, 48, 64, 96 or 128, which keeps X's share of a
// chunk and the reads of the inverse down. Against 64-column tiles throughout, in a graph: 8^3 elements at
// N = 8 11.3 -> 10.9 us, 4^3 7.4 -> 6.3, 2^3 5.7 -> 4.4; 125 elements at N = 7 10.2 -> 7.6.
#include <mutex>
#include <set>

#include "internal.h"
#include "pdl.cuh"
#include "tcgen05.cuh"

namespace dg {

namespace {

constexpr int BM = 128, BK = 32;
constexpr int A_BYTES = BM * BK * 4;  // 16 KiB
constexpr int RING = 96 * 1024;       // two CTAs per SM
constexpr int MAX_STAGES = 5;         // of A_BYTES + nc * 128 bytes: 5 at nc = 16, 4 up to 64, 3 at 96 and 128
constexpr int MAX_CHUNKS = 256;
constexpr int TMEM_COLS = 128;
constexpr int SMEM_BYTES = RING + 1024 + 256;
constexpr int kWidths = 6;
__host__ __device__ constexpr int tile_width(int code) {
  return code < 4 ? 16 * (code + 1) : (code == 4 ? 96 : 128);
}
// instruction descriptor: F32 accumulate, TF32 A and B, both K-major, M = BM; N is added per tile
constexpr uint32_t IDESC = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(BM >> 4) << 24);
static_assert(BM * 128 * 4 <= RING, "split-K partial tile must fit in the idle ring");
static_assert(MAX_CHUNKS * BK >= DG_MAX_N * DG_MAX_N * (DG_MAX_N + 6 * (DG_MAX_N - 1)), "chunk list of the longest column");

struct TcMaps {
  CUtensorMap a, b[kWidths];
};

// SPLIT > 1: the K range of a tile is split across the SPLIT CTAs of a thread-block cluster; each
// keeps its partial 128 x nc tile in shared memory and, after a cluster barrier, every CTA sums a
// 1/SPLIT of the tile's columns over all partials through distributed shared memory in
// rank order, so the result does not depend on timing.
template <int SPLIT>
__global__ void __launch_bounds__(128, 2)
    tc_gemm_kernel(const __grid_constant__ TcMaps maps, float* __restrict__ Y, int ld, const int4* __restrict__ tiles,
                   const int* __restrict__ kchunks, int* __restrict__ err, float alpha) {
  extern __shared__ unsigned char smem_raw[];
  __shared__ int s_k[MAX_CHUNKS];  // this CTA's K chunks
  unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = (uint64_t*)(smem + RING);  // full[MAX_STAGES], empty[MAX_STAGES], acc
  uint32_t* tmem_slot = (uint32_t*)(bars + 2 * MAX_STAGES + 1);
  int* s_issued = (int*)(tmem_slot + 1);    // TMA chunks issued by the producer
  int* s_consumed = (int*)(tmem_slot + 2);  // chunks the MMA thread saw arrive

  const int split = SPLIT > 1 ? (int)cluster_rank() : 0;
  const int4 tile = tiles[blockIdx.x / SPLIT];
  const int wc = (tile.x >> 24) & 7, nc = tile_width(wc);
  const int cls = tile.x & 0xFFFF, row0 = tile.y, col0 = tile.z, ncol = min(tile.w, nc);
  const uint32_t b_bytes = (uint32_t)nc * BK * 4, stage_bytes = A_BYTES + b_bytes;
  const int stages = min(MAX_STAGES, RING / (int)stage_bytes);
  const bool zero = (tile.x >> 30) & 1;  // rows only in the slots of missing neighbours: zeros
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // the K chunks of this class that meet a present slot (the rest of the inverse's row is zero)
  const int* kl = kchunks + (size_t)cls * (ld / BK + 1);
  const int nk_all = zero ? 0 : kl[0];
  const int kc0 = split * nk_all / SPLIT, kc1 = (split + 1) * nk_all / SPLIT;
  const int nk = kc1 - kc0;
  for (int i = threadIdx.x; i < nk; i += 128) s_k[i] = kl[1 + kc0 + i] * BK;
  const uint32_t ring0 = smem_u32(smem), full0 = smem_u32(bars), empty0 = full0 + 8 * MAX_STAGES,
                 accb = empty0 + 8 * MAX_STAGES;

  if (threadIdx.x == 0) {
    *s_issued = 0;
    *s_consumed = 0;
    for (int s = 0; s < MAX_STAGES; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    mbar_init(accb, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  // set-up above overlaps the previous kernel, and so do the first tiles of the inverse, which nothing
  // writes; X (and Y) belong to the stream order from pdl_wait() on
  pdl_launch_dependents();
  if (warp == 0 && lane == 0) {
    for (int kc = 0; kc < nk && kc < stages; ++kc) {
      mbar_expect_tx(full0 + 8 * kc, stage_bytes);
      tma_load_3d(ring0 + kc * stage_bytes, &maps.a, full0 + 8 * kc, s_k[kc], row0, cls);
    }
  }
  pdl_wait();

  if (warp == 0 && lane == 0) {
    // producer: TMA loads into the ring (its first round holds the inverse's tiles already)
    const CUtensorMap* mapB = &maps.b[wc];
    for (int kc = 0, s = 0, round = 0; kc < nk; ++kc) {
      const uint32_t at = ring0 + s * stage_bytes, bar = full0 + 8 * s;
      if (round > 0) {
        if (!mbar_wait(empty0 + 8 * s, (round & 1) ^ 1, err)) break;
        mbar_expect_tx(bar, stage_bytes);
        tma_load_3d(at, &maps.a, bar, s_k[kc], row0, cls);
      }
      tma_load_2d(at + A_BYTES, mapB, bar, s_k[kc], col0);
      *s_issued = kc + 1;
      if (++s == stages) {
        s = 0;
        ++round;
      }
    }
  } else if (warp == 1 && lane == 0) {
    // MMA issuer: 4 instructions of K = 8 per 32-wide K chunk
    const uint32_t idesc = IDESC | ((uint32_t)(nc >> 3) << 17);
    for (int kc = 0, s = 0, round = 0; kc < nk; ++kc) {
      if (!mbar_wait(full0 + 8 * s, round & 1, err)) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t a0 = ring0 + s * stage_bytes, b0 = a0 + A_BYTES;
#pragma unroll
      for (int kk = 0; kk < BK / 8; ++kk)
        mma_tf32(tmem, smem_desc(a0 + 32 * kk), smem_desc(b0 + 32 * kk), idesc, (kc | kk) != 0);
      mma_commit(empty0 + 8 * s);  // frees the stage once these MMAs have read it
      *s_consumed = kc + 1;
      if (++s == stages) {
        s = 0;
        ++round;
      }
    }
    mma_commit(accb);
  }
  __syncwarp();

  // epilogue: warp w owns accumulator lanes (rows) 32 w .. 32 w + 31
  const bool ok = __all_sync(0xffffffffu, mbar_wait(accb, 0, err));
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const int r_local = warp * 32 + lane;
  const int row = row0 + r_local;
  const bool acc = nk > 0;  // the accumulator holds a product (else this CTA's part is zero)
  if (SPLIT == 1) {
    for (int c0 = 0; c0 < nc; c0 += 16) {
      if (!ok) break;
      uint32_t v[16];
      if (acc) tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + c0, v);
      if (row < ld) {
#pragma unroll
        for (int j = 0; j < 16; ++j)
          if (c0 + j < ncol) Y[(size_t)(col0 + c0 + j) * ld + row] = acc ? alpha * __uint_as_float(v[j]) : 0.0f;
      }
    }
  } else {
    // partial tile -> own shared memory (column-major, 128 rows per column; the ring is idle now)
    float* part = reinterpret_cast<float*>(smem);
    for (int c0 = 0; c0 < nc; c0 += 16) {
      uint32_t v[16];
      if (ok && acc) tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + c0, v);
#pragma unroll
      for (int j = 0; j < 16; ++j) part[(c0 + j) * BM + r_local] = ok && acc ? __uint_as_float(v[j]) : 0.0f;
    }
    cluster_sync();
    const int cpr = nc / SPLIT;  // columns reduced by this CTA
    uint32_t peer[SPLIT];
    const uint32_t mine = smem_u32(part + split * cpr * BM + r_local);
#pragma unroll
    for (int p = 0; p < SPLIT; ++p) peer[p] = map_peer(mine, (uint32_t)p);
    // remote loads in groups of up to 32 issued back to back (they are independent), then each column is
    // summed over the partials in rank order
    constexpr int JG = 32 / SPLIT;  // columns per group
    for (int j0 = 0; j0 < cpr; j0 += JG) {
      float v[JG][SPLIT];
#pragma unroll
      for (int j = 0; j < JG; ++j)
#pragma unroll
        for (int p = 0; p < SPLIT; ++p)
          v[j][p] = j0 + j < cpr ? ld_cluster(peer[p] + (uint32_t)((j0 + j) * BM * 4)) : 0.0f;
#pragma unroll
      for (int j = 0; j < JG; ++j) {
        const int c = split * cpr + j0 + j;
        float sum = 0.0f;
#pragma unroll
        for (int p = 0; p < SPLIT; ++p) sum += v[j][p];
        if (j0 + j < cpr && row < ld && c < ncol) Y[(size_t)(col0 + c) * ld + row] = alpha * sum;
      }
    }
    cluster_sync();  // no CTA leaves while a peer still reads its partial tile
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0 && !ok) {
    // a wait gave up: let the copies already issued land (bounded) before the CTA exits
    for (int kc = *s_consumed; kc < *s_issued; ++kc) mbar_wait(full0 + 8 * (kc % stages), (kc / stages) & 1, err);
  }
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
}

CUtensorMap make_map(const float* base, int rank, const cuuint64_t* dims, const cuuint64_t* strides,
                     const cuuint32_t* box) {
  CUtensorMap m;
  auto fn = tensor_map_encoder();
  if (!fn) fail(DG_ERR_CUDA, "cuTensorMapEncodeTiled is unavailable");
  const cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = fn(&m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, rank, (void*)base, dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) fail(DG_ERR_CUDA, "cuTensorMapEncodeTiled failed: " + std::to_string((int)r));
  return m;
}

}  // namespace

PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    else
      (void)cudaGetLastError();
  });
  return fn;
}

bool tc_gemm_available() { return tensor_map_encoder() != nullptr; }

std::vector<int> tc_gemm_splits(int ld) {
  std::vector<int> out;
  for (int split = 1; split <= 8; split *= 2)
    if (split == 1 || (ld / BK) / split >= 4) out.push_back(split);
  return out;
}

int tc_tile_width_code(int columns) {
  for (int c = 0; c < kWidths; ++c)
    if (tile_width(c) >= columns) return c;
  return kWidths - 1;
}
int tc_tile_width(int code) { return tile_width(code); }

// Split K over a cluster of `split` CTAs so that the launch fills one wave of the co-resident CTAs, keeping >= 4 K
// chunks each.
int tc_default_split(int n_tiles, int ld) {
  int split = 1;
  while (split < 8 && n_tiles * split * 2 <= 2 * 152 && ld / BK / (split * 2) >= 4) split *= 2;
  return split;
}

void launch_class_gemm_tc(const float* inv, int n_classes, const float* X, float* Y, int ld, int n_cols,
                          const int4* d_tiles, int n_tiles, int width_mask, const int* d_kchunks, int* err,
                          float alpha, cudaStream_t s, int split) {
  if (n_tiles == 0) return;
  DG_REQUIRE(ld % BK == 0 && ld / BK <= MAX_CHUNKS, "tensor-core GEMM needs a 32-aligned subdomain stride");
  const cuuint64_t dA[3] = {(cuuint64_t)ld, (cuuint64_t)ld, (cuuint64_t)n_classes};
  const cuuint64_t sAr[2] = {(cuuint64_t)ld * 4, (cuuint64_t)ld * ld * 4};
  const cuuint32_t bA[3] = {BK, BM, 1};
  const cuuint64_t dB[2] = {(cuuint64_t)ld, (cuuint64_t)n_cols};
  const cuuint64_t sBr[1] = {(cuuint64_t)ld * 4};
  TcMaps maps;
  maps.a = make_map(inv, 3, dA, sAr, bA);
  for (int w = 0; w < kWidths; ++w) {
    if (!(width_mask >> w & 1)) continue;  // a width no tile of this level has
    const cuuint32_t bB[2] = {BK, (cuuint32_t)tile_width(w)};
    maps.b[w] = make_map(X, 2, dB, sBr, bB);
  }
  {
    // kernel attributes are per device
    static std::mutex mu;
    static std::set<int> done;
    int dev = 0;
    DG_CUDA(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lk(mu);
    if (!done.count(dev)) {
      for (auto k : {tc_gemm_kernel<1>, tc_gemm_kernel<2>, tc_gemm_kernel<4>, tc_gemm_kernel<8>})
        DG_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES));
      done.insert(dev);
    }
  }
  const int nk = ld / BK;
  if (split == 0) split = tc_default_split(n_tiles, ld);
  DG_REQUIRE(split == 1 || split == 2 || split == 4 || split == 8, "GEMM split must be 1, 2, 4 or 8");
  DG_REQUIRE(split == 1 || nk / split >= 1, "GEMM split larger than the K chunks");
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_tiles * split);
  cfg.blockDim = dim3(128);
  cfg.dynamicSmemBytes = SMEM_BYTES;
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
  auto k = split == 1 ? tc_gemm_kernel<1>
                      : (split == 2 ? tc_gemm_kernel<2> : (split == 4 ? tc_gemm_kernel<4> : tc_gemm_kernel<8>));
  DG_CUDA(cudaLaunchKernelEx(&cfg, k, maps, Y, ld, d_tiles, d_kchunks, err, alpha));
  DG_LAUNCHED(1);
}

}  // namespace dg
