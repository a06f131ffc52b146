// kvshot_slab_gemm.cuh -- a table-driven tcgen05 GEMM that writes fp32
// "slabs": for each entry z of a small table, a weight matrix's 256-row block
// times a block of up to 256 token rows,
//   slab[z][t][f] = sum_k W_z[f][wx0 + k] * A_z[t][k]                 (one operand)
//   slab[z][t][f] = sum_k W_z[f][wx0 + k] * (A1_z[t][k] - A0_z[t][k]) (two operands)
// over k in [0, 64 nk).  A difference of bf16 activations is never formed or
// rounded: the two-operand form accumulates both products in fp32 and subtracts
// them when it stores them.  With at most 128 tokens per block, A0's and A1's
// token rows are stacked in one B tile (one MMA of N = 2 x tokens per 16-wide k
// step); with more, there are two MMAs into two accumulators.  Callers add the
// slabs they need and apply their epilogue in a kernel of their own.
//
// A CTA pair (cluster of two, cta_group::2) computes a 256-feature block: each
// CTA stages its own 128 weight rows x 64 k and half of the token rows, and the
// even CTA issues the MMAs (M = 256) for both.  What bounds the kernel is the
// weights' bytes at few tokens and, from some hundred tokens on, the MMAs and shared memory:
// per 64-wide k step and CTA, the tiles written by TMA and the operands read by
// the MMAs.  Sharing the token rows between two CTAs halves both for B: at 192
// tokens and two operands 96 KB per step instead of 144 KB, and ring slots of
// 40 KB instead of 64 KB, so that 5 weight tiles are in flight instead of 3.
// Fusion calls with d = 4096, one CTA per 128 features -> pairs: 1 token 30.4 ->
// 24.9 us, 192 tokens 46.5 -> 38.7 us, 256 tokens 65.5 -> 48.8 us, 1024 tokens 188 ->
// 153 us.  From 129 tokens on, the two-operand CTAs' MMAs are the longest chain.
//
// Shapes: A = 2 x 128 weight rows x 64 k (K-major, 128-byte swizzle, TMA box
// {64, 128}); B = N token rows x 64 k, N = tokens rounded up to 32, in boxes
// {64, N / 2}; fp32 accumulators in TMEM.  Grid (token blocks x 2 CTAs, feature
// blocks of 256, table entries), the token block fastest so that a weight tile's
// token blocks run together and the weights leave HBM once.  128 threads: warp 0
// lane 0 issues the TMA loads, warp 1 owns TMEM and, in the even CTA, its lane 0
// issues the MMAs; all four warps move the accumulators to the slab (thread =
// TMEM lane = output feature; a warp stores 32 consecutive features of one token).
#pragma once

#include <type_traits>

#include "kvshot_attn_common.cuh"
#include "kvshot_tcgen05.cuh"

namespace kvshot {
namespace sg {
namespace {

using namespace dev;
using namespace tc;

constexpr int kFeat = 128;                  // output features per CTA, half the pair's (MMA M = 256)
constexpr int kMaxTok = 256;                // tokens per pair (MMA N)
constexpr int kKT = 64;                     // K per stage: one 128-byte swizzled row
constexpr int kMaxStages = 8;
constexpr int kThreads = 128;
constexpr int kABytes = kFeat * kKT * 2;    // 16 KB
constexpr int kRingBytes = 200 * 1024;
constexpr uint32_t kTmemCols = 512;         // two accumulators of N <= 256 columns
constexpr int kMaxN = 256;                  // the MMA's largest N
constexpr int kMaxEntries = 4;
// Limit on a wait of the pipeline.  (tests/test_gpu_fusion.py builds copies in which both CTAs of a pair, or one, give up
// at once.)
#ifndef KVSHOT_FUSION_WAIT_NS
#define KVSHOT_FUSION_WAIT_NS kWaitLimitNs
#endif

struct Entry {
  int8_t w;    // weight map index
  int8_t a0;   // activation map index
  int8_t a1;   // second activation map index, or -1 (one operand)
  int wx0;     // first weight column (element)
};

struct Params {
  Entry e[kMaxEntries];
  float* slab;   // [entries][T][d_out]
  int32_t* err;
  int T;         // token rows
  int d_out;     // output features (multiple of 128)
  int nk;        // k-tiles of 64
  int box_tok;   // tokens per block: min(T, 256)
};

// MMA N for a token block: a multiple of 32 for a pair; each CTA stages N / 2 token rows per operand.
__host__ __device__ inline int mma_n(int box_tok) { return (box_tok + 31) / 32 * 32; }

struct Maps {
  CUtensorMap w[2];  // weights [d_out, K], boxes {64, 128}
  CUtensorMap a[2];  // activations [T, K], boxes {64, mma_n / 2}
};

inline size_t smem_bytes() { return 1024 + kRingBytes + 8 * (2 * kMaxStages + 1) + 16; }

__device__ __forceinline__ void store_in_pair(uint32_t addr, int rank, int v) {
  asm volatile("{\n\t.reg .u32 ra;\n\tmapa.shared::cluster.u32 ra, %0, %1;\n\tst.shared::cluster.s32 [ra], %2;\n\t}" ::"r"(
                   addr),
               "r"(rank), "r"(v)
               : "memory");
}

__device__ __forceinline__ void pair_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The address, in the cluster's shared memory, of `addr` in the pair's even CTA.
__device__ __forceinline__ uint32_t in_even_cta(uint32_t addr) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(addr));
  return r;
}
// 2-D tiled TMA load into this CTA whose completion is counted on a barrier of either CTA of the pair.
__device__ __forceinline__ void tma_load_pair(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2"
      " [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_load_pair_hint(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar,
                                                   uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2.L2::cache_hint"
      " [%0], [%1, {%2, %3}], [%4], %5;" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar), "l"(policy)
      : "memory");
}

__global__ void __launch_bounds__(kThreads, 1) slab_gemm(const __grid_constant__ Params p, const __grid_constant__ Maps maps) {
  extern __shared__ uint8_t smem_raw[];
  const int rank = blockIdx.x & 1, tt = blockIdx.x >> 1, z = blockIdx.z;
  const int f0 = blockIdx.y * 2 * kFeat + rank * kFeat;  // this CTA's first feature (may lie past d_out)
  const Entry en = p.e[z];
  const bool both = en.a1 >= 0;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  // Ring slot s: the weight tile at base + s * slot, the token tile(s) of N / 2 rows right after it.  Stacked
  // [A0; A1] rows: the even CTA holds all of A0's, the odd one all of A1's.
  const int N = mma_n(p.box_tok), btile = N / 2 * kKT * 2;
  const bool stacked = both && 2 * N <= kMaxN;  // N_mma = 2 N
  const int slot = kABytes + (both ? 2 : 1) * btile;
  const int nst = min(kMaxStages, kRingBytes / slot);
  uint64_t* full = reinterpret_cast<uint64_t*>(base + kRingBytes);  // even CTA: both CTAs' loads of the slot landed
  uint64_t* empty = full + kMaxStages;                              // the slot's MMAs completed (in both CTAs)
  uint64_t* done = empty + kMaxStages;
  uint32_t* tmem_base = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* gave_up = reinterpret_cast<volatile int*>(tmem_base + 1);
  volatile int* peer = gave_up + 1;  // written by the pair's other CTA: k-tiles issued, or -1 - that where it gave up
  if (threadIdx.x == 0) {
    for (int s = 0; s < kMaxStages; ++s) {
      mbar_init(smem_addr(&full[s]), 1);
      mbar_init(smem_addr(&empty[s]), 1);
    }
    mbar_init(smem_addr(done), 1);
    *gave_up = 0;
    fence_mbar_init();
    prefetch_tensormap(&maps.w[en.w]);
    prefetch_tensormap(&maps.a[en.a0]);
    if (both) prefetch_tensormap(&maps.a[en.a1]);
  }
  if (warp == 1) {
    tmem_alloc_pair(smem_addr(tmem_base), kTmemCols);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  __syncthreads();
  pair_sync();  // both CTAs' barriers are initialised
  tc_fence_after();
  const uint32_t tmem = *tmem_base;
  // Launched behind the preceding kernel: nothing before this touches its results.  The kernel that adds the slabs
  // may be placed from here on.
  wait_for_prerequisite_grid();
  if (threadIdx.x == 0) allow_dependent_launch();
  const int nk = p.nk;
  bool ok = true;
  int issued = 0;
  const uint64_t stream_once = l2_policy_evict_first();  // weights: read once
  const uint32_t tx = 2u * static_cast<uint32_t>(slot);  // both CTAs' bytes (rows out of range are filled)
  const int ty = tt * p.box_tok, half = N / 2;
  const uint32_t even0 = in_even_cta(smem_addr(full)), ring = smem_addr(base);
  auto load = [&](int kt, int s) {
    if (rank == 0) mbar_arrive_expect_tx(smem_addr(&full[s]), tx);
    const uint32_t fb = even0 + 8 * s, dst = ring + s * slot, bdst = dst + kABytes;
    tma_load_pair_hint(dst, &maps.w[en.w], en.wx0 + kt * kKT, f0, fb, stream_once);
    if (stacked) {
      const CUtensorMap* a = &maps.a[rank ? en.a1 : en.a0];
      tma_load_pair(bdst, a, kt * kKT, ty, fb);
      tma_load_pair(bdst + btile, a, kt * kKT, ty + half, fb);
    } else {
      tma_load_pair(bdst, &maps.a[en.a0], kt * kKT, ty + rank * half, fb);
      if (both) tma_load_pair(bdst + btile, &maps.a[en.a1], kt * kKT, ty + rank * half, fb);
    }
  };
  if (warp == 0 && lane == 0) {
    const uint32_t empty0 = smem_addr(empty);
    int s = 0;
    uint32_t phase = 1;  // of the empty barriers: their first use needs no wait
    for (int kt = 0; kt < nk; ++kt) {
      if (kt >= nst) ok = mbar_wait(empty0 + 8 * s, phase, p.err, KVSHOT_FUSION_WAIT_NS);
      if (!ok) break;
      load(kt, s);
      issued = kt + 1;
      if (++s == nst) {
        s = 0;
        phase ^= 1u;
      }
    }
    if (!ok) *gave_up = 1;
  } else if (warp == 1 && lane == 0 && rank == 0) {
    const uint32_t idesc = idesc_bf16(2 * kFeat, stacked ? 2 * N : N, false);
    // The issuing thread is on the critical path: a loop for each of one and two MMAs per k step, descriptors,
    // slots and phases by addition.  (d = 4096, 1 / 128 / 192 tokens: 24.9 / 31.3 / 38.7 us per call; with descriptors
    // built and slots divided out at each step 27.6 / 32.1 / 41.8; with a branch between a step's MMAs 35.3 / 39.1 /
    // 41.5.)
    const uint64_t a_desc = smem_desc_sw128(smem_addr(base), 16, 1024);
    const uint32_t full0 = smem_addr(full), empty0 = smem_addr(empty);
    auto issue = [&](auto two) {
      int s = 0;
      uint32_t phase = 0, acc = 0;
      for (int kt = 0; kt < nk; ++kt) {
        ok = mbar_wait(full0 + 8 * s, phase, p.err, KVSHOT_FUSION_WAIT_NS);
        if (!ok) break;
        tc_fence_after();
        // Descriptors hold addresses in units of 16 bytes, and the whole ring stays below their 256 KB.
        const uint64_t a0 = a_desc + static_cast<uint32_t>(s * slot) / 16, b0 = a0 + kABytes / 16;
#pragma unroll
        for (int ks = 0; ks < kKT / 16; ++ks) {
          tc_mma_pair(tmem, a0 + 2 * ks, b0 + 2 * ks, idesc, acc | static_cast<uint32_t>(ks));
          if constexpr (decltype(two)::value)  // W A1 beside W A0
            tc_mma_pair(tmem + N, a0 + 2 * ks, b0 + 2 * ks + btile / 16, idesc, acc | static_cast<uint32_t>(ks));
        }
        acc = 1;
        tc_commit_pair(empty0 + 8 * s);
        if (++s == nst) {
          s = 0;
          phase ^= 1u;
        }
      }
    };
    if (both && !stacked) issue(std::true_type{});
    else issue(std::false_type{});
    if (!ok) *gave_up = 1;
    tc_commit_pair(smem_addr(done));  // every MMA this thread issued has completed
  }
  __syncwarp();
  ok = mbar_wait(smem_addr(done), 0, p.err, KVSHOT_FUSION_WAIT_NS);
  if (!ok) *gave_up = 1;
  tc_fence_after();
  const int f = f0 + warp * 32 + lane;
  const uint32_t trow = tmem + (static_cast<uint32_t>(warp * 32) << 16);
  float* slab = p.slab + static_cast<size_t>(z) * p.T * p.d_out;
  if (f0 < p.d_out) {
#pragma unroll 1
    for (int c = 0; c < N / 32; ++c) {
      const int t0 = tt * p.box_tok + c * 32;
      const int nt = min(32, min(p.T, (tt + 1) * p.box_tok) - t0);
      if (nt <= 0) break;
      uint32_t x[32], y[32];
      tmem_ld32(trow + c * 32, x);
      if (both) tmem_ld32(trow + N + c * 32, y);
      tmem_wait_ld();
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        const float v = both ? __uint_as_float(y[j]) - __uint_as_float(x[j]) : __uint_as_float(x[j]);
        if (j < nt) slab[static_cast<size_t>(t0 + j) * p.d_out + f] = ok ? v : 0.f;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  const bool failed = *gave_up;
  if (threadIdx.x == 0) store_in_pair(smem_addr(tmem_base + 2), rank ^ 1, failed ? -1 - issued : issued);
  pair_sync();  // the pair's MMAs and barriers are used across the two CTAs until here
  if (failed || *peer < 0) {
    // The copies in flight land, and the MMAs end, before the CTAs exit.  A k-tile that one CTA alone has loaded would
    // never complete its barrier, so the other loads it too (no MMA reads the ring any more).
    if (threadIdx.x == 0) {
      const int other = *peer, last = max(issued, other < 0 ? -1 - other : other);
      mbar_wait(smem_addr(done), 0, p.err);
      for (int kt = issued; kt < last; ++kt) load(kt, kt % nst);
      for (int kt = max(0, last - nst); rank == 0 && kt < last; ++kt)
        mbar_wait(smem_addr(&full[kt % nst]), (kt / nst) & 1, p.err);
    }
    __syncthreads();
    pair_sync();
  }
  if (warp == 1) tmem_dealloc_pair(tmem, kTmemCols);
}

// Launches slab_gemm over `entries` table entries.
inline cudaError_t launch(const Params& p, const Maps& maps, int entries, cudaStream_t stream) {
  const size_t smem = smem_bytes();
  cudaError_t e = cudaFuncSetAttribute(slab_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 2;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * ((p.T + p.box_tok - 1) / p.box_tok), (p.d_out + 2 * kFeat - 1) / (2 * kFeat), entries);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, slab_gemm, p, maps);
}

}  // namespace
}  // namespace sg
}  // namespace kvshot
