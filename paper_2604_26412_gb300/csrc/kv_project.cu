// kv_project.cu -- the KV-only drafter's linear projection of multi-layer
// target KV (Sec. 3.2, injection strategy "linear projection", with the
// "Proj + RoPE fix" variant): for every newly verified token t the K (and V)
// vectors of the L_s sampled target layers, each hkv x 128 wide, are
// concatenated and mapped back to one layer's width by learned matrices
// W_K^proj, W_V^proj in R^{d_kv x L_s d_kv} (d_kv = hkv x 128):
//
//   K'(t) = W_K^proj [K^(1)(t); ...; K^(L_s)(t)],   V'(t) = W_V^proj [V^(1)(t); ...; V^(L_s)(t)]
//
// and, with KVSHOT_PROJECT_ROPE, RoPE is re-applied to K'(t) at the token's
// position (the projection mixes keys already rotated by RoPE).  The results
// go to the token's slot of the single reused cache the draft attention reads
// (App. B: verified prefix positions take the target's -- here projected --
// K/V), so the cache is built incrementally, a few tokens per decoding step.
//
// One kernel.  A cluster of up to 8 CTAs owns the 128 output features of one KV head (K or V) for a block of up
// to 128 tokens and splits the L_s d_kv inputs among its CTAs: each runs its part of the GEMM on the tcgen05
// tensor cores (weights as A, tokens as B, fp32 accumulator in tensor memory), leaves its partial sums in its
// shared memory, and after a cluster barrier adds the cluster's partials (in rank order) for its share of the
// tokens, rotates the keys, rounds to bf16 and stores both halves of the head into the cache through the page table.
// What bounds it: the weights' bytes (one decoding step's few tokens, 2 L_s d_kv^2 bf16 values; an SM ingests
// ~44 KB/us) and the fixed latencies of launch, load, MMA and exchange, which slot and angle look-ups overlap.
// Measured, 4 layers of 8 heads, back to back in a graph: 1 token 6.2 us, 32 tokens 7.6, 512 tokens 16.8 us; as a
// GEMM into fp32 slabs per layer and a second kernel to add them 12.5, 12.9 and 21.8 us.
// The angle pos * rope_base^(-2j/128) is formed and reduced modulo 2 pi in fixed point: the position times the frequency
// in turns, a 64-bit fraction from the host, keeps the fraction of a turn in its low 64 bits, of which 32 are turned into
// radians (2^-30; sine, cosine and the rotation are fp32, relative error ~1e-7, far below the bf16 rounding that follows).
// An SM executes two fp64 lanes per clock: with the reduction in fp64 two clusters of 128 tokens on one SM took 26 us for
// it alone (2048 tokens of 1 layer of 8 heads 38.4 us per call, now 32.5).
#include <algorithm>
#include <cmath>

#include "kvshot_attn_common.cuh"
#include "kvshot_tcgen05.cuh"

namespace kvshot {
namespace {

using namespace dev;
using namespace tc;

constexpr int kMaxLayers = 8;
constexpr int kThreads = 256;
constexpr int kFeat = kHeadDim;              // output features per cluster (MMA M): one KV head
constexpr int kTok = 128;                    // most tokens per cluster (MMA N)
constexpr int kKT = 64;                      // inputs per k-tile: one 128-byte swizzled row
constexpr int kABytes = kFeat * kKT * 2;     // a k-tile of weights
// Two CTAs fit an SM: with one (a ring of 192 KB) only 15 clusters of 8 are resident at a time, and the 16 of an
// 8-head cache took a second wave (12.9 against 8.1 us per call, 32 tokens of 4 layers).
constexpr int kRingBytes = 102 * 1024;
constexpr int kMaxStages = 5;
constexpr int kMaxSplit = 8;                 // CTAs per cluster (the portable limit)
constexpr int kProjectCtas = 288;            // CTAs of 8-CTA clusters resident at a time
// Limit on a wait of the pipeline.  (tests/test_gpu_project.py builds a copy whose waits give up at once.)
#ifndef KVSHOT_PROJECT_WAIT_NS
#define KVSHOT_PROJECT_WAIT_NS kWaitLimitNs
#endif
constexpr uint64_t kPipeLimitNs = KVSHOT_PROJECT_WAIT_NS;

struct ProjectParams {
  const int32_t* token_cache;
  const int32_t* positions;
  const int32_t* page_table;  // null: contiguous cache
  __nv_bfloat16* k_out;
  __nv_bfloat16* v_out;
  int32_t* err;
  int T, hkv, C;
  int nk;       // k-tiles: L d_kv / 64
  int box_tok;  // tokens per cluster: min(T, kTok)
  int split;    // CTAs per cluster
  int stages;   // ring slots of a k-tile of weights and one of tokens
  int paged, page_size, max_pages, num_pages, l_cap;
  int rope;
  uint64_t turns[kHeadDim / 2];  // rope_base^(-2j/128) / 2 pi modulo 1, in units of 2^-64
};

// Maps: weights [d_kv, L d_kv] of K and V, boxes {64, 128}; tokens [T, L d_kv], boxes {64, box_tok}.
struct ProjectMaps {
  CUtensorMap w[2], a[2];
};

__host__ __device__ inline int mma_n(int box_tok) { return (box_tok + 15) / 16 * 16; }
__host__ __device__ inline int slot_bytes(int box_tok) { return kABytes + mma_n(box_tok) * kKT * 2; }

// Shared memory: the ring, later the partial sums [tokens][128] fp32; then the barriers.
__host__ __device__ inline size_t ring_bytes(int stages, int box_tok) {
  const size_t ring = static_cast<size_t>(stages) * slot_bytes(box_tok);
  const size_t sums = static_cast<size_t>(mma_n(box_tok) + 31) / 32 * 32 * kFeat * 4;
  return ring > sums ? ring : sums;
}
inline size_t smem_bytes(int stages, int box_tok) {
  return 1024 + (ring_bytes(stages, box_tok) + 1023) / 1024 * 1024 + 8 * (2 * kMaxStages + 1) + 16 + 12 * kTok;
}

__device__ __forceinline__ void tma_load(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::
          "r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Two floats from the shared memory of CTA `rank` of the cluster, at this CTA's address `addr`.
__device__ __forceinline__ float2 cluster_load(uint32_t addr, int rank) {
  float2 v;
  asm volatile(
      "{\n\t.reg .u32 ra;\n\tmapa.shared::cluster.u32 ra, %2, %3;\n\t"
      "ld.shared::cluster.v2.f32 {%0, %1}, [ra];\n\t}"
      : "=f"(v.x), "=f"(v.y)
      : "r"(addr), "r"(rank)
      : "memory");
  return v;
}

__device__ __forceinline__ int cluster_load_int(uint32_t addr, int rank) {
  int v;
  asm volatile("{\n\t.reg .u32 ra;\n\tmapa.shared::cluster.u32 ra, %1, %2;\n\tld.shared::cluster.s32 %0, [ra];\n\t}"
               : "=r"(v)
               : "r"(addr), "r"(rank)
               : "memory");
  return v;
}

// The cache row of a token's head h, or -1 if its cache, position or page id is out of range.
__device__ __forceinline__ int64_t find_row(const ProjectParams& p, int tok, int h) {
  const int c = p.token_cache[tok], pos = p.positions[tok];
  const int cap = p.paged ? p.max_pages * p.page_size : p.l_cap;
  if (c < 0 || c >= p.C || pos < 0 || pos >= cap) return -1;
  if (!p.paged) return (static_cast<int64_t>(c) * p.hkv + h) * p.l_cap + pos;
  const int pid = p.page_table[static_cast<size_t>(c) * p.max_pages + pos / p.page_size];
  if (pid < 0 || pid >= p.num_pages) return -1;
  return (static_cast<int64_t>(pid) * p.hkv + h) * p.page_size + pos % p.page_size;
}

// The angles of the pairs (j, j + 64) and (j + 1, j + 65) at a position.
struct Angles {
  float2 cs, sn;
};
__device__ __forceinline__ Angles angles_at(const ProjectParams& p, int pos, int j) {
  Angles s;
  float r[2];
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const uint64_t turn = static_cast<uint64_t>(static_cast<uint32_t>(pos)) * p.turns[j + e];
    const int32_t x = static_cast<int32_t>((turn + 0x80000000ull) >> 32);  // 2^-32 turns, in [-1/2, 1/2)
    // x * 2 pi / 2^32 rounded about once: x in two exact halves, the constant in two floats
    const float hi = static_cast<float>(x & ~0xffff), lo = static_cast<float>(x & 0xffff);
    constexpr float c = 1.46291807926715968e-9f, c2 = static_cast<float>(1.46291807926715968e-9 - c);
    r[e] = fmaf(hi, c, fmaf(lo, c, hi * c2));
  }
  sincosf(r[0], &s.sn.x, &s.cs.x);
  sincosf(r[1], &s.sn.y, &s.cs.y);
  return s;
}

// Grid (token block x cluster rank, KV head, (0: K, 1: V)).
__global__ void __launch_bounds__(kThreads, 1)
    kv_project_kernel(const __grid_constant__ ProjectParams p, const __grid_constant__ ProjectMaps maps) {
  extern __shared__ uint8_t smem_raw[];
  const int split = p.split, tb = blockIdx.x / split, rank = blockIdx.x - tb * split, h = blockIdx.y, kv = blockIdx.z;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int N = mma_n(p.box_tok), slot = slot_bytes(p.box_tok);
  uint64_t* full = reinterpret_cast<uint64_t*>(base + (ring_bytes(p.stages, p.box_tok) + 1023) / 1024 * 1024);
  uint64_t* empty = full + kMaxStages;
  uint64_t* done = empty + kMaxStages;
  uint32_t* tmem_base = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* gave_up = reinterpret_cast<volatile int*>(tmem_base + 1);  // a wait timed out
  int64_t* rows = reinterpret_cast<int64_t*>(tmem_base + 2);               // [kTok] cache row of each token of the share
  int* pos = reinterpret_cast<int*>(rows + kTok);                          // [kTok] its position
  const int k0 = p.nk * rank / split, n = p.nk * (rank + 1) / split - k0;  // this CTA's k-tiles
  const uint32_t cols = N <= 32 ? 32u : N <= 64 ? 64u : 128u;
  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(smem_addr(&full[s]), 1);
      mbar_init(smem_addr(&empty[s]), 1);
    }
    mbar_init(smem_addr(done), 1);
    *gave_up = 0;
    fence_mbar_init();
    prefetch_tensormap(&maps.w[kv]);
    prefetch_tensormap(&maps.a[kv]);
  }
  if (warp == 1) {
    tmem_alloc(smem_addr(tmem_base), cols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_base;
  wait_for_prerequisite_grid();  // launched behind the preceding kernel: nothing before this touches its results
  if (threadIdx.x == 0) allow_dependent_launch();
  bool ok = true;
  int issued = 0;
  if (warp == 0 && lane == 0) {
    for (int kt = 0; kt < n; ++kt) {
      const int s = kt % p.stages;
      if (kt >= p.stages) ok = mbar_wait(smem_addr(&empty[s]), (kt / p.stages - 1) & 1, p.err, kPipeLimitNs);
      if (!ok) break;
      const uint32_t bar = smem_addr(&full[s]), dst = smem_addr(base + s * slot);
      mbar_arrive_expect_tx(bar, kABytes + p.box_tok * kKT * 2);
      tma_load(dst, &maps.w[kv], (k0 + kt) * kKT, h * kFeat, bar);
      tma_load(dst + kABytes, &maps.a[kv], (k0 + kt) * kKT, tb * p.box_tok, bar);
      issued = kt + 1;
    }
    if (!ok) *gave_up = 1;
  }
  __syncwarp();
  // This CTA's share of the tokens, a warp per token: lane l has pairs (j, j + 64), j = 2 l and 2 l + 1.  While the loads
  // are in flight, a thread per token looks up where it goes, and each warp forms its first token's angles.
  const int tokens = min(p.box_tok, p.T - tb * p.box_tok);
  const int s0 = tokens * rank / split, t0 = s0 + warp, t1 = tokens * (rank + 1) / split, j = 2 * lane;
  const bool rope = p.rope && kv == 0;
  if (threadIdx.x >= kThreads - kTok) {
    const int i = threadIdx.x - (kThreads - kTok);
    if (s0 + i < t1) {
      const int tok = tb * p.box_tok + s0 + i;
      rows[i] = find_row(p, tok, h);
      pos[i] = p.positions[tok];
    }
  }
  Angles ang{};
  if (rope && t0 < t1) ang = angles_at(p, p.positions[tb * p.box_tok + t0], j);
  if (warp == 1 && lane == 0) {
    const uint32_t idesc = idesc_bf16(kFeat, N, false);
    for (int kt = 0; kt < n; ++kt) {
      const int s = kt % p.stages;
      ok = mbar_wait(smem_addr(&full[s]), (kt / p.stages) & 1, p.err, kPipeLimitNs);
      if (!ok) break;
      tc_fence_after();
      const uint32_t a0 = smem_addr(base + s * slot), b0 = a0 + kABytes;
#pragma unroll
      for (int ks = 0; ks < kKT / 16; ++ks)
        tc_mma(tmem, smem_desc_sw128(a0 + ks * 32, 16, 1024), smem_desc_sw128(b0 + ks * 32, 16, 1024), idesc,
               (kt | ks) ? 1u : 0u);
      if (kt + p.stages < n) tc_commit(smem_addr(&empty[s]));
    }
    if (!ok) *gave_up = 1;
    tc_commit(smem_addr(done));  // every MMA this thread issued has completed
  }
  __syncwarp();
  if (!mbar_wait(smem_addr(done), 0, p.err, kPipeLimitNs)) *gave_up = 1;
  tc_fence_after();
  // A producer that gives up makes the MMA thread give up, which says so before its commit: after `done` every warp knows
  // whether all loads were consumed, and leaves the ring alone if not.
  const bool failed = *gave_up;
  if (failed && threadIdx.x == 0) {  // let the copies and MMAs in flight end before the CTA does
    for (int kt = max(0, issued - p.stages); kt < issued; ++kt)
      mbar_wait(smem_addr(&full[kt % p.stages]), (kt / p.stages) & 1, p.err);
    mbar_wait(smem_addr(done), 0, p.err);
  }
  // Partial sums to shared memory, [token][feature], over the ring (every load has been consumed).
  float* sums = reinterpret_cast<float*>(base);
  const int quarter = warp & 3;  // of the TMEM lanes (features); the two warpgroups take alternate chunks of tokens
  const uint32_t trow = tmem + (static_cast<uint32_t>(quarter * 32) << 16);
#pragma unroll 1
  for (int c = warp >> 2; !failed && c * 32 < tokens; c += kThreads / 128) {
    uint32_t x[32];
    tmem_ld32(trow + c * 32, x);
    tmem_wait_ld();
#pragma unroll
    for (int j = 0; j < 32; ++j) sums[(c * 32 + j) * kFeat + quarter * 32 + lane] = __uint_as_float(x[j]);
  }
  tc_fence_before();
  cluster_sync();
  if (warp == 1) tmem_dealloc(tmem, cols);
  // A rank that gave up leaves the cluster's sums incomplete: nothing is stored (the error is recorded already).
  const int rank_failed = lane < split ? cluster_load_int(smem_addr(tmem_base + 1), lane) : 0;
  for (int t = t0; t < t1; t += kThreads / 32) {
    const int64_t row = rows[t - s0];
    const uint32_t at = smem_addr(sums + t * kFeat + j);
    float2 a[kMaxSplit], b[kMaxSplit];
#pragma unroll
    for (int r = 0; r < kMaxSplit; ++r) {  // every load goes out before the first sum
      a[r] = r < split ? cluster_load(at, r) : make_float2(0.f, 0.f);
      b[r] = r < split ? cluster_load(at + 64 * 4, r) : make_float2(0.f, 0.f);
    }
    if (rope && t > t0) ang = angles_at(p, pos[t - s0], j);
    float2 lo = a[0], hi = b[0];
#pragma unroll
    for (int r = 1; r < kMaxSplit; ++r) {
      lo.x += a[r].x;
      lo.y += a[r].y;
      hi.x += b[r].x;
      hi.y += b[r].y;
    }
    if (__any_sync(0xffffffffu, rank_failed)) break;
    if (row < 0) {
      if (lane == 0) set_error(p.err, KVSHOT_ERR_DEVICE_BOUNDS);
      continue;
    }
    if (rope) {
      const float2 x = lo, y = hi;
      lo = make_float2(x.x * ang.cs.x - y.x * ang.sn.x, x.y * ang.cs.y - y.y * ang.sn.y);
      hi = make_float2(y.x * ang.cs.x + x.x * ang.sn.x, y.y * ang.cs.y + x.y * ang.sn.y);
    }
    __nv_bfloat16* out = (kv ? p.v_out : p.k_out) + row * kHeadDim + j;
    *reinterpret_cast<uint32_t*>(out) = pack_bf16x2(lo.x, lo.y);
    *reinterpret_cast<uint32_t*>(out + 64) = pack_bf16x2(hi.x, hi.y);
  }
  cluster_sync();  // the partial sums are read by the other CTAs until here
}

bool aligned(const void* ptr, size_t a) { return (reinterpret_cast<uintptr_t>(ptr) % a) == 0; }

size_t slab_bytes(const kvshot_project_desc* d) {
  return static_cast<size_t>(2) * d->num_layers * static_cast<size_t>(d->num_tokens) * d->hkv * kHeadDim * 4;
}

kvshot_status check_desc(const kvshot_project_desc* d, bool paged) {
  if (d == nullptr) return KVSHOT_ERR_NULL;
  if (d->num_tokens < 0 || d->num_layers < 1 || d->hkv < 1 || d->num_caches < 1) return KVSHOT_ERR_SHAPE;
  if (d->head_dim != kHeadDim || d->num_layers > kMaxLayers || d->hkv > 64) return KVSHOT_ERR_UNSUPPORTED;
  if (!(d->rope_base > 0.f) || !std::isfinite(d->rope_base)) return KVSHOT_ERR_SHAPE;
  if ((d->flags & ~KVSHOT_PROJECT_ROPE) != 0) return KVSHOT_ERR_SHAPE;
  if (static_cast<int64_t>(d->num_tokens) * d->num_layers * d->hkv * kHeadDim >= (int64_t(1) << 31))
    return KVSHOT_ERR_UNSUPPORTED;
  if (paged) {
    if (d->page_size < 1 || d->max_pages_per_seq < 1 || d->num_pages < 1) return KVSHOT_ERR_SHAPE;
  } else if (d->l_cap < 1) {
    return KVSHOT_ERR_SHAPE;
  }
  return KVSHOT_OK;
}

}  // namespace
}  // namespace kvshot

using namespace kvshot;

extern "C" size_t kvshot_kv_project_workspace_size(const kvshot_project_desc* d) {
  if (d == nullptr || check_desc(d, d->page_size > 0) != KVSHOT_OK) return 0;
  return std::max<size_t>(256, slab_bytes(d));
}

extern "C" kvshot_status kvshot_kv_project(const kvshot_project_desc* d, const void* k_in, const void* v_in,
                                           const void* w_k, const void* w_v, const int32_t* token_cache,
                                           const int32_t* positions, const int32_t* page_table, void* k_out,
                                           void* v_out, kvshot_stream_t stream) {
  const bool paged = page_table != nullptr;
  if (kvshot_status st = check_desc(d, paged)) return st;
  if (d->num_tokens == 0) return KVSHOT_OK;
  if (!k_in || !v_in || !w_k || !w_v || !token_cache || !positions || !k_out || !v_out) return KVSHOT_ERR_NULL;
  if (!aligned(k_in, 16) || !aligned(v_in, 16) || !aligned(w_k, 16) || !aligned(w_v, 16) || !aligned(k_out, 16) ||
      !aligned(v_out, 16) || !aligned(token_cache, 4) || !aligned(positions, 4) || (paged && !aligned(page_table, 4)))
    return KVSHOT_ERR_ALIGN;
  if (d->workspace == nullptr || !aligned(d->workspace, 256) || d->workspace_bytes < slab_bytes(d))
    return KVSHOT_ERR_WORKSPACE;
  const int T = d->num_tokens, L = d->num_layers, dkv = d->hkv * kHeadDim;
  ProjectParams p;
  p.token_cache = token_cache;
  p.positions = positions;
  p.page_table = page_table;
  p.k_out = static_cast<__nv_bfloat16*>(k_out);
  p.v_out = static_cast<__nv_bfloat16*>(v_out);
  p.err = d->err_flag;
  p.T = T;
  p.hkv = d->hkv;
  p.C = d->num_caches;
  p.nk = L * dkv / kKT;
  p.paged = paged ? 1 : 0;
  p.page_size = paged ? d->page_size : 0;
  p.max_pages = paged ? d->max_pages_per_seq : 0;
  p.num_pages = paged ? d->num_pages : 0;
  p.l_cap = paged ? 0 : d->l_cap;
  p.rope = (d->flags & KVSHOT_PROJECT_ROPE) ? 1 : 0;
  rope_turns(d->rope_base, p.turns);
  // As many CTAs per cluster as keep the grid within one wave (a k-tile each at least); blocks of equal size.
  auto blocks_of = [&](int box) { return (T + box - 1) / box; };
  auto split_of = [&](int box) {
    const int64_t clusters = static_cast<int64_t>(2) * d->hkv * blocks_of(box);
    int split = kMaxSplit;
    while (split > 1 && (clusters * split > kProjectCtas || split > p.nk)) split /= 2;
    return split;
  };
  // Smaller blocks while a warp has more than one token of a block (its slots and angles are the longest part of a narrow
  // cache's call), and the blocks, which each read the weights again, find free CTAs for it and few weights.  (With
  // the angles still in fp64, 128 tokens of 1 layer of 1 head 11.9 -> 4.4 us per call in blocks of 16, of 8 heads 9.0 ->
  // 8.2 in blocks of 64; beyond 8 k-tiles to a CTA the weights cost more: 512 tokens of 4 layers of 8 heads 19.0 us, in
  // blocks of 64 23.8.)
  int box = std::min(T, kTok);
  while (box > 16 && box > 8 * split_of(box)) {
    const int half = (box / 2 + 15) / 16 * 16;
    const int split = split_of(half);
    if (half >= box || split < std::min(4, p.nk) || (p.nk + split - 1) / split > 8) break;
    box = half;
  }
  const int blocks = blocks_of(box), split = split_of(box);
  p.box_tok = (T + blocks - 1) / blocks;
  p.split = split;
  const int per_cta = (p.nk + split - 1) / split;
  p.stages = std::min({per_cta, kMaxStages, kRingBytes / slot_bytes(p.box_tok)});
  const uint64_t K = static_cast<uint64_t>(L) * dkv;
  ProjectMaps maps;
  if (!encode_bf16_2d(&maps.w[0], w_k, K, dkv, kKT, kFeat) || !encode_bf16_2d(&maps.w[1], w_v, K, dkv, kKT, kFeat) ||
      !encode_bf16_2d(&maps.a[0], k_in, K, T, kKT, static_cast<uint32_t>(p.box_tok)) ||
      !encode_bf16_2d(&maps.a[1], v_in, K, T, kKT, static_cast<uint32_t>(p.box_tok)))
    return KVSHOT_ERR_CUDA;
  const size_t smem = smem_bytes(p.stages, p.box_tok);
  if (cudaFuncSetAttribute(kv_project_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)) !=
      cudaSuccess)
    return KVSHOT_ERR_CUDA;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = static_cast<unsigned>(split);
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(split) * static_cast<unsigned>(blocks), static_cast<unsigned>(d->hkv), 2);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = reinterpret_cast<cudaStream_t>(stream);
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kv_project_kernel, p, maps) == cudaSuccess ? KVSHOT_OK : KVSHOT_ERR_CUDA;
}
