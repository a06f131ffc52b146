// attn_f8.cu -- draft attention over an fp8 e4m3 target cache (KVSHOT_TARGET_FP8)
// on mma.sync tensor cores, for stacks of up to 64 query rows per KV head and
// for the 64-row blocks of larger ones.
//
// What bounds it: at 4 rows per KV head the codes are 256 B per key and the
// arithmetic is small, so HBM; but every code has to become an f16 before it can
// be multiplied (mma.sync's own e4m3 form runs at 20.7 cycles per k32 step and
// SM sub-partition on GB300, against 2 x 8.45 for the two f16 steps, so it buys
// nothing), and that decoding is the instruction cost.  The layout is chosen to
// spend as few instructions per key as possible:
//  - Keys are the M dimension: S^T = K Q^T and O^T = V^T P^T (m16n8k16, f16
//    inputs, fp32 sums).  The query rows are the N dimension in steps of 8, so a
//    4-row stack pads to 8 rows and not to 16, and one decoded fragment serves
//    every row of the warp.
//  - A prefix tile is 128 keys (16 KB of K codes, 16 KB of V codes), 32 keys to
//    a warp, so that the per-tile costs (barrier, cursor, softmax state) are
//    spread over twice the keys of the bf16 kernels' tiles.
//  - The row maxima are exchanged between lanes only when some score exceeds the
//    running maximum (one vote per tile otherwise).
// Fragments.  K: a lane's 16-byte load of one key row (dims 16 (2 q4 + kh) .. + 15)
// feeds four k-steps; the head dimensions of q are taken in the same permuted
// order.  V: a lane pairs the same 16 dims (16 g ..) of two key rows with byte
// permutes, so m-tile mt, rows g and g + 8 are dims 16 g + 2 mt and + 1, and a
// lane owns 16 consecutive dims of its rows in the output.  P^T comes from S^T by
// one 8x8 transpose (movmatrix) per 8 keys x 8 rows.  All shared-memory loads are
// free of bank conflicts under the TMA's 128-byte swizzle.
// e4m3 -> f16 is exact; q, P and the draft K/V are rounded to f16; the cache's
// power-of-two scales are folded into the score scale (keys) and, from 2^-4 to 2^8, into P (values).  Times P (up to 1)
// a larger one would overflow f16 and a smaller one cost P's small values their bits: a form of its own (kWideV) applies
// those to O where a piece leaves the prefix.  (One form for every scale: 1 cache of 300 tokens, 4 rows, 10.5 -> 10.9 us
// per call; 64 caches of 512 to 8192 tokens 0.4%.)
#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>

#include "kvshot_attn_common.cuh"

namespace kvshot {
namespace {

using namespace dev;

constexpr int kPK = kF8PrefixTile;       // keys per prefix tile
constexpr int kCodeBytes = kPK * 128;    // a tile's K (or V) codes
constexpr int kChunk = 32;               // keys a warp takes through QK^T, softmax and P.V at a time
constexpr int kBarConsumers = 1;
constexpr int kCombStride = kHeadDim + 4;  // padded fp32 row in the combine buffer
static_assert(2 * kCodeBytes == kStageBytes, "a stage holds a prefix tile's codes or a bf16 draft tile");

// Four e4m3 codes (a 32-bit word, lowest byte first) -> four f16 values (two f16x2 words).
__device__ __forceinline__ uint2 e4m3x4_to_f16x4(uint32_t codes) {
  uint2 r;
  asm("{\n\t.reg .b16 lo, hi;\n\tmov.b32 {lo, hi}, %2;\n\t"
      "cvt.rn.f16x2.e4m3x2 %0, lo;\n\tcvt.rn.f16x2.e4m3x2 %1, hi;\n\t}"
      : "=r"(r.x), "=r"(r.y)
      : "r"(codes));
  return r;
}

__device__ __forceinline__ uint32_t pack_f16x2(float lo, float hi) {
  __half2 v = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

__device__ __forceinline__ uint32_t bf16x2_to_f16x2(uint32_t w) { return pack_f16x2(bf16_lo(w), bf16_hi(w)); }

// Word t (0..3) of a 16-byte vector; t is a compile-time constant after unrolling.
__device__ __forceinline__ uint32_t word(const uint4& v, int t) {
  return t == 0 ? v.x : t == 1 ? v.y : t == 2 ? v.z : v.w;
}

// 8x8 transpose of b16 elements across the warp.
__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t x) {
  uint32_t y;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
  return y;
}

// D += A * B, m16n8k16, f16 inputs, fp32 accumulate.
__device__ __forceinline__ void mma_f16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                        uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// NR: 8-row steps per warp; RG: row groups (warps that take the same keys for other rows); KS: key
// slices of a tile.
template <int NR, int RG, int KS, int STAGES, int MINB>
struct Cfg {
  static constexpr int kNR = NR;
  static constexpr int kRG = RG;
  static constexpr int kKS = KS;
  static constexpr int kStages = STAGES;
  static constexpr int kMinBlocks = MINB;
  static constexpr int kWarps = RG * KS;  // consumer warps
  static constexpr int kThreads = (kWarps + 1) * 32;
  static constexpr int kKW = kPK / KS;  // keys per warp of a prefix tile
  static constexpr int kWarpRows = 8 * NR;
  static constexpr int kRows = kWarpRows * RG;  // rows per unit
  // Q^T fragments: in registers for 8 rows, else in shared memory (a piece's 32 registers of them spill)
  static constexpr bool kQSmem = NR > 1;
  static constexpr bool kDraftRows = NR == 2 && RG < 4;  // two key slices share a draft tile's keys, each for half of the rows
  static constexpr int kQBytes = kQSmem ? RG * 8 * NR * 32 * 8 : 0;
};

struct Smem {
  uint8_t* ring;
  uint2* qf;      // [RG][8 k-steps][NR][32 lanes] Q^T fragments of the piece (kQSmem)
  uint64_t* full;
  uint64_t* empty;
  uint64_t* anc;
  int* par;
  float* comb_o;  // [kRows][kCombStride]
  float* comb_m;  // [KS][kRows]
  float* comb_l;  // [KS][kRows]
  int* misc;      // [0] abort, [1] issued, [2] consumed
  int* len;
  int* base;
};

template <class CF>
__host__ __device__ constexpr size_t smem_bytes(int C) {
  size_t off = static_cast<size_t>(CF::kStages) * kStageBytes;
  off += CF::kQBytes + 2 * CF::kStages * sizeof(uint64_t);
  off += sizeof(uint64_t) * kMaxTreeNodes + sizeof(int) * kMaxTreeNodes;
  off += sizeof(float) * CF::kRows * kCombStride;
  off += 2 * sizeof(float) * CF::kKS * CF::kRows;
  off += sizeof(int) * 4;
  off += sizeof(int) * (2 * C + 1);
  return off + 1024;
}

template <class CF>
__device__ Smem carve(uint8_t* raw, int C) {
  Smem s;
  uint8_t* p = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~uintptr_t(1023));
  s.ring = p;
  p += CF::kStages * kStageBytes;
  s.comb_o = reinterpret_cast<float*>(p);
  s.qf = reinterpret_cast<uint2*>(s.comb_o + CF::kRows * kCombStride);
  s.full = reinterpret_cast<uint64_t*>(reinterpret_cast<uint8_t*>(s.qf) + CF::kQBytes);
  s.empty = s.full + CF::kStages;
  s.anc = s.empty + CF::kStages;
  s.par = reinterpret_cast<int*>(s.anc + kMaxTreeNodes);
  s.comb_m = reinterpret_cast<float*>(s.par + kMaxTreeNodes);
  s.comb_l = s.comb_m + CF::kKS * CF::kRows;
  s.misc = reinterpret_cast<int*>(s.comb_l + CF::kKS * CF::kRows);
  s.len = s.misc + 4;
  s.base = s.len + C;
  return s;
}

// The producer warp: one stage per tile.  Prefix tiles: boxes of whole 128-byte rows, min(page size,
// 64) rows each, K from lanes 0..15 and V from lanes 16..31.  Draft tiles (bf16, 64 keys): boxes of 8
// rows and one 64-dim half.  Target loads may start while the preceding kernel is still running
// (KVSHOT_OVERLAP_PREVIOUS); draft loads wait for it.
__device__ __forceinline__ void run_producer_codes(const AttnParams& p, const TensorMaps& maps, const Pipe& pipe,
                                                   const int* s_len, Cursor cu) {
  const int lane = threadIdx.x & 31;
  const uint64_t policy = l2_policy_evict_first();
  const int br = p.box_rows, P = p.page_size;
  int stage = 0, issued = 0;
  uint32_t phase = 0;
  bool waited = false;
  PageWindow win;
  for (; cu.t < cu.t_end; cursor_next<kPK>(cu, p, s_len)) {
    const int h = cu.hr / p.row_blocks;
    const TileInfo ti = tile_info<kPK>(cu, p);
    const int i = lane & 15, kv = lane >> 4;
    int y = 0, nbox = 0;
    if (!ti.draft) {
      nbox = (ti.nkeys + br - 1) / br;
      const int row = ti.key0 + min(i, nbox - 1) * br;
      if (p.paged) {
        const int pg0 = ti.key0 / P, pg = row / P;
        win.cover(p, cu.c, (cu.L + P - 1) / P, pg0, (ti.key0 + (nbox - 1) * br) / P - pg0 + 1, lane);
        y = (win.get(pg) * p.hkv + h) * P + (row - pg * P);
      } else {
        y = (cu.c * p.hkv + h) * p.l_cap + row;
      }
    } else if (!waited) {
      wait_for_prerequisite_grid();
      waited = true;
    }
    int ok = 1;
    if (lane == 0) ok = mbar_wait(smem_addr(&pipe.empty[stage]), phase ^ 1u, p.err, p.wait_ns) && !*pipe.abort;
    ok = __shfl_sync(0xffffffffu, ok, 0);
    if (!ok) {
      if (lane == 0) *pipe.abort = 1;
      break;
    }
    const uint32_t bar = smem_addr(&pipe.full[stage]);
    const uint32_t dst = smem_addr(pipe.ring + static_cast<size_t>(stage) * kStageBytes);
    if (!ti.draft) {
      if (lane == 0) mbar_arrive_expect_tx(bar, static_cast<uint32_t>(nbox * br) * 256u);
      __syncwarp();
      if (i < nbox)
        tma_load_2d(dst + kv * kCodeBytes + i * br * 128, kv ? &maps.tv : &maps.tk, 0, y, bar, policy);
    } else {
      const int nb = (ti.nkeys + kDraftBoxRows - 1) / kDraftBoxRows;
      if (lane == 0) mbar_arrive_expect_tx(bar, static_cast<uint32_t>(nb) * kDraftBoxRows * 128 * 4);
      __syncwarp();
      const int dkv = lane & 1, hf = (lane >> 1) & 1, ib = lane >> 2;
      if (ib < nb)
        tma_load_2d(dst + dkv * kKVTileBytes + hf * kHalfBytes + ib * kDraftBoxRows * 128, dkv ? &maps.dv : &maps.dk,
                    hf * 64, (cu.c * p.hkv + h) * p.n_max + ti.key0 + ib * kDraftBoxRows, bar, policy);
    }
    ++issued;
    if (++stage == pipe.stages) {
      stage = 0;
      phase ^= 1u;
    }
  }
  if (lane == 0) *pipe.issued = issued;
}

// Combine the KS key-slice warps of each row group and write the piece: the final bf16 output + lse if
// the piece is the whole unit, else the normalised fp32 partial + log2-domain lse into slot `slot`.
// `o_scale`: what o is still to be multiplied by.  o[mt][nr][2 a + e]: dim 16 g + 2 mt + a of row 8 nr + 2 q4 + e (of the warp's rows).
template <class CF>
__device__ __forceinline__ void finalize(const AttnParams& p, const Smem& sm, int c, int h, int rb, int slot, bool whole,
                                         float o_scale, float (&o)[8][CF::kNR][4], const float (&m_run)[CF::kNR][2],
                                         float (&l_run)[CF::kNR][2]) {
  constexpr int NR = CF::kNR;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rg = warp % CF::kRG, ks = warp / CF::kRG;
  const int g = lane >> 2, q4 = lane & 3;
  const int row0 = rg * CF::kWarpRows + 2 * q4;  // this lane's rows: row0 + 8 nr + e
#pragma unroll
  for (int nr = 0; nr < NR; ++nr)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
#pragma unroll
      for (int d = 4; d < 32; d <<= 1) l_run[nr][e] += __shfl_xor_sync(0xffffffffu, l_run[nr][e], d);
      if (g == 0) {
        sm.comb_m[ks * CF::kRows + row0 + 8 * nr + e] = m_run[nr][e];
        sm.comb_l[ks * CF::kRows + row0 + 8 * nr + e] = l_run[nr][e];
      }
    }
  named_barrier_sync(kBarConsumers, CF::kWarps * 32);
  float M[NR][2], Ls[NR][2];
#pragma unroll
  for (int nr = 0; nr < NR; ++nr)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int row = row0 + 8 * nr + e;
      float mx = -INFINITY, sum = 0.f;
#pragma unroll
      for (int k = 0; k < CF::kKS; ++k) mx = fmaxf(mx, sm.comb_m[k * CF::kRows + row]);
      if (mx != -INFINITY) {
#pragma unroll
        for (int k = 0; k < CF::kKS; ++k) {
          const float mk = sm.comb_m[k * CF::kRows + row];
          sum += (mk == -INFINITY ? 0.f : ex2(mk - mx)) * sm.comb_l[k * CF::kRows + row];
        }
      }
      M[nr][e] = mx;
      Ls[nr][e] = sum;
      const float w = (m_run[nr][e] == -INFINITY || mx == -INFINITY) ? 0.f : ex2(m_run[nr][e] - mx) * o_scale;
#pragma unroll
      for (int mt = 0; mt < 8; ++mt) {
        o[mt][nr][e] *= w;
        o[mt][nr][2 + e] *= w;
      }
    }
  // Key slices accumulate into the buffer one after another; the last one writes out.
#pragma unroll
  for (int k = 0; k < CF::kKS; ++k) {
    if (ks == k) {
#pragma unroll
      for (int nr = 0; nr < NR; ++nr)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int rl = row0 + 8 * nr + e;  // row within the unit
          float4* buf = reinterpret_cast<float4*>(sm.comb_o + rl * kCombStride + 16 * g);
          if (k > 0) {
#pragma unroll
            for (int v = 0; v < 4; ++v) {
              const float4 a = buf[v];
              o[2 * v][nr][e] += a.x;
              o[2 * v][nr][2 + e] += a.y;
              o[2 * v + 1][nr][e] += a.z;
              o[2 * v + 1][nr][2 + e] += a.w;
            }
          }
          if (k < CF::kKS - 1) {
#pragma unroll
            for (int v = 0; v < 4; ++v)
              buf[v] = make_float4(o[2 * v][nr][e], o[2 * v][nr][2 + e], o[2 * v + 1][nr][e], o[2 * v + 1][nr][2 + e]);
          } else {
            const int rr = rb * p.rows_per_unit + rl;  // row within the GQA stack
            if (rl >= p.rows_per_unit || rr >= p.rows_total) continue;
            const float inv = Ls[nr][e] > 0.f ? 1.f / Ls[nr][e] : 0.f;
            const float lse2 = Ls[nr][e] > 0.f ? M[nr][e] + __log2f(Ls[nr][e]) : -INFINITY;
            if (whole) {
              const int nl = rr / p.G, gh = rr - nl * p.G;
              const size_t row = (static_cast<size_t>(c) * p.Nq + nl) * p.hq + h * p.G + gh;
              uint4* dst = reinterpret_cast<uint4*>(p.out + row * kHeadDim + 16 * g);
#pragma unroll
              for (int v = 0; v < 2; ++v) {
                const int m0 = 4 * v;
                dst[v] = make_uint4(pack_bf16x2(o[m0][nr][e] * inv, o[m0][nr][2 + e] * inv),
                                    pack_bf16x2(o[m0 + 1][nr][e] * inv, o[m0 + 1][nr][2 + e] * inv),
                                    pack_bf16x2(o[m0 + 2][nr][e] * inv, o[m0 + 2][nr][2 + e] * inv),
                                    pack_bf16x2(o[m0 + 3][nr][e] * inv, o[m0 + 3][nr][2 + e] * inv));
              }
              if (g == 0) p.lse[row] = lse2 * 0.69314718055994531f;
            } else {
              const size_t row = static_cast<size_t>(slot) * p.rows_per_unit + rl;
              float4* dst = reinterpret_cast<float4*>(p.ws_o + row * kHeadDim + 16 * g);
#pragma unroll
              for (int v = 0; v < 4; ++v)
                dst[v] = make_float4(o[2 * v][nr][e] * inv, o[2 * v][nr][2 + e] * inv, o[2 * v + 1][nr][e] * inv,
                                     o[2 * v + 1][nr][2 + e] * inv);
              if (g == 0) p.ws_lse[row] = lse2;
            }
          }
        }
    }
    named_barrier_sync(kBarConsumers, CF::kWarps * 32);
  }
}

template <class CF, bool kWideV>
__device__ __forceinline__ void run_consumer(const AttnParams& p, const Smem& sm, const Pipe& pipe, Cursor cu) {
  constexpr int NR = CF::kNR;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rg = warp % CF::kRG, ks = warp / CF::kRG;
  const int g = lane >> 2, q4 = lane & 3;
  const int HR = p.hkv * p.row_blocks;
  // This lane's place in a tile of codes (128-byte rows, 16-byte chunk index XOR row index mod 8): chunk
  // 2 q4 + kh of key row g (K), chunk g of key rows 2 q4 and 2 q4 + 1 (V).
  const uint32_t koff0 = g * 128 + (((2 * q4) ^ g) << 4), koff1 = g * 128 + (((2 * q4 + 1) ^ g) << 4);
  const uint32_t voff0 = 2 * q4 * 128 + ((g ^ (2 * q4)) << 4), voff1 = (2 * q4 + 1) * 128 + ((g ^ (2 * q4 + 1)) << 4);
  // Q^T fragments (f16): k-step 4 kh + s on dims 16 (2 q4 + kh) + 4 s + {0, 1}, {2, 3}.
  uint2 qreg[CF::kQSmem ? 1 : 8] = {};
  uint2* qf = sm.qf + rg * (8 * NR * 32) + lane;
  auto q_frag = [&](int kstep, int nr) -> uint2 {
    if constexpr (CF::kQSmem) return qf[(kstep * NR + nr) * 32];
    else return qreg[kstep];
  };
  float o[8][NR][4];
  float m_run[NR][2], l_run[NR][2];  // rows 8 nr + 2 q4 + e; l_run: this lane's keys only
  int stage = 0;
  uint32_t phase = 0;
  int piece_lt0 = 0, anc_seq = -1, consumed = 0;
  int h = 0, rb = 0;
  bool o_codes = kWideV;  // O is in units of the value codes: this warp has had no draft keys of the piece

  for (; cu.t < cu.t_end; cursor_next<kPK>(cu, p, sm.len)) {
    const TileInfo ti = tile_info<kPK>(cu, p);
    if (ti.first) {
      h = cu.hr / p.row_blocks;
      rb = cu.hr - h * p.row_blocks;
      piece_lt0 = cu.lt;
      constexpr int kQV = CF::kQSmem ? 4 / CF::kKS : 4;  // chunks of 8 dims of each lane's 32: the key slices share them
#pragma unroll
      for (int nr = 0; nr < NR; ++nr) {
        const int rr = rb * p.rows_per_unit + rg * CF::kWarpRows + 8 * nr + g;
        const bool ok = rr < p.rows_total;
        const int nl = ok ? rr / p.G : 0, gh = ok ? rr - nl * p.G : 0;
        const uint4* src = reinterpret_cast<const uint4*>(
            p.q + ((static_cast<size_t>(cu.c) * p.Nq + nl) * p.hq + h * p.G + gh) * kHeadDim + 32 * q4);
#pragma unroll
        for (int i = 0; i < kQV; ++i) {
          const int v = CF::kQSmem ? ks * kQV + i : i;  // dims 32 q4 + 8 v .. + 7: k-steps 2 v, 2 v + 1
          const uint4 w = ok ? src[v] : make_uint4(0u, 0u, 0u, 0u);
          const uint2 f0 = make_uint2(bf16x2_to_f16x2(w.x), bf16x2_to_f16x2(w.y));
          const uint2 f1 = make_uint2(bf16x2_to_f16x2(w.z), bf16x2_to_f16x2(w.w));
          if constexpr (CF::kQSmem) {
            qf[(2 * v * NR + nr) * 32] = f0;
            qf[((2 * v + 1) * NR + nr) * 32] = f1;
          } else {
            qreg[2 * i] = f0;
            qreg[2 * i + 1] = f1;
          }
        }
#pragma unroll
        for (int mt = 0; mt < 8; ++mt) o[mt][nr][0] = o[mt][nr][1] = o[mt][nr][2] = o[mt][nr][3] = 0.f;
        m_run[nr][0] = m_run[nr][1] = -INFINITY;
        l_run[nr][0] = l_run[nr][1] = 0.f;
      }
      o_codes = kWideV;
      if constexpr (CF::kQSmem) named_barrier_sync(kBarConsumers, CF::kWarps * 32);  // Q^T is shared by the key slices
    }
    if (ti.draft && p.tree) {
      const int seq = cu.c / (p.C / p.B);
      if (seq != anc_seq) {
        build_ancestor_masks(p, seq, sm.anc, sm.par, threadIdx.x, CF::kWarps * 32, kBarConsumers);
        anc_seq = seq;
      }
    }
    bool live = !*pipe.abort;
    if (live && !mbar_wait(smem_addr(&pipe.full[stage]), phase, p.err, p.wait_ns)) {
      *pipe.abort = 1;
      live = false;
    }
    live = __all_sync(0xffffffffu, live);  // the warp-wide MMA and shuffle steps below need the whole warp
    const uint32_t kbase = smem_addr(pipe.ring + static_cast<size_t>(stage) * kStageBytes);
    const bool codes = !ti.draft;
    const uint32_t vbase = kbase + (codes ? kCodeBytes : kKVTileBytes);
    // The key scale is part of the score scale, the value scale part of P (kWideV: of O); the sum keeps the unscaled P.
    const float qs = codes ? p.qscale * p.k_scale : p.qscale, vs = codes && !kWideV ? p.v_scale : 1.f;
    // 32 keys of the tile from key kw on.  Draft chunks: 8-row step `only` alone (-1: all), and the second 16 keys
    // only where one of them is visible.
    auto chunk = [&](auto draft, int kw, int only) {
      constexpr bool kDraft = decltype(draft)::value;
      const bool full = !kDraft && ti.nkeys == kPK;  // every key of the tile is visible to every row
      const bool wide = !kDraft || ti.nkeys > kw + 16;
      auto skip = [&](int nr) { return kDraft && CF::kDraftRows && nr != only; };
      // S^T = K Q^T for 32 keys: s[m][nr][2 a + e] is key kw + 16 m + 8 a + g, row 8 nr + 2 q4 + e.
      float s[2][NR][4];
#pragma unroll
      for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int nr = 0; nr < NR; ++nr) s[m][nr][0] = s[m][nr][1] = s[m][nr][2] = s[m][nr][3] = 0.f;
      if constexpr (!kDraft) {
#pragma unroll
        for (int kh = 0; kh < 2; ++kh) {
          const uint32_t a = kbase + (kh ? koff1 : koff0) + kw * 128;
          const uint4 w[4] = {lds128(a), lds128(a + 1024), lds128(a + 2048), lds128(a + 3072)};  // keys + 0, 8, 16, 24
#pragma unroll
          for (int st = 0; st < 4; ++st) {
            uint2 q[NR];
#pragma unroll
            for (int nr = 0; nr < NR; ++nr) q[nr] = q_frag(4 * kh + st, nr);
#pragma unroll
            for (int m = 0; m < 2; ++m) {
              const uint2 f0 = e4m3x4_to_f16x4(word(w[2 * m], st)), f1 = e4m3x4_to_f16x4(word(w[2 * m + 1], st));
#pragma unroll
              for (int nr = 0; nr < NR; ++nr) mma_f16(s[m][nr], f0.x, f1.x, f0.y, f1.y, q[nr].x, q[nr].y);
            }
          }
        }
      } else {
#pragma unroll 1
        for (int c8 = 0; c8 < 4; ++c8) {  // dims 32 q4 + 8 c8 .. + 7: k-steps 2 c8, 2 c8 + 1
          const int key = kw + g, ch = 4 * q4 + c8;
          uint4 w[4];
#pragma unroll
          for (int r = 0; r < 4; ++r) w[r] = lds128(kbase + tile_off(key + 8 * r, ch));
#pragma unroll
          for (int st = 0; st < 2; ++st)
#pragma unroll
            for (int nr = 0; nr < NR; ++nr) {
              if (skip(nr)) continue;
              uint2 q;
              if constexpr (CF::kQSmem) q = q_frag(2 * c8 + st, nr);
              else q = c8 == 0 ? qreg[st] : c8 == 1 ? qreg[2 + st] : c8 == 2 ? qreg[4 + st] : qreg[6 + st];
#pragma unroll
              for (int m = 0; m < 2; ++m) {
                if (m == 1 && !wide) break;
                const uint4 &x = w[2 * m], &y = w[2 * m + 1];
                mma_f16(s[m][nr], bf16x2_to_f16x2(word(x, 2 * st)), bf16x2_to_f16x2(word(y, 2 * st)),
                        bf16x2_to_f16x2(word(x, 2 * st + 1)), bf16x2_to_f16x2(word(y, 2 * st + 1)), q.x, q.y);
              }
            }
        }
      }
      float mx[NR][2];
      if (!full) {
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
          for (int nr = 0; nr < NR; ++nr)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int key = kw + 16 * m + 8 * (e >> 1) + g;
              bool valid = key < ti.nkeys && !skip(nr);
              if (kDraft)
                valid = valid && draft_visible(p, sm.anc, rb * p.rows_per_unit + rg * CF::kWarpRows + 8 * nr + 2 * q4 + (e & 1),
                                               ti.key0 + key);
              if (!valid) s[m][nr][e] = -INFINITY;
            }
      }
      bool grow = false;
#pragma unroll
      for (int nr = 0; nr < NR; ++nr)
#pragma unroll
        for (int e = 0; e < 2; ++e) {  // raw maxima (qs > 0)
          mx[nr][e] = fmaxf(fmaxf(s[0][nr][e], s[0][nr][2 + e]), fmaxf(s[1][nr][e], s[1][nr][2 + e])) * qs;
          grow |= mx[nr][e] > m_run[nr][e];
        }
      const bool leave_codes = kWideV && kDraft && o_codes;  // warp-uniform
      if (__any_sync(0xffffffffu, grow || leave_codes)) {
#pragma unroll
        for (int nr = 0; nr < NR; ++nr)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            float v = mx[nr][e];
#pragma unroll
            for (int d = 4; d < 32; d <<= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, d));
            v = fmaxf(v, m_run[nr][e]);
            const float alpha = ex2(m_run[nr][e] - (v == -INFINITY ? 0.f : v));
            m_run[nr][e] = v;
            l_run[nr][e] *= alpha;
            const float o_alpha = leave_codes ? alpha * p.v_scale : alpha;
#pragma unroll
            for (int mt = 0; mt < 8; ++mt) {
              o[mt][nr][e] *= o_alpha;
              o[mt][nr][2 + e] *= o_alpha;
            }
          }
      }
      if (kDraft) o_codes = false;
      // P^T fragments of the chunk's two 16-key steps.
      uint32_t pb[2][NR][2];
#pragma unroll
      for (int nr = 0; nr < NR; ++nr) {
        if (skip(nr)) continue;
        const float m0 = m_run[nr][0] == -INFINITY ? 0.f : m_run[nr][0];
        const float m1 = m_run[nr][1] == -INFINITY ? 0.f : m_run[nr][1];
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
          for (int a = 0; a < 2; ++a) {
            const float e0 = ex2(fmaf(s[m][nr][2 * a], qs, -m0)), e1 = ex2(fmaf(s[m][nr][2 * a + 1], qs, -m1));
            l_run[nr][0] += e0;
            l_run[nr][1] += e1;
            pb[m][nr][a] = movmatrix_trans(pack_f16x2(e0 * vs, e1 * vs));
          }
      }
      // O^T += V^T P^T, 16 keys per step.
#pragma unroll
      for (int kk = 0; kk < 2; ++kk) {
        if (kk == 1 && !wide) break;
        const int k0 = kw + 16 * kk;
        if constexpr (!kDraft) {
          const uint32_t av = vbase + k0 * 128;
          uint4 w[4] = {lds128(av + voff0), lds128(av + voff1), lds128(av + voff0 + 1024), lds128(av + voff1 + 1024)};
          if (!full) {  // rows past the valid keys may hold NaN codes
#pragma unroll
            for (int r = 0; r < 4; ++r)
              if (k0 + 2 * q4 + (r & 1) + 8 * (r >> 1) >= ti.nkeys) w[r] = make_uint4(0u, 0u, 0u, 0u);
          }
#pragma unroll
          for (int t = 0; t < 4; ++t) {  // dims 16 g + 4 t .. + 3: m-tiles 2 t, 2 t + 1
            const uint2 ab0 = e4m3x4_to_f16x4(__byte_perm(word(w[0], t), word(w[1], t), 0x5140));
            const uint2 ab1 = e4m3x4_to_f16x4(__byte_perm(word(w[0], t), word(w[1], t), 0x7362));
            const uint2 cd0 = e4m3x4_to_f16x4(__byte_perm(word(w[2], t), word(w[3], t), 0x5140));
            const uint2 cd1 = e4m3x4_to_f16x4(__byte_perm(word(w[2], t), word(w[3], t), 0x7362));
#pragma unroll
            for (int nr = 0; nr < NR; ++nr) {
              mma_f16(o[2 * t][nr], ab0.x, ab0.y, cd0.x, cd0.y, pb[kk][nr][0], pb[kk][nr][1]);
              mma_f16(o[2 * t + 1][nr], ab1.x, ab1.y, cd1.x, cd1.y, pb[kk][nr][0], pb[kk][nr][1]);
            }
          }
        } else {
#pragma unroll
          for (int hh = 0; hh < 2; ++hh) {  // dims 16 g + 8 hh .. + 7: m-tiles 4 hh .. + 3
            uint4 w[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
              const int key = k0 + 2 * q4 + (r & 1) + 8 * (r >> 1);
              w[r] = lds128(vbase + tile_off(key, 2 * g + hh));
              if (key >= ti.nkeys) w[r] = make_uint4(0u, 0u, 0u, 0u);
            }
#pragma unroll
            for (int t = 0; t < 4; ++t) {  // word t: dims 16 g + 8 hh + 2 t, + 1: m-tile 4 hh + t
              const uint32_t ab = word(w[0], t), bb = word(w[1], t), cb = word(w[2], t), db = word(w[3], t);
              const uint32_t a0 = bf16x2_to_f16x2(__byte_perm(ab, bb, 0x5410));
              const uint32_t a1 = bf16x2_to_f16x2(__byte_perm(ab, bb, 0x7632));
              const uint32_t a2 = bf16x2_to_f16x2(__byte_perm(cb, db, 0x5410));
              const uint32_t a3 = bf16x2_to_f16x2(__byte_perm(cb, db, 0x7632));
#pragma unroll
              for (int nr = 0; nr < NR; ++nr)
                if (!skip(nr)) mma_f16(o[4 * hh + t][nr], a0, a1, a2, a3, pb[kk][nr][0], pb[kk][nr][1]);
            }
          }
        }
      }
    };
    const int kw1 = min(ks * CF::kKW + CF::kKW, ti.nkeys);
    if (live && codes) {
#pragma unroll 1
      for (int kw = ks * CF::kKW; kw < kw1; kw += kChunk) chunk(std::false_type{}, kw, -1);
    } else if (live && CF::kDraftRows) {
      // Two slices take the same draft keys for 8 rows each: few keys would leave one warp all the rows.
#pragma unroll 1
      for (int kw = (ks >> 1) * kChunk; kw < ti.nkeys; kw += CF::kKS / 2 * kChunk) chunk(std::true_type{}, kw, ks & 1);
    } else if (live) {
#pragma unroll 1
      for (int kw = ks * CF::kKW; kw < kw1; kw += kChunk) chunk(std::true_type{}, kw, -1);
    }
    __syncwarp();
    if (live) {
      if (lane == 0) mbar_arrive(smem_addr(&pipe.empty[stage]));
      ++consumed;
    }
    if (++stage == CF::kStages) {
      stage = 0;
      phase ^= 1u;
    }
    if (ti.last) {
      const bool whole = piece_lt0 == 0 && cu.lt == cu.ut - 1;
      finalize<CF>(p, sm, cu.c, h, rb, cu.c * HR + cu.hr + blockIdx.x, whole, o_codes ? p.v_scale : 1.f, o, m_run, l_run);
    }
  }
  if (threadIdx.x == 0) sm.misc[2] = consumed;
}

template <class CF, bool kWideV>
__global__ void __launch_bounds__(CF::kThreads, CF::kMinBlocks)
    attn_f8_kernel(const __grid_constant__ AttnParams p, const __grid_constant__ TensorMaps maps) {
  extern __shared__ uint8_t smem_raw[];
  if (threadIdx.x == 0) allow_dependent_launch();  // the merge may be scheduled as CTAs finish
  const Smem sm = carve<CF>(smem_raw, p.C);
  const int warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    for (int s = 0; s < CF::kStages; ++s) {
      mbar_init(smem_addr(&sm.full[s]), 1);
      mbar_init(smem_addr(&sm.empty[s]), CF::kWarps);
    }
    sm.misc[0] = sm.misc[1] = sm.misc[2] = 0;
    fence_mbar_init();
    prefetch_tensormap(&maps.tk);
    prefetch_tensormap(&maps.tv);
    prefetch_tensormap(&maps.dk);
    prefetch_tensormap(&maps.dv);
  }
  build_plan<kPK>(p, sm.len, sm.base);
  const Cursor cu = cursor_begin<kPK>(p, sm.len, sm.base);
  Pipe pipe{sm.ring, sm.full, sm.empty, CF::kStages, reinterpret_cast<volatile int*>(&sm.misc[0]), &sm.misc[1]};
  if (warp == CF::kWarps) {
    run_producer_codes(p, maps, pipe, sm.len, cu);
  } else {
    // With KVSHOT_OVERLAP_PREVIOUS the kernel may have started before the preceding kernel ended: q is
    // read, and outputs are written, only after it has.
    wait_for_prerequisite_grid();
    run_consumer<CF, kWideV>(p, sm, pipe, cu);
  }
  __syncthreads();
  if (threadIdx.x == 0) drain_after_abort(p, pipe, sm.misc[2]);
}

// Up to 8 rows, up to 16, 32, 48, 64.  What a CTA holds decides how many warps hide the latencies of
// loads, conversions and the softmax: 8 rows fit three CTAs per SM (128 registers; two stages each: 105 us
// per ragged-chain call of 64 caches against 117 us for two CTAs of three stages), 16 rows two (three would
// spill).  48 rows take two key slices: with four, 13 warps are capped at 128 registers and spill (16 caches of 4096 tokens
// 101 us per call, now 85).  Before this kernel the same calls took 185 us (4 rows) and 265 us (16 rows, 16 caches x 32K
// keys, now 173 us): 64-key tiles, query rows as the MMA's M, 18.4 M instead of 13.1 M warp instructions per call of
// 16 caches x 4096 tokens at 16 rows.
// Short units are bound by what a unit costs beside its tiles.  q is converted by all key slices; a draft tile has code of
// its own, apart from the codes' loop, in which two slices share its keys, each for half of the rows, and masked keys
// are left out (16 caches of 32K keys, 16 rows, 178 -> 173 us per call; 40 of 300 to 2500 60.5 -> 50.5; 512 of 50 to
// 400 326 -> 276, 4 rows 136 -> 117).
using Cfg8 = Cfg<1, 1, 4, 2, 3>;
using Cfg16 = Cfg<2, 1, 4, 3, 2>;
using Cfg16Many = Cfg<2, 1, 4, 2, 2>;
using Cfg32 = Cfg<2, 2, 4, 5, 1>;
using Cfg48 = Cfg<2, 3, 2, 5, 1>;
using Cfg64 = Cfg<2, 4, 2, 5, 1>;

// Every plan that kMaxCaches allows fits an SM.
constexpr size_t kMaxSmem = 227 * 1024;
static_assert(smem_bytes<Cfg8>(kMaxCaches) <= kMaxSmem && smem_bytes<Cfg16>(kMaxCaches) <= kMaxSmem &&
                  smem_bytes<Cfg32>(kMaxCaches) <= kMaxSmem && smem_bytes<Cfg48>(kMaxCaches) <= kMaxSmem &&
                  smem_bytes<Cfg64>(kMaxCaches) <= kMaxSmem,
              "shared memory at the largest number of caches");

// The plan takes 8 bytes of shared memory per cache: past this many, two CTAs of three stages no longer fit an SM.
constexpr size_t kSmSmem = 228 * 1024, kCtaReserved = 1024;
constexpr bool many_caches(int C) { return 2 * (smem_bytes<Cfg16>(C) + kCtaReserved) > kSmSmem; }
static_assert(2 * (smem_bytes<Cfg16Many>(kMaxCaches) + kCtaReserved) <= kSmSmem, "two CTAs at any number of caches");

template <class CF>
cudaError_t launch_cfg(const AttnParams& p, const TensorMaps& maps, bool pdl, cudaStream_t stream) {
  const size_t smem = smem_bytes<CF>(p.C);
  auto* kernel = p.v_scale < 0x1p-4f || p.v_scale > 0x1p8f ? attn_f8_kernel<CF, true> : attn_f8_kernel<CF, false>;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  return launch_maybe_pdl(kernel, dim3(p.num_ctas), dim3(CF::kThreads), smem, pdl, stream, p, maps);
}

// (Both forms have the same shared memory, and registers capped by the same launch bounds.)
template <class CF>
cudaError_t occupancy_cfg(int C, int* ctas) {
  const size_t smem = smem_bytes<CF>(C);
  cudaError_t e = cudaFuncSetAttribute(attn_f8_kernel<CF, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas, attn_f8_kernel<CF, false>, CF::kThreads, smem);
}

}  // namespace

int attn_f8_rows(int rows) { return rows <= 8 ? 8 : std::min(64, (rows + 15) / 16 * 16); }

cudaError_t attn_f8_occupancy(int rows_per_unit, int C, int* ctas_per_sm) {
  switch (rows_per_unit) {
    case 8: return occupancy_cfg<Cfg8>(C, ctas_per_sm);
    case 16: return many_caches(C) ? occupancy_cfg<Cfg16Many>(C, ctas_per_sm) : occupancy_cfg<Cfg16>(C, ctas_per_sm);
    case 32: return occupancy_cfg<Cfg32>(C, ctas_per_sm);
    case 48: return occupancy_cfg<Cfg48>(C, ctas_per_sm);
    case 64: return occupancy_cfg<Cfg64>(C, ctas_per_sm);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_attn_f8(const AttnParams& p, const TensorMaps& maps, bool pdl, cudaStream_t stream) {
  switch (p.rows_per_unit) {
    case 8: return launch_cfg<Cfg8>(p, maps, pdl, stream);
    case 16: return many_caches(p.C) ? launch_cfg<Cfg16Many>(p, maps, pdl, stream) : launch_cfg<Cfg16>(p, maps, pdl, stream);
    case 32: return launch_cfg<Cfg32>(p, maps, pdl, stream);
    case 48: return launch_cfg<Cfg48>(p, maps, pdl, stream);
    case 64: return launch_cfg<Cfg64>(p, maps, pdl, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace kvshot
