// merge_append.cu -- the two small kernels of the hot path:
//   * merge:  log-sum-exp merge of the pieces of units that straddled CTAs
//             (softmax over a union of disjoint key sets: lse = log sum_s e^lse_s,
//              out = sum_s e^(lse_s - lse) out_s);
//   * append: RoPE on the drafter's new q and k, then the store of k / v into
//             the draft slots (App. B: draft positions j > t take the drafter's
//             own K/V; Sec. 3.2: RoPE re-applied to drafted keys).
#include <algorithm>

#include "kvshot_attn_common.cuh"

namespace kvshot {
namespace {

using namespace dev;

constexpr int kMergeThreads = 256;
constexpr int kMergeRows = kMergeThreads / 32;  // rows per CTA, one warp per row

// Workspace slot of the piece computed by CTA b is u + b.  One warp per row
// of a unit.  Launched behind the attention kernel with programmatic stream
// serialization, so its CTAs start as the attention CTAs leave.  Each warp
// first rebuilds the attention kernel's plan from the inputs alone (lengths ->
// tiles per unit -> the unit's tile range -> the CTAs that held it): rows of
// units that lived in one CTA leave at once, and the others only then wait
// for the attention grid, with one or a few rounds of loads left: every piece's
// lse (lane k: piece b0 + k) together with the first kMergeBatch pieces' outputs
// (lane: 4 dims; kMergeBatch divides 32), and further pieces a batch at a time.
// The warps take the rows of all units one after another, whatever a unit's rows are (in CTAs of 8 rows of
// one unit, padded to the unit's 16, 64 caches of 4 rows took four times the CTAs: step 1562 -> 1532 us).
// Two forms.  Batches of 16, two CTAs per SM: for the few rows of a small call, each in
// many pieces.  (One piece after another behind the first two, each waiting for its load,
// the calls of a single cache took 2 us longer: 11 pieces, attention and merge 9.8 -> 7.9 us
// in batches of 8, 7.6 of 16; 19 pieces 23.6 us, 22.0, 20.1; of 32 19.7 us.)  Batches of
// 2 in 40 registers, six CTAs per SM: for calls of more CTAs than two per SM, whose units are
// in few pieces and whose waves of CTAs are what costs (16 caches, against batches of 16: 128 rows
// of 32768 tokens 376 -> 369 us per call, 256 rows of 4096 tokens, nothing split, 75.4 -> 73.9,
// with an fp8 cache 185 -> 174; batches of 4 the same, of 8 in four CTAs per SM 1 to 2 us more).
template <int kMergeBatch, int kCtasPerSm>
__global__ void __launch_bounds__(kMergeThreads, kCtasPerSm) merge_kernel(const __grid_constant__ AttnParams p) {
  const uint32_t unit_rows = min(p.rows_per_unit, p.rows_total), row = blockIdx.x * kMergeRows + (threadIdx.x >> 5);
  const int u = row / unit_rows, r = row - u * unit_rows;
  const int lane = threadIdx.x & 31;
  // Rows of unsplit units leave without waiting for the attention grid, so CTA 0 waits for it in any case:
  // a kernel that depends on this grid alone (the next append) then comes after the attention too.
  if (blockIdx.x == 0) wait_for_prerequisite_grid();
  if (threadIdx.x == 0) allow_dependent_launch();
  const int HR = p.hkv * p.row_blocks;
  const int c = u / HR, hr = u - c * HR;
  const int h = hr / p.row_blocks, rb = hr - h * p.row_blocks;
  const int rr = rb * p.rows_per_unit + r;
  if (u >= p.C * HR || rr >= p.rows_total) return;
  const int shift = __ffs(p.prefix_tile) - 1;  // a power of two
  auto tiles = [&](int len) { return ((len + p.prefix_tile - 1) >> shift) + p.draft_tiles; };
  int b0, b1;  // the CTAs that held the unit
  if (p.unit_ctas > 0) {
    const UnitCut cut = unit_cut(p.unit_ctas, tiles(clamp_len(p, 0)));
    b0 = hr * cut.per;
    b1 = b0 + cut.per - 1;
  } else {
    // First tile of cache c and the total (the prefix sums of build_plan): summed per lane, then over the warp once
    // (a reduction per 32 caches and a division per length were 14 of the 88 us of a call of 220 short caches).
    int below = 0, all = 0;
    for (int cc = lane; cc < p.C; cc += 32) {
      const int utc = tiles(clamp_len(p, cc));
      below += cc < c ? utc : 0;
      all += utc;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      below += __shfl_xor_sync(0xffffffffu, below, o);
      all += __shfl_xor_sync(0xffffffffu, all, o);
    }
    const int cbase = below * HR, total = all * HR, ut = tiles(clamp_len(p, c));
    const int gs = cbase + hr * ut;
    const int tpc = tiles_per_cta(total, p.num_ctas);
    b0 = gs / tpc;
    b1 = (gs + ut - 1) / tpc;
  }
  if (b0 == b1) return;  // the unit lived in one CTA, which wrote the output itself
  wait_for_prerequisite_grid();
  const int np = b1 - b0 + 1;
  const int nl = rr / p.G, g = rr - nl * p.G;
  const size_t orow = (static_cast<size_t>(c) * p.Nq + nl) * p.hq + h * p.G + g;
  const size_t row0 = static_cast<size_t>(u + b0) * p.rows_per_unit + r;  // piece k's row: row0 + k * rows
  float ls = lane < np ? p.ws_lse[row0 + static_cast<size_t>(lane) * p.rows_per_unit] : -INFINITY;
  const int ostride = p.rows_per_unit * (kHeadDim / 4);  // float4s from one piece's row to the next's
  const float4* op = reinterpret_cast<const float4*>(p.ws_o + row0 * kHeadDim) + lane;
  float4 x[kMergeBatch];  // the first pieces' outputs, loaded together with the lse (np >= 2 here)
#pragma unroll
  for (int k = 0; k < kMergeBatch; ++k) x[k] = k < np ? op[static_cast<size_t>(k) * ostride] : make_float4(0, 0, 0, 0);
  float M = ls;
  for (int k = lane + 32; k < np; k += 32)  // more than 32 pieces: fold the rest into this lane's max
    M = fmaxf(M, p.ws_lse[row0 + static_cast<size_t>(k) * p.rows_per_unit]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
  float Lsum = 0.f;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  if (M != -INFINITY) {
    float wl = ls == -INFINITY ? 0.f : exp2f(ls - M);  // lane k: piece k's weight, 32 pieces at a time
    for (int k0 = 0; k0 < np; k0 += kMergeBatch) {
      if (k0 > 0) {
        if ((k0 & 31) == 0) {
          const float lk = k0 + lane < np ? p.ws_lse[row0 + static_cast<size_t>(k0 + lane) * p.rows_per_unit] : -INFINITY;
          wl = lk == -INFINITY ? 0.f : exp2f(lk - M);
        }
#pragma unroll
        for (int k = 0; k < kMergeBatch; ++k)
          x[k] = k0 + k < np ? op[static_cast<size_t>(k0 + k) * ostride] : make_float4(0, 0, 0, 0);
      }
#pragma unroll
      for (int k = 0; k < kMergeBatch; ++k) {
        const float w = __shfl_sync(0xffffffffu, wl, (k0 + k) & 31);  // 0 past the last piece
        Lsum += w;
        acc.x += w * x[k].x;
        acc.y += w * x[k].y;
        acc.z += w * x[k].z;
        acc.w += w * x[k].w;
      }
    }
  }
  const float inv = Lsum > 0.f ? 1.f / Lsum : 0.f;
  uint2 packed;
  packed.x = pack_bf16x2(acc.x * inv, acc.y * inv);
  packed.y = pack_bf16x2(acc.z * inv, acc.w * inv);
  *reinterpret_cast<uint2*>(p.out + orow * kHeadDim + 4 * lane) = packed;
  if (lane == 0) p.lse[orow] = Lsum > 0.f ? (M + log2f(Lsum)) * 0.69314718055994531f : -INFINITY;
}

constexpr int kAppendThreads = 128;
// A node is shared out over up to kAppendSplits CTAs while the grid stays within kAppendCtas; from twice as many
// nodes, a CTA takes kAppendGroup.  (Within 256 CTAs: 192 nodes 4.5 us, 1024 nodes 14.1 us; 512: 4.6 and 12.4 us;
// 1024 nodes in CTAs of 4 13.7, of 1 10.8 us alone but 0.7 us slower with the attention behind them.)
constexpr int kAppendCtas = 512;
constexpr int kAppendSplits = 4;
constexpr int kAppendGroup = 2;
constexpr int kNormSplitNodes = 700;
constexpr int kNormOverlapNodes = 384;

__device__ __noinline__ void sincos_far(double theta, double* sn, double* cs) { sincos(theta, sn, cs); }

// An unevaluated sum of two fp32 values, |l| <= half an ulp of h.
struct Pair {
  float h, l;
};
__host__ __device__ constexpr Pair pair_of(double x) {
  return Pair{static_cast<float>(x), static_cast<float>(x - static_cast<double>(static_cast<float>(x)))};
}
// a + b for |a.h| >= |b.h| (or a of larger exponent), to ~2^-46 of the larger.
__device__ __forceinline__ Pair pair_add(Pair a, Pair b) {
  const float s = __fadd_rn(a.h, b.h);
  const float e = __fadd_rn(__fadd_rn(b.h, -__fadd_rn(s, -a.h)), __fadd_rn(a.l, b.l));
  const float h = __fadd_rn(s, e);
  return Pair{h, __fadd_rn(e, -__fadd_rn(h, -s))};
}
__device__ __forceinline__ Pair pair_mul(Pair a, Pair b) {
  const float p = __fmul_rn(a.h, b.h);
  return Pair{p, fmaf(a.h, b.l, fmaf(a.l, b.h, fmaf(a.h, b.h, -p)))};
}

// sin and cos of theta as pairs, to 2^-40 absolute: Cody-Waite reduction to [-pi/4, pi/4] in fp64 by two fused
// steps (pi/2 as an fp64 and its remainder; below 2^40 each step's only error is the rounding of its small
// result), then the Taylor polynomials with their last coefficients in fp32 and the others in fp32 pairs.  An SM
// executes two fp64 lanes per clock and 128 fp32 ones: the angles of a node take 9 fp64 operations per
// frequency, where fp64 polynomials take 31 (4.9 of the 14.6 us of a 1024-node append) and the library more.
__device__ __forceinline__ void sincos_pair(double theta, Pair* sn, Pair* cs) {
  if (!(fabs(theta) < 0x1p40)) {
    double s, c;
    sincos_far(theta, &s, &c);
    *sn = Pair{static_cast<float>(s), static_cast<float>(s - static_cast<double>(static_cast<float>(s)))};
    *cs = Pair{static_cast<float>(c), static_cast<float>(c - static_cast<double>(static_cast<float>(c)))};
    return;
  }
  const double n = rint(theta * 0.63661977236758134308);
  double rd = fma(-n, 1.5707963267948965580, theta);
  rd = fma(-n, 6.1232339957367658860e-17, rd);
  const float rh = static_cast<float>(rd);
  const Pair r{rh, static_cast<float>(rd - static_cast<double>(rh))};
  const int q = static_cast<int>(static_cast<long long>(n) & 3);
  const Pair z = pair_mul(r, r);
  constexpr Pair s1 = pair_of(-1.0 / 6.0), s2 = pair_of(1.0 / 120.0), s3 = pair_of(-1.0 / 5040.0);
  const float s4 = fmaf(z.h, fmaf(z.h, 1.6059044e-10f, -2.5052108e-8f), 2.7557319e-6f);  // 1/9!, -1/11!, 1/13!
  Pair s = pair_add(s3, Pair{z.h * s4, 0.f});
  s = pair_add(s2, pair_mul(z, s));
  s = pair_add(s1, pair_mul(z, s));
  s = pair_add(r, pair_mul(pair_mul(r, z), s));
  constexpr Pair c1{-0.5f, 0.f}, c2 = pair_of(1.0 / 24.0), c3 = pair_of(-1.0 / 720.0), one{1.f, 0.f};
  const float c4 = fmaf(z.h, fmaf(z.h, fmaf(z.h, -1.1470746e-11f, 2.0876757e-9f), -2.7557319e-7f), 2.4801587e-5f);
  Pair c = pair_add(c3, Pair{z.h * c4, 0.f});
  c = pair_add(c2, pair_mul(z, c));
  c = pair_add(c1, pair_mul(z, c));
  c = pair_add(one, pair_mul(z, c));
  const Pair a = (q & 1) ? c : s, b = (q & 1) ? s : c;
  *sn = (q & 2) ? Pair{-a.h, -a.l} : a;
  *cs = (q == 1 || q == 2) ? Pair{-b.h, -b.l} : b;
}

// The append kernels are launched with programmatic stream serialization: their CTAs may be placed while the
// preceding kernel still runs, and touch memory only once it has completed.  A following attention call
// launched with KVSHOT_OVERLAP_PREVIOUS may start its prologue from here on: everything before this kernel
// is complete by now.
__device__ __forceinline__ void begin_after_previous() {
  wait_for_prerequisite_grid();
  if (threadIdx.x == 0) allow_dependent_launch();
}

// cos (or sin) of an angle as two fp32 values: the first with 16 significant bits, so that its product with a
// bf16 is exact, and the rest.
__device__ __forceinline__ float2 split16(Pair x) {
  const float hi = __uint_as_float(__float_as_uint(x.h) & 0xffffff00u);
  return make_float2(hi, __fadd_rn(__fadd_rn(x.h, -hi), x.l));
}
// Place of frequency j in a table of float4: eight lanes that read entries 8 apart hit all banks once.
__device__ __forceinline__ constexpr int angle_at(int j) { return j + (j >> 3); }

// The bits of the bf16 nearest to a * cos + sgn * b * sin, evaluated in fp64 and rounded once.
__device__ __noinline__ uint32_t rope_bf16_fp64(float a, float b, double theta, float sgn) {
  double s, c;
  sincos_far(theta, &s, &c);
  return __bfloat16_as_ushort(__double2bfloat16(static_cast<double>(a) * c + sgn * (static_cast<double>(b) * s)));
}

// One rotated component of RoPE, x' = a * cos + sgn * b * sin: the exact value is r + res to 2^-37 (|a| + |b|).
// a, b are bf16, so a c.x and b s.x are exact in fp32; u + e is their exact sum (two-sum).
struct Rotated {
  float r, res;
};
__device__ __forceinline__ Rotated rotate(float a, float b, float2 c, float2 s, float sgn) {
  const float p = a * c.x, q = sgn * (b * s.x);
  const float u = __fadd_rn(p, q);
  const float bb = __fadd_rn(u, -p);
  const float e = __fadd_rn(__fadd_rn(p, -__fadd_rn(u, -bb)), __fadd_rn(q, -bb));
  const float v = __fadd_rn(e, fmaf(a, c.y, sgn * (b * s.y)));
  const float r = __fadd_rn(u, v);
  return Rotated{r, __fadd_rn(v, -__fadd_rn(r, -u))};
}

// With |r| >= 2^-13 (|a| + |b|) that error is under one fp32 ulp of r, so unless r's low 16 bits are within
// two of the rounding midpoint 0x8000, r rounds to the same bf16 as the exact value: (bits(r) + 0x8000) >> 16.
__device__ __forceinline__ bool rounds_alike(float r, float least) {
  return ((__float_as_uint(r) + 0x8002u) & 0xffffu) > 4u && fabsf(r) >= least;
}

// The bf16 of a component that does not (one in 5,000).  d is its distance past the midpoint above the truncated
// bf16, so |d| beyond the error decides the rounding.  Only the rest (one in millions), values so small that the
// products are not exact, infinities and NaN are evaluated in fp64.
__device__ __noinline__ uint32_t rope_bf16_near(float a, float b, float4 cs, float sgn, double theta) {
  const float2 c = make_float2(cs.x, cs.y), s = make_float2(cs.z, cs.w);
  const Rotated x = rotate(a, b, c, s, sgn);
  const float m = fabsf(a) + fabsf(b);
  if (m == 0.f) return __float_as_uint(__fadd_rn(a * c.x, sgn * (b * s.x))) >> 16;  // a zero, signed as in fp64
  const uint32_t w = __float_as_uint(x.r), e = (w >> 23) & 0xffu;
  if (e > 60u && e < 255u) {
    const float ulp = __uint_as_float((e - 23u) << 23);  // fp32 spacing at r
    const float d = fmaf(static_cast<float>(static_cast<int>(w & 0xffffu) - 0x8000), ulp, x.r < 0.f ? -x.res : x.res);
    if (fabsf(d) > 0x1p-37f * m) return (w >> 16) + (d > 0.f ? 1u : 0u);
  }
  return rope_bf16_fp64(a, b, theta, sgn);
}

// Grid (group of a.group consecutive nodes, split): a node's heads and V chunks are shared out over gridDim.y
// CTAs when there are few nodes; a CTA takes several nodes when there are many, and forms the angles again only
// where the position changes (the nodes of one tree level share theirs).
struct AppendNode {
  int c, i;
  size_t row;  // (cache, node)
};
__device__ __forceinline__ AppendNode append_node(const AppendParams& a, int node) {
  AppendNode t;
  t.c = node / a.n_new;
  t.i = node - t.c * a.n_new;
  t.row = static_cast<size_t>(node);
  return t;
}
__device__ __forceinline__ int share(int n, int k) {  // first of the k-th CTA's items of n
  return static_cast<int>(static_cast<unsigned>(n) * static_cast<unsigned>(k) / gridDim.y);
}
// V: plain copy into the draft slot.
__device__ __forceinline__ void append_v(const AppendParams& a, const AppendNode& t) {
  const int w1 = share(a.hkv * 16, blockIdx.y + 1);
  for (int w = share(a.hkv * 16, blockIdx.y) + threadIdx.x; w < w1; w += kAppendThreads) {
    const int kh = w >> 4, ch = w & 15;
    const uint4 v = *reinterpret_cast<const uint4*>(a.v_in + (t.row * a.hkv + kh) * kHeadDim + ch * 8);
    *reinterpret_cast<uint4*>(a.draft_v + ((static_cast<size_t>(t.c) * a.hkv + kh) * a.n_max + a.n0 + t.i) * kHeadDim +
                              ch * 8) = v;
  }
}

// Work item = (head, 16-byte chunk j0 of the first half): it rotates dims j0..j0+7 together with their
// partners +64.  Latency bound at a few nodes (a thread's first loads go out before the angles are formed, the
// rotations of an item have no branch between them), and by the rotation's instructions at many.  Per call, back
// to back in a graph: 1 node 2.4 us, 16 x 12 nodes 4.5 us, 16 x 64 nodes 12.4 us; with fp64 angles read per
// component, converted there, and an error bound per component: 6.4, 7.1 and 20.8 us.
__global__ void __launch_bounds__(kAppendThreads, 5) append_kernel(const __grid_constant__ AppendParams a) {
  begin_after_previous();
  __shared__ float4 angles[angle_at(kHeadDim / 2)];  // cos and sin, split16
  const int items = (a.hq + a.hkv) * 8, w0 = share(items, blockIdx.y), w1 = share(items, blockIdx.y + 1);
  const int node0 = blockIdx.x * a.group, node1 = min(a.C * a.n_new, node0 + a.group);
  int had = -1;  // the position whose angles are in shared memory
  for (int node = node0; node < node1; ++node) {
    const AppendNode t = append_node(a, node);
    const int pos = a.positions[t.row];
    auto source = [&](int w) {
      const int head = w >> 3;
      return (head < a.hq ? a.q_in + (t.row * a.hq + head) * kHeadDim
                          : a.k_in + (t.row * a.hkv + head - a.hq) * kHeadDim) + (w & 7) * 8;
    };
    uint4 lo = make_uint4(0, 0, 0, 0), hi = lo;
    int w = w0 + threadIdx.x;
    if (w < w1) {
      const __nv_bfloat16* src = source(w);
      lo = *reinterpret_cast<const uint4*>(src);
      hi = *reinterpret_cast<const uint4*>(src + 64);
    }
    append_v(a, t);
    if (node == node0 || pos != had) {  // the same for the whole CTA
      if (node != node0) __syncthreads();
      if (threadIdx.x < kHeadDim / 2) {
        Pair sn, cs;
        sincos_pair(static_cast<double>(pos) * a.inv_freq[threadIdx.x], &sn, &cs);
        const float2 c = split16(cs), s = split16(sn);
        angles[angle_at(threadIdx.x)] = make_float4(c.x, c.y, s.x, s.y);
      }
      __syncthreads();
      had = pos;
    }
    while (w < w1) {
      const int head = w >> 3, j0 = (w & 7) * 8;
      __nv_bfloat16* dst =
          head < a.hq ? a.q_out + (t.row * a.hq + head) * kHeadDim
                      : a.draft_k + ((static_cast<size_t>(t.c) * a.hkv + head - a.hq) * a.n_max + a.n0 + t.i) * kHeadDim;
      const uint32_t wl[4] = {lo.x, lo.y, lo.z, lo.w}, wh[4] = {hi.x, hi.y, hi.z, hi.w};
      w += kAppendThreads;
      if (w < w1) {  // the next item
        const __nv_bfloat16* src = source(w);
        lo = *reinterpret_cast<const uint4*>(src);
        hi = *reinterpret_cast<const uint4*>(src + 64);
      }
      const float4* table = angles + angle_at(j0);  // j0 is a multiple of 8
      // All sixteen components at once, without branches; the few that need a closer look are done again.
      uint32_t ol[4], oh[4], near = 0;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const float x = k & 1 ? bf16_hi(wl[k >> 1]) : bf16_lo(wl[k >> 1]);
        const float y = k & 1 ? bf16_hi(wh[k >> 1]) : bf16_lo(wh[k >> 1]);
        const float4 cs = table[k];
        const float2 c = make_float2(cs.x, cs.y), s = make_float2(cs.z, cs.w);
        const float least = fmaxf((fabsf(x) + fabsf(y)) * 0x1p-13f, 0x1p-60f);
        const float rl = rotate(x, y, c, s, -1.f).r, rh = rotate(y, x, c, s, 1.f).r;
        near |= (rounds_alike(rl, least) ? 0u : 1u << k) | (rounds_alike(rh, least) ? 0u : 256u << k);
        const uint32_t bl = __float_as_uint(rl) + 0x8000u, bh = __float_as_uint(rh) + 0x8000u;
        ol[k >> 1] = k & 1 ? __byte_perm(ol[k >> 1], bl, 0x7632) : bl;
        oh[k >> 1] = k & 1 ? __byte_perm(oh[k >> 1], bh, 0x7632) : bh;
      }
      if (near != 0) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const float x = k & 1 ? bf16_hi(wl[k >> 1]) : bf16_lo(wl[k >> 1]);
          const float y = k & 1 ? bf16_hi(wh[k >> 1]) : bf16_lo(wh[k >> 1]);
          const uint32_t into = k & 1 ? 0x5410u : 0x3254u;  // the new half word over the high or the low one
          const double theta = static_cast<double>(pos) * a.inv_freq[j0 + k];
          if (near >> k & 1u) ol[k >> 1] = __byte_perm(ol[k >> 1], rope_bf16_near(x, y, table[k], -1.f, theta), into);
          if (near >> (8 + k) & 1u) oh[k >> 1] = __byte_perm(oh[k >> 1], rope_bf16_near(y, x, table[k], 1.f, theta), into);
        }
      }
      *reinterpret_cast<uint4*>(dst + j0) = make_uint4(ol[0], ol[1], ol[2], ol[3]);
      *reinterpret_cast<uint4*>(dst + 64 + j0) = make_uint4(oh[0], oh[1], oh[2], oh[3]);
    }
  }
}

// QK-norm variant (Qwen3's per-head RMSNorm of q and k before RoPE): one warp per head, lane l
// holding dims 2l, 2l + 1 and their RoPE partners + 64.  x <- x / sqrt(mean(x^2) + eps) * w (w the
// head-dim weights), then the rotation; fp32 throughout, one rounding to bf16.  One node to a CTA, shared out over
// gridDim.y CTAs when there are few.  Latency bound, and a loop without loads ahead of it fits 32 registers, so sixteen
// CTAs to an SM hide it: per call, 768 nodes of 32 + 8 heads 11.2 -> 8.3 us, 1024 nodes of 64 + 8 heads 17.4 -> 13.0
// against the next head's loads, the weights' and V's ahead of the angles in 48 registers (9.3 and 15.8 us with fp64
// angles and a CTA per node).
__global__ void __launch_bounds__(kAppendThreads) append_qknorm_kernel(const __grid_constant__ AppendParams a) {
  begin_after_previous();
  __shared__ float s_cos[kHeadDim / 2], s_sin[kHeadDim / 2];
  const int heads = a.hq + a.hkv, h0 = share(heads, blockIdx.y), h1 = share(heads, blockIdx.y + 1);
  const int lane = threadIdx.x & 31, j = 2 * lane;
  const AppendNode t = append_node(a, blockIdx.x);
  const int pos = a.positions[t.row];
  if (threadIdx.x < kHeadDim / 2) {
    Pair sn, cs;
    sincos_pair(static_cast<double>(pos) * a.inv_freq[threadIdx.x], &sn, &cs);
    s_cos[threadIdx.x] = cs.h + cs.l;
    s_sin[threadIdx.x] = sn.h + sn.l;
  }
  __syncthreads();
  for (int head = h0 + (threadIdx.x >> 5); head < h1; head += kAppendThreads / 32) {
    const bool query = head < a.hq;
    const __nv_bfloat16* src = (query ? a.q_in + (t.row * a.hq + head) * kHeadDim : a.k_in + (t.row * a.hkv + head - a.hq) * kHeadDim) + j;
    __nv_bfloat16* dst =
        query ? a.q_out + (t.row * a.hq + head) * kHeadDim
              : a.draft_k + ((static_cast<size_t>(t.c) * a.hkv + head - a.hq) * a.n_max + a.n0 + t.i) * kHeadDim;
    const __nv_bfloat16* w = query ? a.q_norm_w : a.k_norm_w;
    const uint32_t lo = *reinterpret_cast<const uint32_t*>(src), hi = *reinterpret_cast<const uint32_t*>(src + 64);
    const uint32_t wl = *reinterpret_cast<const uint32_t*>(w + j);
    const uint32_t wh = *reinterpret_cast<const uint32_t*>(w + 64 + j);
    float x[4] = {bf16_lo(lo), bf16_hi(lo), bf16_lo(hi), bf16_hi(hi)};
    float ss = x[0] * x[0] + x[1] * x[1] + x[2] * x[2] + x[3] * x[3];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    const float r = rsqrtf(ss * (1.f / kHeadDim) + a.eps);
    x[0] *= r * bf16_lo(wl);
    x[1] *= r * bf16_hi(wl);
    x[2] *= r * bf16_lo(wh);
    x[3] *= r * bf16_hi(wh);
    const float c0 = s_cos[j], s0 = s_sin[j], c1 = s_cos[j + 1], s1 = s_sin[j + 1];
    const float y0 = x[0] * c0 - x[2] * s0, y1 = x[1] * c1 - x[3] * s1;   // dims j, j + 1
    const float z0 = x[2] * c0 + x[0] * s0, z1 = x[3] * c1 + x[1] * s1;   // dims j + 64, j + 65
    *reinterpret_cast<uint32_t*>(dst + j) = pack_bf16x2(y0, y1);
    *reinterpret_cast<uint32_t*>(dst + 64 + j) = pack_bf16x2(z0, z1);
  }
  append_v(a, t);
}

}  // namespace

cudaError_t launch_merge(const AttnParams& p, int sms, cudaStream_t stream) {
  const int64_t rows = static_cast<int64_t>(p.C) * p.hkv * p.row_blocks * std::min(p.rows_per_unit, p.rows_total);
  const int blocks = static_cast<int>((rows + kMergeRows - 1) / kMergeRows);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(kMergeThreads);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  // (One cache whose units are in two pieces at most fills no batch of 16: 300 tokens, 4 rows 11.0 -> 10.9 us per call.)
  const bool two_pieces = p.unit_ctas == 1 || p.unit_ctas == 2;
  return cudaLaunchKernelEx(&cfg, blocks <= 2 * sms && !two_pieces ? merge_kernel<16, 2> : merge_kernel<2, 6>, p);
}

cudaError_t launch_append(AppendParams a, cudaStream_t stream) {
  const int nodes = a.C * a.n_new;
  const bool norm = a.q_norm_w != nullptr;
  int splits = std::min(kAppendSplits, kAppendCtas / nodes);
  // With QK-norm the angles weigh less: two CTAs to a node up to 700 nodes (steps of 64 caches with 7 nodes a level 133.9
  // -> 130.8 us; beyond, 768 nodes alone 9.0 against 8.3), and one node to a CTA at any number.
  if (norm) splits = std::max(splits, std::min(2, kNormSplitNodes / nodes * 2));
  splits = std::max(1, splits);
  a.group = norm ? 1 : std::max(1, std::min(kAppendGroup, nodes / kAppendCtas));
  // Launched behind its predecessor; with QK-norm only up to 384 nodes, from where the CTAs that wait cost more than the
  // launch (steps of 64 caches with 7 nodes a level 134.9 us, 130.8 without; 1 cache with 4 nodes a level 38.0, 36.7 with).
  return launch_maybe_pdl(norm ? append_qknorm_kernel : append_kernel,
                          dim3((nodes + a.group - 1) / a.group, splits), dim3(kAppendThreads), 0,
                          !norm || nodes <= kNormOverlapNodes, stream, a);
}

}  // namespace kvshot
