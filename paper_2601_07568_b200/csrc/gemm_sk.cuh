// The matmuls of a decode forward over up to some hundred rows (those that the chain does not take): weights as the MMA's
// row operand on CTA pairs, K ranges cut so that every SM streams the same number of weight bytes, and several matmuls
// that follow one another in one persistent launch.
//
//   D[n, m] = sum_k W[n, k] X[m, k]: a pair of CTAs (cta_group::2, M = 256) owns 256 rows of W (each CTA one
//   pre-swizzled 128 x 64 block per K slab) against up to 256 rows of X (each CTA stages half of them).
//
// Why.  Up to a few hundred rows such a matmul is bound by weight streaming, and 256 x 256 tiles leave most of the
// chip idle: 48 tiles (QKV), 16 (O-proj, down) or 96 (gate/up of the 8B shape, 1.3 waves) for 74 pairs.  Here the
// tiles that do not fill a wave are cut along K: their (tile, slab) units are dealt to all pairs in equal contiguous
// ranges, a range touches at most two tiles, and the partial accumulators meet in global memory (L2).  What a pair
// moves per slab is 16 KB of weights and half of X per CTA, where a lone CTA would stage all of X.
//
// Reduction.  A CTA leaves its accumulators of a cut tile in global memory (L2) as [row of X][128 columns] fp32, gives the
// tensor memory back, raises the tile's counter (release), waits until all contributors have, and finishes its share of
// the rows: the partials added in contributor order (fixed order: the same bits on every run).  All CTAs of the launch
// are resident at once (the host sizes the grid by the occupancy of clusters) and every range ends at about the same
// time, so the wait is short.  It is bounded like every other one.  Cut tiles come first, and the whole ones behind them
// hide the exchange (SkPlan).
//
// Epilogue.  Whole gate/up tiles are finished from tensor memory (swiglu_tile); whole tiles of the other matmuls go through
// global memory like a partial.  From there a warp finishes whole rows of X, four columns a lane, three or four rows at a
// time: all that they need (partials, residual values, cosines) is requested at once, because behind the last MMA of a matmul every trip to L2 is
// on the critical path and takes one to two microseconds beside the next matmul's weights.  Row factors of the folded
// RMSNorm are worked out while the MMAs run, everything that needs an integer division before the launch's dependencies
// are there.  (Forms that were slower, microseconds for O-proj, gate/up, down and QKV of the 8B shape at 128 / 256 rows:
// an output column a lane and sixteen rows unrolled 148 / 190, with the row factors fetched where they are used 108 /
// 139.  With whole tiles in front 107 / 139, as it is 102 / 128, CUDA events around the launch.  Their weights alone take 67
// at the measured copy bandwidth; the rest is mostly the exchanges of the cut tiles, where no whole tile follows to hide
// them (O-proj, down, QKV).  Holding the next matmul's weights back until the exchange is over costs 3 to 6.)
//
// Borders.  A launch runs up to four matmuls in order (O-proj, gate/up, down, the next layer's QKV or the LM head); the next one
// reads what the one before wrote on other SMs, so there is a grid-wide counter between them, as in the chain
// kernel.  The thread that requests weights does not wait at a border: the ring fills with the next matmul's weights
// while the border's dependency resolves.
//
// Per CTA, 480 threads: warp 0 requests weights, warp 1 issues MMAs (leader only) and owns tensor memory, warp 2
// requests rows of X, warps 3-14 epilogue (three per lane quadrant).
#pragma once
#include "chain.cuh"
#include "gemm_pair.cuh"

namespace d3 {
namespace tc {

constexpr int SK_EPI_WARPS = 12;  // three per lane quadrant
constexpr int SK_EPI_THREADS = SK_EPI_WARPS * 32;
constexpr int SK_THREADS = 96 + SK_EPI_THREADS;
constexpr int SK_MAX_OPS = 4;
constexpr int SK_MAX_ROWS = 1024;  // rows of X (the row table lives in shared memory)
constexpr uint32_t SK_W_BYTES = 128u * 128u;  // one weight block

struct SkOp {
  EpiParams ep;
  int epi, N, k_chunks;
  int n_tiles;      // N / 256
  int tiles;        // n_tiles x tiles of tok_n rows of X
  int full_tiles;   // tiles [0, full_tiles) are computed whole, dealt round-robin; the others are cut along K
  unsigned int* part_count;    // [tiles - full_tiles][2] partials written, zero before the launch
  __nv_bfloat16 *k_cache, *v_cache;  // EPI_QKV: this layer's planes
};

struct SkParams {
  CUtensorMap x[SK_MAX_OPS];  // rows of X as [M, K], boxes of tok_n / 2 rows (128-byte swizzle)
  CUtensorMap w[SK_MAX_OPS];  // weight blocks as [N / 128 * k_chunks * 128, 64], boxes of 128 rows, no swizzle
  SkOp op[SK_MAX_OPS];
  int n_ops;
  int M;
  int tok_n, tok_tiles;  // rows of X per tile (a multiple of 32, at most 256) and tiles of them
  int stages;
  float* partial;         // [pairs][3: first cut tile, second, whole tile][2 CTAs][tok_n][128] fp32
  unsigned int* border;   // [n_ops] CTAs that have finished the matmul, zero before the launch
  uint32_t* error_word;
  const float* rope_cos;  // [max_seq][64]
  const float* rope_sin;
  const int* pos_base;
  const int* n_valid;
  int rows_per_seq;
  int rope_rows;          // one of the matmuls is EPI_QKV
  int n_q_heads, n_kv_heads, max_seq;
};

__device__ __forceinline__ void tmem_ld_32x16(uint32_t taddr, float (&v)[16]) {
  uint32_t* r = reinterpret_cast<uint32_t*>(v);
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}

// One segment of a pair's share of a matmul: slabs [k0, k0 + n_k) of a tile.
struct SkSeg {
  int m_t, n_t, k0, n_k;
};
// A segment of a cut tile.  The pairs [first, first + count) share the tile and finish it together.  Where many share one,
// those whose ranges end in it do, an equal share of the rows of X each, so that a pair finishes one tile only (a range
// is no longer than a tile: some range ends in every tile).  Where two or three share one, that would leave all rows of
// some tiles to one pair, and a pair's share of the rows is its share of the slabs.
struct SkCut {
  SkSeg g;
  int index;            // among the cut tiles
  int first, count;
  int first_slot;       // which of its two partials the first pair left in this tile
  int t0, t1;           // rows of X this pair finishes
};
// A pair's share of a matmul: a range of (tile, slab) units that touches up to two cut tiles, then n_whole whole tiles, whose
// MMAs hide the exchange of the cut ones.  Of two cut tiles the one with fewer slabs comes first: its partial goes out
// under the other one's MMAs.  (With the whole tiles in front, and finished by way of L2, every matmul that has both ended in
// an exchange: 3333 against 3270 us for a 32-row step of the 8B shape, 5009 against 4744 for 256 rows of the 7B one.)
// Worked out once per launch, in the prologue: a dozen integer divisions in a row have no place behind a border.
struct SkPlan {
  int n_whole, n_cut;
  int swap;  // the second cut tile comes first
  SkCut cut[2];
};
__device__ inline void sk_plan(const SkOp& o, int pair, int n_pairs, int tok_tiles, int tok_n, SkPlan& s) {
  s.n_whole = pair < o.full_tiles ? (o.full_tiles - pair + n_pairs - 1) / n_pairs : 0;
  const int KC = o.k_chunks, U = (o.tiles - o.full_tiles) * KC;
  const int u0 = U * pair / n_pairs, u1 = U * (pair + 1) / n_pairs;
  s.n_cut = u1 > u0 ? (u1 - 1) / KC - u0 / KC + 1 : 0;
  for (int i = 0; i < s.n_cut; ++i) {
    SkCut& c = s.cut[i];
    c.index = u0 / KC + i;
    const int begin = c.index * KC, end = begin + KC;
    pair_tile_mn(o.full_tiles + c.index, tok_tiles, o.n_tiles, c.g.m_t, c.g.n_t);
    c.g.k0 = max(u0 - begin, 0);
    c.g.n_k = min(u1 - begin, KC) - c.g.k0;
    c.first = ((begin + 1) * n_pairs - 1) / U;
    const int last = (end * n_pairs - 1) / U;
    c.count = last - c.first + 1;
    c.first_slot = U * c.first / n_pairs < begin ? 1 : 0;
    if (2 * U >= KC * n_pairs) {
      c.t0 = tok_n * c.g.k0 / KC;
      c.t1 = tok_n * (c.g.k0 + c.g.n_k) / KC;
    } else {
      const int fin = U * (last + 1) / n_pairs > end ? c.count - 1 : c.count, fi = pair - c.first;
      c.t0 = fi < fin ? tok_n * fi / fin : 0;
      c.t1 = fi < fin ? tok_n * (fi + 1) / fin : 0;
    }
  }
  s.swap = s.n_cut == 2 && s.cut[1].g.n_k < s.cut[0].g.n_k ? 1 : 0;
}
__device__ __forceinline__ SkSeg sk_seg(const SkOp& o, const SkPlan& pl, int i, int pair, int n_pairs, int tok_tiles) {
  if (i < pl.n_cut) return pl.cut[i ^ pl.swap].g;
  SkSeg g;
  pair_tile_mn(pair + (i - pl.n_cut) * n_pairs, tok_tiles, o.n_tiles, g.m_t, g.n_t);
  g.k0 = 0;
  g.n_k = o.k_chunks;
  return g;
}

inline size_t gemm_sk_smem_bytes(int tok_n, int stages) {
  return 1024 + static_cast<size_t>(stages) * (SK_W_BYTES + static_cast<size_t>(tok_n) * 64) + (2 * stages + 4) * 8 + 64 + SK_MAX_OPS * sizeof(SkPlan) + SK_MAX_ROWS * (sizeof(int2) + sizeof(float));
}

// Barrier over the epilogue threads that also tells every one of them whether all are still in order.
__device__ __forceinline__ bool sk_all(bool ok) {
  uint32_t r;
  asm volatile(
      "{\n"
      ".reg .pred p, q;\n"
      "setp.ne.u32 q, %1, 0;\n"
      "barrier.red.and.pred p, 1, %2, q;\n"
      "selp.u32 %0, 1, 0, p;\n"
      "}\n"
      : "=r"(r)
      : "r"(static_cast<uint32_t>(ok)), "n"(SK_EPI_THREADS)
      : "memory");
  return r != 0;
}

// Hands a tensor-memory buffer back to the leader's MMA thread: the loads from it have completed, and nothing else has to
// be visible to that thread, so the arrival need not wait for this thread's stores to reach L2 (a release would).
__device__ __forceinline__ void sk_release_acc(uint64_t* bar) {
  const uint32_t remote = map_to_cta(smem_u32(bar), 0);
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(remote) : "memory");
}

// Rows of a tile to finish.
struct SkFinish {
  int m0, n0;          // first of these rows of X, first of this CTA's 128 columns
  int rows;
  const float* part;   // first contributor's partial of the first row
  int count;           // contributors
  int step0, step;     // floats from the first contributor's partial to the second's, and from there on
};

// Sums over the 32 lanes of 16 values a lane: the lanes halve the values they carry at each exchange; the sum of value
// (lane >> 1) ends up in a[0].
__device__ __forceinline__ void sk_lane_sums16(float (&a)[16], int lane) {
#pragma unroll
  for (int w = 8; w >= 1; w >>= 1) {
    const bool up = (lane & (2 * w)) != 0;
#pragma unroll
    for (int j = 0; j < w; ++j) {
      const float send = up ? a[j] : a[j + w], keep = up ? a[j + w] : a[j];
      a[j] = keep + __shfl_xor_sync(0xffffffffu, send, 2 * w);
    }
  }
  a[0] += __shfl_xor_sync(0xffffffffu, a[0], 1);
}
// Row factors of the folded RMSNorm for rows m0 .. m0 + 15 into rs[0 .. 15] (rows from M on: whatever): a row's chunk
// sums over a warp's lanes, all rows' loads in flight at once.  (A tree of 32-bit sums where row_rstd has a chain: the last
// bits differ from the other kernels', as those of the K-cut sums do.)
__device__ __forceinline__ void sk_row_rstd16(const EpiParams& ep, int m0, int M, int lane, float* rs) {
  float a[16];
  const int chunks = ep.ssq_chunks;  // a multiple of 4
  const float* r = ep.ssq_in + static_cast<size_t>(m0) * chunks + lane * 4;
#pragma unroll
  for (int q = 0; q < 16; ++q) a[q] = 0.f;
#pragma unroll 1
  for (int i = lane * 4; i < chunks; i += 128, r += 128) {
    float4 v[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) v[q] = m0 + q < M ? __ldcg(reinterpret_cast<const float4*>(r + q * chunks)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int q = 0; q < 16; ++q) a[q] += (v[q].x + v[q].y) + (v[q].z + v[q].w);
  }
  sk_lane_sums16(a, lane);
  if ((lane & 1) == 0) rs[lane >> 1] = rsqrtf(a[0] * ep.inv_k + ep.rms_eps);
}

// LM head: softmax statistics of ROWS rows over this CTA's 128 columns, and with a temperature the largest perturbed logit
// (one Philox call covers a lane's four columns).  `l`: the logits.  The head as a launch of its own, in microseconds
// against a row to a thread on 128- or 256-row tiles: 158 against 197 at 32 rows of the 8B shape (weights alone 158), 253
// against 272 at 256 rows, 308 against 388 at 256 rows of the 7B shape.
template <int ROWS>
__device__ __forceinline__ void sk_stats(const SkParams& p, const SkOp& o, float4 (&l)[ROWS], const bool (&live)[ROWS], int m, int n, int lane) {
  const int gone = o.ep.mask_id - n;  // which of the lane's columns is the mask token, if any
  float mx[ROWS], z[ROWS], t[ROWS];
  int a[ROWS];
#pragma unroll
  for (int u = 0; u < ROWS; ++u) {
    float v[4] = {l[u].x, l[u].y, l[u].z, l[u].w};
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (q == gone) v[q] = -INFINITY;
    l[u] = make_float4(v[0], v[1], v[2], v[3]);
    mx[u] = fmaxf(fmaxf(v[0], v[1]), fmaxf(v[2], v[3]));
  }
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1)
#pragma unroll
    for (int u = 0; u < ROWS; ++u) mx[u] = fmaxf(mx[u], __shfl_xor_sync(0xffffffffu, mx[u], d));
#pragma unroll
  for (int u = 0; u < ROWS; ++u) {
    const float v[4] = {l[u].x, l[u].y, l[u].z, l[u].w};
    z[u] = t[u] = 0.f;
    a[u] = 0x7fffffff;
#pragma unroll
    for (int q = 3; q >= 0; --q) {
      if (q == gone) continue;
      const float d = v[q] == INFINITY ? 0.f : v[q] - mx[u], e = __expf(d);
      z[u] += e;
      t[u] += e * d;
      if (v[q] == mx[u]) a[u] = n + q;
    }
    a[u] = __reduce_min_sync(0xffffffffu, a[u]);
  }
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1)
#pragma unroll
    for (int u = 0; u < ROWS; ++u) {
      z[u] += __shfl_xor_sync(0xffffffffu, z[u], d);
      t[u] += __shfl_xor_sync(0xffffffffu, t[u], d);
    }
  const int tile = n >> 7;
#pragma unroll
  for (int u = 0; u < ROWS; ++u)
    if (live[u] && lane == 0)
      o.ep.stat_part[static_cast<size_t>(m + u * SK_EPI_WARPS) * o.ep.n_tiles + tile] = make_float4(mx[u], z[u], t[u], __int_as_float(a[u]));
  if (o.ep.sample_part == nullptr) return;
#pragma unroll 1
  for (int u = 0; u < ROWS; ++u) {
    float4 lu = l[0];
    bool alive = live[0];
#pragma unroll
    for (int q = 1; q < ROWS; ++q)
      if (q == u) { lu = l[q]; alive = live[q]; }
    if (!alive) continue;  // warp-uniform
    const int row = m + u * SK_EPI_WARPS;
    const SampleRow sr = sample_row(o.ep, row);
    const uint4 bits = philox4x32_10(make_uint4(static_cast<uint32_t>(n >> 2), sr.pos, sr.step, sr.seq), o.ep.seed_lo, o.ep.seed_hi);
    const uint32_t w[4] = {bits.x, bits.y, bits.z, bits.w};
    const float v[4] = {lu.x, lu.y, lu.z, lu.w};
    SampleStat sp = sample_empty();
#pragma unroll
    for (int q = 0; q < 4; ++q)  // product and sum rounded separately
      if (q != gone) sample_add(sp, __fadd_rn(v[q], __fmul_rn(o.ep.temperature, gumbel_from_bits(w[q]))), v[q], n + q);
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) {
      SampleStat other;
      other.pm = __shfl_xor_sync(0xffffffffu, sp.pm, d);
      other.la = __shfl_xor_sync(0xffffffffu, sp.la, d);
      other.pa = __shfl_xor_sync(0xffffffffu, sp.pa, d);
      sp = sample_merge(sp, other);
    }
    if (lane == 0) o.ep.sample_part[static_cast<size_t>(row) * o.ep.n_tiles + tile] = make_float4(sp.pm, sp.la, __int_as_float(sp.pa), 0.f);
  }
}

// Warp w takes rows w, w + SK_EPI_WARPS, ..., ROWS at a time with up to BATCH partials of each in flight.  No branch on
// a single row's state but around its stores: the rows' instructions interleave.
template <int ROWS, int BATCH>
__device__ __forceinline__ void sk_finish(const SkParams& p, const SkOp& o, const SkFinish& f, int w, int lane, const int2* row_tab,
                                          const float* rs_tab) {
  const int n = f.n0 + lane * 4, epi = o.epi, ld = o.ep.ldy;
  const int head = f.n0 >> 7, i0 = lane * 2;  // EPI_QKV: a CTA's columns are one head
  const bool rotate = epi == EPI_QKV && head < p.n_q_heads + p.n_kv_heads;
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
  for (int t = w; t < f.rows; t += ROWS * SK_EPI_WARPS) {
    const int m = f.m0 + t;  // rows m, m + SK_EPI_WARPS, ...
    float4 acc[ROWS], aux[ROWS];  // aux: residual values (EPI_RESID), or two cosines and two sines (EPI_QKV)
    bool live[ROWS];
    int2 where[ROWS];  // EPI_QKV: cache slot (-1: no live row), sequence
#pragma unroll
    for (int u = 0; u < ROWS; ++u) {
      live[u] = t + u * SK_EPI_WARPS < f.rows && m + u * SK_EPI_WARPS < p.M;
      acc[u] = aux[u] = zero;
      where[u] = make_int2(0, 0);
    }
    if (epi == EPI_RESID) {
      const float* y = static_cast<const float*>(o.ep.y) + static_cast<size_t>(m) * ld + n;
#pragma unroll
      for (int u = 0; u < ROWS; ++u)
        if (live[u]) aux[u] = __ldcg(reinterpret_cast<const float4*>(y + u * SK_EPI_WARPS * ld));
    } else if (epi == EPI_QKV) {
#pragma unroll
      for (int u = 0; u < ROWS; ++u)
        if (live[u]) where[u] = row_tab[m + u * SK_EPI_WARPS];
#pragma unroll
      for (int u = 0; u < ROWS; ++u) {
        live[u] = live[u] && where[u].x >= 0;
        if (rotate && live[u]) {
          const float2 co = *reinterpret_cast<const float2*>(p.rope_cos + where[u].x * 64 + i0);
          const float2 si = *reinterpret_cast<const float2*>(p.rope_sin + where[u].x * 64 + i0);
          aux[u] = make_float4(co.x, co.y, si.x, si.y);
        }
      }
    }
    const float* src = f.part + t * 128 + lane * 4;
    int step = f.step0;
#pragma unroll 1
    for (int s = 0; s < f.count; s += BATCH) {
      float4 v[BATCH][ROWS];
#pragma unroll
      for (int b = 0; b < BATCH; ++b) {
#pragma unroll
        for (int u = 0; u < ROWS; ++u)
          v[b][u] = s + b < f.count && live[u] ? __ldcg(reinterpret_cast<const float4*>(src + u * SK_EPI_WARPS * 128)) : zero;
        src += step;
        step = f.step;
      }
#pragma unroll
      for (int b = 0; b < BATCH; ++b)
#pragma unroll
        for (int u = 0; u < ROWS; ++u) {
          acc[u].x += v[b][u].x; acc[u].y += v[b][u].y; acc[u].z += v[b][u].z; acc[u].w += v[b][u].w;
        }
    }
    if (epi == EPI_RESID) {
      float* y = static_cast<float*>(o.ep.y) + static_cast<size_t>(m) * ld + n;
      __nv_bfloat16* yb = o.ep.yb + static_cast<size_t>(m) * ld + n;
      float sq[ROWS];
#pragma unroll
      for (int u = 0; u < ROWS; ++u) {
        const float4 v = make_float4(aux[u].x + acc[u].x, aux[u].y + acc[u].y, aux[u].z + acc[u].z, aux[u].w + acc[u].w);
        sq[u] = ((v.x * v.x + v.y * v.y) + v.z * v.z) + v.w * v.w;
        __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
        if (live[u]) {
          *reinterpret_cast<float4*>(y + u * SK_EPI_WARPS * ld) = v;
          if (o.ep.yb != nullptr)
            *reinterpret_cast<uint2*>(yb + u * SK_EPI_WARPS * ld) = make_uint2(*reinterpret_cast<uint32_t*>(&lo), *reinterpret_cast<uint32_t*>(&hi));
        }
      }
      if (o.ep.ssq_out != nullptr) {  // eight neighbouring lanes are a 32-column chunk
#pragma unroll
        for (int d = 1; d <= 4; d <<= 1)
#pragma unroll
          for (int u = 0; u < ROWS; ++u) sq[u] += __shfl_xor_sync(0xffffffffu, sq[u], d);
        const int chunks = (o.N + 31) / 32;
        float* out = o.ep.ssq_out + static_cast<size_t>(m) * chunks + n / 32;
#pragma unroll
        for (int u = 0; u < ROWS; ++u)
          if (live[u] && (lane & 7) == 0) out[u * SK_EPI_WARPS * chunks] = sq[u];
      }
      continue;
    }
#pragma unroll
    for (int u = 0; u < ROWS; ++u) {
      float rs = live[u] ? rs_tab[m + u * SK_EPI_WARPS] : 0.f;
      if (epi == EPI_STATS) rs *= o.ep.scale;  // (one factor, as in the other kernels' logits)
      acc[u] = make_float4(acc[u].x * rs, acc[u].y * rs, acc[u].z * rs, acc[u].w * rs);
    }
    if (epi == EPI_STATS) {
      sk_stats<ROWS>(p, o, acc, live, m, n, lane);
    } else if (epi == EPI_SWIGLU) {
      // packed rows of W: 2j = gate row of hidden unit j, 2j + 1 = its up row
      __nv_bfloat16* y = static_cast<__nv_bfloat16*>(o.ep.y) + static_cast<size_t>(m) * ld + n / 2;
#pragma unroll
      for (int u = 0; u < ROWS; ++u) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(silu_fast(acc[u].x) * acc[u].y, silu_fast(acc[u].z) * acc[u].w);
        if (live[u]) *reinterpret_cast<__nv_bfloat162*>(y + u * SK_EPI_WARPS * ld) = h;
      }
    } else if (rotate) {
      // Packed rows of W inside a q or k head: 2i = dim i, 2i + 1 = dim i + 64
#pragma unroll
      for (int u = 0; u < ROWS; ++u) {
        const __nv_bfloat162 lo = __floats2bfloat162_rn(acc[u].x * aux[u].x - acc[u].y * aux[u].z, acc[u].z * aux[u].y - acc[u].w * aux[u].w);
        const __nv_bfloat162 hi = __floats2bfloat162_rn(acc[u].y * aux[u].x + acc[u].x * aux[u].z, acc[u].w * aux[u].y + acc[u].z * aux[u].w);
        __nv_bfloat16* dst = head < p.n_q_heads
            ? static_cast<__nv_bfloat16*>(o.ep.y) + static_cast<size_t>(m + u * SK_EPI_WARPS) * ld + head * 128
            : o.k_cache + ((static_cast<size_t>(where[u].y) * p.n_kv_heads + (head - p.n_q_heads)) * p.max_seq + where[u].x) * 128;
        if (live[u]) {
          *reinterpret_cast<__nv_bfloat162*>(dst + i0) = lo;
          *reinterpret_cast<__nv_bfloat162*>(dst + 64 + i0) = hi;
        }
      }
    } else {
#pragma unroll
      for (int u = 0; u < ROWS; ++u) {
        if (!live[u]) continue;
        const size_t at = static_cast<size_t>(m + u * SK_EPI_WARPS) * ld + n;
        if (epi == EPI_F32) {
          const float sc = o.ep.scale;
          *reinterpret_cast<float4*>(static_cast<float*>(o.ep.y) + at) = make_float4(acc[u].x * sc, acc[u].y * sc, acc[u].z * sc, acc[u].w * sc);
          continue;
        }
        // bf16 rows; EPI_QKV: a v head keeps its order
        __nv_bfloat16* dst = epi == EPI_T ? static_cast<__nv_bfloat16*>(o.ep.y) + at
            : o.v_cache + ((static_cast<size_t>(where[u].y) * p.n_kv_heads + (head - p.n_q_heads - p.n_kv_heads)) * p.max_seq + where[u].x) * 128 + lane * 4;
        __nv_bfloat162 lo = __floats2bfloat162_rn(acc[u].x, acc[u].y), hi = __floats2bfloat162_rn(acc[u].z, acc[u].w);
        *reinterpret_cast<uint2*>(dst) = make_uint2(*reinterpret_cast<uint32_t*>(&lo), *reinterpret_cast<uint32_t*>(&hi));
      }
    }
  }
}

// grid = 2 x pairs (all resident at once), cluster (2, 1, 1).  Dynamic shared memory (1024-byte aligned inside the
// kernel): [stages] weight blocks, [stages] rows of X, barriers, row table, row factors, plans.
__global__ void __launch_bounds__(SK_THREADS, 1) gemm_sk_kernel(const __grid_constant__ SkParams p) {
  grid_dep_launch();
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int stages = p.stages;
  const uint32_t x_bytes = static_cast<uint32_t>(p.tok_n) * 64u;  // tok_n / 2 rows of 128 bytes
  uint8_t* smem_w = smem;
  uint8_t* smem_x = smem + static_cast<size_t>(stages) * SK_W_BYTES;
  uint64_t* full_bar = reinterpret_cast<uint64_t*>(smem_x + static_cast<size_t>(stages) * x_bytes);
  uint64_t* empty_bar = full_bar + stages;
  uint64_t* acc_full = empty_bar + stages;   // [2]
  uint64_t* acc_empty = acc_full + 2;        // [2], used in the leader only
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int2* row_tab = reinterpret_cast<int2*>(tmem_slot + 4);     // [SK_MAX_ROWS] EPI_QKV: cache slot (-1: no live row) and sequence
  float* rs_tab = reinterpret_cast<float*>(row_tab + SK_MAX_ROWS);   // [SK_MAX_ROWS] row factors of the folded RMSNorm
  SkPlan* plans = reinterpret_cast<SkPlan*>(rs_tab + SK_MAX_ROWS);   // [SK_MAX_OPS]

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = static_cast<int>(cluster_ctarank());
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      mbar_init(&full_bar[s], 2);  // the leader's weight thread and its activation thread each announce both CTAs' bytes
      mbar_init(&empty_bar[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], 2 * SK_EPI_WARPS);  // the epilogue warps of both CTAs
    }
    *abort_flag = 0;
    fence_barrier_init();
    for (int j = 0; j < p.n_ops; ++j) {
      prefetch_tensormap(&p.w[j]);
      prefetch_tensormap(&p.x[j]);
    }
  }
  if (warp == 1) {
    tmem_alloc_pair<512>(tmem_slot);
    tmem_relinquish_pair();
  }
  if (warp == 2 && lane < p.n_ops) sk_plan(p.op[lane], pair, n_pairs, p.tok_tiles, p.tok_n, plans[lane]);
  tc_fence_before();
  cluster_sync_all();  // barriers of both CTAs exist before either signals the other
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const uint32_t lead_full = map_to_cta(smem_u32(full_bar), 0);

  if (warp == 0) {
    // ------------------------------------------------------------------ weights: held back by ring space only
    if (elect_one()) {
      // weights that are read once leave L2 first: partials and activations stay
      const uint64_t stream_policy = l2_evict_first_policy();
      const bool once = p.tok_tiles == 1;
      int s = 0;
      uint32_t ph = 1;  // parity to wait for on the empty barrier (first lap: passes at once)
      bool ok = true;
      for (int j = 0; j < p.n_ops && ok; ++j) {
        const SkOp& o = p.op[j];
        const SkPlan& pl = plans[j];
        const int n_seg = pl.n_whole + pl.n_cut;
        for (int i = 0; i < n_seg && ok; ++i) {
          const SkSeg g = sk_seg(o, pl, i, pair, n_pairs, p.tok_tiles);
          int row = ((g.n_t * 2 + rank) * o.k_chunks + g.k0) * 128;  // first row of the next weight block
          for (int k = 0; k < g.n_k; ++k, row += 128) {
            if (!mbar_wait(&empty_bar[s], ph, abort_flag, p.error_word)) { ok = false; break; }
            if (rank == 0) mbar_arrive_expect_tx(&full_bar[s], 2 * SK_W_BYTES);
            if (once) tma_load_2d_pair_hint(smem_w + static_cast<size_t>(s) * SK_W_BYTES, &p.w[j], lead_full + 8u * s, 0, row, stream_policy);
            else tma_load_2d_pair(smem_w + static_cast<size_t>(s) * SK_W_BYTES, &p.w[j], lead_full + 8u * s, 0, row);
            if (++s == stages) { s = 0; ph ^= 1u; }
          }
        }
      }
    }
  } else if (warp == 2) {
    // ------------------------------------------------------------------ rows of X: behind the border of each matmul
    if (elect_one()) {
      int s = 0;
      uint32_t ph = 1;
      bool ok = true;
      grid_dep_wait();
      for (int j = 0; j < p.n_ops && ok; ++j) {
        const SkOp& o = p.op[j];
        const SkPlan& pl = plans[j];
        const int n_seg = pl.n_whole + pl.n_cut;
        if (j > 0 && n_seg > 0) {
          if (!chain_wait_count(p.border + (j - 1), gridDim.x, abort_flag, p.error_word)) break;
          fence_proxy_async_all();  // the rows were written with ordinary stores; the loads below go through the async proxy
        }
        for (int i = 0; i < n_seg && ok; ++i) {
          const SkSeg g = sk_seg(o, pl, i, pair, n_pairs, p.tok_tiles);
          const int row = g.m_t * p.tok_n + rank * (p.tok_n >> 1);
          for (int k = 0; k < g.n_k; ++k) {
            if (!mbar_wait(&empty_bar[s], ph, abort_flag, p.error_word)) { ok = false; break; }
            if (rank == 0) mbar_arrive_expect_tx(&full_bar[s], 2 * x_bytes);
            tma_load_2d_pair(smem_x + static_cast<size_t>(s) * x_bytes, &p.x[j], lead_full + 8u * s, (g.k0 + k) * BLOCK_K, row);
            if (++s == stages) { s = 0; ph ^= 1u; }
          }
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issue (leader)
    if (rank == 0 && elect_one()) {
      const uint32_t idesc = make_idesc(256, p.tok_n);
      const uint64_t adesc0 = make_smem_desc(smem_u32(smem_w)), bdesc0 = make_smem_desc(smem_u32(smem_x));
      const uint64_t a_step = SK_W_BYTES >> 4, b_step = x_bytes >> 4;
      int s = 0, n_acc = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int j = 0; j < p.n_ops && ok; ++j) {
        const SkOp& o = p.op[j];
        const SkPlan& pl = plans[j];
        const int n_seg = pl.n_whole + pl.n_cut;
        for (int i = 0; i < n_seg && ok; ++i, ++n_acc) {
          const SkSeg g = sk_seg(o, pl, i, pair, n_pairs, p.tok_tiles);
          const int buf = n_acc & 1;
          if (n_acc >= 2) ok = mbar_wait_cluster(&acc_empty[buf], static_cast<uint32_t>((n_acc >> 1) - 1) & 1u, abort_flag, p.error_word);
          if (!ok) break;
          tc_fence_after();
          const uint32_t tmem_d = tmem_base + static_cast<uint32_t>(buf * 256);
          for (int k = 0; k < g.n_k; ++k) {
            ok = mbar_wait_cluster(&full_bar[s], ph, abort_flag, p.error_word);
            if (!ok) break;
            tc_fence_after();
            const uint64_t adesc = adesc0 + a_step * static_cast<uint64_t>(s), bdesc = bdesc0 + b_step * static_cast<uint64_t>(s);
#pragma unroll
            for (int kk = 0; kk < BLOCK_K / UMMA_K; ++kk)
              umma_bf16_pair(tmem_d, adesc + static_cast<uint64_t>(2 * kk), bdesc + static_cast<uint64_t>(2 * kk), idesc,
                             (k > 0 || kk > 0) ? 1u : 0u);
            umma_commit_pair(&empty_bar[s], 3);
            if (++s == stages) { s = 0; ph ^= 1u; }
          }
          if (ok) umma_commit_pair(&acc_full[buf], 3);
        }
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue warps: lane quadrant = warp % 4
    grid_dep_wait();  // residual rows, positions and row sums come from earlier kernels
    const int et = threadIdx.x - 96, ew = warp - 3;
    const int lg = warp & 3;
    const uint32_t lane_addr = tmem_base + (static_cast<uint32_t>(lg * 32) << 16);
    const int part_ld = p.tok_n * 128;  // floats of one partial
    float* part = p.partial + static_cast<size_t>(rank) * part_ld;
    // The accumulator of segment `acc_i` goes to `dst` as [row of X][128 columns] and its buffer back to the MMA thread.
    auto dump = [&](int acc_i, float* dst) {
      const int buf = acc_i & 1;
      bool ok = mbar_wait(&acc_full[buf], static_cast<uint32_t>(acc_i >> 1) & 1u, abort_flag, p.error_word);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) return false;
      tc_fence_after();
      dst += lg * 32 + lane;
#pragma unroll 1
      for (int c = (ew >> 2) * 16; c < p.tok_n; c += SK_EPI_WARPS * 4) {
        float v[16];
        tmem_ld_32x16(lane_addr + static_cast<uint32_t>(buf * 256 + c), v);
        tmem_ld_wait();
#pragma unroll
        for (int q = 0; q < 16; ++q) __stcg(dst + (c + q) * 128, v[q]);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) sk_release_acc(&acc_empty[buf]);
      return true;
    };
    // A whole tile of gate and up rows straight from tensor memory: lane = packed row of W (even: gate row of a hidden unit,
    // odd: its up row), column = row of X.  The even lane of a unit finishes the even rows of X, the odd lane the odd ones.
    // (By way of L2 and sk_finish, the last whole tile of a pair held up the border for 8.6 us at 256 rows.)
    auto swiglu_tile = [&](const SkOp& o, int acc_i, const SkSeg& g) {
      const int buf = acc_i & 1;
      bool ok = mbar_wait(&acc_full[buf], static_cast<uint32_t>(acc_i >> 1) & 1u, abort_flag, p.error_word);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) return false;
      tc_fence_after();
      const bool odd = (lane & 1) != 0;
      __nv_bfloat16* y = static_cast<__nv_bfloat16*>(o.ep.y) + ((g.n_t * 256 + rank * 128 + lg * 32 + lane) >> 1);
#pragma unroll 1
      for (int c = (ew >> 2) * 16; c < p.tok_n; c += SK_EPI_WARPS * 4) {
        float v[16];
        tmem_ld_32x16(lane_addr + static_cast<uint32_t>(buf * 256 + c), v);
        tmem_ld_wait();
        const int m0 = g.m_t * p.tok_n + c + (odd ? 1 : 0);
#pragma unroll
        for (int q = 0; q < 16; q += 2) {
          const float mine = odd ? v[q + 1] : v[q];
          const float other = __shfl_xor_sync(0xffffffffu, odd ? v[q] : v[q + 1], 1);
          const int m = m0 + q;
          if (m < p.M) {
            const float rs = rs_tab[m];
            const float gate = (odd ? other : mine) * rs, up = (odd ? mine : other) * rs;
            y[static_cast<size_t>(m) * o.ep.ldy] = __float2bfloat16_rn(silu_fast(gate) * up);
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) sk_release_acc(&acc_empty[buf]);
      return true;
    };
    if (p.rope_rows) {
      for (int m = et; m < p.M; m += SK_EPI_THREADS) {
        const int b = m / p.rows_per_seq, r = m % p.rows_per_seq;
        int pos = -1;
        if (r < p.n_valid[b]) {
          pos = p.pos_base[b] + r;
          if (pos < 0 || pos >= p.max_seq) {
            atomicOr(p.error_word, ERRW_BAD_POSITION);
            pos = -1;
          }
        }
        row_tab[m] = make_int2(pos, b);
      }
    }
    int n_acc = 0;
    bool alive = true;
    for (int j = 0; j < p.n_ops && alive; ++j) {
      const SkOp& o = p.op[j];
      const SkPlan& pl = plans[j];
      if (j > 0 && pl.n_whole + pl.n_cut > 0) {
        bool ok = true;
        if (et == 0) ok = chain_wait_count(p.border + (j - 1), gridDim.x, abort_flag, p.error_word);
        if (!sk_all(ok)) { alive = false; break; }
      }
      // Row factors, while the MMAs run (visible to the other warps behind the barriers below).
      if (o.epi != EPI_RESID && pl.n_whole + pl.n_cut > 0) {
        for (int m = ew * 16; m < p.M; m += SK_EPI_WARPS * 16) {
          if (o.ep.ssq_in != nullptr) sk_row_rstd16(o.ep, m, p.M, lane, rs_tab + m);
          else if (lane < 16) rs_tab[m + lane] = 1.f;
        }
      }
      bool ok = true;
      // ---- cut tiles: partials go out, then this pair's shares are finished
      if (pl.n_cut > 0) {
        for (int k = 0; k < pl.n_cut; ++k) ok = ok && dump(n_acc + k, part + static_cast<size_t>(pair * 6 + (k ^ pl.swap) * 2) * part_ld);
        if (!sk_all(ok)) { alive = false; break; }  // every thread's partials are ordered before the releases below
        if (et < pl.n_cut) {
          unsigned int* count = o.part_count + pl.cut[et].index * 2 + rank;
          chain_arrive(count);
          if (pl.cut[et].t1 > pl.cut[et].t0) ok = chain_wait_count(count, static_cast<unsigned int>(pl.cut[et].count), abort_flag, p.error_word);
        }
        if (!sk_all(ok)) { alive = false; break; }
        const int step = 6 * part_ld;  // (a later contributor's range begins in this tile: its first partial)
        for (int k = 0; k < pl.n_cut; ++k) {
          const SkCut& c = pl.cut[k];
          if (c.t1 <= c.t0) continue;
          const SkFinish f{c.g.m_t * p.tok_n + c.t0, c.g.n_t * 256 + rank * 128, c.t1 - c.t0,
                           part + static_cast<size_t>(c.first * 6 + c.first_slot * 2) * part_ld + c.t0 * 128, c.count, step - c.first_slot * 2 * part_ld, step};
          if (c.count <= 3) sk_finish<3, 3>(p, o, f, ew, lane, row_tab, rs_tab);
          else sk_finish<3, 5>(p, o, f, ew, lane, row_tab, rs_tab);
        }
      }
      // ---- whole tiles
      if (o.epi == EPI_SWIGLU) {
        if (pl.n_whole > 0 && pl.n_cut == 0 && !sk_all(true)) { alive = false; break; }  // the row factors are there
        for (int i = 0; i < pl.n_whole && ok; ++i) ok = swiglu_tile(o, n_acc + pl.n_cut + i, sk_seg(o, pl, pl.n_cut + i, pair, n_pairs, p.tok_tiles));
      } else {
        for (int i = 0; i < pl.n_whole; ++i) {
          const SkSeg g = sk_seg(o, pl, pl.n_cut + i, pair, n_pairs, p.tok_tiles);
          float* mine = part + static_cast<size_t>(pair * 6 + 4) * part_ld;
          if (i > 0 && !sk_all(true)) { alive = false; break; }  // every warp has finished the tile before
          if (!sk_all(dump(n_acc + pl.n_cut + i, mine))) { alive = false; break; }
          const SkFinish f{g.m_t * p.tok_n, g.n_t * 256 + rank * 128, p.tok_n, mine, 1, 0, 0};
          sk_finish<4, 1>(p, o, f, ew, lane, row_tab, rs_tab);
        }
      }
      if (!alive) break;
      n_acc += pl.n_whole + pl.n_cut;
      // ---- border: this CTA's stores of the matmul are done
      if (j + 1 < p.n_ops) {
        if (!sk_all(ok)) { alive = false; break; }
        if (et == 0) chain_arrive(p.border + j);  // (a release: the barrier put every thread's stores before it)
      }
    }
  }
  // Neither CTA may leave (its shared memory is an operand of the leader's MMAs, its barriers a target of the
  // leader's commits) nor give back tensor memory before both are through.
  __syncwarp();
  tc_fence_before();
  cluster_sync_all();
  if (warp == 1) tmem_dealloc_pair<512>(tmem_base);
}

}  // namespace tc
}  // namespace d3
