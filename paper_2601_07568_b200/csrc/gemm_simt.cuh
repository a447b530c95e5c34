// Plain SIMT matmul Y[M,N] = X[M,K] . W[N,K]^T with fp32 accumulation and the same epilogues as the
// tensor-core kernel.  It is the fp32 path (TF32 tensor cores cannot hold 1e-4 relative on logits)
// and a debugging cross-check for bf16.  Tile 32 x 128, K slabs of 32, 256 threads, 4 x 4 outputs each.
#pragma once
#include "common.cuh"
#include "ptx_sm100.cuh"

namespace d3 {
namespace simt {

constexpr int BM = 32, BN = 128, BK = 32, THREADS = 256;

// Epilogue of a BM_ x BN_ tile of sums in shared memory whose first element is (m0, n0).  (EPI_STATS: BN_ is 128.)
template <typename T, int EPI, int BM_, int BN_>
__device__ __forceinline__ void simt_epilogue(const float (*Cs)[BN_ + 1], int m0, int n0, int M, int N, const EpiParams& ep) {
  const int t = threadIdx.x;
  if constexpr (EPI == EPI_F32 || EPI == EPI_RESID || EPI == EPI_T) {
    for (int e = t; e < BM_ * BN_; e += THREADS) {
      int r = e / BN_, c = e % BN_;
      int m = m0 + r, n = n0 + c;
      if (m < M && n < N) {
        size_t o = static_cast<size_t>(m) * ep.ldy + n;
        if constexpr (EPI == EPI_F32) static_cast<float*>(ep.y)[o] = Cs[r][c] * ep.scale;
        else if constexpr (EPI == EPI_RESID) static_cast<float*>(ep.y)[o] += Cs[r][c];
        else static_cast<T*>(ep.y)[o] = TypeOps<T>::from_f(Cs[r][c]);
      }
    }
  } else if constexpr (EPI == EPI_SWIGLU) {
    // packed rows of W: 2j = gate row of hidden unit j, 2j+1 = its up row
    const int F = N / 2;
    for (int e = t; e < BM_ * (BN_ / 2); e += THREADS) {
      int r = e / (BN_ / 2), c = e % (BN_ / 2);
      int m = m0 + r, h = n0 / 2 + c;
      if (m < M && h < F)
        static_cast<T*>(ep.y)[static_cast<size_t>(m) * ep.ldy + h] =
            TypeOps<T>::from_f(silu_f(Cs[r][2 * c]) * Cs[r][2 * c + 1]);
    }
  } else if constexpr (EPI == EPI_STATS) {
    // one warp per row (8 warps, 4 rows each): lanes stride the 128 columns, fixed shuffle tree
    const int warp = t / 32, lane = t % 32;
    for (int r = warp; r < BM_; r += THREADS / 32) {
      int m = m0 + r;
      SoftStat st = stat_empty();
      for (int c = lane; c < BN_; c += 32) {
        int n = n0 + c;
        if (n < N && n != ep.mask_id) stat_add(st, Cs[r][c] * ep.scale, n);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        SoftStat other;
        other.m = __shfl_xor_sync(0xffffffffu, st.m, o);
        other.z = __shfl_xor_sync(0xffffffffu, st.z, o);
        other.s = __shfl_xor_sync(0xffffffffu, st.s, o);
        other.a = __shfl_xor_sync(0xffffffffu, st.a, o);
        st = (lane & o) ? stat_merge(other, st) : stat_merge(st, other);
      }
      if (lane == 0 && m < M)
        ep.stat_part[static_cast<size_t>(m) * ep.n_tiles + blockIdx.x] =
            make_float4(st.m, st.z, st.s, __int_as_float(st.a));
      if (ep.sample_part != nullptr && m < M) {  // temperature sampling: largest l + T * g of the tile
        SampleStat sp = sample_empty();
        const SampleRow sr = sample_row(ep, m);
        for (int c = lane; c < BN_; c += 32) {
          const int n = n0 + c;
          if (n < N && n != ep.mask_id) {
            const uint4 bits = philox4x32_10(make_uint4(static_cast<uint32_t>(n >> 2), sr.pos, sr.step, sr.seq), ep.seed_lo, ep.seed_hi);
            const uint32_t w = (n & 3) == 0 ? bits.x : (n & 3) == 1 ? bits.y : (n & 3) == 2 ? bits.z : bits.w;
            const float l = Cs[r][c] * ep.scale;
            sample_add(sp, __fadd_rn(l, __fmul_rn(ep.temperature, gumbel_from_bits(w))), l, n);
          }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          SampleStat other;
          other.pm = __shfl_xor_sync(0xffffffffu, sp.pm, o);
          other.la = __shfl_xor_sync(0xffffffffu, sp.la, o);
          other.pa = __shfl_xor_sync(0xffffffffu, sp.pa, o);
          sp = sample_merge(sp, other);
        }
        if (lane == 0)
          ep.sample_part[static_cast<size_t>(m) * ep.n_tiles + blockIdx.x] = make_float4(sp.pm, sp.la, __int_as_float(sp.pa), 0.f);
      }
    }
  }
}

// EPI_QKV on small fp32 tiles: what rope_kv_kernel does with the projected rows, from the tile (its columns 2k and 2k + 1 of a
// q or k head are the dims k and k + d_head / 2).  A launch fewer per layer.
struct SimtQkv {
  float *k_cache, *v_cache;  // this layer's planes
  const float *rope_cos, *rope_sin;
  const int *pos_base, *n_valid;
  int rows_per_seq, hq, hkv, dh, max_seq;
  uint32_t* error_word;
};
template <int BM_, int BN_>
__device__ __forceinline__ void simt_qkv_epilogue(const float (*Cs)[BN_ + 1], int m0, int n0, int M, int N, const EpiParams& ep, const SimtQkv& q) {
  const int half = q.dh / 2;
  for (int e = threadIdx.x; e < BM_ * (BN_ / 2); e += THREADS) {
    const int r = e / (BN_ / 2), c = e % (BN_ / 2) * 2, m = m0 + r, n = n0 + c;
    if (m >= M || n >= N) continue;
    const int b = m / q.rows_per_seq, row = m - b * q.rows_per_seq;
    if (row >= q.n_valid[b]) continue;
    const int pos = q.pos_base[b] + row;
    if (pos < 0 || pos >= q.max_seq) {
      if (n == 0) atomicOr(q.error_word, ERRW_BAD_POSITION);
      continue;
    }
    const int head = n / q.dh, d = n - head * q.dh;
    const float x = Cs[r][c], y = Cs[r][c + 1];
    if (head >= q.hq + q.hkv) {  // a v head keeps its order
      float* dst = q.v_cache + ((static_cast<size_t>(b) * q.hkv + (head - q.hq - q.hkv)) * q.max_seq + pos) * q.dh + d;
      dst[0] = x;
      dst[1] = y;
      continue;
    }
    const int k = d >> 1;
    const float co = q.rope_cos[static_cast<size_t>(pos) * half + k], si = q.rope_sin[static_cast<size_t>(pos) * half + k];
    float* dst = head < q.hq ? static_cast<float*>(ep.y) + static_cast<size_t>(m) * ep.ldy + head * q.dh
                             : q.k_cache + ((static_cast<size_t>(b) * q.hkv + (head - q.hq)) * q.max_seq + pos) * q.dh;
    dst[k] = x * co - y * si;
    dst[k + half] = y * co + x * si;
  }
}

template <typename T, int EPI>
__global__ void __launch_bounds__(THREADS) gemm_simt_kernel(const T* __restrict__ X, const T* __restrict__ W, int M,
                                                            int N, int K, EpiParams ep) {
  ptx::grid_dep_wait();
  ptx::grid_dep_launch();
  __shared__ float Xs[BM][BK + 1];
  __shared__ float Ws[BN][BK + 1];
  __shared__ float Cs[BM][BN + 1];
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const int t = threadIdx.x, ty = t / 32, tx = t % 32;
  float acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;

  for (int k0 = 0; k0 < K; k0 += BK) {
    for (int e = t; e < BM * BK; e += THREADS) {
      int r = e / BK, c = e % BK;
      int m = m0 + r, k = k0 + c;
      Xs[r][c] = (m < M && k < K) ? TypeOps<T>::to_f(X[static_cast<size_t>(m) * K + k]) : 0.f;
    }
    for (int e = t; e < BN * BK; e += THREADS) {
      int r = e / BK, c = e % BK;
      int n = n0 + r, k = k0 + c;
      Ws[r][c] = (n < N && k < K) ? TypeOps<T>::to_f(W[static_cast<size_t>(n) * K + k]) : 0.f;
    }
    __syncthreads();
#pragma unroll 8
    for (int kk = 0; kk < BK; ++kk) {
      float a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = Xs[ty * 4 + i][kk];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Ws[tx + 32 * j][kk];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) Cs[ty * 4 + i][tx + 32 * j] = acc[i][j];
  __syncthreads();

  simt_epilogue<T, EPI, BM, BN>(Cs, m0, n0, M, N, ep);
}

// The same sums, bit for bit (one chain of fused multiply-adds per output, ascending in k), for matmuls whose 32 x 128 tiles
// would leave most SMs idle: BM_ x BN_ tiles, 256 threads, KC columns of X and W in shared memory at a time, read four at
// a time.  What bounds it is the chain of K multiply-adds and, per KC columns, one trip to memory.  A 16 x 128 x 512
// product took 50 us as one 32 x 128 tile on one SM; as 8 tiles of 16 x 16 it takes 6.  K % 4 == 0, rows aligned to 4 elements.
// NORM (fp32): the rows of X are those in front of an RMSNorm with the gains ep.norm_gain; every block works out the factors of
// its few rows (the bits of rmsnorm_kernel) while its first columns are on their way.  (An instance of its own: with the norm as a
// branch the LM head without one took 26.1 us instead of 22.9 at 4 x 9000 x 1024 and 15.8 instead of 14.2 at 16 x 2000 x 512.)
template <typename T, int EPI, int BM_, int BN_, int KC, bool NORM>
__global__ void __launch_bounds__(THREADS) gemm_simt_small_kernel(const T* __restrict__ X, const T* __restrict__ W, int M, int N, int K, EpiParams ep, const SimtQkv qkv) {
  ptx::grid_dep_wait();
  ptx::grid_dep_launch();
  constexpr int OUT = BM_ * BN_ / THREADS, ROWS = THREADS / BN_;
  __shared__ __align__(16) float Xs[BM_][KC + 4];
  __shared__ __align__(16) float Ws[BN_][KC + 4];
  __shared__ float Cs[BM_][BN_ + 1];
  const int m0 = blockIdx.y * BM_, n0 = blockIdx.x * BN_;
  const int t = threadIdx.x, c = t % BN_, r0 = t / BN_;
  float acc[OUT];
#pragma unroll
  for (int i = 0; i < OUT; ++i) acc[i] = 0.f;
  // A thread's pieces of the next KC columns are requested before the products of the present ones.
  constexpr int XN = BM_ * (KC / 4), WN = BN_ * (KC / 4), XP = (XN + THREADS - 1) / THREADS, WP = WN / THREADS;
  static_assert(WN % THREADS == 0 && (XN % THREADS == 0 || XN < THREADS), "pieces deal out evenly");
  float4 xv[XP], wv[WP];
  auto piece = [&](const T* src, int row, int rows, int k) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (row < rows && k < K) {
      if constexpr (sizeof(T) == 4) {
        v = *reinterpret_cast<const float4*>(src + static_cast<size_t>(row) * K + k);
      } else {
        const uint2 w = *reinterpret_cast<const uint2*>(src + static_cast<size_t>(row) * K + k);
        v = make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u), __uint_as_float(w.y << 16), __uint_as_float(w.y & 0xffff0000u));
      }
    }
    return v;
  };
  auto request = [&](int k0) {
#pragma unroll
    for (int i = 0; i < XP; ++i)
      if (XN >= THREADS || t < XN) xv[i] = piece(X, m0 + (t + i * THREADS) / (KC / 4), M, k0 + (t + i * THREADS) % (KC / 4) * 4);
#pragma unroll
    for (int i = 0; i < WP; ++i) wv[i] = piece(W, n0 + (t + i * THREADS) / (KC / 4), N, k0 + (t + i * THREADS) % (KC / 4) * 4);
  };
  request(0);
  __shared__ float rstd[NORM ? BM_ : 1];
  if constexpr (NORM) {
    const int lane = t & 31, n4 = K >> 2;
    for (int r = t >> 5; r < BM_; r += THREADS / 32) {
      const float4* row = reinterpret_cast<const float4*>(X + static_cast<size_t>(min(m0 + r, M - 1)) * K);
      float tot = 0.f;
      for (int w = 0; w < 8 && w * 32 < n4; ++w) {  // what warp w of rmsnorm_kernel adds up
        float ss = 0.f;
        for (int i = w * 32 + lane; i < n4; i += 256) {
          const float4 v = row[i];
          ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
        tot += ss;
      }
      if (lane == 0) rstd[r] = rsqrtf(tot / static_cast<float>(K) + ep.rms_eps);
    }
    __syncthreads();
  }
  for (int k0 = 0; k0 < K; k0 += KC) {
    if constexpr (NORM) {
#pragma unroll
      for (int i = 0; i < XP; ++i) {
        const int e = t + i * THREADS, k = k0 + e % (KC / 4) * 4;
        if ((XN >= THREADS || t < XN) && k < K) {
          const float f = rstd[e / (KC / 4)];
          const float4 g = *reinterpret_cast<const float4*>(ep.norm_gain + k);
          xv[i] = make_float4(xv[i].x * f * g.x, xv[i].y * f * g.y, xv[i].z * f * g.z, xv[i].w * f * g.w);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < XP; ++i)
      if (XN >= THREADS || t < XN) *reinterpret_cast<float4*>(&Xs[(t + i * THREADS) / (KC / 4)][(t + i * THREADS) % (KC / 4) * 4]) = xv[i];
#pragma unroll
    for (int i = 0; i < WP; ++i) *reinterpret_cast<float4*>(&Ws[(t + i * THREADS) / (KC / 4)][(t + i * THREADS) % (KC / 4) * 4]) = wv[i];
    __syncthreads();
    if (k0 + KC < K) request(k0 + KC);
    // (up to the last column in whole slabs of the other kernel, the same bits: 1 x 5842 x 4 takes 5.2 us, all KC of them 10.4)
    const int columns = min(KC, (K - k0 + BK - 1) / BK * BK);
#pragma unroll 1
    for (int k1 = 0; k1 < columns; k1 += BK) {
#pragma unroll
      for (int k = k1; k < k1 + BK; k += 4) {
        const float4 w = *reinterpret_cast<const float4*>(&Ws[c][k]);
#pragma unroll
        for (int i = 0; i < OUT; ++i) {
          const float4 x = *reinterpret_cast<const float4*>(&Xs[r0 + i * ROWS][k]);
          acc[i] = fmaf(x.x, w.x, acc[i]);
          acc[i] = fmaf(x.y, w.y, acc[i]);
          acc[i] = fmaf(x.z, w.z, acc[i]);
          acc[i] = fmaf(x.w, w.w, acc[i]);
        }
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < OUT; ++i) Cs[r0 + i * ROWS][c] = acc[i];
  __syncthreads();
  if constexpr (EPI == EPI_QKV) simt_qkv_epilogue<BM_, BN_>(Cs, m0, n0, M, N, ep, qkv);
  else simt_epilogue<T, EPI, BM_, BN_>(Cs, m0, n0, M, N, ep);
}

}  // namespace simt
}  // namespace d3
