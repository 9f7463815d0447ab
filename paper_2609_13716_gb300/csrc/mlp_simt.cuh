// mlp_simt.cuh -- fp32 CUDA-core forward of a tile of M policy rows (Sec. 3 policy pi_i).
//
// z = W3 tanh(W2 tanh(W1 o + b1) + b2) + b3 for M rows that share one policy, computed by
// a group of threads (a whole CTA, or the warps of one seat).  Weights are the packed fp32
// (transposed) copy, read through L1/L2.  Every output is bias + sum_k x_k w_k accumulated
// with fmaf in increasing k, so a row's result does not depend on which tile, slot or
// thread layout it gets.
//
// Layout.  Activations sit in shared memory transposed, a column of M rows per unit (+ 4 of
// padding, which spreads the column stores over the banks).  A thread owns one or two output
// columns for all M rows: it reads each of its weights from global memory once (a warp's are
// consecutive), 2 x 8 rows of W^T ahead, and a unit's rows as 16-byte broadcast loads; the
// products run as packed fma.rn.f32x2 over row pairs.  The packed fma has half the rate of the
// scalar one (measured), so it halves the issue slots, not the FMA time, and lets two warps
// per scheduler saturate the pipe.  No barrier inside a layer: warps run apart and hide each
// other's latencies.  (Weights staged through a shared-memory ring by asynchronous copies,
// with 4 x 4 or 2 x 4 blocks per thread, took twice as long: a barrier per stage keeps the
// warps in phase, loading and then multiplying together.)
//
// What bounds it: at 8 rows the FMA pipe and the shared-memory port both need ~32 cycles per
// unit (two groups, 256 columns); 66 are measured, the rest is the L2 latency that 2 x 8 rows
// ahead do not cover (2 x 16 spill).  Before, a tile was 32 to 64 rows with 4 x 4 blocks per
// thread, every feature multiplied and no load in flight ahead: few SMs busy, each waiting
// for L2 at every fourth k.  Kitchen collection (520-256-256-7, 1000 envs x 64 steps) 16.1 ->
// 1.13 ms, Hanabi policy outputs (660-512-512-21, n = 3001) 421 -> 111 us.
#pragma once
#include "aht_common.cuh"
#include "tc_common.cuh"

namespace aht {

extern __shared__ __align__(16) uint8_t tile_smem_[];

// The threads that compute one tile together: thread `tid` of `n` (a multiple of 32), with
// the named barrier `bar` over exactly these threads.
struct Group {
  int tid, n, bar;
  __device__ __forceinline__ void sync() const {
    asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(n) : "memory");
  }
};

// Shared memory of one tile: observations, activations, outputs; TileOffsets are the byte
// offsets in the CTA's dynamic shared memory (see smem_layout).
struct TileOffsets {
  int32_t X, A, B, Z, ks, list, cnt;
  TileCfg cfg;
};
struct TileBufs {
  uint8_t* X;      // observation bytes [M][KP], or bit rows [M][bit_words(K)]
  float* A;        // [max(K, H1)][M + 4]: the observation's listed features, then layer 2
  float* B;        // [H0][M + 4]: layer 1
  float* Z;        // [M][NOP] outputs
  uint16_t* ks;    // [K] listed features
  uint32_t* list;  // sparse first layer: [M][kSparseCap]
  int* cnt;        // [8]
};

__device__ __forceinline__ TileBufs tile_bufs(const TileOffsets& o) {
  uint8_t* p = tile_smem_;
  return TileBufs{p + o.X,
                  reinterpret_cast<float*>(p + o.A),
                  reinterpret_cast<float*>(p + o.B),
                  reinterpret_cast<float*>(p + o.Z),
                  reinterpret_cast<uint16_t*>(p + o.ks),
                  reinterpret_cast<uint32_t*>(p + o.list),
                  reinterpret_cast<int*>(p + o.cnt)};
}

__host__ __device__ constexpr inline int bit_words(int K) { return (K + 31) / 32; }

// out[c][r] = tanh(bias[c] + sum_j in[j][r] * Wt[k_j][c]) for r < M, c < N (N % C == 0), k_j =
// ks[j] (kList) or j, j < n.
constexpr int kActPad = 4;
template <int M, int C, bool kList>
__device__ __forceinline__ void dense_cols(const Group& g, const float* in, int n, const uint16_t* ks,
                                           const float* __restrict__ Wt, const float* __restrict__ bias, int N,
                                           float* out) {
  constexpr int ld = M + kActPad, U = 8;
  struct Wv {
    float v[C];
  };
#pragma unroll 1
  for (int c0 = C * g.tid; c0 < N; c0 += C * g.n) {
    uint64_t acc[M / 2][C];  // rows 2 i, 2 i + 1
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const float b = __ldg(bias + c0 + c);
#pragma unroll
      for (int i = 0; i < M / 2; ++i) acc[i][c] = tc::f2_pack(b, b);
    }
    auto weight = [&](int j) {
      const int k = kList ? (int)ks[j] : j;
      const float* p = Wt + (uint32_t)(k * N + c0);
      Wv w;
      if constexpr (C == 2) {
        const float2 v = __ldg(reinterpret_cast<const float2*>(p));
        w.v[0] = v.x, w.v[1] = v.y;
      } else {
        w.v[0] = __ldg(p);
      }
      return w;
    };
    auto fetch = [&](Wv (&w)[U], int j) {
#pragma unroll
      for (int u = 0; u < U; ++u) w[u] = weight(j + u);
    };
    auto use = [&](const Wv& w, const float* x) {
      uint64_t ww[C];
#pragma unroll
      for (int c = 0; c < C; ++c) ww[c] = tc::f2_pack(w.v[c], w.v[c]);
#pragma unroll
      for (int i = 0; i < M / 2; i += 2) {
        const ulonglong2 xv = *reinterpret_cast<const ulonglong2*>(x + 2 * i);
#pragma unroll
        for (int c = 0; c < C; ++c) {
          acc[i][c] = tc::f2_fma(xv.x, ww[c], acc[i][c]);
          acc[i + 1][c] = tc::f2_fma(xv.y, ww[c], acc[i + 1][c]);
        }
      }
    };
    const int full = n / U * U;
    Wv wa[U], wb[U];
    int j = 0;
    if (full > 0) fetch(wa, 0);
    const float* x = in;
#pragma unroll 1
    for (; j + 2 * U <= full; j += 2 * U, x += 2 * U * ld) {  // two batches a turn: the buffers swap by name
      fetch(wb, j + U);
#pragma unroll
      for (int u = 0; u < U; ++u) use(wa[u], x + u * ld);
      if (j + 2 * U < full) fetch(wa, j + 2 * U);
#pragma unroll
      for (int u = 0; u < U; ++u) use(wb[u], x + (U + u) * ld);
    }
    if (j < full) {
#pragma unroll
      for (int u = 0; u < U; ++u) use(wa[u], x + u * ld);
      j += U, x += U * ld;
    }
#pragma unroll 1
    for (; j < n; ++j, x += ld) use(weight(j), x);
#pragma unroll
    for (int c = 0; c < C; ++c) {
      float* o = out + (c0 + c) * ld;
#pragma unroll
      for (int i = 0; i < M / 2; i += 2) {
        float4 v;
        tc::f2_unpack(acc[i][c], v.x, v.y);
        tc::f2_unpack(acc[i + 1][c], v.z, v.w);
        *reinterpret_cast<float4*>(o + 2 * i) = make_float4(tanhf(v.x), tanhf(v.y), tanhf(v.z), tanhf(v.w));
      }
    }
  }
}

// Two columns per thread where that still occupies the group, else one.
template <int M, bool kList>
__device__ __forceinline__ void dense_tile(const Group& g, const float* in, int n, const uint16_t* ks,
                                           const float* __restrict__ Wt, const float* __restrict__ bias, int N,
                                           float* out) {
  if (N >= 2 * g.n) dense_cols<M, 2, kList>(g, in, n, ks, Wt, bias, N, out);
  else dense_cols<M, 1, kList>(g, in, n, ks, Wt, bias, N, out);
}

// The output layer: Z[r][c] = bias[c] + sum_k in[k][r] W3[k][c], one thread per output (few
// columns: a block of rows x columns per thread would leave most threads idle).  W3 is the
// copy in shared memory where the caller keeps one (kShared), else W3^T itself.
template <int M, int kNOP, bool kShared>
__device__ __forceinline__ void dense_out(const Group& g, const float* in, int K, const float* W3,
                                          const float* __restrict__ bias, float* Z) {
  constexpr int ld = M + kActPad;
#pragma unroll 1
  for (int o = g.tid; o < M * kNOP; o += g.n) {
    const int c = o / M, r = o - c * M;
    float acc = __ldg(bias + c);
    const float *x = in + r, *w = W3 + c;
#pragma unroll 1
    for (int k = 0; k < K; k += 16, x += 16 * ld, w += 16 * kNOP) {  // K is a multiple of 16
      float xv[16], wv[16];
#pragma unroll
      for (int u = 0; u < 16; ++u) {
        xv[u] = x[u * ld];
        wv[u] = kShared ? w[u * kNOP] : __ldg(w + u * kNOP);
      }
#pragma unroll
      for (int u = 0; u < 16; ++u) acc = fmaf(xv[u], wv[u], acc);
    }
    Z[r * kNOP + c] = acc;
  }
}
template <int M, bool kShared>
__device__ __forceinline__ void dense_out_n(const Group& g, const float* in, int K, const float* W3,
                                            const float* __restrict__ bias, int NOP, float* Z) {
  if (NOP == 8) dense_out<M, 8, kShared>(g, in, K, W3, bias, Z);         // 6 actions + value
  else if (NOP == 12) dense_out<M, 12, kShared>(g, in, K, W3, bias, Z);  // Mini Hanabi
  else dense_out<M, 24, kShared>(g, in, K, W3, bias, Z);                 // Hanabi
}

// A policy's W3^T [H1][NOP] into shared memory (a rollout tile keeps its policies' where
// there is room, TileCfg::w3).
__device__ __forceinline__ void load_w3(const Group& g, const float* __restrict__ w, const MlpDims& m, float* W3) {
  const float* src = w + m.oW3;
  for (int i = 4 * g.tid; i < m.H1 * m.NOP; i += 4 * g.n)
    *reinterpret_cast<float4*>(W3 + i) = __ldg(reinterpret_cast<const float4*>(src + i));
}

// The features that are nonzero in some row of the tile, in increasing order, and their
// values as fp32 columns: a zero feature adds 0 x w, which changes no sum while w is
// finite, so the first layer runs over the listed ones only (a kitchen tile of 8 rows lists
// 60-100 of 520).  all: every feature is listed (W1 holds an infinity or a NaN).
// From bit rows (binary games): one lane per 32-feature word (K <= 1024).
template <int M>
__device__ __forceinline__ void list_bits(const Group& g, const TileBufs& t, int K, bool all) {
  const uint32_t* bits = reinterpret_cast<const uint32_t*>(t.X);
  const int nw = bit_words(K);
  if (g.tid < 32) {
    uint32_t u = 0;
    if (g.tid < nw) {
      for (int r = 0; r < M; ++r) u |= bits[r * nw + g.tid];
      if (all) u = 0xFFFFFFFFu;
      const int left = K - 32 * g.tid;
      if (left < 32) u &= (1u << left) - 1u;
    }
    const int own = __popc(u);
    int incl = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (g.tid >= o) incl += y;
    }
    int pos = incl - own;
    while (u) {
      t.ks[pos++] = (uint16_t)(32 * g.tid + __ffs(u) - 1);
      u &= u - 1;
    }
    if (g.tid == 31) t.cnt[0] = incl;
  }
  g.sync();
  constexpr int ld = M + kActPad;
  const int n = t.cnt[0];
#pragma unroll 2
  for (int i = g.tid; i < n * M; i += g.n) {
    const int j = i / M, r = i - j * M, k = t.ks[j];
    t.A[j * ld + r] = (float)((bits[r * nw + (k >> 5)] >> (k & 31)) & 1u);
  }
}
// From byte rows [M][KP] (any values; K % 4 == 0, K <= 1024): one lane per 4-feature word,
// a warp per 32 words.
template <int M>
__device__ __forceinline__ void list_bytes(const Group& g, const TileBufs& t, int K, int KP, bool all) {
  const int words = K >> 2, chunks = (words + 31) >> 5, lane = g.tid & 31;
  auto flags = [&](int ch) {
    const int w = 32 * ch + lane;
    if (w >= words) return 0u;
    uint32_t u = 0;
    for (int r = 0; r < M; ++r) u |= *reinterpret_cast<const uint32_t*>(t.X + r * KP + 4 * w);
    if (all) u = 0xFFFFFFFFu;
    return (u & 0xFFu ? 1u : 0u) | (u & 0xFF00u ? 2u : 0u) | (u & 0xFF0000u ? 4u : 0u) | (u >> 24 ? 8u : 0u);
  };
  for (int ch = g.tid >> 5; ch < chunks; ch += g.n >> 5) {
    const int c = __reduce_add_sync(0xFFFFFFFFu, __popc(flags(ch)));
    if (lane == 0) t.cnt[ch] = c;
  }
  g.sync();
  int n = 0;
  for (int ch = 0; ch < chunks; ++ch) n += t.cnt[ch];
  for (int ch = g.tid >> 5; ch < chunks; ch += g.n >> 5) {
    int base = 0;
    for (int q = 0; q < ch; ++q) base += t.cnt[q];
    const uint32_t f = flags(ch);
    const int c = __popc(f);
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += y;
    }
    int pos = base + incl - c;
#pragma unroll
    for (int b = 0; b < 4; ++b)
      if ((f >> b) & 1u) t.ks[pos++] = (uint16_t)(4 * (32 * ch + lane) + b);
  }
  g.sync();
  constexpr int ld = M + kActPad;
#pragma unroll 2
  for (int i = g.tid; i < n * M; i += g.n) {
    const int j = i / M, r = i - j * M;
    t.A[j * ld + r] = (float)t.X[r * KP + t.ks[j]];
  }
  if (g.tid == 0) t.cnt[7] = n;
}

// First layer for m.sparse observations: each row is the default pattern (every word
// kSparseDefaultWord) except a few bytes, so W1 o + b1 = c + sum over the changed
// features f of (o_f - default_f) W1[:, f], with c = b1 + W1 x_default packed per policy.
// One warp per row lists the changed features in increasing order (list[r][0] = count,
// entries (f << 8) | (delta & 0xFF)); then every output adds its row's entries in that
// order, so the result is deterministic.  A row with more changed bytes than the list
// holds (any observation that is not of the pattern) takes the dense sum b1 + W1 o.
// Rows from `live` on are not computed.
template <int M>
__device__ __forceinline__ void sparse_l1_tile(const Group& g, const TileBufs& t, const MlpDims& m, int live,
                                               const float* __restrict__ Wt, const float* __restrict__ b1,
                                               const float* __restrict__ c) {
  constexpr int ld = M + kActPad;
  const int lane = g.tid & 31, warp = g.tid >> 5, nw = g.n >> 5;
  const uint8_t* X = t.X;
  const int words = m.K >> 2;
  for (int r = warp; r < live; r += nw) {
    const uint32_t* row = reinterpret_cast<const uint32_t*>(X + r * m.KP);
    uint32_t* L = t.list + r * kSparseCap;
    int base = 0;
    for (int w0 = 0; w0 < words; w0 += 32) {
      const int wi = w0 + lane;
      const uint32_t v = wi < words ? row[wi] : kSparseDefaultWord;
      int d[4], n = 0;
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        d[kk] = (int)((v >> (8 * kk)) & 0xFFu) - (int)((kSparseDefaultWord >> (8 * kk)) & 0xFFu);
        n += d[kk] != 0;
      }
      int incl = n;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += y;
      }
      int pos = base + incl - n;
#pragma unroll
      for (int kk = 0; kk < 4; ++kk)
        if (d[kk] != 0) {
          if (pos < kSparseCap - 1) L[1 + pos] = ((uint32_t)(4 * wi + kk) << 8) | ((uint32_t)d[kk] & 0xFFu);
          ++pos;
        }
      base += __shfl_sync(0xFFFFFFFFu, incl, 31);
    }
    if (lane == 0) L[0] = (uint32_t)base;
  }
  g.sync();
  const int ncb = m.H0 >> 2;
#pragma unroll 1
  for (int blk = g.tid; blk < live * ncb; blk += g.n) {
    const int r = blk / ncb, c0 = (blk - r * ncb) << 2;
    const uint32_t* L = t.list + r * kSparseCap;
    const int n = (int)L[0];
    float4 acc;
    if (n > kSparseCap - 1) {  // not of the pattern: the dense sum
      acc = __ldg(reinterpret_cast<const float4*>(b1 + c0));
      for (int k = 0; k < m.K; ++k) {
        const float x = (float)X[r * m.KP + k];
        const float4 wv = __ldg(reinterpret_cast<const float4*>(Wt + (int64_t)k * m.H0 + c0));
        acc.x = fmaf(x, wv.x, acc.x);
        acc.y = fmaf(x, wv.y, acc.y);
        acc.z = fmaf(x, wv.z, acc.z);
        acc.w = fmaf(x, wv.w, acc.w);
      }
    } else {
      acc = __ldg(reinterpret_cast<const float4*>(c + c0));
#pragma unroll 4
      for (int j = 1; j <= n; ++j) {
        const uint32_t e = L[j];
        const float dv = (float)(int8_t)(e & 0xFFu);
        const float4 wv = __ldg(reinterpret_cast<const float4*>(Wt + (int64_t)(e >> 8) * m.H0 + c0));
        acc.x = fmaf(dv, wv.x, acc.x);
        acc.y = fmaf(dv, wv.y, acc.y);
        acc.z = fmaf(dv, wv.z, acc.z);
        acc.w = fmaf(dv, wv.w, acc.w);
      }
    }
    float* o = t.B + c0 * ld + r;
    o[0] = tanhf(acc.x);
    o[ld] = tanhf(acc.y);
    o[2 * ld] = tanhf(acc.z);
    o[3 * ld] = tanhf(acc.w);
  }
}

// Whole policy forward for a tile: the observation buffer (bytes, or
// bit rows for kBits) -> Z.  The sparse first layer computes rows < live only (the others'
// outputs are then undefined).  o_tile and o_dims: shared-memory offsets of the tile's
// TileOffsets and of the MlpDims; o_w3: of load_w3's copy, or -1.  The group has synchronised
// since all of these were written; it synchronises between layers and at the end.  A
// function of its own, called once a step, keeps the compiler from carrying its address
// arithmetic through the rollout kernels' step loop (255 registers and spills when inlined
// there); it takes offsets because a pointer argument would make every shared-memory
// access a generic one (four times the time).
template <int M, bool kBits>
__device__ __forceinline__ void mlp_rows(const Group& g, const float* __restrict__ w, int o_w3, const MlpDims& m,
                                         const TileBufs& t, int live) {
  if (!kBits && m.sparse) {
    sparse_l1_tile<M>(g, t, m, live, w + m.oW1, w + m.ob1, w + m.oC);
  } else {
    const bool all = __ldg(w + m.oFin) == 0.0f;
    if constexpr (kBits) list_bits<M>(g, t, m.K, all);
    else list_bytes<M>(g, t, m.K, m.KP, all);
    g.sync();
    dense_tile<M, true>(g, t.A, t.cnt[kBits ? 0 : 7], t.ks, w + m.oW1, w + m.ob1, m.H0, t.B);
  }
  g.sync();
  dense_tile<M, false>(g, t.B, m.H0, nullptr, w + m.oW2, w + m.ob2, m.H1, t.A);
  g.sync();
  if (o_w3 >= 0)
    dense_out_n<M, true>(g, t.A, m.H1, reinterpret_cast<const float*>(tile_smem_ + o_w3), w + m.ob3, m.NOP, t.Z);
  else
    dense_out_n<M, false>(g, t.A, m.H1, w + m.oW3, w + m.ob3, m.NOP, t.Z);
  g.sync();
}
template <bool kBits>
__device__ __noinline__ void mlp_tile(int tid, int n, int bar, const float* __restrict__ w, int o_w3, int o_dims,
                                      int o_tile, int live) {
  const Group g{tid, n, bar};
  const MlpDims m = *reinterpret_cast<const MlpDims*>(tile_smem_ + o_dims);
  const TileOffsets to = *reinterpret_cast<const TileOffsets*>(tile_smem_ + o_tile);
  const TileBufs t = tile_bufs(to);
  switch (to.cfg.M) {  // tile_rows()
    case 8: mlp_rows<8, kBits>(g, w, o_w3, m, t, live); break;
    case 16: mlp_rows<16, kBits>(g, w, o_w3, m, t, live); break;
    default: mlp_rows<24, kBits>(g, w, o_w3, m, t, live); break;
  }
}

// Masked categorical inverse-CDF sample in fp32: a = min{k : u*Z < S_k} over the legal
// actions (S_k = sum_{j<=k} exp(z_j - max)), else the last legal action.  A compile-time
// action count keeps everything in registers.
template <int K, int N>
__device__ __forceinline__ int sample_k(const float (&z)[N], uint32_t legal, float u, float& logp) {
  static_assert(K <= N, "logit array shorter than the action count");
  float m = -INFINITY;
#pragma unroll
  for (int k = 0; k < K; ++k)
    if ((legal >> k) & 1u) m = fmaxf(m, z[k]);
  float S[K];
  float run = 0.0f;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    if ((legal >> k) & 1u) run = __fadd_rn(run, expf(z[k] - m));
    S[k] = run;
  }
  const float target = u * run;
  int a = -1;
#pragma unroll
  for (int k = K - 1; k >= 0; --k)
    if (target < S[k]) a = k;
  if (a < 0) {
#pragma unroll
    for (int k = 0; k < K; ++k)
      if ((legal >> k) & 1u) a = k;
  }
  float za = z[0];
#pragma unroll
  for (int k = 1; k < K; ++k)
    if (a == k) za = z[k];
  logp = za - m - logf(run);
  return a;
}

}  // namespace aht
