// rollout_impl.cuh -- fused persistent rollout kernels on CUDA cores, templated on the env
// rules.
//
// One CTA owns a tile of M envs for the whole call.  Env state lives in shared memory
// from the first step to the last; each step the CTA builds the observations of its
// envs in shared memory, runs the acting policies' MLPs over the tile, samples actions
// with Philox draws, steps the envs and streams the trajectory out.  Nothing but the
// trajectory (PPO) or the final returns (cross-play) goes back to HBM.
//
// Simultaneous games run the two seats at once, a group of kSeatThreads threads each with
// its own observation and activation buffers (Group, TileBufs): their policies are
// independent until the env step, and one seat's barriers, output layer and sampling hide
// under the other's products.  Turn-based games run the acting seat on the whole CTA.
#pragma once
#include "kernels.h"
#include "mlp_simt.cuh"

namespace aht {

constexpr int kTileThreads = 256;  // a CTA of the rollout kernels
constexpr int kSeatThreads = kTileThreads / 2;

// Shared memory of a CTA: the tile's states and per-env values, then `groups` sets of
// tile buffers (TileBufs) group_stride bytes apart from g0.
struct SmemLayout {
  int32_t st, envid, act, lp, val, alive, steps, bufs, dims, g0, group_stride, total;
  TileOffsets t;  // within a group
  int32_t w3, w3_bytes;  // W3 of the CTA's policies, w3_bytes apart
};

// policies: whose W3 cfg.w3 keeps here; bits: bit rows.
__host__ __device__ inline SmemLayout smem_layout(const TileCfg& cfg, const MlpDims& m, int state_bytes, int groups,
                                                  int policies, bool bits) {
  SmemLayout L;
  auto up16 = [](int32_t x) { return (x + 15) & ~15; };
  const int32_t M = cfg.M, ld = M + kActPad;
  int32_t o = 0;
  L.t.X = o;     o = up16(o + (bits ? (int32_t)M * bit_words(m.K) * 4 : (int32_t)M * m.KP));
  const int32_t cols = m.sparse ? m.H1 : (m.K > m.H1 ? m.K : m.H1);
  L.t.A = o;     o = up16(o + cols * ld * 4);
  L.t.B = o;     o = up16(o + (int32_t)m.H0 * ld * 4);
  L.t.Z = o;     o = up16(o + (int32_t)M * m.NOP * 4);
  L.t.ks = o;    o = up16(o + (m.sparse ? 0 : (int32_t)m.K * 2));
  L.t.list = o;  o = up16(o + (m.sparse ? (int32_t)M * kSparseCap * 4 : 0));
  L.t.cnt = o;   o = up16(o + 8 * 4);
  L.t.cfg = cfg;
  L.group_stride = o;
  o = 0;
  L.st = o;    o = up16(o + (int32_t)M * state_bytes);
  L.envid = o; o = up16(o + (int32_t)M * 4);
  L.act = o;   o = up16(o + (int32_t)M * 2);
  L.lp = o;    o = up16(o + (int32_t)M * 4);
  L.val = o;   o = up16(o + (int32_t)M * 4);
  L.alive = o; o = up16(o + (int32_t)M * 4);
  L.steps = o; o = up16(o + (int32_t)M * 4);
  L.bufs = o; o = up16(o + 2 * (int32_t)sizeof(TileOffsets));  // the groups' buffers and the dims, as
  L.dims = o; o = up16(o + (int32_t)sizeof(MlpDims));          // mlp_tile reads them
  L.w3 = o;
  L.w3_bytes = cfg.w3 ? up16(m.H1 * m.NOP * 4) : 0;
  o += policies * L.w3_bytes;
  L.g0 = o;
  L.total = o + groups * L.group_stride;
  return L;
}

__device__ __forceinline__ TileOffsets group_offsets(const SmemLayout& L, int group) {
  const int d = L.g0 + group * L.group_stride;
  return TileOffsets{L.t.X + d,  L.t.A + d,    L.t.B + d,   L.t.Z + d,
                     L.t.ks + d, L.t.list + d, L.t.cnt + d, L.t.cfg};
}

// All of an env's state words are requested at once (one memory latency, not one per
// word): the loads complete into registers before any is stored.
template <class S>
__device__ __forceinline__ void load_state(const uint32_t* __restrict__ g, int64_t n, int64_t e,
                                           S& s) {
  constexpr int kW = (int)(sizeof(S) / 4);
  uint32_t v[kW];
#pragma unroll
  for (int w = 0; w < kW; ++w) v[w] = __ldg(g + (int64_t)w * n + e);
  uint32_t* p = reinterpret_cast<uint32_t*>(&s);
#pragma unroll
  for (int w = 0; w < kW; ++w) p[w] = v[w];
}

template <class S>
__device__ __forceinline__ void store_state(uint32_t* __restrict__ g, int64_t n, int64_t e,
                                            const S& s) {
  const uint32_t* p = reinterpret_cast<const uint32_t*>(&s);
#pragma unroll
  for (int w = 0; w < (int)(sizeof(S) / 4); ++w) g[(int64_t)w * n + e] = p[w];
}

// The tile's observation rows for `seat`, rows i < count of st (a row with alive[i] == 0 is
// empty), zero (bit rows) or untouched (byte rows) past them.  The group synchronises at
// the end.  Bit rows: one thread per row, the env's word writer; byte rows (LBF): the
// row's words divided among the group's g.n / M threads per row.
template <class Env>
__device__ __forceinline__ void build_obs(const Group& g, const DevEnv& env, const typename Env::State* st, int seat,
                                          int count, int M, const MlpDims& m, const TileBufs& t,
                                          const int32_t* alive) {
  if constexpr (Env::kBinaryObs) {
    const int bw = bit_words(m.K);
    uint32_t* bits = reinterpret_cast<uint32_t*>(t.X);
    for (int i = g.tid; i < M; i += g.n) {
      ObsBits wr{bits + i * bw, bw};
      if (i < count && (!alive || alive[i])) Env::obs_into(env, st[i], seat, wr);
      else wr.clear();
    }
  } else {
    const int words = m.K >> 2, per_row = g.n / M > 0 ? g.n / M : 1;
    const int chunk = (words + per_row - 1) / per_row;
    for (int q = g.tid; q < count * per_row; q += g.n) {
      const int i = q / per_row, p = q - i * per_row, w0 = min(p * chunk, words);
      if (!alive || alive[i])
        Env::obs_words(env, st[i], seat, reinterpret_cast<uint32_t*>(t.X + i * m.KP), w0, min(w0 + chunk, words));
    }
  }
  g.sync();
}

// Copies `count` observation rows (row i goes to dst row ids[i]) as 32-bit words of bytes.
template <bool kBits>
__device__ __forceinline__ void copy_obs_rows(const Group& g, const TileBufs& t, const MlpDims& m, int count,
                                              const int32_t* ids, uint8_t* dst) {
  const int wpr = m.K >> 2, bw = bit_words(m.K);
  uint32_t* d = reinterpret_cast<uint32_t*>(dst);
  for (int idx = g.tid; idx < count * wpr; idx += g.n) {
    const int i = idx / wpr, w = idx - i * wpr;
    uint32_t v;
    if constexpr (kBits) {  // four features: bit b of the nibble to byte b
      const uint32_t nib = (reinterpret_cast<const uint32_t*>(t.X)[i * bw + (w >> 3)] >> (4 * (w & 7))) & 15u;
      v = (nib * 0x00204081u) & 0x01010101u;
    } else {
      v = reinterpret_cast<const uint32_t*>(t.X + i * m.KP)[w];
    }
    d[(int64_t)ids[i] * wpr + w] = v;
  }
}

// ---- PPO rollout collection ------------------------------------------------------------
template <class Env>
__global__ void __launch_bounds__(kTileThreads, 1) ppo_kernel(const PpoArgs a) {
  using State = typename Env::State;
  constexpr int NA = Env::kNumActions;
  constexpr bool kBits = Env::kBinaryObs;
  uint8_t* const smem = tile_smem_;
  const int4 tile = a.tiles[blockIdx.x];
  const int count = tile.y;
  if (count == 0) return;
  const int M = a.cfg.M;
  const MlpDims& m = a.b.mlp;
  const SmemLayout L = smem_layout(a.cfg, m, sizeof(State), 2, 2, kBits);
  State* st = reinterpret_cast<State*>(smem + L.st);
  int32_t* envid = reinterpret_cast<int32_t*>(smem + L.envid);
  uint8_t* act = smem + L.act;
  float* lp = reinterpret_cast<float*>(smem + L.lp);
  float* val = reinterpret_cast<float*>(smem + L.val);
  const int tid = threadIdx.x, seat = tid / kSeatThreads;
  const Group g{tid - seat * kSeatThreads, kSeatThreads, 1 + seat};
  TileOffsets* bufs = reinterpret_cast<TileOffsets*>(smem + L.bufs);
  MlpDims* dims = reinterpret_cast<MlpDims*>(smem + L.dims);
  const TileOffsets to = group_offsets(L, seat);
  const TileBufs t = tile_bufs(to);
  if (g.tid == 0) bufs[seat] = to;
  if (tid == 0) *dims = m;
  const int64_t N = a.n_envs;
  const int od = a.b.env.obs_dim;
  const TrajPtrs& traj = seat == 0 ? a.traj : a.traj1;  // this seat's learner fields

  for (int i = tid; i < count; i += blockDim.x) {
    const int env = a.perm[tile.x + i];
    envid[i] = env;
    load_state(a.state, N, env, st[i]);
  }
  if (!kBits)  // padding columns and the rows past count stay zero
    for (int i = g.tid; i < M * (m.KP >> 2); i += g.n) reinterpret_cast<uint32_t*>(t.X)[i] = 0u;
  const float* w_pol = a.b.weights + (int64_t)(seat == 0 ? a.ego : tile.z) * m.stride;
  const int o_w3 = a.cfg.w3 ? L.w3 + seat * L.w3_bytes : -1;
  if (o_w3 >= 0) load_w3(g, w_pol, m, reinterpret_cast<float*>(smem + o_w3));
  __syncthreads();

  // Steps 0..T-1, then the bootstrap value V_T of the state after the last step where asked.
  for (int s = 0; s <= a.T; ++s) {
    const bool boot = s == a.T;
    const uint32_t gt = a.step0 + (uint32_t)s;
    if (!boot || traj.last_value) {
      build_obs<Env>(g, a.b.env, st, seat, count, M, m, t, nullptr);
      if (!boot && traj.obs) copy_obs_rows<kBits>(g, t, m, count, envid, traj.obs + (int64_t)s * N * od);
      mlp_tile<kBits>(g.tid, g.n, g.bar, w_pol, o_w3, L.dims, L.bufs + seat * (int)sizeof(TileOffsets), count);
    }
    if (boot) {
      if (traj.last_value)
        for (int i = g.tid; i < count; i += g.n) traj.last_value[envid[i]] = t.Z[i * m.NOP + NA];
      break;
    }
    for (int i = g.tid; i < count; i += g.n) {
      const float u = u01(draw0(a.b.key, (uint32_t)envid[i], gt, kStreamAct0 + seat));
      float z[NA];
#pragma unroll
      for (int o = 0; o < NA; ++o) z[o] = t.Z[i * m.NOP + o];
      float logp;
      act[i * 2 + seat] = (uint8_t)sample_k<NA>(z, 0xFFFFFFFFu >> (32 - NA), u, logp);
      const float v = t.Z[i * m.NOP + NA];
      if (seat == 0) {
        lp[i] = logp;
        val[i] = v;
      } else {
        const int64_t o = (int64_t)s * N + envid[i];
        if (traj.logp) traj.logp[o] = logp;
        if (traj.values) traj.values[o] = v;
      }
    }
    __syncthreads();
    for (int i = tid; i < count; i += blockDim.x) {
      const int env = envid[i];
      float r0, r1, team;
      const int done = Env::step(a.b.env, st[i], act[2 * i], act[2 * i + 1], r0, r1, team);
      const int64_t o = (int64_t)s * N + env;
      if (a.traj.actions) a.traj.actions[o] = act[2 * i];
      if (a.traj.tm_actions) a.traj.tm_actions[o] = act[2 * i + 1];
      if (a.traj.logp) a.traj.logp[o] = lp[i];
      if (a.traj.values) a.traj.values[o] = val[i];
      if (a.traj.rewards) a.traj.rewards[o] = team;
      if (a.traj.dones) a.traj.dones[o] = (uint8_t)(done > 0);
      if (a.traj1.actions) a.traj1.actions[o] = act[2 * i + 1];
      if (a.traj1.tm_actions) a.traj1.tm_actions[o] = act[2 * i];
      if (a.traj1.rewards) a.traj1.rewards[o] = team;
      if (a.traj1.dones) a.traj1.dones[o] = (uint8_t)(done > 0);
      if (done > 0) {
        Env::reset(a.b.env, a.b.key, (uint32_t)env, gt + 1, st[i]);
        if (a.ep_step) a.ep_step[env] = gt + 1;
      }
    }
    __syncthreads();
  }
  for (int i = tid; i < count; i += blockDim.x) store_state(a.state, N, envid[i], st[i]);
}

// ---- cross-play evaluation --------------------------------------------------------------
template <class Env>
__global__ void __launch_bounds__(kTileThreads, 1) xplay_kernel(const XpArgs a) {
  using State = typename Env::State;
  constexpr int NA = Env::kNumActions;
  constexpr bool kBits = Env::kBinaryObs, kTurn = Env::kTurnBased;
  uint8_t* const smem = tile_smem_;
  const int M = a.cfg.M;
  const MlpDims& m = a.b.mlp;
  const SmemLayout L = smem_layout(a.cfg, m, sizeof(State), kTurn ? 1 : 2, 2, kBits);
  State* st = reinterpret_cast<State*>(smem + L.st);
  uint8_t* act = smem + L.act;
  int32_t* alive = reinterpret_cast<int32_t*>(smem + L.alive);
  int32_t* nsteps = reinterpret_cast<int32_t*>(smem + L.steps);
  const int tid = threadIdx.x, half = tid / kSeatThreads;
  const Group g = kTurn ? Group{tid, kTileThreads, 1} : Group{tid - half * kSeatThreads, kSeatThreads, 1 + half};
  TileOffsets* bufs = reinterpret_cast<TileOffsets*>(smem + L.bufs);
  MlpDims* dims = reinterpret_cast<MlpDims*>(smem + L.dims);
  const int set = kTurn ? 0 : half;
  const TileOffsets to = group_offsets(L, set);
  const TileBufs t = tile_bufs(to);
  if (g.tid == 0) bufs[set] = to;
  if (tid == 0) *dims = m;

  const int pair = blockIdx.x / a.tiles_per_pair;
  const int first = (blockIdx.x - pair * a.tiles_per_pair) * M;
  const int count = min(M, a.P - first);
  const int64_t e0 = (int64_t)pair * a.P + first;
  const int64_t n_total = (int64_t)a.n_ego * a.n_tm * a.P;
  const float* w_pol[2] = {a.b.weights + (int64_t)a.ego_ids[pair / a.n_tm] * m.stride,
                           a.b.weights + (int64_t)a.tm_ids[pair % a.n_tm] * m.stride};

  for (int i = tid; i < M; i += blockDim.x) {
    if (i < count) Env::reset(a.b.env, a.b.key, (uint32_t)(e0 + i), a.step0, st[i]);
    alive[i] = i < count;
    nsteps[i] = 0;
  }
  if (!kBits)
    for (int i = g.tid; i < M * (m.KP >> 2); i += g.n) reinterpret_cast<uint32_t*>(t.X)[i] = 0u;
  const bool w3s = a.cfg.w3 != 0;
  for (int p = 0; w3s && p < 2; ++p)
    load_w3(Group{tid, kTileThreads, 0}, w_pol[p], m, reinterpret_cast<float*>(smem + L.w3 + p * L.w3_bytes));
  __syncthreads();

  for (int s = 0; s < a.max_steps; ++s) {
    if (!__syncthreads_or(tid < count && alive[tid])) break;
    const uint32_t gt = a.step0 + (uint32_t)s;
    const int actor = kTurn ? (s & 1) : -1;
    const int seat = kTurn ? actor : half;
    build_obs<Env>(g, a.b.env, st, seat, count, M, m, t, alive);
    mlp_tile<kBits>(g.tid, g.n, g.bar, seat ? w_pol[1] : w_pol[0], w3s ? L.w3 + seat * L.w3_bytes : -1, L.dims,
                    L.bufs + set * (int)sizeof(TileOffsets), count);
    for (int i = g.tid; i < count; i += g.n) {
      if (!alive[i]) continue;
      uint32_t legal = 0xFFFFFFFFu >> (32 - NA);
      if (kTurn) {
        legal = Env::legal(st[i]);
        if (Env::actor(st[i]) != seat) atomicOr(a.b.status, kStatusActorMismatch);
      }
      const float u = u01(draw0(a.b.key, (uint32_t)(e0 + i), gt, kStreamAct0 + seat));
      float z[NA];
#pragma unroll
      for (int o = 0; o < NA; ++o) z[o] = t.Z[i * m.NOP + o];
      float logp;
      act[i * 2 + seat] = (uint8_t)sample_k<NA>(z, legal, u, logp);
    }
    __syncthreads();
    for (int i = tid; i < count; i += blockDim.x) {
      const int64_t e = e0 + i;
      // (the host pre-fills the optional action record with 255 = no action)
      uint8_t* rec = a.actions ? a.actions + ((int64_t)s * n_total + e) * 2 : nullptr;
      if (!alive[i]) continue;
      const int a0 = (actor < 0 || actor == 0) ? act[2 * i] : 0;
      const int a1 = (actor < 0 || actor == 1) ? act[2 * i + 1] : 0;
      if (rec) {
        rec[0] = (actor < 0 || actor == 0) ? (uint8_t)a0 : 255;
        rec[1] = (actor < 0 || actor == 1) ? (uint8_t)a1 : 255;
      }
      float r0, r1, team;
      const int done = Env::step(a.b.env, st[i], a0, a1, r0, r1, team);
      if (done < 0) {
        atomicOr(a.b.status, kStatusIllegalAction);
        alive[i] = 0;
        continue;
      }
      nsteps[i] += 1;
      if (done) alive[i] = 0;
    }
    __syncthreads();
  }
  for (int i = tid; i < count; i += blockDim.x) {
    a.returns[e0 + i] = Env::ret(st[i]);
    if (a.steps) a.steps[e0 + i] = nsteps[i];
  }
}

// ---- forced step, reset, policy forward --------------------------------------------------
template <class Env>
__global__ void forced_kernel(const ForcedArgs a) {
  using State = typename Env::State;
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= a.n_envs) return;
  State s;
  load_state(a.state, a.n_envs, e, s);
  float r0, r1, team;
  int done = Env::step(a.b.env, s, a.actions[2 * e], a.actions[2 * e + 1], r0, r1, team);
  if (done < 0) {
    atomicOr(a.b.status, kStatusIllegalAction);
    load_state(a.state, a.n_envs, e, s);
    done = 0;
    r0 = r1 = team = 0.0f;
  }
  if (done) {
    Env::reset(a.b.env, a.b.key, (uint32_t)e, a.step + 1, s);
    if (a.ep_step) a.ep_step[e] = a.step + 1;
  }
  if (a.rewards) { a.rewards[2 * e] = r0; a.rewards[2 * e + 1] = r1; }
  if (a.team) a.team[e] = team;
  if (a.dones) a.dones[e] = (uint8_t)done;
  if (a.obs) {
    const int od = a.b.env.obs_dim;
    Env::obs(a.b.env, s, 0, a.obs + (2 * e) * od);
    Env::obs(a.b.env, s, 1, a.obs + (2 * e + 1) * od);
  }
  store_state(a.state, a.n_envs, e, s);
}

template <class Env>
__global__ void reset_kernel(const ResetArgs a) {
  using State = typename Env::State;
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= a.n_envs) return;
  State s;
  Env::reset(a.b.env, a.b.key, (uint32_t)e, a.step, s);
  store_state(a.state, a.n_envs, e, s);
  if (a.ep_step) a.ep_step[e] = a.step;
}

template <class Env>
struct Launch {
  using State = typename Env::State;
  static cudaError_t ppo(const PpoArgs& a, int grid, size_t smem, cudaStream_t s) {
    ppo_kernel<Env><<<grid, kTileThreads, smem, s>>>(a);
    return cudaGetLastError();
  }
  static cudaError_t xplay(const XpArgs& a, int grid, size_t smem, cudaStream_t s) {
    xplay_kernel<Env><<<grid, kTileThreads, smem, s>>>(a);
    return cudaGetLastError();
  }
  static cudaError_t forced(const ForcedArgs& a, cudaStream_t s) {
    const int blocks = (int)((a.n_envs + 127) / 128);
    forced_kernel<Env><<<blocks, 128, 0, s>>>(a);
    return cudaGetLastError();
  }
  static cudaError_t reset(const ResetArgs& a, cudaStream_t s) {
    const int blocks = (int)((a.n_envs + 127) / 128);
    reset_kernel<Env><<<blocks, 128, 0, s>>>(a);
    return cudaGetLastError();
  }
  static cudaError_t smem_limit(size_t bytes) {
    cudaError_t e = cudaFuncSetAttribute(ppo_kernel<Env>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(xplay_kernel<Env>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  }
};

#define AHT_DEFINE_ENV_LAUNCHERS(name, EnvT)                                                   \
  cudaError_t name##_ppo(const PpoArgs& a, int g, size_t sm, cudaStream_t s) {                  \
    return Launch<EnvT>::ppo(a, g, sm, s);                                                     \
  }                                                                                            \
  cudaError_t name##_xplay(const XpArgs& a, int g, size_t sm, cudaStream_t s) {                 \
    return Launch<EnvT>::xplay(a, g, sm, s);                                                   \
  }                                                                                            \
  cudaError_t name##_forced(const ForcedArgs& a, cudaStream_t s) { return Launch<EnvT>::forced(a, s); } \
  cudaError_t name##_reset(const ResetArgs& a, cudaStream_t s) { return Launch<EnvT>::reset(a, s); }    \
  int name##_state_words() { return (int)(sizeof(EnvT::State) / 4); }                          \
  int name##_state_bytes() { return (int)sizeof(EnvT::State); }                                \
  cudaError_t name##_set_smem_limit(size_t b) { return Launch<EnvT>::smem_limit(b); }            \
  int name##_occupancy(int which, size_t sm) {                                                 \
    int n = 0;                                                                                 \
    if (which == 0) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, ppo_kernel<EnvT>, kTileThreads, sm); \
    else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, xplay_kernel<EnvT>, kTileThreads, sm);  \
    cudaGetLastError();                                                                        \
    return n;                                                                                  \
  }

}  // namespace aht
