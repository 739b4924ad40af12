// Actor kernel of the linear-Gaussian env on the FP32 pipes (FP32 contexts, and the environment half of BF16 contexts whose shape
// no fused tensor-core actor takes): policy inference, selection, environment step and the version-tagged record for a tile of
// environments, looped over n_steps inside one launch; and the initial states of every env.  CartPole and Acrobot: tj_actor_fma.cu.
//
// Environments are independent, so a thread block keeps its TE environments (state in shared memory) for the whole call and no
// block ever waits on another.  The ring cursor advances by N per step, which every block can compute on its own.
#include "tj_async.cuh"
#include "tj_device.cuh"
#include "tj_internal.h"
#include "tj_mlp.cuh"

namespace tj {

namespace {

struct ActorSmem {
  float *xs, *h1, *h2, *out, *nxt, *rew;
  int *act, *done;
};

inline size_t actor_smem_floats(int TE, int D, int Hp, int Ap) {
  const int Dx = (D + 3) & ~3;
  return 2 * (size_t)Dx * TE + 2 * (size_t)Hp * TE + (size_t)Ap * TE + 3 * TE;   // + rew, act, done
}

__device__ inline ActorSmem carve(float* base, int TE, int D, int Hp, int Ap) {
  const int Dx = (D + 3) & ~3;
  ActorSmem s;
  s.xs = base; base += (size_t)Dx * TE;
  s.h1 = base; base += (size_t)Hp * TE;
  s.h2 = base; base += (size_t)Hp * TE;
  s.out = base; base += (size_t)Ap * TE;
  s.nxt = base; base += (size_t)Dx * TE;
  s.rew = base; base += TE;
  s.act = reinterpret_cast<int*>(base); base += TE;
  s.done = reinterpret_cast<int*>(base);
  return s;
}

__device__ __forceinline__ float4 reset4(uint2 seed, uint32_t block, uint32_t e, unsigned long long step, float lo,
                                         float width) {
  const uint4 w = stream_words(seed, STREAM_RESET, block, e, step);
  return make_float4(uniform_range(w.x, lo, width), uniform_range(w.y, lo, width), uniform_range(w.z, lo, width),
                     uniform_range(w.w, lo, width));
}

// ------------------------------------------------------------------------------------------------
// Linear-Gaussian env: the state (= observation) of the tile lives in shared memory, k-major.
// ------------------------------------------------------------------------------------------------
template <int TE, int NT>
__global__ void __launch_bounds__(NT) actor_lingauss_kernel(const ActorParams p) {
  extern __shared__ __align__(128) float smem[];
  const bool ext = p.logits_in != nullptr;   // network outputs come from the tensor-core kernel
  const ActorSmem sm = carve(smem, TE, p.D, ext ? 0 : p.Hp, ext ? 0 : p.Ap);
  __shared__ uint64_t unused_bar;
  const MlpWeights mw = stage_mlp_weights<0>(p, p.W, nullptr, &unused_bar, false);
  const int tid = threadIdx.x;
  const int e0 = blockIdx.x * TE;
  const int D = p.D, Dp = (p.D + 3) & ~3;
  const int n_here = min(TE, p.N - e0);
  chain_begin();

  // state -> xs[k][e]
  for (int i = tid; i < TE * D; i += NT) {
    const int el = i / D, k = i % D;
    sm.xs[k * TE + el] = el < n_here ? p.state[(size_t)(e0 + el) * D + k] : 0.f;
  }
  int ep = 0;
  float ep_ret = 0.f;
  if (tid < n_here) {
    ep = p.ep_step[e0 + tid];
    ep_ret = p.ep_return[e0 + tid];
  }
  unsigned long long n_episodes = 0;
  double ret_sum = 0.0;
  __syncthreads();

  for (int step = 0; step < p.n_steps; ++step) {
    const unsigned long long t = (unsigned long long)p.t0 + step;
    if (!ext) mlp_forward_tile<TE, NT, 4, false, false>(mw, D, p.H, p.Hp, p.Aout, p.Ap, sm.xs, sm.h1, sm.h2, sm.out);
    if (tid < TE) {
      int a = 0;
      if (tid < n_here) {
        const int e = e0 + tid;
        auto logit = [&](int i) { return ext ? p.logits_in[(size_t)e * p.A + i] : sm.out[i * TE + tid]; };
        if (p.dbg_logits) {
          float* dl = p.dbg_logits + ((size_t)step * p.N + e) * p.A;
          for (int i = 0; i < p.A; ++i) dl[i] = logit(i);
        }
        const uint4 w = stream_words(p.seed, STREAM_ACTION, 0, (uint32_t)e, t);
        a = select_eps_greedy(p.A, logit, w, p.explore_thr);
      }
      sm.act[tid] = a;
    }
    __syncthreads();
    // s' = tanh(A s + B[a]) ...
    dense_layer<TE, NT, 4, ACT_TANH, true, false>(p.lgAt, p.lgB, Dp, D, D, sm.xs, sm.nxt, sm.act);
    __syncthreads();
    // ... + noise_std * n, four normals per Philox call
    for (int i = tid; i < TE * (D / 4); i += NT) {
      const int el = i % TE, b = i / TE;
      if (el < n_here) {
        const uint4 w = stream_words(p.seed, STREAM_NOISE, (uint32_t)b, (uint32_t)(e0 + el), t);
        const float2 z01 = box_muller(w.x, w.y), z23 = box_muller(w.z, w.w);
        sm.nxt[(4 * b + 0) * TE + el] += p.lg_noise_std * z01.x;
        sm.nxt[(4 * b + 1) * TE + el] += p.lg_noise_std * z01.y;
        sm.nxt[(4 * b + 2) * TE + el] += p.lg_noise_std * z23.x;
        sm.nxt[(4 * b + 3) * TE + el] += p.lg_noise_std * z23.y;
      }
    }
    __syncthreads();
    if (tid < TE) {
      int done = 0;
      float rew = 0.f;
      if (tid < n_here) {
        float sq = 0.f;
        for (int k = 0; k < D; ++k) {
          const float v = sm.nxt[k * TE + tid];
          sq = fmaf(v, v, sq);
        }
        rew = -sq / (float)D;
        ep += 1;
        done = (sqrtf(sq) > p.lg_done_norm || ep >= p.max_ep) ? 1 : 0;
        ep_ret += rew;
        if (done) {
          n_episodes += 1;
          ret_sum += (double)ep_ret;
          ep_ret = 0.f;
          ep = 0;
        }
      }
      sm.done[tid] = done;
      sm.rew[tid] = rew;
    }
    __syncthreads();
    // record rows: [obs D][next_obs D][act, rew, done, ver]
    {
      const int rw = p.rec_words;
      for (int i = tid; i < n_here * rw; i += NT) {
        const int el = i / rw, w = i % rw;
        const unsigned long long slot = (p.cursor0 + (unsigned long long)step * p.N + (e0 + el)) % (unsigned long long)p.C;
        float v;
        if (w < D) v = sm.xs[w * TE + el];
        else if (w < 2 * D) v = sm.nxt[(w - D) * TE + el];
        else if (w == 2 * D) v = __int_as_float(sm.act[el]);
        else if (w == 2 * D + 1) v = sm.rew[el];
        else if (w == 2 * D + 2) v = __int_as_float(sm.done[el]);
        else v = __int_as_float(p.version);
        p.ring[slot * rw + w] = v;
      }
    }
    if (blockIdx.x == 0 && tid == 0)
      p.block_ver[((p.cursor0 + (unsigned long long)step * p.N) % (unsigned long long)p.C) / p.N] = p.version;
    __syncthreads();
    // next state: the stepped state, or a fresh draw for finished episodes
    for (int i = tid; i < TE * (D / 4); i += NT) {
      const int el = i % TE, b = i / TE;
      float4 v;
      if (el < n_here && sm.done[el]) {
        v = reset4(p.seed, (uint32_t)b, (uint32_t)(e0 + el), t, -0.1f, 0.2f);
      } else {
        v = make_float4(sm.nxt[(4 * b + 0) * TE + el], sm.nxt[(4 * b + 1) * TE + el], sm.nxt[(4 * b + 2) * TE + el],
                        sm.nxt[(4 * b + 3) * TE + el]);
      }
      sm.xs[(4 * b + 0) * TE + el] = v.x;
      sm.xs[(4 * b + 1) * TE + el] = v.y;
      sm.xs[(4 * b + 2) * TE + el] = v.z;
      sm.xs[(4 * b + 3) * TE + el] = v.w;
    }
    __syncthreads();
  }
  for (int i = tid; i < n_here * D; i += NT) {
    const int el = i / D, k = i % D;
    p.state[(size_t)(e0 + el) * D + k] = sm.xs[k * TE + el];
  }
  if (tid < n_here) {
    p.ep_step[e0 + tid] = ep;
    p.ep_return[e0 + tid] = ep_ret;
    if (n_episodes) {
      atomicAdd(&p.stats->episodes, n_episodes);
      atomicAdd(&p.stats->return_sum, ret_sum);
    }
  }
}

__global__ void init_env_kernel(int env_kind, int N, int S_d, uint2 seed, float* state, int* ep_step, float* ep_return) {
  chain_begin();
  const int nb = S_d / 4;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (long long)N * nb) return;
  const int e = (int)(i / nb), b = (int)(i % nb);
  const float lo = env_kind == TJ_ENV_CARTPOLE ? -0.05f : -0.1f, width = env_kind == TJ_ENV_CARTPOLE ? 0.1f : 0.2f;
  reinterpret_cast<float4*>(state + (size_t)e * S_d)[b] = reset4(seed, (uint32_t)b, (uint32_t)e, ~0ull, lo, width);
  if (b == 0) {
    ep_step[e] = 0;
    ep_return[e] = 0.f;
  }
}

constexpr size_t kSmemMax = 227 * 1024 - 1024;   // per block, leaving room for static shared memory
}  // namespace

cudaError_t launch_init_env(int env_kind, int N, int S_d, uint2 seed, float* state, int* ep_step, float* ep_return,
                            cudaStream_t s) {
  const long long n = (long long)N * (S_d / 4);
  return launch_chained(init_env_kernel, (unsigned)((n + 255) / 256), 256, 0, s, env_kind, N, S_d, seed, state, ep_step, ep_return);
}

cudaError_t launch_actor(int env_kind, const ActorParams& p, int sm_count, cudaStream_t s) {
  if (env_kind != TJ_ENV_LINGAUSS) return launch_actor_fma(env_kind, p, sm_count, s);
  constexpr int TE = 32, NT = 256;
  const bool ext = p.logits_in != nullptr;
  const size_t smem = actor_smem_floats(TE, p.D, ext ? 0 : p.Hp, ext ? 0 : p.Ap) * sizeof(float);
  if (smem > kSmemMax) return cudaErrorInvalidConfiguration;
  return launch_chained<1024>(actor_lingauss_kernel<TE, NT>, (p.N + TE - 1) / TE, NT, smem, s, p);
}

}  // namespace tj
