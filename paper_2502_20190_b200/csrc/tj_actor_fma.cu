// FP32 actor for CartPole and Acrobot: policy inference, action selection, environment step and the version-tagged trajectory
// write for a tile of environments, looped over n_steps inside one launch.  Environments are independent, so a block keeps its
// E environments (state in shared memory) for the whole call and no block waits on another.
//
// The fixed FMA order makes every output a chain of K dependent FMAs, so a small number of environments is bound by that latency
// and by everything else a step does one after the other; a large one by the FP32 pipes and the operand loads that feed them.  E is
// the number of environments that spreads the call over the SMs once, and the threads' register tile grows with it: 4 rows x 1
// neuron while the chain is the bound, 8 x 4 where the FMAs are (tj_fma.cuh).  The hidden x hidden matrix sits in shared memory where
// it fits beside the activations; wider ones (hidden 256: 256 KB) stream through a ring of 16 KB chunks once per step for all E
// environments.
// The head's outputs and the environment step belong to the same lanes, four per environment: lane a sums output a, the four
// outputs meet by shuffle, all four lanes step the environment (the same instructions; Acrobot's sines are spread over them) and
// each writes its quarter of the record.  Three block barriers per step.  Positions in the ring and the segment advance by additions
// (64-bit divisions by the capacity cost 500 cycles per step), and the Philox words of the next step are drawn by warps that the head
// leaves idle.
#include "tj_async.cuh"
#include "tj_device.cuh"
#include "tj_fma.cuh"
#include "tj_internal.h"

namespace tj {

namespace {

constexpr int AF_SLOTS = 4;
enum { AF_SMEM = 0, AF_RING = 1 };   // where W2 is read from

struct AfPlan {
  int E, EG, NG, half, n_compute;           // environments per block; row quads x neuron groups; computing threads
  int nt, ldh, overlap, kc;                         // threads; row stride of h2; h2 lies over h1; rows of W2 per chunk
  int gap;                                          // floats of the packed parameters that are not staged (W2 in a ring)
  int w, w2, xs, h1, h2, w3, pw, env, bar;          // offsets in shared memory, floats
  long long slot0;                                  // ring slot of env 0 in the first step
  int blk0, n_blk;                                  // its ring block, blocks of the ring
  int pos0, seg0;                                   // position in the running segment, its slot
};

__device__ __forceinline__ float4 reset4(uint2 seed, uint32_t block, uint32_t e, unsigned long long step, float lo, float width) {
  const uint4 w = stream_words(seed, STREAM_RESET, block, e, step);
  return make_float4(uniform_range(w.x, lo, width), uniform_range(w.y, lo, width), uniform_range(w.z, lo, width),
                     uniform_range(w.w, lo, width));
}

// Acrobot's angles with their sines spread over the four lanes of an environment: lane 0 takes th1, lane 1 th1 + th2, the others th2
struct AcrobotAngles { float4 trig; float s12, c12; };       // trig = (cos th1, sin th1, cos th2, sin th2)
__device__ __forceinline__ AcrobotAngles acrobot_angles4(float4 s, int lane) {
  const int a = lane & 3, base = lane & ~3;
  float sn, cs;
  sincosf(a == 0 ? s.x : (a == 1 ? s.x + s.y : s.y), &sn, &cs);
  AcrobotAngles r;
  r.trig = make_float4(__shfl_sync(0xffffffffu, cs, base), __shfl_sync(0xffffffffu, sn, base), __shfl_sync(0xffffffffu, cs, base + 2),
                       __shfl_sync(0xffffffffu, sn, base + 2));
  r.s12 = __shfl_sync(0xffffffffu, sn, base + 1);
  r.c12 = __shfl_sync(0xffffffffu, cs, base + 1);
  return r;
}

// one RK4 step as in acrobot_step; `at`: the angles of s on entry (the first stage's), of the new state on return (its observation and tip)
__device__ __forceinline__ StepResult acrobot_step4(float4 s, AcrobotAngles& at, int act, int lane, float4& sn) {
  constexpr float dt = 0.2f, PI = 3.14159265358979323846f;
  const float torque = (float)(act - 1);
  float4 k1, acc, y = s;
  k1 = acc = make_float4(0.f, 0.f, 0.f, 0.f);
  // stages 1 .. 4 in one copy of the derivative's code; the sums keep acrobot_step's order k1 + 2 k2 + 2 k3 + k4
#pragma unroll 1
  for (int st = 0; st < 4; ++st) {
    if (st > 0) at = acrobot_angles4(y, lane);
    k1 = acrobot_deriv(y, torque, at.trig.y, at.s12, at.trig.w, at.trig.z);
    if (st == 0) acc = k1;
    else if (st == 3) acc = make_float4(acc.x + k1.x, acc.y + k1.y, acc.z + k1.z, acc.w + k1.w);
    else acc = make_float4(acc.x + 2.0f * k1.x, acc.y + 2.0f * k1.y, acc.z + 2.0f * k1.z, acc.w + 2.0f * k1.w);
    y = axpy4(s, st == 2 ? dt : 0.5f * dt, k1);
  }
  y.x = s.x + dt / 6.0f * acc.x;
  y.y = s.y + dt / 6.0f * acc.y;
  y.z = s.z + dt / 6.0f * acc.z;
  y.w = s.w + dt / 6.0f * acc.w;
  sn.x = wrap_pi(y.x);
  sn.y = wrap_pi(y.y);
  sn.z = fminf(fmaxf(y.z, -4.0f * PI), 4.0f * PI);
  sn.w = fminf(fmaxf(y.w, -9.0f * PI), 9.0f * PI);
  at = acrobot_angles4(sn, lane);
  const float tip = -at.trig.x - at.c12;
  StepResult r;
  r.terminated = tip > 1.0f;
  r.reward = r.terminated ? 0.0f : -1.0f;
  return r;
}

// one environment between steps; trig = (cos th1, sin th1, cos th2, sin th2) and s12 = sin(th1 + th2) of an Acrobot state
struct __align__(16) AfEnv { float4 s, trig; int ep; float ret; int episodes; float s12; double ret_sum, pad2; };

// One chunk of W2 (kc rows, chunk c of a step, number g of the stream) into slot g mod AF_SLOTS; the chunk that was there is used up
__device__ __forceinline__ void af_queue_chunk(float* ring, const float* W2, uint64_t* full, uint32_t g, uint32_t c, int kc, int H, int Hp) {
  const uint32_t s = g % AF_SLOTS, bytes = (uint32_t)(min(kc, H - (int)c * kc) * Hp * 4);
  mbar_expect_tx(full + s, bytes);
  bulk_copy_g2s(ring + s * (kc * Hp), W2 + (size_t)c * kc * Hp, bytes, full + s);
}

template <int EPT, int NPT>
__device__ __forceinline__ void af_layer1(const float* b1, const float* W1t, const float* xs, float* h1, int E, int Hp, int D, const FmaTile t,
                                          bool computes) {
  if (!computes) return;
  FmaAcc<EPT, NPT> acc;
  fma_bias<EPT, NPT>(acc, b1, t);
  fma_accumulate<EPT, NPT, (EPT * NPT > 16 ? 1 : 6)>(acc, W1t, Hp, xs, E, D, t);
  fma_store_kmajor(acc, h1, E, t);
}

struct AfHidden {
  const float *w, *src, *b, *h1;                    // W2 in shared memory (or the ring) and in global memory
  float* h2;
  uint64_t* full;                                   // full[SLOTS], empty[SLOTS]
  unsigned long long* error;
  int E, H, Hp, ldh, kc, overlap, warps, n_chunks;
  uint32_t g0;                                      // number of the step's first chunk in the stream
  bool more, computes;                              // another step follows
  FmaTile t;
};

// The hidden layer.  Chunks of the ring are queued by thread 0 two ahead of their use, into the slot of the chunk before last.  A wait
// that runs out is flagged and the thread goes on, in this and later steps, with meaningless numbers and without further waits;
// thread 0, which waits for every chunk it queues, first lets the queued ones arrive and queues no more.
template <int EPT, int NPT, int SRC>
__device__ __forceinline__ void af_hidden(const AfHidden& a, bool& ok) {
  FmaAcc<EPT, NPT> acc;
  if (a.computes) fma_bias<EPT, NPT>(acc, a.b, a.t);
  if (SRC == AF_RING) {
    if ((int)(threadIdx.x >> 5) < a.warps) {
      uint64_t* empty = a.full + AF_SLOTS;
      const bool ok_before = ok;
      uint32_t g = a.g0;
#pragma unroll 1
      for (int c = 0; c < a.n_chunks; ++c, ++g) {
        const uint32_t sl = g % AF_SLOTS;
        const bool live = ok;
        uint32_t queued = g + (c + 1 < a.n_chunks || a.more ? 2 : 1);         // chunks queued so far
        if (threadIdx.x == 0 && ok && (c + 2 < a.n_chunks || a.more)) {
          const uint32_t n = g + 2;
          if (n >= AF_SLOTS) ok = mbar_wait_bounded(empty + n % AF_SLOTS, ((n / AF_SLOTS) - 1) & 1);
          queued += ok ? 1 : 0;
          if (ok) af_queue_chunk(const_cast<float*>(a.w), a.src, a.full, n, (uint32_t)(c + 2 < a.n_chunks ? c + 2 : c + 2 - a.n_chunks), a.kc, a.H, a.Hp);
        }
        __syncwarp();
        ok = ok && mbar_wait_bounded(a.full + sl, (g / AF_SLOTS) & 1);
        if (threadIdx.x == 0 && live && !ok)
          for (uint32_t n = g; n < queued; ++n) mbar_settle(a.full + n % AF_SLOTS, (n / AF_SLOTS) & 1);
        if (a.computes) fma_accumulate<EPT, NPT, 4>(acc, a.w + sl * (a.kc * a.Hp), a.Hp, a.h1 + c * a.kc * a.E, a.E, min(a.kc, a.H - c * a.kc), a.t);
        __syncwarp();
        if ((threadIdx.x & 31) == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(empty + sl)) : "memory");
      }
      if (ok_before && !ok) atomicExch(a.error, 1ull);
    }
  } else if (a.computes) {
    fma_accumulate<EPT, NPT, (EPT * NPT > 8 ? 4 : 8)>(acc, a.w, a.Hp, a.h1, a.E, a.H, a.t);
  }
  if (a.overlap) __syncthreads();                   // every read of h1 is done: h2 takes its place
  if (a.computes) fma_store_rows(acc, a.h2, a.ldh, a.t);
}

// most threads of a register tile: 448 for the largest (128 registers each), else 512
constexpr int af_most(int ept, int npt) { return ept * npt >= 32 ? 448 : 512; }

template <int ENV, int EPT, int NPT, int SRC>
__global__ void __launch_bounds__(af_most(EPT, NPT), 1) actor_fma_kernel(const ActorParams p, const AfPlan q) {
  extern __shared__ __align__(128) float af_sm[];
  constexpr int D = ENV == TJ_ENV_CARTPOLE ? 4 : 6;
  float* sm = af_sm;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, a = lane & 3;
  const int E = q.E, e0 = blockIdx.x * E;
  uint64_t* bar = reinterpret_cast<uint64_t*>(sm + q.bar);    // [0] small parameters, [1] W2 or unused, then full[SLOTS], empty[SLOTS]
  uint64_t *full = bar + 2, *empty = full + AF_SLOTS;
  const int cw = (q.n_compute + 31) / 32;                     // warps that compute
  if (tid == 0) {
    mbar_init(bar, 1);
    mbar_init(bar + 1, 1);
    for (int i = 0; i < AF_SLOTS; ++i) { mbar_init(full + i, 1); mbar_init(empty + i, cw); }
  }
  __syncthreads();
  chain_begin();
  const bool on_policy = p.C == 0;
  const int n_iters = p.n_steps + (on_policy && (q.pos0 + p.n_steps) % p.T == 0 ? 1 : 0);   // a last pass for the bootstrap value alone

  // layer 1 with the rows fastest over the lanes (its k-major stores are then contiguous), the hidden layer with the neurons
  FmaTile t1, t;
  t1.ng = tid / q.EG; t1.eg = tid - t1.ng * q.EG;
  t.eg = tid / q.NG; t.ng = tid - t.eg * q.NG;
  t.half = t1.half = q.half;
  const bool computes = tid < q.n_compute;
  if (tid == 0) {
    const size_t head = p.off_W2t, tail = p.w_total - p.off_b2;
    mbar_expect_tx(bar, (uint32_t)((head + tail) * 4));
    bulk_copy_chunks(sm + q.w, p.W, head * 4, bar);
    bulk_copy_chunks(sm + q.w + p.off_b2 - q.gap, p.W + p.off_b2, tail * 4, bar);
    if (SRC == AF_SMEM) {
      mbar_expect_tx(bar + 1, (uint32_t)((p.off_b2 - p.off_W2t) * 4));
      bulk_copy_chunks(sm + q.w + p.off_W2t, p.W + p.off_W2t, (p.off_b2 - p.off_W2t) * 4, bar + 1);
    }
  }
  const float *W1t = sm + q.w + p.off_W1t, *b1 = sm + q.w + p.off_b1, *b2 = sm + q.w + p.off_b2 - q.gap;
  float *xs = sm + q.xs, *h1 = sm + q.h1, *h2 = sm + q.h2, *w3 = sm + q.w3;
  uint2* pw = reinterpret_cast<uint2*>(sm + q.pw);            // [2][E]: the step's ACTION words, by step parity

  // head lanes: environment el, output a.  The environment lives in shared memory between steps: its registers are the layers'
  const int el = warp * 8 + (lane >> 2), e = e0 + el;
  const bool head_warp = warp * 8 < E, owner = el < E && e < p.N;
  AfEnv* env = reinterpret_cast<AfEnv*>(sm + q.env) + (el < E ? el : 0);
  auto put_obs = [&](const float4 s, const float4 trig) {     // observation of state s -> xs[k][el]
    if (ENV == TJ_ENV_CARTPOLE) {
      const float v = a == 0 ? s.x : (a == 1 ? s.y : (a == 2 ? s.z : s.w));
      if (el < E) xs[a * E + el] = owner ? v : 0.f;
    } else {
      const float v = a == 0 ? trig.x : (a == 1 ? trig.y : (a == 2 ? trig.z : trig.w));
      if (el < E) {
        xs[a * E + el] = owner ? v : 0.f;
        if (a < 2) xs[(4 + a) * E + el] = owner ? (a == 0 ? s.z : s.w) : 0.f;
      }
    }
  };
  // draws for step `it` by the last warps (those the head leaves idle, where there are any)
  auto draw = [&](int it) {
    const int d = q.nt - 1 - tid;
    if (d < E) {
      const uint4 w = stream_words(p.seed, STREAM_ACTION, 0, (uint32_t)(e0 + d), (unsigned long long)p.t0 + it);
      pw[(it & 1) * E + d] = make_uint2(w.x, w.y);
    }
  };
  draw(0);
  if (head_warp) {
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    AcrobotAngles at{s, 0.f, 0.f};
    if (owner) s = reinterpret_cast<const float4*>(p.state)[e];
    if (ENV == TJ_ENV_ACROBOT) at = acrobot_angles4(s, lane);
    put_obs(s, at.trig);
    if (el < E && a == 0) {
      env->s = s;
      env->trig = at.trig;
      env->s12 = at.s12;
      env->ep = owner ? p.ep_step[e] : 0;
      env->ret = owner ? p.ep_return[e] : 0.f;
      env->episodes = 0;
      env->ret_sum = 0.0;
    }
  }
  // a wait that runs out is flagged and the thread goes on, with meaningless numbers, through the same barriers
  bool ok = true;
  auto wait = [&](uint64_t* b, uint32_t parity) {
    if (ok && !mbar_wait_bounded(b, parity)) {
      ok = false;
      atomicExch(&p.stats->error, 1ull);
      if (tid == 0) {                                         // the copies queued so far have to arrive before the block leaves
        mbar_settle(bar, 0);
        if (SRC == AF_SMEM) mbar_settle(bar + 1, 0);
      }
    }
  };
  wait(bar, 0);
  {
    const float* W3t = sm + q.w + p.off_W3t - q.gap;          // rows of four outputs -> one row of weights per output
    for (int i = tid; i < 4 * p.Hp; i += q.nt) w3[(i & 3) * q.ldh + (i >> 2)] = (i >> 2) < p.H ? W3t[i] : 0.f;
  }
  __syncthreads();

  const int n_chunks = (p.H + q.kc - 1) / q.kc;
  if (SRC == AF_RING && tid == 0 && ok)
    for (uint32_t g = 0; g < 2; ++g) af_queue_chunk(sm + q.w2, p.W + p.off_W2t, full, g, g, q.kc, p.H, p.Hp);
  long long slot = q.slot0;                                   // ring slot of env 0 in this step
  int blk = q.blk0, pos = q.pos0, seg = q.seg0;
  for (int it = 0; it < n_iters; ++it) {
    af_layer1<EPT, NPT>(b1, W1t, xs, h1, E, p.Hp, D, t1, computes);
    __syncthreads();
    if (SRC == AF_SMEM && it == 0) wait(bar + 1, 0);
    AfHidden hd;
    hd.w = SRC == AF_SMEM ? sm + q.w + p.off_W2t : sm + q.w2;
    hd.src = p.W + p.off_W2t;
    hd.b = b2; hd.h1 = h1; hd.h2 = h2; hd.full = full; hd.error = &p.stats->error;
    hd.E = E; hd.H = p.H; hd.Hp = p.Hp; hd.ldh = q.ldh; hd.kc = q.kc; hd.overlap = q.overlap; hd.warps = cw; hd.n_chunks = n_chunks;
    hd.g0 = (uint32_t)(it * n_chunks); hd.more = it + 1 < n_iters;
    hd.t = t; hd.computes = computes;
    af_hidden<EPT, NPT, SRC>(hd, ok);
    __syncthreads();
    draw(it + 1);
    if (head_warp) {
      const float* b3 = sm + q.w + p.off_b3 - q.gap;
      const float out = fma_head<(EPT * NPT > 16 ? 4 : 8)>(b3[a], w3 + a * q.ldh, h2 + (el < E ? el : 0) * q.ldh, p.Hp / 4);
      float l[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) l[i] = __shfl_sync(0xffffffffu, out, (lane & ~3) + i);
      if (on_policy && it > 0 && pos == 0 && owner && a == p.A)   // the state after a segment's last step: its bootstrap value
        p.seg_val[((size_t)(seg == 0 ? p.G - 1 : seg - 1) * (p.T + 1) + p.T) * p.N + e] = out;
      if (it < p.n_steps) {
        if (owner && p.dbg_logits && a < p.A) p.dbg_logits[((size_t)it * p.N + e) * p.A + a] = out;
        auto logit = [&](int i) { return i == 0 ? l[0] : (i == 1 ? l[1] : (i == 2 ? l[2] : l[3])); };
        const uint2 pwv = pw[(it & 1) * E + (el < E ? el : 0)];
        const uint4 w = make_uint4(pwv.x, pwv.y, 0u, 0u);
        const float4 s = env->s, trig = ENV == TJ_ENV_ACROBOT ? env->trig : s;
        const int ep = env->ep + 1;
        int act;
        float logp = 0.f;
        if (p.policy_kind == TJ_POLICY_EPS_GREEDY) act = select_eps_greedy(p.A, logit, w, p.explore_thr);
        else act = select_categorical(p.A, logit, u01(w.x), logp);
        float4 sn;
        AcrobotAngles at{trig, ENV == TJ_ENV_ACROBOT ? env->s12 : 0.f, 0.f};   // of s, then of the new state
        StepResult r;
        if (ENV == TJ_ENV_CARTPOLE) {
          r = cartpole_step(s, act, sn);
        } else {
          r = acrobot_step4(s, at, act, lane, sn);
        }
        const int done = (r.terminated || ep >= p.max_ep) ? 1 : 0;
        if (owner) {
          if (on_policy) {
            const size_t i = ((size_t)seg * p.T + pos) * p.N + e;
            if (ENV == TJ_ENV_CARTPOLE) {
              if (a == 0) *reinterpret_cast<float4*>(p.seg_obs + i * 4) = s;
            } else if (a < 3) {
              *reinterpret_cast<float2*>(p.seg_obs + i * 6 + 2 * a) =
                  a == 0 ? make_float2(trig.x, trig.y) : (a == 1 ? make_float2(trig.z, trig.w) : make_float2(s.z, s.w));
            }
            if (a == 1) { p.seg_act[i] = act; p.seg_done[i] = (uint8_t)done; }
            if (a == 2) p.seg_rew[i] = r.reward;
            if (a == 3) p.seg_logp[i] = logp;
            if (a == p.A) p.seg_val[((size_t)seg * (p.T + 1) + pos) * p.N + e] = out;   // value head = output A
          } else {
            long long sl = slot + e;
            if (sl >= p.C) sl -= p.C;
            float4* rec = reinterpret_cast<float4*>(p.ring + (size_t)sl * p.rec_words);
            const float4 tail = make_float4(__int_as_float(act), r.reward, __int_as_float(done), __int_as_float(p.version));
            if (ENV == TJ_ENV_CARTPOLE) {
              if (a < 3) rec[a] = a == 0 ? s : (a == 1 ? sn : tail);
            } else {
              rec[a] = a == 0 ? trig : (a == 1 ? make_float4(s.z, s.w, at.trig.x, at.trig.y)
                                               : (a == 2 ? make_float4(at.trig.z, at.trig.w, sn.z, sn.w) : tail));
            }
          }
        }
        const float ret = env->ret + r.reward;
        float4 next = sn;
        if (done) {
          const unsigned long long t_now = (unsigned long long)p.t0 + it;
          next = ENV == TJ_ENV_CARTPOLE ? reset4(p.seed, 0, (uint32_t)e, t_now, -0.05f, 0.1f) : reset4(p.seed, 0, (uint32_t)e, t_now, -0.1f, 0.2f);
        }
        if (ENV == TJ_ENV_ACROBOT && __any_sync(0xffffffffu, done)) {
          const AcrobotAngles fresh = acrobot_angles4(next, lane);
          if (done) at = fresh;
        }
        put_obs(next, at.trig);
        __syncwarp();                                         // the other lanes of the environment have read it
        if (el < E && a == 0) {
          env->s = next;
          if (ENV == TJ_ENV_ACROBOT) { env->trig = at.trig; env->s12 = at.s12; }
          env->ep = done ? 0 : ep;
          env->ret = done ? 0.f : ret;
          if (done) { env->episodes += 1; env->ret_sum += (double)ret; }
        }
      }
    }
    if (it < p.n_steps) {
      if (on_policy) {
        if (++pos == p.T) { pos = 0; seg = seg + 1 == p.G ? 0 : seg + 1; }
      } else {
        if (blockIdx.x == 0 && tid == 0) p.block_ver[blk] = p.version;
        slot += p.N;
        if (slot >= p.C) slot -= p.C;
        if (++blk == q.n_blk) blk = 0;
      }
    }
    __syncthreads();
  }
  if (owner && a == 0) {
    reinterpret_cast<float4*>(p.state)[e] = env->s;
    p.ep_step[e] = env->ep;
    p.ep_return[e] = env->ret;
    if (env->episodes) {
      atomicAdd(&p.stats->episodes, (unsigned long long)env->episodes);
      atomicAdd(&p.stats->return_sum, env->ret_sum);
    }
  }
}

template <int ENV, int EPT, int NPT>
cudaError_t launch_af(const ActorParams& p, const AfPlan& q, int src, int grid, size_t smem, cudaStream_t s) {
  if (src == AF_SMEM) return launch_chained(actor_fma_kernel<ENV, EPT, NPT, AF_SMEM>, grid, q.nt, smem, s, p, q);
  return launch_chained(actor_fma_kernel<ENV, EPT, NPT, AF_RING>, grid, q.nt, smem, s, p, q);
}

}  // namespace

cudaError_t launch_actor_fma(int env_kind, const ActorParams& p, int sm_count, cudaStream_t s) {
  if (p.Ap != 4) return cudaErrorInvalidConfiguration;        // at most four outputs: one float4 per row of the head
  const int sms = sm_count > 0 ? sm_count : 148, Hp = p.Hp;
  // Environments per block: the call spread over the SMs in as few rounds as 56 per SM allow.  (More per round need 8 x 8 tiles.  With one
  // input's operands in flight on 224 threads of 255 registers they take 252 us for four steps of 16,384 Acrobot envs, hidden 256, against 261
  // with two rounds of 8 x 4, and 277 against 409 at 4,096 envs, hidden 512, but 99-121 against 99 at 6,000 envs, where they pad; with more
  // threads or loads in flight they spill, 333-410 us.)
  const int rounds = (p.N + sms * 56 - 1) / (sms * 56);
  int want = (p.N + sms * rounds - 1) / (sms * rounds);
  // Two blocks per SM where both fit with W2 in shared memory: one steps its environments while the other multiplies (4,096 CartPole
  // envs, hidden 128, four steps: 35 us with one block per SM).
  int per_sm = want >= 12 ? 2 : 1;
  if (per_sm == 2) want = (want + 1) / 2;
  AfPlan q{};
  int ept = 0, npt = 0, src = AF_SMEM;
  size_t smem = 0;
  const size_t small = p.w_total - (p.off_b2 - p.off_W2t);
  bool fits = false;
  for (; !fits; want = per_sm == 2 ? 2 * want : (want > 8 ? want / 2 : want - 4), per_sm = 1) {
    if (want < 1) return cudaErrorInvalidConfiguration;
    // Register tile by the number of environments: few of them are bound by the chain of dependent FMAs, so small tiles on many
    // threads; from 17 per SM on the operand loads bound the layer, and larger tiles load less per FMA (figures in tj_fma.cuh).
    static const int tiles[4][3] = {{4, 1, 8}, {4, 2, 16}, {4, 4, 32}, {8, 4, 56}};   // rows x neurons, most rows per SM
    int k = 0;
    for (; k < 4; ++k) {
      ept = tiles[k][0]; npt = tiles[k][1];
      q.E = (want + ept - 1) / ept * ept;
      if (want * per_sm <= tiles[k][2] && q.E / ept * (Hp / npt) <= af_most(ept, npt)) break;
    }
    if (k == 4) continue;
    q.EG = q.E / ept;
    q.NG = Hp / npt;
    q.n_compute = q.EG * q.NG;
    q.half = q.E / 2;
    q.nt = (q.n_compute + 31) / 32 * 32;
    if (q.nt < (q.E + 7) / 8 * 32) q.nt = (q.E + 7) / 8 * 32;     // a head warp per eight environments
    if (q.nt < (q.E + 31) / 32 * 32 + 32) q.nt = (q.E + 31) / 32 * 32 + 32;
    if (q.nt > af_most(ept, npt)) continue;
    q.ldh = 4 * ((Hp / 4) | 1);
    q.kc = Hp <= 256 ? 16 : (Hp <= 512 ? 8 : 4);
    // W2 in shared memory if it fits beside the activations (h2 over h1 if need be), else through the ring
    for (int c = 0; c < (per_sm == 2 ? 2 : 4) && !fits; ++c) {
      src = c < 2 ? AF_SMEM : AF_RING;
      q.overlap = c & 1;
      size_t o = 0;
      auto take = [&](size_t n) { const size_t r = o; o += (n + 31) / 32 * 32; return (int)r; };
      q.gap = src == AF_SMEM ? 0 : (int)(p.off_b2 - p.off_W2t);
      q.w = take(src == AF_SMEM ? p.w_total : small);
      q.w2 = src == AF_RING ? take((size_t)AF_SLOTS * q.kc * Hp) : 0;
      q.xs = take((size_t)8 * q.E);
      const size_t n1 = (size_t)Hp * q.E, n2 = (size_t)q.E * q.ldh;
      q.h1 = take(q.overlap ? (n1 > n2 ? n1 : n2) : n1);
      q.h2 = q.overlap ? q.h1 : take(n2);
      q.w3 = take((size_t)4 * q.ldh);
      q.pw = take((size_t)4 * q.E);
      q.env = take(sizeof(AfEnv) / 4 * (size_t)q.E);
      q.bar = take(2 * (2 + 2 * AF_SLOTS));
      smem = o * sizeof(float);
      fits = smem <= (per_sm == 2 ? 112 : 226) * 1024;
    }
  }
  const int grid = (p.N + q.E - 1) / q.E;
  if (p.C > 0) {
    q.slot0 = (long long)(p.cursor0 % (unsigned long long)p.C);
    q.blk0 = (int)(q.slot0 / p.N);
    q.n_blk = (int)(p.C / p.N);
  } else {
    q.pos0 = (int)(p.t0 % p.T);
    q.seg0 = (int)((p.t0 / p.T) % p.G);
  }
#define TJ_AF(ENV)                                                                                        \
  (ept == 4 ? (npt == 1 ? launch_af<ENV, 4, 1>(p, q, src, grid, smem, s)                                  \
                        : (npt == 2 ? launch_af<ENV, 4, 2>(p, q, src, grid, smem, s) : launch_af<ENV, 4, 4>(p, q, src, grid, smem, s))) \
            : launch_af<ENV, 8, 4>(p, q, src, grid, smem, s))
  return env_kind == TJ_ENV_CARTPOLE ? TJ_AF(TJ_ENV_CARTPOLE) : TJ_AF(TJ_ENV_ACROBOT);
#undef TJ_AF
}

}  // namespace tj
