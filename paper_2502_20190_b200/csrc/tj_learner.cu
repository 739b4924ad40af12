// Learner-side kernels: staleness-bounded sampling and gather, TD error / Huber loss, and the GAE reverse scan.
#include <mutex>

#include "tj_async.cuh"
#include "tj_device.cuh"
#include "tj_internal.h"
#include "tj_mlp.cuh"

namespace tj {

namespace {

__global__ void transpose_pad_kernel(const float* __restrict__ src, float* __restrict__ dst, int rows, int cols,
                                     int ld_dst) {
  // dst[c][r] = src[r][c], dst rows padded to ld_dst with zeros
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (size_t)cols * ld_dst) return;
  const int c = (int)(i / ld_dst), r = (int)(i % ld_dst);
  dst[i] = r < rows ? src[(size_t)r * cols + c] : 0.f;
}

// Staleness-bounded sampling in two kernels.  One ring block = the N records of one actor step, all with one version, and
// blocks are written with non-decreasing versions, so the blocks within the bound are the newest ones: in slot order one
// interval of blocks, or two where it wraps round the ring's end (p.n_lo blocks from 0, the rest from p.b_hi on).  The host
// knows both from its own bookkeeping, and E[r] is arithmetic: no list of eligible blocks is built or read.
//
// draw_slots_kernel: draw j takes E[mulhi(x0, |E|)]; one thread per draw, bound by one launch's latency (the arithmetic
// reads no memory and runs before the wait for the kernel in front).
__device__ __forceinline__ int eligible_slot(const SampleParams& p, uint32_t r) {
  const uint32_t i = r / (uint32_t)p.N, e = r % (uint32_t)p.N;
  const uint32_t block = i < (uint32_t)p.n_lo ? i : (uint32_t)p.b_hi + (i - (uint32_t)p.n_lo);
  return (int)(block * (uint32_t)p.N + e);
}

__global__ void __launch_bounds__(256) draw_slots_kernel(const SampleParams p) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  const uint4 w = stream_words(p.seed, STREAM_SAMPLE, 0, (uint32_t)j, (unsigned long long)p.k);
  const int slot = eligible_slot(p, __umulhi(w.x, p.n_elig));
  chain_begin();
  chain_next();
  if (j >= p.B) return;
  p.slots[j] = slot;
  if (p.idx_out) p.idx_out[j] = slot;
}

// gather_kernel: LPD lanes share a draw and copy its record in 16-byte chunks -- obs, next_obs, then the (act, rew, done, ver)
// tail -- into the dense arrays (whole chunks where the rows allow it, word by word for obs_dim 6 or unaligned arrays).  The
// loads of UNR draws are in flight at once: bound by the latency of the scattered rows for short records, by HBM for the
// 1,040-byte ones.  The staleness counts are taken per block in shared memory first: one global atomic per draw on the
// handful of bins in use serialised in L2 (8,192 draws of 1,040 bytes: 10.4 us before, 4.9 us with the counts per block).
template <int LPD, int UNR, bool VEC>
__global__ void __launch_bounds__(256) gather_kernel(const SampleParams p) {
  __shared__ unsigned int bins[33];
  __shared__ unsigned long long most;
  constexpr int DPW = 32 / LPD;                              // draws a warp covers at a time
  const int lane = threadIdx.x & 31, sub = lane % LPD, warp = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < 33; i += blockDim.x) bins[i] = 0u;
  if (threadIdx.x == 0) most = 0ull;
  chain_begin();
  chain_next();
  __syncthreads();
  const int chunks = p.rec_words / 4, dq = p.D / 4;
  const int j0 = (blockIdx.x * (int)(blockDim.x >> 5) + warp) * (DPW * UNR) + lane / LPD;
  int slot[UNR];
#pragma unroll
  for (int u = 0; u < UNR; ++u) {
    const int j = j0 + u * DPW;
    slot[u] = j < p.B ? p.slots[j] : -1;
  }
  for (int c = sub; c < chunks; c += LPD) {
    float4 v[UNR];
#pragma unroll
    for (int u = 0; u < UNR; ++u)                            // sampled rows are not reused: streaming loads
      if (slot[u] >= 0) v[u] = __ldcs(reinterpret_cast<const float4*>(p.ring + (size_t)slot[u] * p.rec_words) + c);
#pragma unroll
    for (int u = 0; u < UNR; ++u) {
      if (slot[u] < 0) continue;
      const size_t j = (size_t)(j0 + u * DPW);
      if (c == chunks - 1) {
        const int ver = __float_as_int(v[u].w);
        p.act[j] = __float_as_int(v[u].x);
        p.rew[j] = v[u].y;
        p.done[j] = __float_as_int(v[u].z);
        p.ver[j] = ver;
        long long stale = p.v_learner - (long long)ver;
        if (stale < 0) stale = 0;
        atomicAdd(&bins[stale > 32 ? 32 : stale], 1u);
        if (stale >= 32) atomicMax(&most, (unsigned long long)stale);
      } else if (VEC) {
        if (c < dq) reinterpret_cast<float4*>(p.obs + j * p.D)[c] = v[u];
        else reinterpret_cast<float4*>(p.next_obs + j * p.D)[c - dq] = v[u];
      } else {
        const float w[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int k = 4 * c + i;
          if (k < p.D) p.obs[j * p.D + k] = w[i];
          else p.next_obs[j * p.D + (k - p.D)] = w[i];
        }
      }
    }
  }
  __syncthreads();
  if (threadIdx.x < 33 && bins[threadIdx.x]) {
    atomicAdd(&p.stats->hist[threadIdx.x], (unsigned long long)bins[threadIdx.x]);
    atomicMax(&p.stats->max_stale, threadIdx.x < 32 ? (unsigned long long)threadIdx.x : most);
  }
}

// A staging wait that ran out, for the whole block: latch the context's error word and leave defined outputs (NaN) for this block's rows
// and its partial sum, so that neither the caller nor the loss reduction reads what an earlier call left there; the staged
// parameters have to arrive before the block leaves.
__device__ __forceinline__ void td_give_up(const TdParams& p, int n_here, int j0, uint64_t* bar, uint32_t parity) {
  const float nan = __int_as_float(0x7FC00000);
  if (threadIdx.x == 0) {
    mbar_settle(bar, parity);
    if (p.error) atomicExch(p.error, 3ull);
    p.partial[blockIdx.x] = nan;
  }
  if ((int)threadIdx.x < n_here) {
    if (p.td_out) p.td_out[j0 + threadIdx.x] = nan;
    if (p.huber_out) p.huber_out[j0 + threadIdx.x] = nan;
  }
}

// TD error on a tile of TE samples: online forward on obs, target forward on next_obs.  STAGE: what of the parameters lies in shared
// memory (stage_mlp_weights); the staging buffer is filled twice (online, then target parameters).
template <int TE, int NT, int EPT, int NPT, int STAGE>
__global__ void __launch_bounds__(NT) td_kernel(const TdParams p) {
  extern __shared__ __align__(128) float smem[];
  __shared__ __align__(8) uint64_t wbar;
  const size_t staged = STAGE == 2 ? p.w_total : (STAGE == 1 ? p.w_total - (p.off_b2 - p.off_W2t) : 0);
  const int Dx = (p.D + 3) & ~3;
  float* wsm = smem;
  float* xs = wsm + staged;
  float* h1 = xs + (size_t)Dx * TE;
  float* h2 = h1 + (size_t)p.Hp * TE;
  float* out = h2 + (size_t)p.Hp * TE;
  float* qsel = out + (size_t)p.Ap * TE;
  float* hub = qsel + TE;
  const int tid = threadIdx.x, j0 = blockIdx.x * TE, n_here = min(TE, p.n - j0), D = p.D;
  chain_begin();
  if (STAGE > 0) {
    if (tid == 0) mbar_init(&wbar, 1);
    __syncthreads();
  }
  MlpWeights mw = stage_mlp_weights<STAGE>(p, p.Wonline, wsm, &wbar, tid == 0);

  for (int i = tid; i < TE * D; i += NT) {
    const int el = i / D, k = i % D;
    xs[k * TE + el] = el < n_here ? p.obs[(size_t)(j0 + el) * D + k] : 0.f;
  }
  if (!__syncthreads_and(STAGE == 0 || mbar_wait_bounded(&wbar, 0))) { td_give_up(p, n_here, j0, &wbar, 0); return; }
  mlp_forward_tile<TE, NT, EPT, (STAGE > 0), (STAGE == 2), NPT>(mw, D, p.H, p.Hp, p.A, p.Ap, xs, h1, h2, out);
  if (tid < n_here) {
    int a = p.act[j0 + tid];
    a = a < 0 ? 0 : (a >= p.A ? p.A - 1 : a);
    qsel[tid] = out[a * TE + tid];
  }
  __syncthreads();  // every thread is done with the online parameters: the buffer may be refilled
  mw = stage_mlp_weights<STAGE>(p, p.Wtarget, wsm, &wbar, tid == 0);
  for (int i = tid; i < TE * D; i += NT) {
    const int el = i / D, k = i % D;
    xs[k * TE + el] = el < n_here ? p.next_obs[(size_t)(j0 + el) * D + k] : 0.f;
  }
  if (!__syncthreads_and(STAGE == 0 || mbar_wait_bounded(&wbar, 1))) { td_give_up(p, n_here, j0, &wbar, 1); return; }
  mlp_forward_tile<TE, NT, EPT, (STAGE > 0), (STAGE == 2), NPT>(mw, D, p.H, p.Hp, p.A, p.Ap, xs, h1, h2, out);
  if (tid < TE) {
    float h = 0.f;
    if (tid < n_here) {
      const int j = j0 + tid;
      float qmax = out[tid];
      for (int i = 1; i < p.A; ++i) qmax = fmaxf(qmax, out[i * TE + tid]);
      const float y = p.rew[j] + p.gamma * (p.done[j] ? 0.f : 1.f) * qmax;
      const float delta = y - qsel[tid];
      const float ad = fabsf(delta);
      h = ad <= p.kappa ? 0.5f * delta * delta : p.kappa * (ad - 0.5f * p.kappa);
      if (p.td_out) p.td_out[j] = delta;
      if (p.huber_out) p.huber_out[j] = h;
    }
    hub[tid] = h;
  }
  __syncthreads();
  if (tid == 0) {
    float sum = 0.f;
    for (int i = 0; i < n_here; ++i) sum += hub[i];
    p.partial[blockIdx.x] = sum;
  }
}

// Fixed-order sum of the per-block partial losses: thread i adds partials i, i + 256, ... (independent loads), then a tree.  One block,
// bound by one memory latency (a warp that added them in index order, one shuffle each, took 6-8 us for 512 partials).
__global__ void __launch_bounds__(256) td_finish_kernel(const float* __restrict__ partial, int n_partial, int n, float* __restrict__ loss_out,
                                                        const UpdateWatch watch) {
  __shared__ float ws[8];
  chain_begin();
  chain_next();
  const unsigned asked = watch.failed ? update_ask(watch.failed, watch.number) : ~watch.number;    // the loss of a TD error has no update
  float s = 0.f;
#pragma unroll 4
  for (int i = threadIdx.x; i < n_partial; i += 256) s += __ldcg(partial + i);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
  const bool valid = update_valid(watch.number, asked);
  if (threadIdx.x == 0) {
    s = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) s += ws[w];
    *loss_out = valid ? s / (float)n : __int_as_float(0x7FC00000);
  }
}

// GAE: one thread per environment walks its column backwards; a warp reads 32 consecutive environments, so
// every access is a full 128-byte line.  The recurrence is serial in t, but its inputs are not: each thread
// fetches the next GAE_U time steps' rewards, values and done flags before it needs them, which keeps enough
// loads in flight to stream at HBM speed.
constexpr int GAE_U = 8;
__global__ void __launch_bounds__(128) gae_kernel(const float* __restrict__ rew, const float* __restrict__ val,
                                                  const uint8_t* __restrict__ done, int T, int N, float gamma,
                                                  float lambda, float* __restrict__ adv, float* __restrict__ ret) {
  chain_begin();
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= N) return;
  float next_adv = 0.f;
  float v_next = __ldcs(val + (size_t)T * N + e);
  const float gl = gamma * lambda;
  int t = T - 1;
  for (; t >= GAE_U - 1; t -= GAE_U) {
    float r[GAE_U], v[GAE_U];
    uint8_t d[GAE_U];
#pragma unroll
    for (int u = 0; u < GAE_U; ++u) {
      const size_t i = (size_t)(t - u) * N + e;
      r[u] = __ldcs(rew + i);
      v[u] = __ldcs(val + i);
      d[u] = __ldcs(done + i);
    }
#pragma unroll
    for (int u = 0; u < GAE_U; ++u) {
      const size_t i = (size_t)(t - u) * N + e;
      const float nd = d[u] ? 0.f : 1.f;
      const float delta = r[u] + gamma * nd * v_next - v[u];
      const float a = delta + gl * nd * next_adv;
      __stcs(adv + i, a);
      __stcs(ret + i, a + v[u]);
      next_adv = a;
      v_next = v[u];
    }
  }
  for (; t >= 0; --t) {
    const size_t i = (size_t)t * N + e;
    const float nd = done[i] ? 0.f : 1.f;
    const float v = val[i];
    const float delta = rew[i] + gamma * nd * v_next - v;
    const float a = delta + gl * nd * next_adv;
    adv[i] = a;
    ret[i] = a + v;
    next_adv = a;
    v_next = v;
  }
}

constexpr int kTdTile = 16;
constexpr int kTdThreads = 128;

}  // namespace

cudaError_t launch_transpose_pad(const float* src, float* dst, int rows, int cols, int ld_dst, cudaStream_t s) {
  const size_t n = (size_t)cols * ld_dst;
  transpose_pad_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(src, dst, rows, cols, ld_dst);
  return cudaGetLastError();
}

template <int LPD, int UNR>
static cudaError_t launch_gather(const SampleParams& p, bool vec, cudaStream_t s) {
  const int per_block = 8 * (32 / LPD) * UNR;                // draws of a block of eight warps
  const int grid = (p.B + per_block - 1) / per_block;
  return launch_chained(vec ? gather_kernel<LPD, UNR, true> : gather_kernel<LPD, UNR, false>, grid, 256, 0, s, p);
}

cudaError_t launch_sample_gather(const SampleParams& p, cudaStream_t s) {
  const cudaError_t e = launch_chained(draw_slots_kernel, (p.B + 255) / 256, 256, 0, s, p);
  if (e != cudaSuccess) return e;
  const bool vec = p.D % 4 == 0 && ((reinterpret_cast<uintptr_t>(p.obs) | reinterpret_cast<uintptr_t>(p.next_obs)) & 15) == 0;
  // lanes per draw by the record's length in 16-byte chunks (3 or 4 for the small envs, 65 for obs_dim 128), so that few
  // lanes idle and a warp's loads stay contiguous per record
  if (p.rec_words <= 16) return launch_gather<4, 1>(p, vec, s);
  if (p.rec_words <= 64) return launch_gather<8, 2>(p, vec, s);
  return launch_gather<32, 4>(p, vec, s);
}

int td_grid(int n) { return (n + kTdTile - 1) / kTdTile; }

template <int TE, int NT, int EPT, int NPT, int STAGE>
cudaError_t launch_td_stage(const TdParams& p, size_t smem, int grid, cudaStream_t s) {
  return launch_chained<1024>(td_kernel<TE, NT, EPT, NPT, STAGE>, grid, NT, smem, s, p);
}

// tile: 16 rows x 128 threads with 4 x 4 register tiles; wide layers (hidden >= 192) 32 rows x 128 threads, 8 x 8
template <int TE, int NT, int EPT, int NPT>
cudaError_t launch_td_tile(const TdParams& p, cudaStream_t s, int* grid_out) {
  const int Dx = (p.D + 3) & ~3;
  const size_t acts = (size_t)Dx * TE + 2 * (size_t)p.Hp * TE + (size_t)p.Ap * TE + 2 * TE;
  const size_t limit = 226 * 1024;
  const size_t smem2 = (acts + p.w_total) * sizeof(float);
  const size_t smem1 = (acts + p.w_total - (p.off_b2 - p.off_W2t)) * sizeof(float);
  const size_t smem0 = acts * sizeof(float);
  const int grid = (p.n + TE - 1) / TE;
  *grid_out = grid;
  if (smem2 <= 112 * 1024) return launch_td_stage<TE, NT, EPT, NPT, 2>(p, smem2, grid, s);
  if (smem1 <= limit) return launch_td_stage<TE, NT, EPT, NPT, 1>(p, smem1, grid, s);
  if (smem0 <= limit) return launch_td_stage<TE, NT, EPT, NPT, 0>(p, smem0, grid, s);
  return cudaErrorInvalidConfiguration;
}

// Parameters of both networks in shared memory where they fit; else, up to four outputs, layer by layer where the context's update
// scratch holds the activations (whole calls, hidden 256: 4,096 rows 64 us by 32-row tiles that read W2 through L2, 47 as layers; 300
// rows 63 and 18); else those tiles.  All of them sum in the same order (tj_mlp.cuh), the layers' loss partials over the tiles' rows too:
// the route depends on the configured minibatch, the bits do not.
cudaError_t launch_td(const TdParams& p, int sm_count, cudaStream_t s, int* launches) {
  int grid = 0;
  cudaError_t err = launch_td_fma(p, sm_count, &grid, s);
  int n_launches = 1;
  if (err == cudaSuccess && grid == 0 && p.layers && p.A <= 4) {
    err = launch_td_layers(p, sm_count, &grid, s);
    n_launches = 3;
  }
  if (launches) *launches = n_launches + (p.loss_out ? 1 : 0);
  if (err == cudaSuccess && grid == 0)
    err = td_tile_rows(p.H) == 32 ? launch_td_tile<32, 128, 8, 8>(p, s, &grid) : launch_td_tile<kTdTile, kTdThreads, 4, 4>(p, s, &grid);
  if (err != cudaSuccess) return err;
  if (p.loss_out) {
    err = launch_td_finish(p.partial, grid, p.n, p.loss_out, s);
  }
  return err;
}

// Scratch for tj_td_error_static: it is part of the library image, so every GPU that loads the library
// holds these 32 KB until the process exits and nobody has to allocate it.
constexpr int kStaticTdPartials = 8192;
static __device__ __align__(256) float g_td_static_partial[kStaticTdPartials];

int td_static_max_rows() { return 65536; }

cudaError_t launch_td_static(const TdParams& p_in, int device, int sm_count, cudaStream_t s, int* launches, bool* too_large) {
  *too_large = p_in.n > td_static_max_rows() || td_grid(p_in.n) > kStaticTdPartials;
  if (*too_large) return cudaSuccess;
  // In host code the array's name is only a stand-in; the device address has to be asked for, once per device, with
  // that device current.  The table is keyed by the context's device and filled under a lock, so first calls from
  // several threads (one context each) do not race.
  static float* addr_by_device[64] = {};
  static std::mutex addr_lock;
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (device < 0 || device >= 64 || dev != device) return cudaErrorInvalidDevice;
  float* scratch = nullptr;
  {
    std::lock_guard<std::mutex> hold(addr_lock);
    if (!addr_by_device[device]) {
      float* q = nullptr;
      e = cudaGetSymbolAddress(reinterpret_cast<void**>(&q), g_td_static_partial);
      if (e != cudaSuccess) return e;
      addr_by_device[device] = q;
    }
    scratch = addr_by_device[device];
  }
  TdParams p = p_in;
  p.partial = scratch;
  return launch_td(p, sm_count, s, launches);
}

cudaError_t launch_td_finish(const float* partial, int n_partial, int n, float* loss_out, cudaStream_t s, const UpdateWatch& watch) {
  return launch_chained(td_finish_kernel, 1, 256, 0, s, partial, n_partial, n, loss_out, watch);
}

cudaError_t launch_gae(const float* rew, const float* val, const uint8_t* done, int T, int N, float gamma, float lambda,
                       float* adv, float* ret, cudaStream_t s) {
  return launch_chained(gae_kernel, (N + 127) / 128, 128, 0, s, rew, val, done, T, N, gamma, lambda, adv, ret);
}

}  // namespace tj
