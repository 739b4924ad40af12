// TD error and Huber loss for networks whose parameters fit in shared memory twice (at most four outputs, hidden up to about 150): the
// online network on obs and the target network on next_obs at the same time, each on its own half of the block's threads, in the
// fixed FMA order of tj_fma.cuh.
//
// A minibatch of a few hundred to a few thousand rows is bound by the chain parameters -> layers -> head, not by the FMAs (1,024
// rows of 4-128-128-2 are 9 us of one SM's FMA time spread over 148).  So a block takes the rows that spread the minibatch over
// the SMs once, both networks run side by side instead of one after the other with the parameters staged in between (21 us for those
// rows with 16-row blocks), and the head's outputs meet by shuffle in the lanes that sum them.
#include "tj_async.cuh"
#include "tj_fma.cuh"
#include "tj_internal.h"

namespace tj {

namespace {

struct TfPlan {
  int E, EG, NG, half, n_half;                      // rows per tile; row quads x neuron groups; threads per network (whole warps)
  int nt, ldh, w, xs, h1, h2, w3, q, bar;           // threads; row stride of h2; offsets in shared memory, floats
  int s_w, s_xs, s_h1, s_h2, s_w3;                  // distance between the two networks' parts, floats
};

constexpr int TF_NT = 512;

template <int EPT, int NPT>
__global__ void __launch_bounds__(TF_NT, 1) td_fma_kernel(const TdParams p, const TfPlan q) {
  extern __shared__ __align__(128) float tf_sm[];
  float* sm = tf_sm;
  const int tid = threadIdx.x, lane = tid & 31, E = q.E;
  uint64_t* bar = reinterpret_cast<uint64_t*>(sm + q.bar);    // [0] all but the hidden matrices, [1] those
  if (tid < 2) mbar_init(bar + tid, 1);
  __syncthreads();
  chain_begin();
  const int net = tid >= q.n_half ? 1 : 0, t0 = tid - net * q.n_half;
  const bool computes = tid < 2 * q.n_half && t0 < q.EG * q.NG;
  FmaTile t1, t;
  t1.ng = t0 / q.EG; t1.eg = t0 - t1.ng * q.EG;               // rows fastest: layer 1's k-major stores are contiguous
  t.eg = t0 / q.NG; t.ng = t0 - t.eg * q.NG;                  // neurons fastest: the hidden layer's row operand is a broadcast
  t.half = t1.half = q.half;
  if (tid == 0) {
    const size_t head = p.off_W2t, mid = p.off_b2 - p.off_W2t, tail = p.w_total - p.off_b2;
    mbar_expect_tx(bar, (uint32_t)(2 * (head + tail) * 4));
    mbar_expect_tx(bar + 1, (uint32_t)(2 * mid * 4));
    for (int n = 0; n < 2; ++n) {
      const float* W = n ? p.Wtarget : p.Wonline;
      float* d = sm + q.w + n * q.s_w;
      bulk_copy_chunks(d, W, head * 4, bar);
      bulk_copy_chunks(d + p.off_b2, W + p.off_b2, tail * 4, bar);
    }
    for (int n = 0; n < 2; ++n)
      bulk_copy_chunks(sm + q.w + n * q.s_w + p.off_W2t, (n ? p.Wtarget : p.Wonline) + p.off_W2t, mid * 4, bar + 1);
  }
  const float* W = sm + q.w + net * q.s_w;
  float *xs = sm + q.xs + net * q.s_xs, *h1 = sm + q.h1 + net * q.s_h1, *h2 = sm + q.h2 + net * q.s_h2;
  const int D = p.D, n_tiles = (p.n + E - 1) / E;
  bool ok = true;
  float sum = 0.f;
  for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const int j0 = tile * E, here = min(E, p.n - j0);
    if (tid < 2 * q.n_half) {
      const float* x = net ? p.next_obs : p.obs;
      for (int i = t0; i < E * D; i += q.n_half) {
        const int r = i / D, k = i - r * D;
        xs[k * E + r] = r < here ? __ldg(x + (size_t)(j0 + r) * D + k) : 0.f;
      }
    }
    int act = 0, done = 0;
    float rew = 0.f;
    if (tid < here) { act = p.act[j0 + tid]; rew = p.rew[j0 + tid]; done = p.done[j0 + tid]; }   // fetched ahead of their use
    if (tile == (int)blockIdx.x) {
      ok = mbar_wait_bounded(bar, 0);
      for (int i = tid; i < 8 * p.Hp; i += q.nt) {            // rows of four outputs -> one row of weights per output
        const int n = i >= 4 * p.Hp ? 1 : 0, j = i - n * 4 * p.Hp;
        sm[q.w3 + n * q.s_w3 + (j & 3) * q.ldh + (j >> 2)] = (j >> 2) < p.H ? sm[q.w + n * q.s_w + p.off_W3t + j] : 0.f;
      }
    }
    __syncthreads();
    if (computes) {
      FmaAcc<EPT, NPT> acc;
      fma_bias<EPT, NPT>(acc, W + p.off_b1, t1);
      fma_accumulate<EPT, NPT, 1>(acc, W + p.off_W1t, p.Hp, xs, E, D, t1);
      fma_store_kmajor(acc, h1, E, t1);
    }
    __syncthreads();
    ok = ok && mbar_wait_bounded(bar + 1, 0);
    if (computes) {
      FmaAcc<EPT, NPT> acc;
      fma_bias<EPT, NPT>(acc, W + p.off_b2, t);
      fma_accumulate<EPT, NPT, (EPT * NPT > 8 ? 4 : 8)>(acc, W + p.off_W2t, p.Hp, h1, E, p.H, t);
      fma_store_rows(acc, h2, q.ldh, t);
    }
    __syncthreads();
    // heads: lane a of a group of four sums output a of (network, row)
    for (int g = tid >> 2; g < (2 * E + 7) / 8 * 8; g += q.nt >> 2) {
      const int n = g >= E ? 1 : 0, r = g < 2 * E ? g - n * E : 0, a = lane & 3;
      const float out = fma_head<4>(sm[q.w + n * q.s_w + p.off_b3 + a], sm + q.w3 + n * q.s_w3 + a * q.ldh, sm + q.h2 + n * q.s_h2 + r * q.ldh, p.Hp / 4);
      if (g < 2 * E) sm[q.q + 4 * g + a] = out;
    }
    ok = __syncthreads_and(ok);                               // whichever thread's wait ran out, none of the block's rows is valid
    if (tid < 64) {
      float h = 0.f;
      if (tid < here) {
        act = act < 0 ? 0 : (act >= p.A ? p.A - 1 : act);
        const float* qt = sm + q.q + 4 * (E + tid);
        float qmax = qt[0];
        for (int i = 1; i < p.A; ++i) qmax = fmaxf(qmax, qt[i]);
        const float y = rew + p.gamma * (done ? 0.f : 1.f) * qmax;
        float delta = y - sm[q.q + 4 * tid + act];
        const float ad = fabsf(delta);
        h = ad <= p.kappa ? 0.5f * delta * delta : p.kappa * (ad - 0.5f * p.kappa);
        if (!ok) delta = h = __int_as_float(0x7FC00000);      // the parameters never arrived: defined outputs
        if (p.td_out) p.td_out[j0 + tid] = delta;
        if (p.huber_out) p.huber_out[j0 + tid] = h;
      }
      for (int o = 16; o > 0; o >>= 1) h += __shfl_xor_sync(0xffffffffu, h, o);
      if (tid == 32) sm[q.q + 8 * E] = h;
      sum += h;
    }
    __syncthreads();
    if (tid == 0) sum += sm[q.q + 8 * E];
  }
  if (tid == 0) {
    p.partial[blockIdx.x] = sum;
    if (!ok) {
      if (p.error) atomicExch(p.error, 3ull);
      mbar_settle(bar, 0);
      mbar_settle(bar + 1, 0);
    }
  }
}

}  // namespace

// Rows per tile and register tile as in the FP32 actor; false where the two networks do not fit (the caller has another kernel).
static bool plan_td_fma(const TdParams& p, int sms, TfPlan& q, int& ept, int& npt, size_t& smem) {
  if (p.Ap != 4) return false;
  const int Hp = p.Hp;
  int want = (p.n + sms - 1) / sms;
  if (want > 56) want = 56;
  for (; want >= 1; want = want > 8 ? want / 2 : want - 4) {
    static const int tiles[4][3] = {{4, 1, 8}, {4, 2, 16}, {4, 4, 32}, {8, 4, 56}};   // rows x neurons, most rows per tile
    int k = 0;
    for (; k < 4; ++k) {
      ept = tiles[k][0]; npt = tiles[k][1];
      q.E = (want + ept - 1) / ept * ept;
      if (want <= tiles[k][2] && 2 * ((q.E / ept * (Hp / npt) + 31) / 32 * 32) <= TF_NT) break;
    }
    if (k == 4) continue;
    q.EG = q.E / ept;
    q.NG = Hp / npt;
    q.n_half = (q.EG * q.NG + 31) / 32 * 32;
    q.half = q.E / 2;
    q.nt = 2 * q.n_half < 128 ? 128 : 2 * q.n_half;
    q.ldh = 4 * ((Hp / 4) | 1);
    size_t o = 0;
    auto take = [&](size_t n) { const size_t r = o; o += (n + 31) / 32 * 32; return (int)r; };
    auto both = [&](int& first, int& step, size_t n) { first = take(n); step = take(n) - first; };
    both(q.w, q.s_w, p.w_total);
    both(q.xs, q.s_xs, (size_t)p.D * q.E);
    both(q.h1, q.s_h1, (size_t)Hp * q.E);
    both(q.h2, q.s_h2, (size_t)q.E * q.ldh);
    both(q.w3, q.s_w3, (size_t)4 * q.ldh);
    q.q = take((size_t)8 * q.E + 4);
    q.bar = take(8);
    smem = o * sizeof(float);
    if (smem <= 226 * 1024) return true;
  }
  return false;
}

// *grid_out = 0: nothing launched, the networks do not fit
cudaError_t launch_td_fma(const TdParams& p, int sm_count, int* grid_out, cudaStream_t s) {
  TfPlan q{};
  int ept = 0, npt = 0;
  size_t smem = 0;
  const int sms = sm_count > 0 ? sm_count : 148;
  *grid_out = 0;
  if (!plan_td_fma(p, sms, q, ept, npt, smem)) return cudaSuccess;
  const int tiles = (p.n + q.E - 1) / q.E, grid = tiles < sms ? tiles : sms;
  *grid_out = grid;
  return launch_chained(ept == 8 ? td_fma_kernel<8, 4> : (npt == 4 ? td_fma_kernel<4, 4> : (npt == 2 ? td_fma_kernel<4, 2> : td_fma_kernel<4, 1>)), grid,
                        q.nt, smem, s, p, q);
}

}  // namespace tj
