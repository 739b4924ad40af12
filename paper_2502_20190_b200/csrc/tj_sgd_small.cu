// Learner update for small networks (obs_dim <= 8, hidden <= 128, at most four outputs: CartPole and Acrobot): forward of
// both networks (or PPO's one), loss, backward and this block's share of every gradient in ONE kernel, then the apply pass.
//
// Such a minibatch is a few microseconds of FP32 work (6-64-64-2 at 1,024 rows: 37 MFLOP) that the layered kernels spent on
// launches, on global round trips of the activations and on 16-row tiles that left most SMs idle (66 us per update).  Here a
// block keeps all parameters of both networks in shared memory (135 KB at hidden 128) and takes R rows, R the smallest of
// 4, 8, 16, 32 that leaves at most one block per SM, so that the whole minibatch is in flight at once; what bounds it then is
// the latency of the chain of layers.  Activations are stored row by row, so that both operands of a layer are 16-byte words
// along the contraction and the products run as packed pairs (fma.rn.f32x2: each half rounds as fmaf does); where a layer
// has fewer 4 x 4 output tiles than threads the contraction is split over the idle ones.
// Gradients leave as one partial per block, laid out like the parameter blob; the apply kernel adds them in a fixed order.
#include "tj_async.cuh"
#include "tj_fma.cuh"
#include "tj_internal.h"

namespace tj {

namespace {

constexpr int FS_NT = 512;
constexpr int FS_MAX_H = 128;
constexpr int FS_MAX_PARTS = SGD_FUSED_MAX_PARTS;

// row strides: a multiple of four floats, odd in 16-byte units, so that eight lanes on consecutive rows touch all banks
__host__ __device__ inline int fs_ld(int k) {
  const int q = (k + 3) / 4;
  return 4 * (q | 1);
}

// One parameter matrix: rows x cols of the blob at float offset `src` to shared memory at `dst` (row stride ld), zeros up to
// rows_pad x 4 ceil(cols / 4).
struct FsLoad { int src, dst, ld, rows, cols, rows_pad; };

__device__ __forceinline__ void load_matrix(float* sm, const float* blob, const FsLoad& m) {
  const int cp = (m.cols + 3) & ~3;
  const float* src = blob + m.src;
  const bool vec = (m.cols & 3) == 0 && (reinterpret_cast<uintptr_t>(src) & 15) == 0;
  const int step = vec ? 4 : 1, items = cp / step;
  int shift = 0;                                   // 2^shift lanes per row, all 32 of a warp in use for narrow matrices
  while ((1 << shift) < items && shift < 5) ++shift;
  const int c0 = (threadIdx.x & ((1 << shift) - 1)) * step, r0 = threadIdx.x >> shift, dr = FS_NT >> shift;
#pragma unroll 1
  for (int r = r0; r < m.rows_pad; r += dr)
#pragma unroll 1
    for (int c = c0; c < cp; c += step << shift) {
      float* d = sm + m.dst + r * m.ld + c;
      if (r < m.rows && c < m.cols) {
        const float* g = src + r * m.cols + c;
        if (vec) cp_async16(d, g);
        else cp_async4(d, g);
      } else {
        for (int i = 0; i < step; ++i) d[i] = 0.f;
      }
    }
}

// where everything lies in shared memory, in floats
struct FsLayout {
  int ldD, ldH, Hp;
  int W2, W3, b2, b3, T2, T3, tb2, tb3, xs, xn, h1, h2, d1, d2, g, q, part, one, red, bar, total;
  int G, T, KS, KB;                                // neuron quads; 4 x 4 output tiles of a hidden layer; shares of a contraction, of the backward one
  int words16;                                     // rows of the parameter blobs are whole 16-byte words
};

inline FsLayout fs_layout(int D, int H, int R, bool ppo) {
  FsLayout L;
  L.Hp = (H + 3) / 4 * 4;
  L.ldD = fs_ld(D);
  L.ldH = fs_ld(H);
  int o = 0;
  auto take = [&](int n) { const int r = o; o += (n + 3) / 4 * 4; return r; };
  L.W2 = take(L.Hp * L.ldH); L.W3 = take(4 * L.ldH); L.b2 = take(L.Hp); L.b3 = take(4);
  if (ppo) {
    L.T2 = L.T3 = L.tb2 = L.tb3 = 0;
  } else {
    L.T2 = take(L.Hp * L.ldH); L.T3 = take(4 * L.ldH); L.tb2 = take(L.Hp); L.tb3 = take(4);
  }
  L.xs = take(R * L.ldD);
  L.xn = ppo ? 0 : take(R * L.ldD);
  L.h1 = take(R * L.ldH); L.h2 = take(R * L.ldH); L.d1 = take(R * L.ldH); L.d2 = take(R * L.ldH);
  L.g = take(R * 4); L.q = take(2 * R * 4); L.part = take(5 * R); L.one = take(4);
  L.G = L.Hp / 4;
  L.T = L.G * (R / 4);
  const int nets = ppo ? 1 : 2;                    // the hidden layers of both networks run side by side
  L.KS = FS_NT / (nets * L.T);
  L.KB = FS_NT / L.T;
  L.KS = L.KS < 1 ? 1 : (L.KS > 4 ? 4 : L.KS);   // a whole update, us, with up to 2 / 4 / 8 / 16 shares:
                                                   // hidden 64, 256 rows 13.1 / 12.3 / 12.2 / 12.5, 1,024 rows 13.8 / 12.8 / 12.9 / 13.6;
                                                   // hidden 128, 256 rows 16.8 / 14.6 / 14.4 / 14.8
  L.KB = L.KB < 1 ? 1 : (L.KB > 4 ? 4 : L.KB);
  if (L.KS > L.G) L.KS = L.G;
  if (L.KB > L.G) L.KB = L.G;
  auto red = [&] { const int f = L.KS > 1 ? L.KS * nets * L.T * 16 : 0, b = L.KB > 1 ? L.KB * L.T * 16 : 0; return f > b ? f : b; };
  if (o + red() + 8 > 227 * 256) L.KS = L.KB = 1;
  L.red = take(red());                             // only where a layer's contraction is split
  L.bar = take(8);
  L.words16 = 0;
  L.total = o;
  return L;
}

// this thread's part in a layer's product, the same for all hidden layers: output tile (row group rg, neuron group g), share
struct FsTile { int T, KS, tile, share, rg, g; bool active; };   // T, tile: over all networks of the product

// the partial sums of a split contraction: 4 x 4 values per tile and share; slot j of a tile is finished by share j mod KS
template <typename F>
__device__ __forceinline__ void reduce_shares(float* red, const float (&v)[4][4], const FsTile& t, int KS, bool active, F finish) {
  if (KS == 1) {
    if (active) {
#pragma unroll
      for (int j = 0; j < 4; ++j) finish(j, make_float4(v[j][0], v[j][1], v[j][2], v[j][3]));
    }
    return;
  }
  if (active) {
#pragma unroll
    for (int j = 0; j < 4; ++j)
      *reinterpret_cast<float4*>(red + ((t.share * 4 + j) * t.T + t.tile) * 4) = make_float4(v[j][0], v[j][1], v[j][2], v[j][3]);
  }
  __syncthreads();
  if (!active) return;
#pragma unroll 1
  for (int j = t.share; j < 4; j += KS) {
    const float* col = red + (j * t.T + t.tile) * 4;
    float4 s = *reinterpret_cast<const float4*>(col);
#pragma unroll 1
    for (int k = 1; k < KS; ++k) {
      col += 16 * t.T;
      const float4 o = *reinterpret_cast<const float4*>(col);
      s.x += o.x; s.y += o.y; s.z += o.z; s.w += o.w;
    }
    finish(j, s);
  }
}

// out[r][n] = relu(bias[n] + sum_k W[n][k] in[r][k]) for R rows; a thread owns neurons g + G j and rows rg + RG i, j, i < 4
template <int R>
__device__ __noinline__ void dense_rows(const float* W, int ldw, const float* bias, const float* in, int ldi, float* out, int ldo, int K4,
                                        int G, const FsTile t, float* red) {
  constexpr int RG = R / 4;
  const int KS = t.KS < K4 ? t.KS : K4;
  const bool active = t.share < KS;
  const int rg = t.rg, g = t.g;
  f32x2 acc[4][4];
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[j][i] = 0ull;
  if (active) {
#pragma unroll 1
    for (int k4 = t.share; k4 < K4; k4 += KS) {
      ulonglong2 w[4], x[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) w[j] = ld_pairs(W + (g + G * j) * ldw + 4 * k4);
#pragma unroll
      for (int i = 0; i < 4; ++i) x[i] = ld_pairs(in + (rg + RG * i) * ldi + 4 * k4);
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) { fma2(acc[j][i], w[j].x, x[i].x); fma2(acc[j][i], w[j].y, x[i].y); }
    }
  }
  float v[4][4];
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int i = 0; i < 4; ++i) { const float2 h = halves(acc[j][i]); v[j][i] = h.x + h.y; }
  reduce_shares(red, v, t, KS, active, [&](int j, float4 s) {
    float* o = out + rg * ldo + g + G * j;
    const float b = bias[g + G * j];
    o[0] = fmaxf(s.x + b, 0.f);
    o[RG * ldo] = fmaxf(s.y + b, 0.f);
    o[2 * RG * ldo] = fmaxf(s.z + b, 0.f);
    o[3 * RG * ldo] = fmaxf(s.w + b, 0.f);
  });
  __syncthreads();
}

// d1[r][k] = sum_i d2[r][i] W[i][k] where h1[r][k] > 0; a thread owns the input quad g and rows rg + RG i
template <int R>
__device__ __forceinline__ void dense_back(const float* W, int ldw, const float* d2, const float* h1, float* d1, int ld, int I4, const FsTile t,
                                           float* red) {
  constexpr int RG = R / 4;
  const int rg = t.rg, g = t.g;
  f32x2 acc[4][2];                                 // [row][pair of inputs]
#pragma unroll
  for (int i = 0; i < 4; ++i) acc[i][0] = acc[i][1] = 0ull;
  if (t.active) {
#pragma unroll 1
    for (int i4 = t.share; i4 < I4; i4 += t.KS) {
      ulonglong2 w[4];
      float4 d[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) w[j] = ld_pairs(W + (4 * i4 + j) * ldw + 4 * g);
#pragma unroll
      for (int i = 0; i < 4; ++i) d[i] = *reinterpret_cast<const float4*>(d2 + (rg + RG * i) * ld + 4 * i4);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const f32x2 a = dup2(d[i].x), b = dup2(d[i].y), c = dup2(d[i].z), e = dup2(d[i].w);
        fma2(acc[i][0], a, w[0].x); fma2(acc[i][1], a, w[0].y);
        fma2(acc[i][0], b, w[1].x); fma2(acc[i][1], b, w[1].y);
        fma2(acc[i][0], c, w[2].x); fma2(acc[i][1], c, w[2].y);
        fma2(acc[i][0], e, w[3].x); fma2(acc[i][1], e, w[3].y);
      }
    }
  }
  float v[4][4];                                   // [row slot][input of the quad]
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 a = halves(acc[i][0]), b = halves(acc[i][1]);
    v[i][0] = a.x; v[i][1] = a.y; v[i][2] = b.x; v[i][3] = b.y;
  }
  reduce_shares(red, v, t, t.KS, t.active, [&](int i, float4 s) {
    const int o = (rg + RG * i) * ld + 4 * g;
    const float4 h = *reinterpret_cast<const float4*>(h1 + o);
    *reinterpret_cast<float4*>(d1 + o) = make_float4(h.x > 0.f ? s.x : 0.f, h.y > 0.f ? s.y : 0.f, h.z > 0.f ? s.z : 0.f, h.w > 0.f ? s.w : 0.f);
  });
  __syncthreads();
}

// partial gradients: the block's first chunk of rows stores, later ones add
struct FsOut {
  float* P;
  bool add;
  __device__ __forceinline__ void one(int i, float v) const { P[i] = add ? P[i] + v : v; }
  __device__ __forceinline__ void quad(int i, float4 v, bool vec) const {
    if (vec) {
      float4* d = reinterpret_cast<float4*>(P + i);
      if (add) { const float4 o = *d; v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w; }
      *d = v;
    } else {
      one(i, v.x); one(i + 1, v.y); one(i + 2, v.z); one(i + 3, v.w);
    }
  }
};

// dW2[i][k] = sum_r d2[r][i] h1[r][k]: a thread owns TI quads of neurons (half the width apart) x one quad of inputs
template <int R, int TI>
__device__ __forceinline__ void grad_hidden(const float* d2, const float* h1, int ld, int H, int G, int off, const FsOut& out) {
  const int QH = (G + TI - 1) / TI;
  const int ti = threadIdx.x / G, tk = threadIdx.x - ti * G;
  if (ti >= QH) return;
  f32x2 acc[4 * TI][2];
#pragma unroll
  for (int a = 0; a < 4 * TI; ++a) acc[a][0] = acc[a][1] = 0ull;
  const float* hp = h1 + 4 * tk;
  const float* dp = d2 + 4 * ti;
  const int second = TI > 1 && ti + QH < G ? 4 * QH : 0;     // an odd width has no second quad in its last tile: computed, not written
#pragma unroll 1
  for (int r = 0; r < R; ++r, hp += ld, dp += ld) {
    const ulonglong2 h = ld_pairs(hp);
#pragma unroll
    for (int u = 0; u < TI; ++u) {
      const float4 d = *reinterpret_cast<const float4*>(dp + u * second);
      const float dv[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const f32x2 dd = dup2(dv[a]);
        fma2(acc[4 * u + a][0], dd, h.x);
        fma2(acc[4 * u + a][1], dd, h.y);
      }
    }
  }
  const bool vec = (H & 3) == 0 && (off & 3) == 0;
#pragma unroll
  for (int u = 0; u < TI; ++u) {
    if (u == 1 && !second) break;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const int i = 4 * (ti + u * QH) + a;
      const float2 lo = halves(acc[4 * u + a][0]), hi = halves(acc[4 * u + a][1]);
      if (vec) {
        out.quad(off + i * H + 4 * tk, make_float4(lo.x, lo.y, hi.x, hi.y), true);
      } else if (i < H) {
        const float v[4] = {lo.x, lo.y, hi.x, hi.y};
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (4 * tk + c < H) out.one(off + i * H + 4 * tk + c, v[c]);
      }
    }
  }
}

// W1, the biases of the hidden layers and the head, one sum per thread and turn: neuron n of a column -- an input (times d1), ones
// (times d1, then d2), an output's gradient (times h2).  Lanes run along the neurons; the column's value is a broadcast.  The block's
// threads from `first` on (a multiple of 128) share the columns.
template <int R>
__device__ __forceinline__ void grad_narrow(const FsLayout& L, const float* sm, int D, int H, int A, int vh, int first, const FsOut& out) {
  const int shift = H > 64 ? 7 : (H > 32 ? 6 : 5), id = (int)threadIdx.x - first, n = id & ((1 << shift) - 1), n_cols = D + 2 + A + vh;
  if (id < 0 || n >= H) return;
#pragma unroll 1
  for (int c = id >> shift; c < n_cols; c += (FS_NT - first) >> shift) {
    const int a = c - D - 2;
    const float* d = sm + (c <= D ? L.d1 : (a < 0 ? L.d2 : L.h2)) + n;
    const float* x = sm + (c < D ? L.xs + c : (a < 0 ? L.one : L.g + a));
    const int ldx = c < D ? L.ldD : (a < 0 ? 0 : 4);
    float s = 0.f;
#pragma unroll 8
    for (int r = 0; r < R; ++r, d += L.ldH, x += ldx) s = fmaf(*d, *x, s);
    const int o_b1 = H * D, o_b2 = o_b1 + H + H * H, o_W3 = o_b2 + H;
    // the value head's row follows the action heads' rows and their biases
    out.one(c < D ? n * D + c : (a < 0 ? (a == -2 ? o_b1 : o_b2) + n : o_W3 + a * H + (a == A ? A : 0) + n), s);
  }
}

template <int R, bool PPO>
__global__ void __launch_bounds__(FS_NT, 1) sgd_fused_kernel(const SgdParams p, const FsLayout L, int stride) {
  extern __shared__ __align__(128) float fs_sm[];
  const int D = p.D, H = p.H, A = p.A, tid = threadIdx.x, G = L.G, Dq = (D + 3) / 4, Dp = 4 * Dq;
  float* sm = fs_sm;
  uint64_t* bar = reinterpret_cast<uint64_t*>(sm + L.bar);   // the parameters are here
  FsTile t, tb;                                    // of the forward layers and of the backward one
  t.T = (PPO ? 1 : 2) * L.T; t.KS = L.KS;
  t.share = tid / t.T; t.tile = tid - t.share * t.T;
  t.active = t.share < L.KS;
  const bool target = !PPO && t.tile >= L.T;               // this thread's network in the forward layers
  t.g = (t.tile - (target ? L.T : 0)) / (R / 4); t.rg = t.tile % (R / 4);
  tb.T = L.T; tb.KS = L.KB;
  tb.share = tid / L.T; tb.tile = tid - tb.share * L.T; tb.g = tb.tile / (R / 4); tb.rg = tb.tile % (R / 4);
  tb.active = tb.share < L.KB;
  if (L.words16 && tid == 0) mbar_init(bar, FS_NT);
  __syncthreads();
  chain_begin();
  const int o_b1 = H * D, o_W2 = o_b1 + H, o_b2 = o_W2 + H * H, o_W3 = o_b2 + H, o_b3 = o_W3 + A * H;
  // every load of the prologue is in flight before the first result is used: a load that waits for another costs a round trip
  // to L2 (0.45 us), and four of them in a row were a third of the kernel.  What layer 1 needs goes first: the hidden matrices, which every
  // block reads at the same time, hold up whatever is queued behind them.
  // layer 1: a thread owns neuron n for rows r0, r0 + dr, ...; its weights and biases of both networks go straight to registers
  const int shift = H > 64 ? 7 : (H > 32 ? 6 : 5), n = tid & ((1 << shift) - 1), r0 = tid >> shift, dr = FS_NT >> shift;
  float w1[8], t1[8], c1 = 0.f, e1 = 0.f, head_bias = 0.f, head_value = 0.f;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const bool live = n < H && k < D;
    w1[k] = live ? __ldg(p.theta + n * D + k) : 0.f;
    t1[k] = !PPO && live ? __ldg(p.theta_target + n * D + k) : 0.f;
  }
  if (n < H) {
    c1 = __ldg(p.theta + o_b1 + n);
    if (!PPO) e1 = __ldg(p.theta_target + o_b1 + n);
  }
  if (tid < (PPO ? 4 : 8)) {
    const int a = tid & 3;
    if (a < A) head_bias = __ldg((tid >> 2 ? p.theta_target : p.theta) + o_b3 + a);
    else if (PPO && a == A) head_bias = __ldg(p.theta + o_b3 + A + H);
  }
  if (PPO && L.words16 && tid < H) head_value = __ldg(p.theta + o_b3 + A + tid);
  // a chunk's rows: element k of row r by thread 8 r + k, the row's scalars by thread r
  float x = 0.f, y = 0.f, rew = 0.f, adv = 0.f, ret = 0.f;
  int act = 0, done = 0;
  auto fetch_rows = [&](int chunk) {
    const int row0 = chunk * R, rows = min(R, p.n - row0), r = tid >> 3, k = tid & 7;
    x = y = 0.f;
    if (r < rows && k < D) {
      x = __ldg(p.obs + (size_t)(row0 + r) * D + k);
      if (!PPO) y = __ldg(p.next_obs + (size_t)(row0 + r) * D + k);
    }
    if (tid < rows) {
      act = p.act[row0 + tid];
      if (PPO) {
        rew = p.logp_old[row0 + tid];
        adv = p.adv[row0 + tid];
        ret = p.ret[row0 + tid];
      } else {
        rew = p.rew[row0 + tid];
        done = p.done[row0 + tid];
      }
    }
  };
  fetch_rows(blockIdx.x);
  if (L.words16) {
    // a thread copies one 16-byte column of every RP-th row of the hidden matrices, the first rows' threads the head and the biases too.
    // (One bulk copy per row, issued by a thread per row, took 32 cycles each, one after the other: 4,400 cycles for two networks at
    // hidden 64, a quarter of the kernel.)
    const int RP = FS_NT / G, first = tid / G, c = 4 * (tid - first * G);
    if (first < RP) {
#pragma unroll 1
      for (int net = PPO ? 0 : 1; net >= 0; --net) {
        const float* blob = net ? p.theta_target : p.theta;
        if (first < A) cp_async16(sm + (net ? L.T3 : L.W3) + first * L.ldH + c, blob + o_W3 + first * H + c);
        else if (first == 4) cp_async16(sm + (net ? L.tb2 : L.b2) + c, blob + o_b2 + c);
        const float* src = blob + o_W2 + first * H + c;
        float* dst = sm + (net ? L.T2 : L.W2) + first * L.ldH + c;
#pragma unroll 4
        for (int r = first; r < H; r += RP, src += RP * H, dst += RP * L.ldH) cp_async16(dst, src);
      }
    }
    cp_async_arrive(bar);
  } else {
#pragma unroll 1
    for (int net = PPO ? 0 : 1; net >= 0; --net) {
#pragma unroll 1
      for (int m = 0; m < (PPO ? 4 : 3); ++m) {
        FsLoad ld;
        if (m == 0) ld = FsLoad{o_b2, net ? L.tb2 : L.b2, L.Hp, 1, H, 1};
        else if (m == 1) ld = FsLoad{o_W3, net ? L.T3 : L.W3, L.ldH, A, H, PPO ? A : 4};
        else if (m == 2) ld = FsLoad{o_W2, net ? L.T2 : L.W2, L.ldH, H, H, L.Hp};
        else ld = FsLoad{o_b3 + A, L.W3 + A * L.ldH, L.ldH, 1, H, 4 - A};
        load_matrix(sm, net ? p.theta_target : p.theta, ld);
      }
    }
    cp_async_commit();
  }
  if (tid < (PPO ? 4 : 8)) sm[(tid >> 2 ? L.tb3 : L.b3) + (tid & 3)] = head_bias;
  if (L.words16 && tid < H)
    for (int a = A; a < 4; ++a) {                  // zeros for the head's unused outputs (PPO's value head is output A)
      sm[L.W3 + a * L.ldH + tid] = PPO && a == A ? head_value : 0.f;
      if (!PPO) sm[L.T3 + a * L.ldH + tid] = 0.f;
    }
  if (tid == 0) sm[L.one] = 1.f;
  const int n_chunks = (p.n + R - 1) / R;
  bool ok = true;                                  // a wait that runs out: the thread goes on with meaningless numbers
  FsOut out{p.grad_partial + (size_t)blockIdx.x * stride, false};
  const int lane = tid & 31;
  float part[5] = {0.f, 0.f, 0.f, 0.f, 0.f};       // the block's loss terms, in one of its warps
  for (int chunk = blockIdx.x; chunk < n_chunks; chunk += gridDim.x, out.add = true) {
    const int rows = min(R, p.n - chunk * R);
    if (tid < 8 * R && (tid & 7) < Dp) {
      sm[L.xs + (tid >> 3) * L.ldD + (tid & 7)] = x;
      if (!PPO) sm[L.xn + (tid >> 3) * L.ldD + (tid & 7)] = y;
    }
    if (!L.words16) cp_async_wait<0>();
    __syncthreads();
    if (n < L.Hp) {
#pragma unroll 1
      for (int r = r0; r < R; r += dr) {
        const float* xr = sm + L.xs + r * L.ldD;
        const float* yr = sm + L.xn + r * L.ldD;
        float a = c1, b = e1;
#pragma unroll
        for (int k = 0; k < 8; ++k)
          if (k < 4 || D > 4) {
            a = fmaf(w1[k], xr[k], a);
            if (!PPO) b = fmaf(t1[k], yr[k], b);
          }
        sm[L.h1 + r * L.ldH + n] = fmaxf(a, 0.f);
        if (!PPO) sm[L.d1 + r * L.ldH + n] = fmaxf(b, 0.f);
      }
    }
    __syncthreads();
    if (L.words16) ok = ok && mbar_wait_bounded(bar, 0);
    // both networks side by side: the target's activations lie in d1, d2
    dense_rows<R>(sm + (target ? L.T2 : L.W2), L.ldH, sm + (target ? L.tb2 : L.b2), sm + (target ? L.d1 : L.h1), L.ldH, sm + (target ? L.d2 : L.h2),
                  L.ldH, G, G, t, sm + L.red);
    // heads: eight lanes per (network, row)
    for (int slot = tid >> 3; slot < (PPO ? R : 2 * R); slot += FS_NT / 8) {
      const int net = PPO ? 0 : slot / R, r = PPO ? slot : slot % R, s = tid & 7;
      const float* h = sm + (net ? L.d2 : L.h2) + r * L.ldH;
      const float* w = sm + (net ? L.T3 : L.W3);
      float o[4] = {0.f, 0.f, 0.f, 0.f};
      for (int q = s; q < G; q += 8) {
        const float4 x = *reinterpret_cast<const float4*>(h + 4 * q);
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          const float4 c = *reinterpret_cast<const float4*>(w + a * L.ldH + 4 * q);
          o[a] = fmaf(x.x, c.x, o[a]); o[a] = fmaf(x.y, c.y, o[a]); o[a] = fmaf(x.z, c.z, o[a]); o[a] = fmaf(x.w, c.w, o[a]);
        }
      }
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        o[a] += __shfl_xor_sync(0xffffffffu, o[a], 4);
        o[a] += __shfl_xor_sync(0xffffffffu, o[a], 2);
        o[a] += __shfl_xor_sync(0xffffffffu, o[a], 1);
      }
      if (s == 0) {
        const float4 b = *reinterpret_cast<const float4*>(sm + (net ? L.tb3 : L.b3));
        *reinterpret_cast<float4*>(sm + L.q + (net * R + r) * 4) = make_float4(o[0] + b.x, o[1] + b.y, o[2] + b.z, o[3] + b.w);
      }
    }
    __syncthreads();
    // loss and its gradient at the outputs, one thread per row
    if (tid < R) {
      const int r = tid;
      // outputs in registers: an array indexed at run time is a shared-memory latency per access
      const float4 q4 = *reinterpret_cast<const float4*>(sm + L.q + r * 4);
      const float q[4] = {q4.x, q4.y, q4.z, q4.w};
      auto pick = [](const float (&v)[4], int i) { return i == 0 ? v[0] : (i == 1 ? v[1] : (i == 2 ? v[2] : v[3])); };
      act = act < 0 ? 0 : (act >= A ? A - 1 : act);
      float g[4] = {0.f, 0.f, 0.f, 0.f}, l[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
      if (r < rows) {
        if (PPO) {
          float lmax = q[0];
#pragma unroll
          for (int i = 1; i < 4; ++i)
            if (i < A) lmax = fmaxf(lmax, q[i]);
          float Z = 0.f;
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (i < A) Z += expf(q[i] - lmax);
          const float logZ = lmax + logf(Z);
          float ent = 0.f, lp[4] = {0.f, 0.f, 0.f, 0.f}, pi[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (i < A) {
              lp[i] = q[i] - logZ;
              pi[i] = expf(lp[i]);
              ent -= pi[i] * lp[i];
            }
          const float logp = pick(q, act) - logZ, ratio = expf(logp - rew);
          const float rc = fminf(fmaxf(ratio, 1.f - p.clip_eps), 1.f + p.clip_eps);
          const float t1 = ratio * adv, t2 = rc * adv;
          const bool unclipped = t1 <= t2;
          const float dv = pick(q, A) - ret;
          l[1] = -(unclipped ? t1 : t2);
          l[2] = 0.5f * dv * dv;
          l[3] = ent;
          l[4] = unclipped ? 0.f : 1.f;
          l[0] = l[1] + p.c_v * l[2] - p.c_e * l[3];
          const float g_logp = unclipped ? -adv * ratio : 0.f, inv_n = 1.f / (float)p.n;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float dlogp = (i == act ? 1.f : 0.f) - pi[i], dent = -pi[i] * (lp[i] + ent);
            if (i < A) g[i] = (g_logp * dlogp - p.c_e * dent) * inv_n;
            else if (i == A) g[i] = p.c_v * dv * inv_n;
          }
        } else {
          const float4 t4 = *reinterpret_cast<const float4*>(sm + L.q + (R + r) * 4);
          const float qt[4] = {t4.x, t4.y, t4.z, t4.w};
          float qmax = qt[0];
#pragma unroll
          for (int i = 1; i < 4; ++i)
            if (i < A) qmax = fmaxf(qmax, qt[i]);
          const float y = rew + p.gamma * (done ? 0.f : 1.f) * qmax;
          const float delta = y - pick(q, act), ad = fabsf(delta);
          l[0] = ad <= p.kappa ? 0.5f * delta * delta : p.kappa * (ad - 0.5f * p.kappa);
          const float ga = -fminf(fmaxf(delta, -p.kappa), p.kappa) / (float)p.n;
#pragma unroll
          for (int i = 0; i < 4; ++i) g[i] = i == act ? ga : 0.f;
        }
      }
      *reinterpret_cast<float4*>(sm + L.g + r * 4) = make_float4(g[0], g[1], g[2], g[3]);
#pragma unroll
      for (int k = 0; k < (PPO ? 5 : 1); ++k) sm[L.part + k * R + r] = l[k];
    }
    __syncthreads();
    // d2[r][i] = sum_a g[r][a] W3[a][i] where h2 > 0 (the target network's activations in d1, d2 are used up)
#pragma unroll 1
    for (int i = tid; i < R * 32; i += FS_NT) {
      const int r = i >> 5, q = i & 31;
      if (q >= G) continue;
      const float4 g = *reinterpret_cast<const float4*>(sm + L.g + r * 4), h = *reinterpret_cast<const float4*>(sm + L.h2 + r * L.ldH + 4 * q);
      const float ga[4] = {g.x, g.y, g.z, g.w};
      float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const float4 w = *reinterpret_cast<const float4*>(sm + L.W3 + a * L.ldH + 4 * q);
        d.x = fmaf(ga[a], w.x, d.x); d.y = fmaf(ga[a], w.y, d.y); d.z = fmaf(ga[a], w.z, d.z); d.w = fmaf(ga[a], w.w, d.w);
      }
      d.x = h.x > 0.f ? d.x : 0.f; d.y = h.y > 0.f ? d.y : 0.f; d.z = h.z > 0.f ? d.z : 0.f; d.w = h.w > 0.f ? d.w : 0.f;
      *reinterpret_cast<float4*>(sm + L.d2 + r * L.ldH + 4 * q) = d;
    }
    // the block's loss terms and the output biases' gradients (column sums of g), a warp each, lane r row r: added by one thread row after
    // row they kept this phase at 2,070 cycles for 32 rows of PPO
    if (tid >> 5 == FS_NT / 32 - 2) {
      float v[5];
#pragma unroll
      for (int k = 0; k < (PPO ? 5 : 1); ++k) v[k] = lane < R ? sm[L.part + k * R + lane] : 0.f;
#pragma unroll
      for (int k = 0; k < (PPO ? 5 : 1); ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
        part[k] += v[k];
      }
    } else if (tid >> 5 == FS_NT / 32 - 1) {
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (lane < R) v = *reinterpret_cast<const float4*>(sm + L.g + lane * 4);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o); v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
        v.z += __shfl_xor_sync(0xffffffffu, v.z, o); v.w += __shfl_xor_sync(0xffffffffu, v.w, o);
      }
      const int off = H * D + H + H * H + H + A * H;
      const float s = lane == 0 ? v.x : (lane == 1 ? v.y : (lane == 2 ? v.z : v.w));
      if (lane < A) out.one(off + lane, s);
      else if (PPO && lane == A) out.one(off + A + H, s);
    }
    __syncthreads();
    dense_back<R>(sm + L.W2, L.ldH, sm + L.d2, sm + L.h1, sm + L.d1, L.ldH, G, tb, sm + L.red);
    if (G * G <= FS_NT) grad_hidden<R, 1>(sm + L.d2, sm + L.h1, L.ldH, H, G, H * D + H, out);
    else grad_hidden<R, 2>(sm + L.d2, sm + L.h1, L.ldH, H, G, H * D + H, out);
    if (chunk + (int)gridDim.x < n_chunks) fetch_rows(chunk + gridDim.x);
    // where the hidden matrix's gradient leaves half of the threads idle (up to hidden 64), they do the narrow ones meanwhile
    grad_narrow<R>(L, sm, D, H, A, PPO ? 1 : 0, G * G <= FS_NT / 2 ? FS_NT / 2 : 0, out);
    __syncthreads();
  }
  if (tid == FS_NT - 64) {
    float* pp = p.partial + (size_t)blockIdx.x * 5;
#pragma unroll
    for (int k = 0; k < (PPO ? 5 : 1); ++k) pp[k] = part[k];
  }
  if (!ok) {
    update_failed(p.watch);
    if (L.words16) mbar_settle(bar, 0);
  }
}

// theta from the sums of the blocks' partial gradients: a block takes 128 parameters, sixteen warps a share of the partials each
// (sixteen bytes per lane and partial), added in a fixed order; block 0 also adds up the loss terms
constexpr int FA_SHARES = 16, FA_NT = 32 * FA_SHARES;
//
// The parameters are 96 bytes on purpose: with 24 more the kernel's first look at the last of them missed the constant cache once more
// and the launch took 4.75 us instead of 4.0 (hidden 64, 1,024 rows).
struct FaParams {
  float *theta, *m, *v;
  const float *P, *loss_parts;
  float* loss_out;
  float lr, beta1, beta2, eps, c1, c2;
  int stride, count, n_parts, n_terms, n_rows;
  unsigned number;                                 // of the update; the number of the last one that failed lies in front of P
};
static_assert(sizeof(FaParams) <= 96, "a fourth constant line");
template <bool ADAM>
__global__ void __launch_bounds__(FA_NT) sgd_fused_apply_kernel(const FaParams p) {
  __shared__ float4 sums[FA_SHARES][32];
  const int tid = threadIdx.x, lane = tid & 31, share = tid >> 5, q = blockIdx.x * 32 + lane;
  chain_begin();
  chain_next();
  // this thread's parameter and moments are on their way while the partials are added
  const int i = blockIdx.x * 128 + tid;
  const bool mine = tid < 128 && i < p.count;
  const unsigned asked = update_ask(reinterpret_cast<const unsigned*>(p.P) - 4, p.number);
  float theta_i = 0.f, m_i = 0.f, v_i = 0.f;
  if (mine) {
    theta_i = p.theta[i];
    if (ADAM) { m_i = p.m[i]; v_i = p.v[i]; }
  }
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
  if (4 * q < p.count) {
#pragma unroll 8
    for (int b = share; b < p.n_parts; b += FA_SHARES) {
      const float4 v = __ldcg(reinterpret_cast<const float4*>(p.P + (size_t)b * p.stride) + q);
      s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
    }
  }
  sums[share][lane] = s;
  const bool valid = update_valid(p.number, asked);   // and the sums are there
  if (tid < 128) {
    if (mine && valid) {                           // else parameters and moments stay as they were
      const float* col = reinterpret_cast<const float*>(&sums[0][0]) + tid;
      float g = 0.f;
#pragma unroll
      for (int k = 0; k < FA_SHARES; ++k) g += col[k * 128];
      if (ADAM) {
        const float mi = fmaf(p.beta1, m_i, (1.f - p.beta1) * g);
        const float vi = fmaf(p.beta2, v_i, (1.f - p.beta2) * g * g);
        p.m[i] = mi;
        p.v[i] = vi;
        p.theta[i] = theta_i - p.lr * (mi / p.c1) / (sqrtf(vi / p.c2) + p.eps);
      } else {
        p.theta[i] = theta_i - p.lr * g;
      }
    }
  } else if (blockIdx.x == 0 && p.loss_out && share >= 4 && share - 4 < p.n_terms) {
    const int k = share - 4;
    float t = 0.f;
    for (int b = lane; b < p.n_parts; b += 32) t += p.loss_parts[(size_t)b * 5 + k];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) p.loss_out[k] = valid ? t / (float)p.n_rows : __int_as_float(0x7FC00000);
  }
}

int fs_rows(int n, int sm_count) {
  for (int R = 4; R < 32; R *= 2)
    if ((n + R - 1) / R <= sm_count) return R;
  return 32;
}

template <int R, bool PPO>
cudaError_t launch_fused(const SgdParams& p, int stride, int grid, cudaStream_t s) {
  FsLayout L = fs_layout(p.D, p.H, R, PPO);
  // H a multiple of four makes every row and the start of W2, W3 and the hidden biases whole 16-byte words of the blob
  L.words16 = p.H % 4 == 0 && ((reinterpret_cast<uintptr_t>(p.theta) | reinterpret_cast<uintptr_t>(p.theta_target)) & 15) == 0;
  return launch_chained(sgd_fused_kernel<R, PPO>, grid, FS_NT, (size_t)L.total * sizeof(float), s, p, L, stride);
}

}  // namespace

// sizes whose parameters (of both networks) fit in shared memory beside the activations of 32 rows
bool sgd_fused_ok(int D, int H, int A, int value_head) { return D <= 8 && H <= FS_MAX_H && A + value_head <= 4; }

int sgd_fused_stride(int D, int H) {
  const int blob = H * D + H + H * H + H + 17 * H + 17;
  return (blob + 3) / 4 * 4;
}

cudaError_t launch_sgd_fused(const SgdParams& p, float lr, const AdamParams* adam, float* loss_out, cudaStream_t s) {
  const int R = fs_rows(p.n, p.sm_count), chunks = (p.n + R - 1) / R, grid = chunks < FS_MAX_PARTS ? chunks : FS_MAX_PARTS;
  const int stride = sgd_fused_stride(p.D, p.H), H = p.H, D = p.D, A = p.A;
  const int count = H * D + H + H * H + H + A * H + A + (p.value_head ? H + 1 : 0);
  cudaError_t e;
  if (p.value_head) {
    e = R == 4 ? launch_fused<4, true>(p, stride, grid, s) : R == 8 ? launch_fused<8, true>(p, stride, grid, s)
      : R == 16 ? launch_fused<16, true>(p, stride, grid, s) : launch_fused<32, true>(p, stride, grid, s);
  } else {
    e = R == 4 ? launch_fused<4, false>(p, stride, grid, s) : R == 8 ? launch_fused<8, false>(p, stride, grid, s)
      : R == 16 ? launch_fused<16, false>(p, stride, grid, s) : launch_fused<32, false>(p, stride, grid, s);
  }
  if (e != cudaSuccess) return e;
  FaParams a{p.theta, nullptr, nullptr, p.grad_partial, p.partial, loss_out};
  if (adam) { a.m = adam->m; a.v = adam->v; a.beta1 = adam->beta1; a.beta2 = adam->beta2; a.eps = adam->eps; a.c1 = adam->c1; a.c2 = adam->c2; }
  a.lr = lr; a.stride = stride; a.count = count; a.n_parts = grid; a.n_terms = p.value_head ? 5 : 1; a.n_rows = p.n; a.number = p.watch.number;
  return launch_chained(adam ? sgd_fused_apply_kernel<true> : sgd_fused_apply_kernel<false>, (count + 127) / 128, FA_NT, 0, s, a);
}

}  // namespace tj
