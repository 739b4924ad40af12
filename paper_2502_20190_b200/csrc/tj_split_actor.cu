// FP32-accuracy tensor-core actor for the small environments (CartPole, Acrobot) with hidden widths of 64 .. 256: the
// hidden x hidden layer -- the one dense contraction of these networks (Algorithm 1, task 1: 65,536 of a 6-256-256-3
// network's 67,840 multiply-adds per env step) -- runs on the tensor cores as three FP16 products of split operands,
//   W2 h1 = W_hi h_hi + W_hi h_lo + W_lo h_hi,   x = x_hi + x_lo with x_hi the 11 leading bits of the (power-of-two scaled) value,
// with FP32 accumulation in tensor memory (error about 2^-22 per term, the dropped lo x lo term; FP16 runs at twice the rate
// of the 3 x TF32 form of the same idea).  Layer 1 (4 or 6 inputs) and the head (2-4 outputs) stay on the FP32 pipes.
//
// One thread block keeps its tiles of 128 environments for all n_steps of the call (environments are independent): eight worker
// warps, one MMA-issuing warp, one copy warp; per step and tile:
//   workers: layer 1 in the fixed FMA order of the FP32 path, ReLU, split -> FP16 A operand, 32 hidden units (one K chunk of
//     the next layer) at a time, each chunk handed to the issuing lane through its own mbarrier;
//   copy lane: streams W2's parts in 32-column chunks (bulk copies, four ring slots, the stream running on across steps), or, for a pair
//     of blocks, brings its half of both parts once;
//   issuing lane: per K chunk, issues W_hi x (h_hi, h_lo) and W_lo x h_hi (M = 128 or a pair's 256, N = H) as soon as that chunk of h1
//     exists, so the tensor pipe works underneath layer 1;
//   workers: accumulator -> + b2, ReLU, head sums -> outputs;
//   then exactly the FP32 kernel's selection, env step, record / segment write and reset.
// The FP32 work per step (layer 1 with its split, drain, env step: about 14,000 warp instructions a tile) and the MMAs (6,100 cycles at
// hidden 256) are of one size; what a step takes beyond them is latency.
// Every wait is bounded; a timeout latches the context's error word and the block leaves after its copies and matrix instructions in
// flight are over and its tensor memory is free.
#include <cuda_fp16.h>

#include "tj_fma.cuh"
#include "tj_internal.h"
#include "tj_tc.cuh"

namespace tj {

namespace {

constexpr int SA_TE = 128;            // envs per tile = rows of the MMA
constexpr int SA_KC = 32;             // K columns per streamed chunk of W2
constexpr int SA_SLOTS = 4;
constexpr float SA_H_SCALE = 16.0f;   // hidden activations are split after this scaling (|h1| < 4,094 stays inside FP16)

__device__ __forceinline__ float4 sa_reset4(uint2 seed, uint32_t e, unsigned long long step, float lo, float width) {
  const uint4 w = stream_words(seed, STREAM_RESET, 0, e, step);
  return make_float4(uniform_range(w.x, lo, width), uniform_range(w.y, lo, width), uniform_range(w.z, lo, width),
                     uniform_range(w.w, lo, width));
}

template <int ENV>
__device__ __forceinline__ void sa_observe(float4 s, float* obs) {
  if (ENV == TJ_ENV_CARTPOLE) {
    obs[0] = s.x; obs[1] = s.y; obs[2] = s.z; obs[3] = s.w; obs[4] = obs[5] = 0.f;
  } else {
    const float4 t = acrobot_trig(s);
    obs[0] = t.x; obs[1] = t.y; obs[2] = t.z; obs[3] = t.w; obs[4] = s.z; obs[5] = s.w;
  }
}

// ------------------------------------------------------------------------------------------------------------------------
// The actor.  A thread owns an environment for the whole call: observation, layer 1, head sums, selection and environment step stay
// in its registers, so the workers meet nobody but the issuing lane.  TPR threads per environment:
//   1  two groups of four warps, each on a tile of its own: while one tile's MMAs run, the other tile's threads drain, step and
//      compute layer 1 (calls with more tiles than SMs).  Two blocks of a cluster share every product (cta_group::2, 256 rows): each holds half
//      of W2's rows, which then stay in shared memory for the whole call instead of passing through it once per tile and step, and a product
//      reads 64 of the 128 bytes per cycle instead of 96;
//   2  eight warps on one tile: each thread takes half the rows of layer 1 and two of the outputs, the two exchange their outputs once per
//      step and both step the environment (one tile per SM: the chain of one step is the bound).
// 65,536 CartPole envs, hidden 256, 128 steps: 3.55 ms with a block per tile whose threads computed layer 1 each for its own env, 2.86 as
// pairs.  A step of two tiles is then about 20,000 cycles, 12,300 of them MMAs: what bounds it is the chain layer 1 (5,500; a fence and an
// arrival per chunk) -> MMA of the last chunk (2,000 with its signals) -> drain -> environment (3,000) of four warps per tile.  More of them
// do not fit: eight warps per tile (one thread of two steps the environment) spill at 96 registers.  Arrivals of the second block through
// a relaying warp: 4.26.
// Layer 1 hands 32 hidden units (one K chunk) at a time to the issuing lane through a ring of A-operand slots.
constexpr int S2_NT = 320;                // eight worker warps (on one tile or on two), the issuing warp, the copy warp
constexpr int S2_A_SLOTS = 8;             // most A-operand slots of a block, 16 KB each
constexpr int S2_A_PART = SA_TE * SA_KC * 2;
constexpr int S2_A_SLOT = 2 * S2_A_PART;  // high part, low part

struct S2Ctl {
  uint64_t full[SA_SLOTS], empty[SA_SLOTS];
  uint64_t a_ready[S2_A_SLOTS], a_free[S2_A_SLOTS];
  uint64_t acc_full[2], settled, w_ready;  // w_ready: a pair's halves of W2 are in shared memory
  uint32_t tmem_base, copies;             // copies: bulk copies queued so far
  int abort_flag, range_flag;
};

struct S2Plan {
  long long slot0;                        // ring slot of env 0 in the first step
  int blk0, n_blk;                        // its ring block, blocks of the ring
  int pos0, seg0;                         // position in the running segment, its slot
  int n_pass;                             // forward passes per tile: steps, and one per segment end inside the call
};

__device__ __forceinline__ f32x2 pair2(float a, float b) {
  f32x2 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
  return d;
}

// Eight hidden units of layer 1 for ROWS rows, eight apart, in the canonical order (bias, then inputs in index order; weights and biases
// come scaled by SA_H_SCALE, a power of two, which leaves every rounding where it was), ReLU, split -> a 16-byte row segment of each part
// of the A operand per row; returns the largest scaled activation.
template <int D, int ROWS>
__device__ __forceinline__ float s2_layer1(const f32x2 (&w)[D][4], const f32x2 (&b)[4], const f32x2 (&x)[ROWS][D], uint8_t* hi_dst, float vmax) {
  const f32x2 minus1 = dup2(-1.f);
#pragma unroll
  for (int r = 0; r < ROWS; ++r) {
    f32x2 acc[4] = {b[0], b[1], b[2], b[3]};
#pragma unroll
    for (int k = 0; k < D; ++k)
#pragma unroll
      for (int i = 0; i < 4; ++i) fma2(acc[i], w[k][i], x[r][k]);
    uint32_t hi[4], lo[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      // The ReLU is a maximum, which takes a NaN to 0 as in the other weight modes (a clamping conversion hands it on).  The high part is the
      // value cut to 11 bits, then converted: below 2^-14, where FP16 has fewer, rounding that is exact to 2^-25, a truncating conversion of
      // the whole value to 2^-24.
      const float2 a = halves(acc[i]);
      const float v0 = fmaxf(a.x, 0.f), v1 = fmaxf(a.y, 0.f);
      vmax = max3(vmax, v0, v1);
      const float h0 = __uint_as_float(__float_as_uint(v0) & 0xFFFFE000u), h1 = __uint_as_float(__float_as_uint(v1) & 0xFFFFE000u);
      f32x2 rest = pair2(v0, v1);
      fma2(rest, pair2(h0, h1), minus1);
      const float2 d = halves(rest);
      hi[i] = pack_f16x2(h0, h1);
      lo[i] = pack_f16x2(d.x, d.y);
    }
    *reinterpret_cast<uint4*>(hi_dst + r * ((SA_KC / 8) * 128)) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    *reinterpret_cast<uint4*>(hi_dst + S2_A_PART + r * ((SA_KC / 8) * 128)) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
  }
  return vmax;
}

// where everything lies in shared memory
template <int D, int H, int TPR>
struct S2Smem {
  static constexpr bool PAIR = TPR == 1;                      // two blocks share every product
  static constexpr int GROUPS = PAIR ? 2 : 1;                 // tiles in flight per block
  static constexpr uint32_t CHUNK_BYTES = H * SA_KC * 2;      // one chunk of one part of W2
  static constexpr uint32_t W_CHUNK = PAIR ? CHUNK_BYTES / 2 : CHUNK_BYTES;      // what of it lies in this block
  static constexpr int NKC = H / SA_KC, NSTREAM = 2 * NKC;
  static constexpr int W_SLOTS = PAIR ? NSTREAM : SA_SLOTS;
  // A slots: one ring that the groups' passes go through in turn.  A worker waits only for the chunks whose slots it takes over, so
  // the one two rounds of the ring back must be known to be used up: the ring holds more than half of two passes' chunks, and products are
  // signalled complete in the order of their issue, so a worker that has seen a pass or a chunk end knows every earlier chunk used up
  static constexpr int AS = PAIR && H > 192 ? 5 : S2_A_SLOTS;
  static_assert(2 * AS > NKC || !PAIR, "the phase of a slot's barrier is unambiguous");
  static constexpr uint32_t ACC_COLS = H <= 128 ? 128 : 256;
  uint8_t *a_ring, *w_ring;
  float *w1, *b1;         // [D][H] and [H], scaled
  float* hw;              // second-layer biases and head weights as the drain reads them.  TPR 1, per column c < H / 2: biases, head weights of
                          // outputs 0, 1, 2 of hidden units c and c + H / 2; TPR 2: [2][H] head weights of outputs 0, 1 and of outputs 2, 3
  float* hw3;             // TPR 1: head weights of output 3 of units c and c + H / 2; TPR 2: [H] second-layer biases
  float* b3;              // [4]
  float* part;            // TPR 2: outputs [pass parity][pair of outputs][TE][2]
  S2Ctl* ctl;
  __device__ __forceinline__ explicit S2Smem(uint8_t* base) {
    a_ring = base;
    w_ring = a_ring + AS * S2_A_SLOT;
    w1 = reinterpret_cast<float*>(w_ring + W_SLOTS * W_CHUNK);
    b1 = w1 + D * H; hw = b1 + H; hw3 = hw + 4 * H; b3 = hw3 + H; part = b3 + 4;
    ctl = reinterpret_cast<S2Ctl*>(part + (TPR == 2 ? 2 * 2 * SA_TE * 2 : 0));
  }
  static size_t bytes() {
    return (size_t)AS * S2_A_SLOT + (size_t)W_SLOTS * W_CHUNK +
           ((size_t)(D + 6) * H + 4 + (TPR == 2 ? 2 * 2 * SA_TE * 2 : 0)) * sizeof(float) + sizeof(S2Ctl) + 64;
  }

  // barriers and tensor memory; returns its base.  Ends with a block barrier.
  __device__ __forceinline__ uint32_t set_up() const {
    if (threadIdx.x == 0) {
      for (int s = 0; s < SA_SLOTS; ++s) { mbar_init(&ctl->full[s], 1); mbar_init(&ctl->empty[s], 1); }
      for (int s = 0; s < S2_A_SLOTS; ++s) { mbar_init(&ctl->a_ready[s], 4 * TPR * (PAIR ? 2 : 1)); mbar_init(&ctl->a_free[s], 1); }
      mbar_init(&ctl->acc_full[0], 1);
      mbar_init(&ctl->acc_full[1], 1);
      mbar_init(&ctl->settled, 1);
      mbar_init(&ctl->w_ready, 2);
      ctl->copies = 0;
      ctl->abort_flag = ctl->range_flag = 0;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
      if (PAIR) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&ctl->tmem_base)), "r"(GROUPS * ACC_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
      } else {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&ctl->tmem_base)), "r"(GROUPS * ACC_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
      }
    }
    tc_fence_before();
    if (PAIR) cluster_sync_all();                             // the other block's barriers are set up too
    else __syncthreads();
    tc_fence_after();
    return ctl->tmem_base;
  }
  __device__ __forceinline__ void tear_down(uint32_t tmem) const {
    tc_fence_before();
    __syncthreads();
    const bool issuing_warp = (int)(threadIdx.x >> 5) == S2_NT / 32 - 2;  // the last but one
    if (PAIR) {
      // Neither block leaves before the products that read both blocks' operands are over and the last arrival has reached the first one.
      // Where one block gives up, the other follows: a warp whose wait ran out arrives no more, so the first block's issuing warp waits in
      // vain and stops, and with it every completion that the second block waits for.  If nothing but the last waits is left, the other
      // block's results are whole and its own; the error word is set by either.
      if (ctl->abort_flag) {
        if (issuing_warp && cluster_rank() == 0) {
          umma_commit_pair(&ctl->settled, elect_one());
          mbar_settle(&ctl->settled, 0);
        }
        if (threadIdx.x == 0 && ctl->copies) mbar_settle(&ctl->full[0], 0);
        __syncwarp();                                         // a wait's lanes leave it one by one
      }
      cluster_sync_all();
    } else if (ctl->abort_flag) {
      tc_settle(&ctl->settled, issuing_warp, ctl->full, SA_SLOTS, ctl->copies);
      __syncthreads();
    }
    if (threadIdx.x < 32) {
      __syncwarp();
      tc_fence_after();
      if (PAIR) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(GROUPS * ACC_COLS) : "memory");
      else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(GROUPS * ACC_COLS) : "memory");
    }
  }
  // the parameters around the hidden matrix, from the packed FP32 layout P describes
  template <typename P>
  __device__ __forceinline__ void stage(const P& p, const float* W, int Aout) const {
    for (int i = threadIdx.x; i < H; i += S2_NT) {
      float wk[D];
#pragma unroll
      for (int k = 0; k < D; ++k) wk[k] = __ldg(W + p.off_W1t + k * H + i);
      const float c1 = __ldg(W + p.off_b1 + i), c2 = __ldg(W + p.off_b2 + i);
      const float4 w = __ldg(reinterpret_cast<const float4*>(W + p.off_W3t) + i);
#pragma unroll
      for (int k = 0; k < D; ++k) w1[k * H + i] = SA_H_SCALE * wk[k];
      b1[i] = SA_H_SCALE * c1;
      if (TPR == 1) {
        const int c = i % (H / 2), upper = i / (H / 2);
        float* d = hw + 8 * c + upper;
        d[0] = c2; d[2] = w.x; d[4] = w.y; d[6] = w.z;
        hw3[2 * c + upper] = w.w;
      } else {
        reinterpret_cast<float2*>(hw)[i] = make_float2(w.x, w.y);
        reinterpret_cast<float2*>(hw)[H + i] = make_float2(w.z, w.w);
        hw3[i] = c2;
      }
    }
    if (threadIdx.x >= S2_NT - 4) {
      const int a = threadIdx.x - (S2_NT - 4);
      b3[a] = a < Aout ? __ldg(W + p.off_b3 + a) : 0.f;
    }
  }
  // Issuing warp of a pair's first block: the products of n_pass passes over each of `tiles` tiles of 256 rows, the groups' passes in turn
  __device__ __forceinline__ void issue_pair(uint32_t tmem, int tiles, int n_pass) const {
    volatile int* abort_flag = &ctl->abort_flag;
    const uint32_t leader = elect_one();
    const uint32_t idesc = make_idesc_f16_m256(H);
    const uint32_t a0 = desc_lo(smem_addr(a_ring), 128u), w0 = desc_lo(smem_addr(w_ring), 128u);
    const uint32_t hiword = desc_hi((uint32_t)(SA_KC / 8) * 128u);            // A slots and W2 chunks: 32 columns wide
    uint32_t as = 0, round = 0;                               // slot of the ring, rounds of it
    bool alive = tc_wait_warp<true>(&ctl->w_ready, 0, abort_flag);
    for (int r = 0; r * GROUPS < tiles && alive; ++r)
      for (int i = 0; i < n_pass && alive; ++i)
#pragma unroll
        for (int g = 0; g < GROUPS; ++g) {
          if (!alive || r * GROUPS + g >= tiles) break;
          const uint32_t acc = tmem + (uint32_t)g * ACC_COLS;
#pragma unroll 1
          for (int kc = 0; kc < NKC; ++kc) {
            if (!tc_wait_warp<true>(&ctl->a_ready[as], round & 1, abort_flag)) { alive = false; break; }
            tc_fence_after();
            const uint32_t a_hi = a0 + as * (S2_A_SLOT / 16), a_lo = a_hi + S2_A_PART / 16, b = w0 + 2 * kc * (W_CHUNK / 16);
#pragma unroll
            for (int j = 0; j < SA_KC / 16; ++j) {
              umma_ss_pair(acc, a_hi + 16u * j, hiword, b + 16u * j, hiword, idesc, (kc | j) != 0, leader);
              umma_ss_pair(acc, a_lo + 16u * j, hiword, b + 16u * j, hiword, idesc, 1u, leader);
            }
#pragma unroll
            for (int j = 0; j < SA_KC / 16; ++j)
              umma_ss_pair(acc, a_hi + 16u * j, hiword, b + W_CHUNK / 16 + 16u * j, hiword, idesc, 1u, leader);
            umma_commit_both(&ctl->a_free[as], leader);
            if (++as == AS) { as = 0; ++round; }
          }
          if (alive) umma_commit_both(&ctl->acc_full[g], leader);
        }
  }
  // Copy lane of a block of a pair: its half of W2's rows, both parts, once
  __device__ __forceinline__ void copy_half(const uint16_t* parts) const {
    mbar_expect_tx(&ctl->full[0], NSTREAM * W_CHUNK);
    for (uint32_t c = 0; c < NSTREAM; ++c)
      bulk_copy_g2s(w_ring + c * W_CHUNK, reinterpret_cast<const uint8_t*>(parts) + (size_t)c * CHUNK_BYTES + cluster_rank() * W_CHUNK, W_CHUNK,
                    &ctl->full[0]);
    ctl->copies = NSTREAM;
    if (tc_wait(&ctl->full[0], 0, &ctl->abort_flag)) mbar_arrive_cluster(&ctl->w_ready, 0);
  }
  // Issuing warp of a block on its own: the MMAs of `passes` passes, one after the other
  __device__ __forceinline__ void issue(uint32_t tmem, uint32_t passes) const {
    volatile int* abort_flag = &ctl->abort_flag;
    const uint32_t leader = elect_one();
    const uint32_t idesc = make_idesc_f16(H);
    const uint32_t a0 = desc_lo(smem_addr(a_ring), 128u), w0 = desc_lo(smem_addr(w_ring), 128u);
    const uint32_t hiword = desc_hi((uint32_t)(SA_KC / 8) * 128u);            // A slots and W2 chunks: 32 columns wide
    uint32_t wc = 0, ac = 0;
    bool alive = true;
    for (uint32_t i = 0; i < passes && alive; ++i) {
#pragma unroll 1
      for (int kc = 0; kc < NKC; ++kc, ++ac) {
        const uint32_t as = ac % AS;
        if (!tc_wait_warp(&ctl->a_ready[as], (ac / AS) & 1, abort_flag)) { alive = false; break; }
        tc_fence_after();
        const uint32_t a_hi = a0 + as * (S2_A_SLOT / 16), a_lo = a_hi + S2_A_PART / 16;
#pragma unroll
        for (int half = 0; half < 2; ++half, ++wc) {
          const uint32_t s = wc % SA_SLOTS;
          if (!tc_wait_warp(&ctl->full[s], (wc / SA_SLOTS) & 1, abort_flag)) { alive = false; break; }
          tc_fence_after();
          const uint32_t b = w0 + s * (CHUNK_BYTES / 16);
#pragma unroll
          for (int j = 0; j < SA_KC / 16; ++j) {
            umma_ss(tmem, a_hi + 16u * j, hiword, b + 16u * j, hiword, idesc, (kc | half | j) != 0, leader);
            if (half == 0) umma_ss(tmem, a_lo + 16u * j, hiword, b + 16u * j, hiword, idesc, 1u, leader);
          }
          umma_commit(&ctl->empty[s], leader);
        }
        if (!alive) break;
        umma_commit(&ctl->a_free[as], leader);
      }
      umma_commit(&ctl->acc_full[0], leader);
    }
  }
  // Copy lane: W2's parts, chunk by chunk, `passes` times
  __device__ __forceinline__ void copy(const uint16_t* parts, uint32_t passes) const {
    volatile int* abort_flag = &ctl->abort_flag;
    const uint32_t total = passes * NSTREAM;
    uint32_t c = 0;
    for (uint32_t in_pass = 0; c < total; ++c, in_pass = in_pass + 1 == NSTREAM ? 0 : in_pass + 1) {
      const uint32_t s = c % SA_SLOTS;
      if (c >= SA_SLOTS && !tc_wait(&ctl->empty[s], ((c / SA_SLOTS) - 1) & 1, abort_flag)) break;
      mbar_expect_tx(&ctl->full[s], CHUNK_BYTES);
      bulk_copy_g2s(w_ring + s * CHUNK_BYTES, reinterpret_cast<const uint8_t*>(parts) + (size_t)in_pass * CHUNK_BYTES, CHUNK_BYTES, &ctl->full[s]);
      ctl->copies = c + 1;
    }
  }
};

// A worker thread's side of the forward passes.  After a timeout the abort flag is up: the thread neither waits nor hands operands over any
// more and runs to its end on meaningless numbers, through the same barriers as the others.
template <int D, int H, int TPR>
struct S2Worker {
  using M = S2Smem<D, H, TPR>;
  const M& m;
  int g, half, row;                                           // tile in flight (TPR 2: 0), which thread of its env, row of the tile = TMEM lane
  uint32_t t_row, pass = 0;
  float inv_scale, vmax = 0.f;                                // 1 / (activation scale x weight scale); largest scaled activation
  bool ok = true;
  __device__ __forceinline__ S2Worker(const M& mm, uint32_t tmem, float inv) : m(mm) {
    const int warp = threadIdx.x >> 5;
    g = TPR == 1 ? warp >> 2 : 0;
    half = TPR == 2 ? (warp >> 2) & 1 : 0;
    row = threadIdx.x & (SA_TE - 1);
    t_row = tmem + (uint32_t)g * M::ACC_COLS + ((uint32_t)((warp & 3) * 32) << 16);
    inv_scale = inv;
  }
  // Network outputs of one observation.  What a thread keeps in registers decides what the layers read from shared memory, whose read path
  // returns a word per lane and cycle, broadcast or not.
  //   Layer 1: a lane takes eight hidden units of four (TPR 2: two) rows of its warp, eight apart, whose observations come by shuffle, so a
  //   weight read serves four rows.  (A thread per environment read every weight for every environment.)
  //   Drain: an output is (b3 + sum over the lower half of the hidden units) + sum over the upper half, both in column order from zero, in
  //   every form and for every width.  The order is part of the result: with another one of the same rounding error about one categorical
  //   draw in 17 million falls the other way.  It leaves a weight read two rows at most: TPR 2 gives a lane one half of the columns of two
  //   rows and two of the outputs (actor call of four steps, 16,384 Acrobot envs, hidden 256: 45.1 us; a row and all outputs per lane, 45.7;
  //   four rows per weight read by sums of every fourth pair of columns, 43.2).  TPR 1, where every warp has a tile's rows to itself, has a
  //   row per lane and both halves side by side in one instruction: 65,536 CartPole envs, 128 steps 2.77 ms; two rows and one half per
  //   lane read half as much but issue more, 3.27; double-buffered loads of 8 columns take 6 % longer, blocks of 32 columns the same.
  // `chunk`: number of this pass's first chunk in the ring's order.
  __device__ __forceinline__ void forward(const float (&obs)[6], int Aout, uint32_t chunk, float (&out)[4]) {
    constexpr int ROWS = 4 / TPR;
    volatile int* abort_flag = &m.ctl->abort_flag;
    const int lane = threadIdx.x & 31, first = (row & ~31) + (TPR == 2 ? half * 16 : 0);   // first row of this warp's share
    tc_fence_before();                                        // this thread's accumulator reads of the previous pass are complete
    f32x2 x[ROWS][D];
#pragma unroll
    for (int r = 0; r < ROWS; ++r)
#pragma unroll
      for (int k = 0; k < D; ++k) x[r][k] = dup2(__shfl_sync(0xffffffffu, obs[k], (first & 31) + 8 * r + (lane & 7)));
    const float *w1 = m.w1 + (lane >> 3) * 8, *b1 = m.b1 + (lane >> 3) * 8;
    uint8_t* dst = m.a_ring + (first >> 3) * ((SA_KC / 8) * 128) + (lane & 7) * 16 + (lane >> 3) * 128;
#pragma unroll 1
    for (int kc = 0; kc < M::NKC; ++kc, ++chunk) {
      const uint32_t as = chunk % M::AS;
      f32x2 w[D][4], b[4];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const ulonglong2 bb = ld_pairs(b1 + kc * SA_KC + 4 * i);
        b[2 * i] = bb.x; b[2 * i + 1] = bb.y;
#pragma unroll
        for (int k = 0; k < D; ++k) {
          const ulonglong2 ww = ld_pairs(w1 + k * H + kc * SA_KC + 4 * i);
          w[k][2 * i] = ww.x; w[k][2 * i + 1] = ww.y;
        }
      }
      if (chunk >= M::AS) ok = ok && tc_wait_elect<M::PAIR>(&m.ctl->a_free[as], ((chunk / M::AS) - 1) & 1, abort_flag);
      vmax = s2_layer1<D, ROWS>(w, b, x, dst + as * S2_A_SLOT, vmax);
      fence_async_smem();
      if (M::PAIR) {
        __syncwarp();
        if (lane == 0 && ok) mbar_arrive_cluster(&m.ctl->a_ready[as], 0);
      } else if (ok) {
        mbar_arrive_warp(&m.ctl->a_ready[as]);
      }
    }
    ok = ok && tc_wait_elect<M::PAIR>(&m.ctl->acc_full[g], pass & 1, abort_flag);
    tc_fence_after();
    // h2 = relu(acc / scale + b2) and the head's sums
    if (TPR == 1) {
      const f32x2 inv2 = dup2(inv_scale);
      f32x2 s[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll 1
      for (int c0 = 0; c0 < H / 2; c0 += 16) {
        uint32_t u[16], v[16];
        tmem_ld16(t_row + (uint32_t)c0, u);
        tmem_ld16(t_row + (uint32_t)(c0 + H / 2), v);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const ulonglong2 p01 = ld_pairs(m.hw + 8 * (c0 + i)), p23 = ld_pairs(m.hw + 8 * (c0 + i) + 4);
          f32x2 h = p01.x;
          fma2(h, pair2(__uint_as_float(u[i]), __uint_as_float(v[i])), inv2);
          const float2 t = halves(h);
          h = pair2(fmaxf(t.x, 0.f), fmaxf(t.y, 0.f));
          fma2(s[0], p01.y, h);
          fma2(s[1], p23.x, h);
          fma2(s[2], p23.y, h);
          if (Aout > 3) fma2(s[3], *reinterpret_cast<const unsigned long long*>(m.hw3 + 2 * (c0 + i)), h);
        }
      }
#pragma unroll
      for (int a = 0; a < 4; ++a) { const float2 t = halves(s[a]); out[a] = (m.b3[a] + t.x) + t.y; }
    } else {
      // lanes r and r + 16: rows r and r + 16 of the warp's 32, lower and upper half of the columns; this warp: outputs 2 half and 2 half + 1
      const int upper = lane >> 4;
      const float *w = m.hw + half * 2 * H + upper * H, *b2 = m.hw3 + upper * (H / 2);
      float s[2][2] = {{0.f, 0.f}, {0.f, 0.f}};                // [row][output]
#pragma unroll 1
      for (int c0 = 0; c0 < H / 2; c0 += 16) {
        uint32_t u[2][16];
        tmem_ld16_halves<H / 2>(t_row + (uint32_t)c0, u[0]);
        tmem_ld16_halves<H / 2>(t_row + (16u << 16) + (uint32_t)c0, u[1]);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 16; i += 4) {
          const float4 b = *reinterpret_cast<const float4*>(b2 + c0 + i), wa = *reinterpret_cast<const float4*>(w + 2 * (c0 + i)),
                       wb = *reinterpret_cast<const float4*>(w + 2 * (c0 + i) + 4);
          const float bv[4] = {b.x, b.y, b.z, b.w}, w0[4] = {wa.x, wa.z, wb.x, wb.z}, w1[4] = {wa.y, wa.w, wb.y, wb.w};
#pragma unroll
          for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int r = 0; r < 2; ++r) {
              const float h = fmaxf(fmaf(__uint_as_float(u[r][i + j]), inv_scale, bv[j]), 0.f);
              s[r][0] = fmaf(w0[j], h, s[r][0]);
              s[r][1] = fmaf(w1[j], h, s[r][1]);
            }
        }
      }
      float o[2];
#pragma unroll
      for (int a = 0; a < 2; ++a) {                            // this lane's row: one half's sum is here, the other in the lane 16 away
        const float own = upper ? s[1][a] : s[0][a], other = __shfl_xor_sync(0xffffffffu, upper ? s[0][a] : s[1][a], 16);
        o[a] = (m.b3[2 * half + a] + (upper ? other : own)) + (upper ? own : other);
      }
      float2* px = reinterpret_cast<float2*>(m.part) + (size_t)(pass & 1) * 2 * SA_TE;
      px[half * SA_TE + row] = make_float2(o[0], o[1]);
      asm volatile("bar.sync 1, 256;" ::: "memory");
      const float2 o01 = px[row], o23 = px[SA_TE + row];
      out[0] = o01.x; out[1] = o01.y; out[2] = o23.x; out[3] = o23.y;
    }
    ++pass;
  }
};

template <int ENV, int H, int TPR>
__global__ void __launch_bounds__(S2_NT, 1) actor_split_tc_kernel(const ActorParams p, const S2Plan pl, const uint16_t* __restrict__ w2parts,
                                                                  const float* __restrict__ w2scale) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  constexpr int D = ENV == TJ_ENV_CARTPOLE ? 4 : 6;
  constexpr int WW = S2_NT / 32 - 2;                          // worker warps, then the issuing warp and the copy warp
  using M = S2Smem<D, H, TPR>;
  constexpr int GROUPS = M::GROUPS;
  const M m(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // a pair of blocks walks tiles of 256 envs, each block its 128 of them
  constexpr int BLOCKS = M::PAIR ? 2 : 1;
  const int n_tiles = (p.N + SA_TE * BLOCKS - 1) / (SA_TE * BLOCKS), walker = (int)blockIdx.x / BLOCKS, walkers = (int)gridDim.x / BLOCKS;
  const bool on_policy = p.C == 0;
  const uint32_t tmem = m.set_up();
  chain_begin();
  m.stage(p, p.W, p.Aout);
  const int my_tiles = walker < n_tiles ? (n_tiles - 1 - walker) / walkers + 1 : 0;
  __syncthreads();
  if (warp == WW + 1) {
    if (lane == 0) {
      if constexpr (M::PAIR) m.copy_half(w2parts);
      else m.copy(w2parts, (uint32_t)my_tiles * (uint32_t)pl.n_pass);
    }
    __syncwarp();
  } else if (warp == WW) {
    if constexpr (M::PAIR) {
      if (cluster_rank() == 0) m.issue_pair(tmem, my_tiles, pl.n_pass);
    } else {
      m.issue(tmem, (uint32_t)my_tiles * (uint32_t)pl.n_pass);
    }
  } else {
    S2Worker<D, H, TPR> wk(m, tmem, __ldg(w2scale + 1));
    const int g = wk.g, half = wk.half, row = wk.row;
    unsigned long long n_episodes = 0;
    double ret_sum = 0.0;
    const bool first = half == 0;                             // of an environment's threads the one that writes what is written once
#pragma unroll 1
    for (int tl = g; tl < my_tiles; tl += GROUPS) {
      const int e = ((walker + tl * walkers) * BLOCKS + (int)blockIdx.x % BLOCKS) * SA_TE + row;
      const bool owner = e < p.N;
      // the passes of the tiles in flight alternate: this tile's first chunk, and from one of its passes to the next
      uint32_t chunk = (uint32_t)((tl - g) * pl.n_pass + g) * M::NKC;
      const uint32_t next_pass = (uint32_t)min(GROUPS, my_tiles - (tl - g)) * M::NKC;
      float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
      int ep = 0;
      float ep_ret = 0.f;
      if (owner) {
        s = reinterpret_cast<const float4*>(p.state)[e];
        ep = p.ep_step[e];
        ep_ret = p.ep_return[e];
      }
      float obs[6];
      sa_observe<ENV>(s, obs);
      long long slot = pl.slot0;                              // ring slot of env 0 in this step
      int blk = pl.blk0, pos = pl.pos0, seg = pl.seg0;
#pragma unroll 1
      for (int step = 0; step < p.n_steps; ++step) {
        const unsigned long long t = (unsigned long long)p.t0 + step;
        float out[4];
        const uint4 w = stream_words(p.seed, STREAM_ACTION, 0, (uint32_t)e, t);
        wk.forward(obs, p.Aout, chunk, out);
        chunk += next_pass;
        auto logit = [&](int i) { return i == 0 ? out[0] : (i == 1 ? out[1] : (i == 2 ? out[2] : out[3])); };
        if (p.dbg_logits && owner && first) {
          float* dl = p.dbg_logits + ((size_t)step * p.N + e) * p.A;
          for (int i = 0; i < p.A; ++i) dl[i] = logit(i);
        }
        int a;
        float logp = 0.f;
        if (p.policy_kind == TJ_POLICY_EPS_GREEDY) a = select_eps_greedy(p.A, logit, w, p.explore_thr);
        else a = select_categorical(p.A, logit, u01(w.x), logp);
        float4 sn;
        float obs_n[6];
        StepResult r;
        if (ENV == TJ_ENV_CARTPOLE) {
          r = cartpole_step(s, a, sn);
          sa_observe<ENV>(sn, obs_n);
        } else {
          float4 trig_n;
          r = acrobot_step(s, make_float4(obs[0], obs[1], obs[2], obs[3]), a, sn, trig_n);
          obs_n[0] = trig_n.x; obs_n[1] = trig_n.y; obs_n[2] = trig_n.z; obs_n[3] = trig_n.w; obs_n[4] = sn.z; obs_n[5] = sn.w;
        }
        ep += 1;
        const int done = (r.terminated || ep >= p.max_ep) ? 1 : 0;
        if (owner) {
          if (on_policy) {
            const size_t i = ((size_t)seg * p.T + pos) * p.N + e;
            if (first) {
              if (ENV == TJ_ENV_CARTPOLE) {
                *reinterpret_cast<float4*>(p.seg_obs + i * 4) = s;
              } else {
                float2* so = reinterpret_cast<float2*>(p.seg_obs + i * 6);
                so[0] = make_float2(obs[0], obs[1]); so[1] = make_float2(obs[2], obs[3]); so[2] = make_float2(obs[4], obs[5]);
              }
            }
            if (TPR == 1 || !first) {
              p.seg_act[i] = a;
              p.seg_rew[i] = r.reward;
              p.seg_done[i] = (uint8_t)done;
              p.seg_logp[i] = logp;
              p.seg_val[((size_t)seg * (p.T + 1) + pos) * p.N + e] = logit(p.A);  // value head = output A
            }
          } else {
            long long sl = slot + e;
            if (sl >= p.C) sl -= p.C;
            float4* rec = reinterpret_cast<float4*>(p.ring + (size_t)sl * p.rec_words);
            const float4 tail = make_float4(__int_as_float(a), r.reward, __int_as_float(done), __int_as_float(p.version));
            if (ENV == TJ_ENV_CARTPOLE) {
              if (first) rec[0] = s;
              if (TPR == 1 || !first) { rec[1] = sn; rec[2] = tail; }
            } else {
              if (first) { rec[0] = make_float4(obs[0], obs[1], obs[2], obs[3]); rec[1] = make_float4(obs[4], obs[5], obs_n[0], obs_n[1]); }
              if (TPR == 1 || !first) { rec[2] = make_float4(obs_n[2], obs_n[3], obs_n[4], obs_n[5]); rec[3] = tail; }
            }
          }
        }
        ep_ret += r.reward;
        s = sn;
#pragma unroll
        for (int k = 0; k < 6; ++k) obs[k] = obs_n[k];
        if (done) {
          n_episodes += 1;
          ret_sum += (double)ep_ret;
          ep_ret = 0.f;
          ep = 0;
          s = (ENV == TJ_ENV_CARTPOLE) ? sa_reset4(p.seed, (uint32_t)e, t, -0.05f, 0.1f) : sa_reset4(p.seed, (uint32_t)e, t, -0.1f, 0.2f);
          sa_observe<ENV>(s, obs);
        }
        if (on_policy) {
          if (++pos == p.T) {                                 // bootstrap value of the state each env is now in
            wk.forward(obs, p.Aout, chunk, out);
            chunk += next_pass;
            if (owner && first) p.seg_val[((size_t)seg * (p.T + 1) + p.T) * p.N + e] = logit(p.A);
            pos = 0;
            seg = seg + 1 == p.G ? 0 : seg + 1;
          }
        } else {
          if (blockIdx.x == 0 && tid == 0 && tl == 0) p.block_ver[blk] = p.version;
          slot += p.N;
          if (slot >= p.C) slot -= p.C;
          if (++blk == pl.n_blk) blk = 0;
        }
      }
      if (owner && first) {
        reinterpret_cast<float4*>(p.state)[e] = s;
        p.ep_step[e] = ep;
        p.ep_return[e] = ep_ret;
      } else {
        n_episodes = 0;                                       // rows beyond the last env, and the other half's count
        ret_sum = 0.0;
      }
      if (n_episodes) {
        atomicAdd(&p.stats->episodes, n_episodes);
        atomicAdd(&p.stats->return_sum, ret_sum);
      }
      n_episodes = 0;
      ret_sum = 0.0;
    }
    // 65,504 is FP16's largest finite value
    if (wk.vmax > 65504.f) m.ctl->range_flag = 1;
  }
  m.tear_down(tmem);
  if (tid == 0) {
    if (m.ctl->abort_flag) atomicExch(&p.stats->error, 4ull);
    else if (m.ctl->range_flag) atomicExch(&p.stats->error, 5ull);
  }
}

// TD error (Algorithm 1, TD-error line; Huber loss on it) for a context in this weight mode: a pair of thread blocks (a cluster) per 128
// sampled rows, block 0 with the online network on obs, block 1 with the target network on next_obs at the same time; block 1 leaves
// max_a q' in block 0's shared memory.  (One block that ran the two networks one after the other took 25 us for 4,096 rows.)
// Outputs and the per-tile loss partial as in the FP32 TD kernel.
template <int D, int H>
__global__ void __launch_bounds__(S2_NT, 1) td_split_tc_kernel(const TdParams p, const uint16_t* __restrict__ parts_online,
                                                              const float* __restrict__ scale_online,
                                                              const uint16_t* __restrict__ parts_target,
                                                              const float* __restrict__ scale_target) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const S2Smem<D, H, 2> m(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int net = (int)(blockIdx.x & 1u), tile = (int)(blockIdx.x >> 1);   // the cluster is blocks 2 t and 2 t + 1
  const int j = tile * SA_TE + (tid & (SA_TE - 1));
  float* qmax = m.part + 2 * SA_TE * 2;                       // the exchange area of the pass that never comes
  const uint32_t tmem = m.set_up();
  chain_begin();
  m.stage(p, net ? p.Wtarget : p.Wonline, p.A);
  cluster_sync_all();                                         // block 0 is running before block 1 writes to it
  float out[4] = {0.f, 0.f, 0.f, 0.f};
  const bool row_thread = tid < SA_TE, live = j < p.n;
  int act = 0, done = 0;
  float rew = 0.f;
  if (warp == 9) {
    if (lane == 0) m.copy(net ? parts_target : parts_online, 1u);
    __syncwarp();
  } else if (warp == 8) {
    m.issue(tmem, 1u);
  } else {
    S2Worker<D, H, 2> wk(m, tmem, __ldg((net ? scale_target : scale_online) + 1));
    const float* x = net ? p.next_obs : p.obs;
    float obs[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (live) {
#pragma unroll
      for (int k = 0; k < D; ++k) obs[k] = __ldg(x + (size_t)j * D + k);
      if (row_thread && net == 0) {
        act = p.act[j];
        rew = p.rew[j];
        done = p.done[j];
      }
    }
    wk.forward(obs, p.A, 0u, out);
    if (wk.vmax > 65504.f) m.ctl->range_flag = 1;
    if (row_thread && net == 1) {
      float q = out[0];
      for (int i = 1; i < p.A; ++i) q = fmaxf(q, i == 1 ? out[1] : (i == 2 ? out[2] : out[3]));
      if (!wk.ok) q = __int_as_float(0x7FC00000);             // after a timeout: defined outputs (NaN), never what an earlier call left
      cluster_store_f32(qmax + tid, 0u, q);
    }
    if (!wk.ok) out[0] = out[1] = out[2] = out[3] = __int_as_float(0x7FC00000);
  }
  cluster_sync_all();
  if (row_thread && net == 0) {
    float h = 0.f;
    if (live) {
      act = act < 0 ? 0 : (act >= p.A ? p.A - 1 : act);
      const float q = act == 0 ? out[0] : (act == 1 ? out[1] : (act == 2 ? out[2] : out[3]));
      const float y = rew + p.gamma * (done ? 0.f : 1.f) * qmax[tid];
      const float delta = y - q, ad = fabsf(delta);
      h = ad <= p.kappa ? 0.5f * delta * delta : p.kappa * (ad - 0.5f * p.kappa);
      if (p.td_out) p.td_out[j] = delta;
      if (p.huber_out) p.huber_out[j] = h;
    }
    for (int o = 16; o > 0; o >>= 1) h += __shfl_xor_sync(0xffffffffu, h, o);
    if (lane == 0) m.part[warp] = h;
  }
  m.tear_down(tmem);
  if (tid == 0) {
    if (net == 0) p.partial[tile] = (m.part[0] + m.part[1]) + (m.part[2] + m.part[3]);
    if (m.ctl->abort_flag && p.error) atomicExch(p.error, 4ull);
    else if (m.ctl->range_flag && p.error) atomicExch(p.error, 5ull);
  }
}

// launch_chained for a kernel of block pairs
template <typename... P, typename... A>
cudaError_t launch_pairs(void (*kernel)(P...), int grid, int threads, size_t smem, cudaStream_t s, A&&... args) {
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2; at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

template <int ENV, int H>
cudaError_t launch_split(const ActorParams& p, const S2Plan& pl, const uint16_t* w2parts, const float* w2scale, int grid, bool pairs, cudaStream_t s) {
  constexpr int D = ENV == TJ_ENV_CARTPOLE ? 4 : 6;
  if (pairs) return launch_pairs(actor_split_tc_kernel<ENV, H, 1>, grid, S2_NT, S2Smem<D, H, 1>::bytes(), s, p, pl, w2parts, w2scale);
  return launch_chained(actor_split_tc_kernel<ENV, H, 2>, grid, S2_NT, S2Smem<D, H, 2>::bytes(), s, p, pl, w2parts, w2scale);
}

template <int ENV>
cudaError_t launch_split_env(const ActorParams& p, const S2Plan& pl, const uint16_t* w2parts, const float* w2scale, int grid, bool pairs, cudaStream_t s) {
  switch (p.H) {
    case 64: return launch_split<ENV, 64>(p, pl, w2parts, w2scale, grid, pairs, s);
    case 128: return launch_split<ENV, 128>(p, pl, w2parts, w2scale, grid, pairs, s);
    case 192: return launch_split<ENV, 192>(p, pl, w2parts, w2scale, grid, pairs, s);
    case 256: return launch_split<ENV, 256>(p, pl, w2parts, w2scale, grid, pairs, s);
    default: return cudaErrorInvalidConfiguration;
  }
}

}  // namespace

bool split_actor_supported(int env_kind, int D, int H, int Aout) {
  const bool env_ok = (env_kind == TJ_ENV_CARTPOLE && D == 4) || (env_kind == TJ_ENV_ACROBOT && D == 6);
  return env_ok && H >= 64 && H <= 256 && H % 64 == 0 && Aout <= 4;   // Aout <= 4: rows of the head matrix are one float4
}

size_t split_weight_halfs(int H) { return (size_t)2 * H * H; }

float split_hidden_scale() { return SA_H_SCALE; }

cudaError_t launch_actor_split(int env_kind, const ActorParams& p, const uint16_t* w2parts, const float* w2scale, int sm_count,
                               cudaStream_t s) {
  if (p.N <= 0) return cudaSuccess;
  if (!split_actor_supported(env_kind, p.D, p.H, p.Aout)) return cudaErrorInvalidConfiguration;
  const int n_tiles = (p.N + SA_TE - 1) / SA_TE;
  const bool pairs = n_tiles > sm_count && sm_count > 1;     // more tiles than SMs: pairs of blocks with two tiles each in flight
  const int grid = pairs ? sm_count & ~1 : (n_tiles < sm_count ? n_tiles : sm_count);
  S2Plan pl{};
  pl.n_pass = p.n_steps;
  if (p.C > 0) {
    pl.slot0 = (long long)(p.cursor0 % (unsigned long long)p.C);
    pl.blk0 = (int)(pl.slot0 / p.N);
    pl.n_blk = (int)(p.C / p.N);
  } else {
    pl.pos0 = (int)(p.t0 % p.T);
    pl.seg0 = (int)((p.t0 / p.T) % p.G);
    pl.n_pass += (pl.pos0 + p.n_steps) / p.T;
  }
  return env_kind == TJ_ENV_CARTPOLE ? launch_split_env<TJ_ENV_CARTPOLE>(p, pl, w2parts, w2scale, grid, pairs, s)
                                     : launch_split_env<TJ_ENV_ACROBOT>(p, pl, w2parts, w2scale, grid, pairs, s);
}

int td_split_grid(int n) { return (n + SA_TE - 1) / SA_TE; }

template <int D, int H>
static cudaError_t launch_td_split_dh(const TdParams& p, const uint16_t* po, const float* so, const uint16_t* pt, const float* st, cudaStream_t s) {
  return launch_pairs(td_split_tc_kernel<D, H>, 2 * td_split_grid(p.n), S2_NT, S2Smem<D, H, 2>::bytes(), s, p, po, so, pt, st);
}

template <int D>
static cudaError_t launch_td_split_d(const TdParams& p, const uint16_t* po, const float* so, const uint16_t* pt, const float* st, cudaStream_t s) {
  switch (p.H) {
    case 64: return launch_td_split_dh<D, 64>(p, po, so, pt, st, s);
    case 128: return launch_td_split_dh<D, 128>(p, po, so, pt, st, s);
    case 192: return launch_td_split_dh<D, 192>(p, po, so, pt, st, s);
    case 256: return launch_td_split_dh<D, 256>(p, po, so, pt, st, s);
    default: return cudaErrorInvalidConfiguration;
  }
}

cudaError_t launch_td_split(const TdParams& p, const uint16_t* parts_online, const float* scale_online, const uint16_t* parts_target,
                            const float* scale_target, cudaStream_t s) {
  if (p.n <= 0) return cudaSuccess;
  if (!(p.D == 4 || p.D == 6) || p.A > 4 || p.Ap != 4) return cudaErrorInvalidConfiguration;
  return p.D == 4 ? launch_td_split_d<4>(p, parts_online, scale_online, parts_target, scale_target, s)
                  : launch_td_split_d<6>(p, parts_online, scale_online, parts_target, scale_target, s);
}

}  // namespace tj
