// FP32-accuracy tensor-core actor for the small environments (CartPole, Acrobot) with hidden widths of 64 .. 256: the
// hidden x hidden layer -- the one dense contraction of these networks (Algorithm 1, task 1: 65,536 of a 6-256-256-3
// network's 67,840 multiply-adds per env step) -- runs on the tensor cores as three FP16 products of split operands,
//   W2 h1 = W_hi h_hi + W_hi h_lo + W_lo h_hi,   x = x_hi + x_lo with x_hi the 11 leading bits of the (power-of-two scaled) value,
// with FP32 accumulation in tensor memory (error about 2^-22 per term, the dropped lo x lo term; FP16 runs at twice the rate
// of the 3 x TF32 form of the same idea).  Layer 1 (4 or 6 inputs) and the head (2-4 outputs) stay on the FP32 pipes.
//
// One thread block keeps a tile of 128 environments for all n_steps of the call (environments are independent): thread e
// owns env e's state in registers.  Eight worker warps, one MMA-issuing warp, one copy warp; per step:
//   observation -> shared memory;
//   workers: layer 1 in the fixed FMA order of the FP32 path, ReLU, split -> FP16 A operand, 32 hidden units (one K chunk of
//     the next layer) at a time, each chunk handed to the issuing lane through its own mbarrier;
//   copy lane: streams W2's parts in 32-column chunks (bulk copies, four ring slots, the stream running on across steps);
//   issuing lane: per K chunk, issues W_hi x (h_hi, h_lo) and W_lo x h_hi (M = 128, N = H) as soon as that chunk of h1 exists, so
//     the tensor pipe works underneath layer 1;
//   workers: accumulator -> + b2, ReLU, head partial sums by two threads per row -> outputs;
//   then exactly the FP32 kernel's selection, env step, record / segment write and reset.
// Every wait is bounded; a timeout latches the context's error word and the block leaves after freeing its tensor memory.
#include <cuda_fp16.h>

#include "tj_fma.cuh"
#include "tj_internal.h"
#include "tj_mlp.cuh"
#include "tj_tc.cuh"

namespace tj {

namespace {

constexpr int SA_TE = 128;            // envs per tile = rows of the MMA
constexpr int SA_WORKERS = 256;       // threads of the worker warps; one more warp issues
constexpr int SA_NT = SA_WORKERS + 64;   // + the MMA-issuing warp and the copy warp
constexpr int SA_KC = 32;             // K columns per streamed chunk of W2
constexpr int SA_SLOTS = 4;
constexpr int SA_MAX_KC = 256 / SA_KC;
constexpr float SA_H_SCALE = 16.0f;   // hidden activations are split after this scaling (|h1| < 4,094 stays inside FP16)

struct SaCtl {
  uint64_t full[SA_SLOTS], empty[SA_SLOTS];
  uint64_t a_ready[SA_MAX_KC];   // K chunk of the A operand written (one arrival per worker warp)
  uint64_t wbar;                 // small parameters staged
  uint64_t acc_full;             // all MMAs of a forward pass complete
  uint32_t tmem_base;
  int abort_flag;
  int range_flag;               // a scaled hidden activation left FP16's range: the outputs of that pass are meaningless
};

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
    float s1, c1, s2, c2;
    sincosf(s.x, &s1, &c1);
    sincosf(s.y, &s2, &c2);
    obs[0] = c1; obs[1] = s1; obs[2] = c2; obs[3] = s2; obs[4] = s.z; obs[5] = s.w;
  }
}

struct SaShared {
  uint8_t *a_hi, *a_lo, *ring;
  float *xs, *out, *part;
  SaCtl* ctl;
};

// eight hidden units n0 .. n0+7 of layer 1 for one env, in the canonical order (bias, then inputs in index order), ReLU,
// scaling, split; one 16-byte row segment of each part of the A operand
template <int D>
__device__ __forceinline__ float sa_layer1_block(const MlpWeights& mw, int Hp, const float* x, int n0, uint8_t* a_hi, uint8_t* a_lo, size_t off) {
  float acc[8];
  const float4 b0 = *reinterpret_cast<const float4*>(mw.b1 + n0), b1 = *reinterpret_cast<const float4*>(mw.b1 + n0 + 4);
  acc[0] = b0.x; acc[1] = b0.y; acc[2] = b0.z; acc[3] = b0.w; acc[4] = b1.x; acc[5] = b1.y; acc[6] = b1.z; acc[7] = b1.w;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    const float4 w0 = *reinterpret_cast<const float4*>(mw.W1t + (size_t)k * Hp + n0);
    const float4 w1 = *reinterpret_cast<const float4*>(mw.W1t + (size_t)k * Hp + n0 + 4);
    acc[0] = fmaf(w0.x, x[k], acc[0]); acc[1] = fmaf(w0.y, x[k], acc[1]); acc[2] = fmaf(w0.z, x[k], acc[2]); acc[3] = fmaf(w0.w, x[k], acc[3]);
    acc[4] = fmaf(w1.x, x[k], acc[4]); acc[5] = fmaf(w1.y, x[k], acc[5]); acc[6] = fmaf(w1.z, x[k], acc[6]); acc[7] = fmaf(w1.w, x[k], acc[7]);
  }
  uint32_t hi2[4], lo2[4];
  float vmax = 0.f;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float v0 = fmaxf(acc[2 * i], 0.f) * SA_H_SCALE, v1 = fmaxf(acc[2 * i + 1], 0.f) * SA_H_SCALE;
    vmax = fmaxf(vmax, fmaxf(v0, v1));
    const float h0 = __uint_as_float(__float_as_uint(v0) & 0xFFFFE000u), h1 = __uint_as_float(__float_as_uint(v1) & 0xFFFFE000u);
    hi2[i] = pack_f16x2(h0, h1);
    lo2[i] = pack_f16x2(v0 - h0, v1 - h1);
  }
  *reinterpret_cast<uint4*>(a_hi + off) = make_uint4(hi2[0], hi2[1], hi2[2], hi2[3]);
  *reinterpret_cast<uint4*>(a_lo + off) = make_uint4(lo2[0], lo2[1], lo2[2], lo2[3]);
  return vmax;
}

// Network outputs of the observations in xs -> out[i][e], i < Aout.  Called by every thread of the block; `pass` counts the
// calls, `copied` is the copy lane's position in the chunk stream: pass q reads the split matrix parts[q & 1] (the actor
// passes the same matrix twice, the TD kernel the online and the target network's).  Returns false after a timeout.
template <int D, int H>
__device__ __forceinline__ bool sa_forward(int Hp, int Aout, const MlpWeights& mw, const SaShared& sh, const uint16_t* parts0,
                                           const uint16_t* parts1, float inv_scale, uint32_t tmem, uint32_t pass, uint32_t& copied,
                                           volatile int* abort_flag) {
  constexpr int NKC = H / SA_KC;                 // K chunks of the hidden x hidden layer
  constexpr uint32_t NSTREAM = 2 * NKC;          // chunks of W2 per pass: (high, low) per K chunk
  constexpr uint32_t CHUNK_BYTES = H * SA_KC * 2;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  SaCtl* ctl = sh.ctl;
  if (tid < SA_WORKERS) {
    const int e = tid & (SA_TE - 1), half = tid >> 7;
    float x[D];
#pragma unroll
    for (int k = 0; k < D; ++k) x[k] = sh.xs[k * SA_TE + e];
    tc_fence_before();                            // this thread's accumulator reads of the previous pass are complete
    float vmax = 0.f;
#pragma unroll 1
    for (int kc = 0; kc < NKC; ++kc) {
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const int n0 = kc * SA_KC + half * 16 + b * 8;
        const size_t off = ((size_t)(e >> 3) * (H / 8) + (n0 >> 3)) * 128 + (e & 7) * 16;
        vmax = fmaxf(vmax, sa_layer1_block<D>(mw, Hp, x, n0, sh.a_hi, sh.a_lo, off));
      }
      fence_async_smem();
      mbar_arrive_warp(&ctl->a_ready[kc]);
    }
    // 65,504 is FP16's largest finite value (a NaN activation also lands here: the comparison is written to catch it)
    if (!(vmax <= 65504.f)) ctl->range_flag = 1;
  } else if (warp == SA_WORKERS / 32) {
    // The issuing lane's warp-mates wait at the warp barrier, not in a polling loop: lanes of one warp that poll while
    // another lane of it issues take turns with that lane, and every blocked poll then stalls the issue.
    if (lane == 0) {
      // The stream position at the start of a pass is pass x NSTREAM, a multiple of the slot count: chunk c of any pass sits
      // in slot c % SLOTS, and only the barrier parities depend on the pass.
      const uint32_t idesc = make_idesc_f16(H);
      const uint32_t ahi_lo = desc_lo(smem_addr(sh.a_hi), 128u), alo_lo = desc_lo(smem_addr(sh.a_lo), 128u);
      const uint32_t a_hiword = desc_hi((uint32_t)(H / 8) * 128u), b_hiword = desc_hi((uint32_t)(SA_KC / 8) * 128u);
      const uint32_t ring_lo = desc_lo(smem_addr(sh.ring), 128u);
      const uint32_t round0 = pass * (NSTREAM / SA_SLOTS);           // trips around the ring before this pass
      bool alive = true;
#pragma unroll
      for (int kc = 0; kc < NKC; ++kc) {
        if (!alive) break;
        if (!tc_wait(&ctl->a_ready[kc], pass & 1, abort_flag)) { alive = false; break; }
        tc_fence_after();
        const uint32_t a_off = (uint32_t)kc * (SA_KC / 8) * 8u;     // in 16-byte units: 8 per core matrix, 4 core matrices per chunk
#pragma unroll
        for (int part = 0; part < 2; ++part) {
          const int c = 2 * kc + part, s = c % SA_SLOTS;
          if (!tc_wait(&ctl->full[s], (round0 + c / SA_SLOTS) & 1, abort_flag)) { alive = false; break; }
          tc_fence_after();
          const uint32_t b_lo = ring_lo + (uint32_t)s * (CHUNK_BYTES / 16);
#pragma unroll
          for (int j = 0; j < SA_KC / 16; ++j) {
            umma_ss(tmem, ahi_lo + a_off + 16u * j, a_hiword, b_lo + 16u * j, b_hiword, idesc, (c | j) != 0);
            if (part == 0) umma_ss(tmem, alo_lo + a_off + 16u * j, a_hiword, b_lo + 16u * j, b_hiword, idesc, 1u);
          }
          umma_commit(&ctl->empty[s]);
        }
      }
      umma_commit(&ctl->acc_full);
    }
    __syncwarp();
  } else {
    // copy lane: keeps the ring full -- chunk g of the stream follows chunk g - SLOTS into its slot once that one is consumed
    if (lane == 0) {
#pragma unroll 1
      for (uint32_t c = 0; c < NSTREAM; ++c, ++copied) {
        const uint32_t sp = copied % SA_SLOTS;
        if (!tc_wait(&ctl->empty[sp], ((copied / SA_SLOTS) - 1) & 1, abort_flag)) break;
        mbar_expect_tx(&ctl->full[sp], CHUNK_BYTES);
        const uint16_t* src = ((copied / NSTREAM) & 1u) ? parts1 : parts0;
        bulk_copy_g2s(sh.ring + (size_t)sp * CHUNK_BYTES, reinterpret_cast<const uint8_t*>(src) + (size_t)(copied % NSTREAM) * CHUNK_BYTES,
                      CHUNK_BYTES, &ctl->full[sp]);
      }
    }
    __syncwarp();
  }
  // after a timeout the abort flag is up: the pass runs to its end on meaningless numbers (every thread keeps to the same
  // barriers) and the caller leaves
  tc_wait_elect(&ctl->acc_full, pass & 1, abort_flag);
  tc_fence_after();
  // drain: two threads per row (the two column halves); h2 = relu(acc / scale + b2), head partial sums in column order
  if (tid < SA_WORKERS) {
    const int q = warp & 3, half = warp >> 2, r = q * 32 + lane;
    float pa[4] = {0.f, 0.f, 0.f, 0.f};
    const uint32_t t_row = tmem + ((uint32_t)(q * 32) << 16);
#pragma unroll 2
    for (int c0 = half * (H / 2); c0 < (half + 1) * (H / 2); c0 += 16) {
      uint32_t v[16];
      tmem_ld16(t_row + (uint32_t)c0, v);
      tmem_ld_wait();
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const float h2 = fmaxf(fmaf(__uint_as_float(v[i]), inv_scale, mw.b2[c0 + i]), 0.f);
        const float4 w = *reinterpret_cast<const float4*>(mw.W3t + (size_t)(c0 + i) * 4);   // a row of W3t (Ap = 4)
        pa[0] = fmaf(w.x, h2, pa[0]); pa[1] = fmaf(w.y, h2, pa[1]); pa[2] = fmaf(w.z, h2, pa[2]); pa[3] = fmaf(w.w, h2, pa[3]);
      }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
      if (a < Aout) sh.part[((size_t)half * 4 + a) * SA_TE + r] = pa[a];
  }
  __syncthreads();
  if (tid < SA_TE)
    for (int a = 0; a < Aout; ++a)
      sh.out[a * SA_TE + tid] = (mw.b3[a] + sh.part[(size_t)a * SA_TE + tid]) + sh.part[((size_t)4 + a) * SA_TE + tid];
  __syncthreads();
  return *abort_flag == 0;
}

// ------------------------------------------------------------------------------------------------------------------------
// The actor.  A thread owns an environment for the whole call: observation, layer 1, head sums, selection and environment step stay
// in its registers, so the workers meet nobody but the issuing lane.  TPR threads per environment:
//   1  two groups of four warps, each on a tile of its own: while one tile's MMAs run, the other tile's threads drain, step and
//      compute layer 1 (calls with more tiles than SMs);
//   2  eight warps on one tile: each thread takes half the neurons and half the columns of the drain, the two exchange their head
//      sums once per step and both step the environment (one tile per SM: the chain of one step is the bound).
// Layer 1 hands 32 hidden units (one K chunk) at a time to the issuing lane through a ring of A-operand slots.
constexpr int S2_NT = 320;                // eight worker warps, the issuing warp, the copy warp
constexpr int S2_A_SLOTS = 8;             // A-operand slots of a block, 16 KB each: four per group, or eight for the one tile
constexpr int S2_A_PART = SA_TE * SA_KC * 2;
constexpr int S2_A_SLOT = 2 * S2_A_PART;  // high part, low part

struct S2Ctl {
  uint64_t full[SA_SLOTS], empty[SA_SLOTS];
  uint64_t a_ready[S2_A_SLOTS], a_free[S2_A_SLOTS];
  uint64_t acc_full[2];
  uint32_t tmem_base;
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

// eight hidden units n0 .. n0 + 7 of layer 1 in the canonical order (bias, then inputs in index order; weights and biases come scaled by
// SA_H_SCALE, a power of two, which leaves every rounding where it was), ReLU, split; returns the largest scaled activation
template <int D, int H>
__device__ __forceinline__ float s2_layer1_block(const float* w1, const float* b1, const f32x2 (&x)[D], int n0, uint8_t* hi_dst, uint8_t* lo_dst, float vmax) {
  f32x2 acc[4];
  {
    const ulonglong2 b0 = ld_pairs(b1 + n0), b4 = ld_pairs(b1 + n0 + 4);
    acc[0] = b0.x; acc[1] = b0.y; acc[2] = b4.x; acc[3] = b4.y;
  }
#pragma unroll
  for (int k = 0; k < D; ++k) {
    const ulonglong2 w0 = ld_pairs(w1 + k * H + n0), w4 = ld_pairs(w1 + k * H + n0 + 4);
    fma2(acc[0], w0.x, x[k]); fma2(acc[1], w0.y, x[k]); fma2(acc[2], w4.x, x[k]); fma2(acc[3], w4.y, x[k]);
  }
  uint32_t hi[4], lo[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 a = halves(acc[i]);
    const float v0 = fmaxf(a.x, 0.f), v1 = fmaxf(a.y, 0.f);
    vmax = fmaxf(vmax, fmaxf(a.x, a.y));
    const float h0 = __uint_as_float(__float_as_uint(v0) & 0xFFFFE000u), h1 = __uint_as_float(__float_as_uint(v1) & 0xFFFFE000u);
    hi[i] = pack_f16x2(h0, h1);
    lo[i] = pack_f16x2(v0 - h0, v1 - h1);
  }
  *reinterpret_cast<uint4*>(hi_dst) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
  *reinterpret_cast<uint4*>(lo_dst) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
  return vmax;
}

template <int ENV, int H, int TPR>
__global__ void __launch_bounds__(S2_NT, 1) actor_split_tc_kernel(const ActorParams p, const S2Plan pl, const uint16_t* __restrict__ w2parts,
                                                                 const float* __restrict__ w2scale) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  constexpr int D = ENV == TJ_ENV_CARTPOLE ? 4 : 6;
  constexpr uint32_t CHUNK_BYTES = H * SA_KC * 2;             // one chunk of one part of W2
  constexpr int NKC = H / SA_KC, NSTREAM = 2 * NKC;
  constexpr int GROUPS = 3 - TPR, AS = S2_A_SLOTS / GROUPS;   // tiles in flight; A slots of each
  constexpr uint32_t ACC_COLS = H <= 128 ? 128 : 256;
  uint8_t* a_ring = smem_raw;
  uint8_t* w_ring = a_ring + S2_A_SLOTS * S2_A_SLOT;
  float* w1 = reinterpret_cast<float*>(w_ring + SA_SLOTS * CHUNK_BYTES);   // [D][H], scaled
  float* b1 = w1 + D * H;                                     // [H], scaled
  float* b2 = b1 + H;                                         // [H]
  float* w3 = b2 + H;                                         // TPR 1: [4][H / 2] pairs (column c, column c + H / 2); 2: [H][4]
  float* b3 = w3 + 4 * H;                                     // [4]
  float* part = b3 + 4;                                       // TPR 2: head sums [step parity][half][TE][4]
  S2Ctl* ctl = reinterpret_cast<S2Ctl*>(part + (TPR == 2 ? 2 * 2 * SA_TE * 4 : 0));
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n_tiles = (p.N + SA_TE - 1) / SA_TE;
  const bool on_policy = p.C == 0;
  if (tid == 0) {
    for (int s = 0; s < SA_SLOTS; ++s) { mbar_init(&ctl->full[s], 1); mbar_init(&ctl->empty[s], 1); }
    for (int s = 0; s < S2_A_SLOTS; ++s) { mbar_init(&ctl->a_ready[s], 4 * TPR); mbar_init(&ctl->a_free[s], 1); }
    mbar_init(&ctl->acc_full[0], 1);
    mbar_init(&ctl->acc_full[1], 1);
    ctl->abort_flag = ctl->range_flag = 0;
  }
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&ctl->tmem_base)), "r"(GROUPS * ACC_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = ctl->tmem_base;
  volatile int* abort_flag = &ctl->abort_flag;
  chain_begin();
  for (int i = tid; i < D * H; i += S2_NT) w1[i] = SA_H_SCALE * __ldg(p.W + p.off_W1t + i);
  for (int i = tid; i < H; i += S2_NT) {
    b1[i] = SA_H_SCALE * __ldg(p.W + p.off_b1 + i);
    b2[i] = __ldg(p.W + p.off_b2 + i);
    const float4 w = __ldg(reinterpret_cast<const float4*>(p.W + p.off_W3t) + i);
    if (TPR == 2) {
      reinterpret_cast<float4*>(w3)[i] = w;
    } else {
      float* d = w3 + 2 * (i % (H / 2)) + i / (H / 2);
      d[0] = w.x; d[H] = w.y; d[2 * H] = w.z; d[3 * H] = w.w;
    }
  }
  if (tid < 4) b3[tid] = tid < p.Aout ? __ldg(p.W + p.off_b3 + tid) : 0.f;
  __syncthreads();
  const int my_tiles = ((int)blockIdx.x < n_tiles) ? (n_tiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;

  if (warp == 8) {
    // The issuing lane's warp-mates wait at the block's last barrier: lanes of one warp that poll while another lane of it issues
    // take turns with that lane, and every blocked poll then stalls the issue.
    if (lane == 0) {
      const uint32_t idesc = make_idesc_f16(H);
      const uint32_t a0 = desc_lo(smem_addr(a_ring), 128u), w0 = desc_lo(smem_addr(w_ring), 128u);
      const uint32_t hiword = desc_hi((uint32_t)(SA_KC / 8) * 128u);          // A slots and W2 chunks: 32 columns wide
      uint32_t wc = 0, ac[2] = {0, 0};
      bool alive = true;
      for (int r = 0; r * GROUPS < my_tiles && alive; ++r)
        for (int i = 0; i < pl.n_pass && alive; ++i)
#pragma unroll
          for (int g = 0; g < GROUPS; ++g) {
            if (!alive || r * GROUPS + g >= my_tiles) break;
            const uint32_t acc = tmem + (uint32_t)g * ACC_COLS;
#pragma unroll 1
            for (int kc = 0; kc < NKC; ++kc, ++ac[g]) {
              const uint32_t as = (uint32_t)g * AS + ac[g] % AS;
              if (!tc_wait(&ctl->a_ready[as], (ac[g] / AS) & 1, abort_flag)) { alive = false; break; }
              tc_fence_after();
              const uint32_t a_hi = a0 + as * (S2_A_SLOT / 16), a_lo = a_hi + S2_A_PART / 16;
#pragma unroll
              for (int half = 0; half < 2; ++half, ++wc) {
                const uint32_t s = wc % SA_SLOTS;
                if (!tc_wait(&ctl->full[s], (wc / SA_SLOTS) & 1, abort_flag)) { alive = false; break; }
                tc_fence_after();
                const uint32_t b = w0 + s * (CHUNK_BYTES / 16);
#pragma unroll
                for (int j = 0; j < SA_KC / 16; ++j) {
                  umma_ss(acc, a_hi + 16u * j, hiword, b + 16u * j, hiword, idesc, (kc | half | j) != 0);
                  if (half == 0) umma_ss(acc, a_lo + 16u * j, hiword, b + 16u * j, hiword, idesc, 1u);
                }
                umma_commit(&ctl->empty[s]);
              }
              if (!alive) break;
              umma_commit(&ctl->a_free[as]);
            }
            umma_commit(&ctl->acc_full[g]);
          }
    }
    __syncwarp();
  } else if (warp == 9) {
    // copy lane: W2's parts, chunk by chunk and pass after pass (the same for every tile)
    if (lane == 0) {
      const uint32_t total = (uint32_t)my_tiles * (uint32_t)pl.n_pass * NSTREAM;
      uint32_t c = 0;
      for (uint32_t in_pass = 0; c < total; ++c, in_pass = in_pass + 1 == NSTREAM ? 0 : in_pass + 1) {
        const uint32_t s = c % SA_SLOTS;
        if (c >= SA_SLOTS && !tc_wait(&ctl->empty[s], ((c / SA_SLOTS) - 1) & 1, abort_flag)) break;
        mbar_expect_tx(&ctl->full[s], CHUNK_BYTES);
        bulk_copy_g2s(w_ring + s * CHUNK_BYTES, reinterpret_cast<const uint8_t*>(w2parts) + (size_t)in_pass * CHUNK_BYTES, CHUNK_BYTES, &ctl->full[s]);
      }
      // after a timeout the last copies may still be on their way: they must land before the block gives its shared memory back
      if (*abort_flag)
        for (uint32_t i = c > SA_SLOTS ? c - SA_SLOTS : 0; i < c; ++i)
          if (!mbar_wait_bounded(&ctl->full[i % SA_SLOTS], (i / SA_SLOTS) & 1)) break;
    }
    __syncwarp();
  } else {
    const int g = TPR == 1 ? warp >> 2 : 0, half = TPR == 2 ? warp >> 2 : 0;
    const int row = tid & (SA_TE - 1);                        // row of the tile = TMEM lane
    const uint32_t t_row = tmem + (uint32_t)g * ACC_COLS + ((uint32_t)((warp & 3) * 32) << 16);
    const float inv_scale = __ldg(w2scale + 1);               // 1 / (activation scale x weight scale)
    uint32_t ac = 0, pass = 0;
    bool ok = true;
    float vmax = 0.f;

    // network outputs of one observation
    auto forward = [&](const float (&obs)[6], float (&out)[4]) {
      tc_fence_before();                                      // this thread's accumulator reads of the previous pass are complete
      f32x2 x[D];
#pragma unroll
      for (int k = 0; k < D; ++k) x[k] = dup2(obs[k]);
#pragma unroll 1
      for (int kc = 0; kc < NKC; ++kc, ++ac) {
        const uint32_t as = (uint32_t)g * AS + ac % AS;
        if (ac >= AS) ok = ok && tc_wait_elect(&ctl->a_free[as], ((ac / AS) - 1) & 1, abort_flag);
        uint8_t* dst = a_ring + as * S2_A_SLOT + (row >> 3) * ((SA_KC / 8) * 128) + (row & 7) * 16;
#pragma unroll
        for (int b = 0; b < 4 / TPR; ++b) {
          const int kg = half * 2 + b;
          vmax = s2_layer1_block<D, H>(w1, b1, x, kc * SA_KC + kg * 8, dst + kg * 128, dst + S2_A_PART + kg * 128, vmax);
        }
        fence_async_smem();
        mbar_arrive_warp(&ctl->a_ready[as]);
      }
      ok = ok && tc_wait_elect(&ctl->acc_full[g], pass & 1, abort_flag);
      tc_fence_after();
      if (TPR == 1) {
        // h2 = relu(acc / scale + b2); the sums over the two halves of the columns side by side, each in column order
        f32x2 s[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll 1
        for (int c0 = 0; c0 < H / 2; c0 += 16) {
          uint32_t u[16], v[16];
          tmem_ld16(t_row + (uint32_t)c0, u);
          tmem_ld16(t_row + (uint32_t)(c0 + H / 2), v);
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 16; i += 4) {
            const float4 ba = *reinterpret_cast<const float4*>(b2 + c0 + i), bb = *reinterpret_cast<const float4*>(b2 + c0 + i + H / 2);
            const float b_lo[4] = {ba.x, ba.y, ba.z, ba.w}, b_hi[4] = {bb.x, bb.y, bb.z, bb.w};
            f32x2 h[4];
#pragma unroll
            for (int j = 0; j < 4; ++j)
              h[j] = pair2(fmaxf(fmaf(__uint_as_float(u[i + j]), inv_scale, b_lo[j]), 0.f), fmaxf(fmaf(__uint_as_float(v[i + j]), inv_scale, b_hi[j]), 0.f));
#pragma unroll
            for (int a = 0; a < 4; ++a) {
              if (a >= 3 && p.Aout <= 3) break;
              const ulonglong2 wa = ld_pairs(w3 + a * H + 2 * (c0 + i)), wb = ld_pairs(w3 + a * H + 2 * (c0 + i) + 4);
              fma2(s[a], wa.x, h[0]); fma2(s[a], wa.y, h[1]); fma2(s[a], wb.x, h[2]); fma2(s[a], wb.y, h[3]);
            }
          }
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) { const float2 t = halves(s[a]); out[a] = (b3[a] + t.x) + t.y; }
      } else {
        f32x2 s01 = 0ull, s23 = 0ull;
        const int c_begin = half * (H / 2);
#pragma unroll 1
        for (int c0 = c_begin; c0 < c_begin + H / 2; c0 += 32) {
          uint32_t u[32];
          tmem_ld16(t_row + (uint32_t)c0, u);
          tmem_ld16(t_row + (uint32_t)c0 + 16u, u + 16);
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 32; i += 4) {
            const float4 ba = *reinterpret_cast<const float4*>(b2 + c0 + i);
            const float bv[4] = {ba.x, ba.y, ba.z, ba.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const f32x2 h = dup2(fmaxf(fmaf(__uint_as_float(u[i + j]), inv_scale, bv[j]), 0.f));
              const ulonglong2 w = ld_pairs(w3 + 4 * (c0 + i + j));
              fma2(s01, w.x, h);
              fma2(s23, w.y, h);
            }
          }
        }
        const float2 a = halves(s01), b = halves(s23);
        float4* px = reinterpret_cast<float4*>(part) + (size_t)(pass & 1) * 2 * SA_TE;
        px[half * SA_TE + row] = make_float4(a.x, a.y, b.x, b.y);
        asm volatile("bar.sync 1, 256;" ::: "memory");
        const float4 l = px[row], h = px[SA_TE + row];
        out[0] = (b3[0] + l.x) + h.x; out[1] = (b3[1] + l.y) + h.y; out[2] = (b3[2] + l.z) + h.z; out[3] = (b3[3] + l.w) + h.w;
      }
      ++pass;
    };

    unsigned long long n_episodes = 0;
    double ret_sum = 0.0;
    const bool first = half == 0;                             // of an environment's threads the one that writes what is written once
#pragma unroll 1
    for (int tl = g; tl < my_tiles; tl += GROUPS) {
      const int e = ((int)blockIdx.x + tl * (int)gridDim.x) * SA_TE + row;
      const bool owner = e < p.N;
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
        forward(obs, out);
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
        const StepResult r = (ENV == TJ_ENV_CARTPOLE) ? cartpole_step(s, a, sn) : acrobot_step(s, a, sn);
        ep += 1;
        const int done = (r.terminated || ep >= p.max_ep) ? 1 : 0;
        float obs_n[6];
        sa_observe<ENV>(sn, obs_n);
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
            forward(obs, out);
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
    // 65,504 is FP16's largest finite value (the comparison is written to catch a NaN too)
    if (!(vmax <= 65504.f)) ctl->range_flag = 1;
  }
  tc_fence_before();
  __syncthreads();
  if (tid == 0) {
    if (ctl->abort_flag) atomicExch(&p.stats->error, 4ull);
    else if (ctl->range_flag) atomicExch(&p.stats->error, 5ull);
  }
  if (warp == 0) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(GROUPS * ACC_COLS) : "memory");
  }
}

// TD error (Algorithm 1, TD-error line; Huber loss on it) for a context in this weight mode: a tile of 128 sampled rows per
// block, the online network on obs (pass 0), the target network on next_obs (pass 1), both with the split-operand hidden
// layer above; the small parameters are staged twice, the chunk stream alternates between the two split matrices.
// Outputs and the per-block loss partial as in the FP32 TD kernel (one partial per 128 rows, summed in row order).
template <int D, int H>
__global__ void __launch_bounds__(SA_NT, 1) td_split_tc_kernel(const TdParams p, const uint16_t* __restrict__ parts_online,
                                                              const float* __restrict__ scale_online,
                                                              const uint16_t* __restrict__ parts_target,
                                                              const float* __restrict__ scale_target) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  constexpr int A_BYTES = SA_TE * H * 2;
  constexpr uint32_t CHUNK_BYTES = H * SA_KC * 2;
  constexpr uint32_t NSTREAM = 2 * (H / SA_KC);
  SaShared sh;
  sh.a_hi = smem_raw;
  sh.a_lo = sh.a_hi + A_BYTES;
  sh.ring = sh.a_lo + A_BYTES;
  float* wsm = reinterpret_cast<float*>(sh.ring + SA_SLOTS * CHUNK_BYTES);
  const size_t staged = p.w_total - (p.off_b2 - p.off_W2t);
  sh.xs = wsm + staged;
  sh.out = sh.xs + (size_t)8 * SA_TE;
  sh.part = sh.out + (size_t)4 * SA_TE;
  sh.ctl = reinterpret_cast<SaCtl*>(sh.part + 2 * (size_t)4 * SA_TE);
  SaCtl* ctl = sh.ctl;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int j0 = blockIdx.x * SA_TE, n_here = min(SA_TE, p.n - j0);
  if (tid == 0) {
    for (int s = 0; s < SA_SLOTS; ++s) { mbar_init(&ctl->full[s], 1); mbar_init(&ctl->empty[s], 1); }
    for (int k = 0; k < SA_MAX_KC; ++k) mbar_init(&ctl->a_ready[k], SA_WORKERS / 32);
    mbar_init(&ctl->wbar, 1);
    mbar_init(&ctl->acc_full, 1);
    ctl->abort_flag = 0;
    ctl->range_flag = 0;
  }
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&ctl->tmem_base)), "r"(256u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = ctl->tmem_base;
  chain_begin();
  MlpWeights mw = stage_mlp_weights<1>(p, p.Wonline, wsm, &ctl->wbar, tid == 0);
  for (int i = tid; i < SA_TE * D; i += SA_NT) {
    const int el = i / D, k = i % D;
    sh.xs[k * SA_TE + el] = el < n_here ? p.obs[(size_t)(j0 + el) * D + k] : 0.f;
  }
  volatile int* abort_flag = &ctl->abort_flag;
  bool ok = tc_wait_elect(&ctl->wbar, 0, abort_flag);
  ok = __syncthreads_and(ok);
  uint32_t copied = 0;
  if (tid == SA_WORKERS + 32 && ok) {
    for (; copied < SA_SLOTS; ++copied) {
      mbar_expect_tx(&ctl->full[copied], CHUNK_BYTES);
      bulk_copy_g2s(sh.ring + (size_t)copied * CHUNK_BYTES, reinterpret_cast<const uint8_t*>(parts_online) + (size_t)copied * CHUNK_BYTES,
                    CHUNK_BYTES, &ctl->full[copied]);
    }
  }
  uint32_t passes = 0;
  float qsel = 0.f;
  if (ok) {
    ok = sa_forward<D, H>(p.Hp, p.A, mw, sh, parts_online, parts_target, scale_online[1], tmem, 0u, copied, abort_flag);
    passes = 1;
    ok = __syncthreads_and(ok);
  }
  if (ok) {
    if (tid < n_here) {
      int a = p.act[j0 + tid];
      a = a < 0 ? 0 : (a >= p.A ? p.A - 1 : a);
      qsel = sh.out[a * SA_TE + tid];
    }
    __syncthreads();   // every thread is done with the online parameters and outputs: the staging buffer may be refilled
    mw = stage_mlp_weights<1>(p, p.Wtarget, wsm, &ctl->wbar, tid == 0);
    for (int i = tid; i < SA_TE * D; i += SA_NT) {
      const int el = i / D, k = i % D;
      sh.xs[k * SA_TE + el] = el < n_here ? p.next_obs[(size_t)(j0 + el) * D + k] : 0.f;
    }
    ok = tc_wait_elect(&ctl->wbar, 1, abort_flag);
    ok = __syncthreads_and(ok);
  }
  if (ok) {
    ok = sa_forward<D, H>(p.Hp, p.A, mw, sh, parts_online, parts_target, scale_target[1], tmem, 1u, copied, abort_flag);
    passes = 2;
    ok = __syncthreads_and(ok);
  }
  const float nan = __int_as_float(0x7FC00000);
  float* hub = sh.part;                       // free again after the pass
  if (tid < SA_TE) {
    float h = 0.f;
    if (tid < n_here) {
      const int j = j0 + tid;
      float delta = nan;
      h = nan;
      if (ok) {
        float qmax = sh.out[tid];
        for (int i = 1; i < p.A; ++i) qmax = fmaxf(qmax, sh.out[i * SA_TE + tid]);
        const float y = p.rew[j] + p.gamma * (p.done[j] ? 0.f : 1.f) * qmax;
        delta = y - qsel;
        const float ad = fabsf(delta);
        h = ad <= p.kappa ? 0.5f * delta * delta : p.kappa * (ad - 0.5f * p.kappa);
      }
      if (p.td_out) p.td_out[j] = delta;        // after a timeout: defined outputs (NaN), never what an earlier call left
      if (p.huber_out) p.huber_out[j] = h;
    }
    hub[tid] = h;
  }
  __syncthreads();
  if (tid == 0) {
    float sum = 0.f;
    for (int i = 0; i < n_here; ++i) sum += hub[i];
    p.partial[blockIdx.x] = sum;
    if (ctl->abort_flag && p.error) atomicExch(p.error, 4ull);
    else if (ctl->range_flag && p.error) atomicExch(p.error, 5ull);
  }
  // the copies still in flight must land before the block gives its shared memory back
  if (tid == SA_WORKERS + 32) {
    for (uint32_t g = passes * NSTREAM; g < copied; ++g)
      if (!tc_wait(&ctl->full[g % SA_SLOTS], (g / SA_SLOTS) & 1, abort_flag)) break;
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256u) : "memory");
  }
}

template <int ENV, int H>
cudaError_t launch_split(const ActorParams& p, const S2Plan& pl, const uint16_t* w2parts, const float* w2scale, int grid, int tpr, cudaStream_t s) {
  constexpr int D = ENV == TJ_ENV_CARTPOLE ? 4 : 6;
  const size_t smem = (size_t)S2_A_SLOTS * S2_A_SLOT + (size_t)SA_SLOTS * H * SA_KC * 2 +
                      ((size_t)(D + 6) * H + 4 + (tpr == 2 ? 2 * 2 * SA_TE * 4 : 0)) * sizeof(float) + sizeof(S2Ctl) + 64;
  return tpr == 1 ? launch_chained(actor_split_tc_kernel<ENV, H, 1>, grid, S2_NT, smem, s, p, pl, w2parts, w2scale)
                  : launch_chained(actor_split_tc_kernel<ENV, H, 2>, grid, S2_NT, smem, s, p, pl, w2parts, w2scale);
}

template <int ENV>
cudaError_t launch_split_env(const ActorParams& p, const S2Plan& pl, const uint16_t* w2parts, const float* w2scale, int grid, int tpr, cudaStream_t s) {
  switch (p.H) {
    case 64: return launch_split<ENV, 64>(p, pl, w2parts, w2scale, grid, tpr, s);
    case 128: return launch_split<ENV, 128>(p, pl, w2parts, w2scale, grid, tpr, s);
    case 192: return launch_split<ENV, 192>(p, pl, w2parts, w2scale, grid, tpr, s);
    case 256: return launch_split<ENV, 256>(p, pl, w2parts, w2scale, grid, tpr, s);
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
  const int grid = n_tiles < sm_count ? n_tiles : sm_count;
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
  const int tpr = n_tiles > sm_count ? 1 : 2;                // a second tile per SM hides the first one's chain
  return env_kind == TJ_ENV_CARTPOLE ? launch_split_env<TJ_ENV_CARTPOLE>(p, pl, w2parts, w2scale, grid, tpr, s)
                                     : launch_split_env<TJ_ENV_ACROBOT>(p, pl, w2parts, w2scale, grid, tpr, s);
}

template <int D>
static cudaError_t launch_td_split_d(const TdParams& p, const uint16_t* po, const float* so, const uint16_t* pt, const float* st, int grid,
                                     size_t smem, cudaStream_t s) {
#define TJ_TD_SPLIT_CASE(HH) \
  case HH: return launch_chained(td_split_tc_kernel<D, HH>, grid, SA_NT, smem, s, p, po, so, pt, st);
  switch (p.H) {
    TJ_TD_SPLIT_CASE(64)
    TJ_TD_SPLIT_CASE(128)
    TJ_TD_SPLIT_CASE(192)
    TJ_TD_SPLIT_CASE(256)
    default: return cudaErrorInvalidConfiguration;
  }
#undef TJ_TD_SPLIT_CASE
}

int td_split_grid(int n) { return (n + SA_TE - 1) / SA_TE; }

cudaError_t launch_td_split(const TdParams& p, const uint16_t* parts_online, const float* scale_online, const uint16_t* parts_target,
                            const float* scale_target, cudaStream_t s) {
  if (p.n <= 0) return cudaSuccess;
  if (!(p.D == 4 || p.D == 6) || p.A > 4 || p.Ap != 4) return cudaErrorInvalidConfiguration;
  const size_t staged = p.w_total - (p.off_b2 - p.off_W2t);
  const size_t smem = (size_t)2 * SA_TE * p.H * 2 + (size_t)SA_SLOTS * p.H * SA_KC * 2 +
                      (staged + (size_t)(8 + 4 + 8) * SA_TE) * sizeof(float) + sizeof(SaCtl) + 64;
  if (smem > 227 * 1024) return cudaErrorInvalidConfiguration;
  const int grid = td_split_grid(p.n);
  return p.D == 4 ? launch_td_split_d<4>(p, parts_online, scale_online, parts_target, scale_target, grid, smem, s)
                  : launch_td_split_d<6>(p, parts_online, scale_online, parts_target, scale_target, grid, smem, s);
}

}  // namespace tj
