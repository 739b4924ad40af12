// Pipelined tensor-core actor step for the linear-Gaussian workload (obs_dim 128, hidden a multiple of 128 up to 512):
// network, action selection, z = A s, env epilogue, record and reset in one persistent kernel whose roles overlap.
//
// A thread block owns 128 rows (envs) per tile, one row per TMEM lane, and walks its tiles once per step of the call: a tile stays with
// its block, so no step waits for another block, and the weights' ring, the pipeline and the launch are set up once (four steps of
// 20,000 envs, hidden 512: 206 us as four launches, 171 as one).  Roles:
//   warp 0, one lane    producer: streams 32 KB operand chunks (weights, the env matrix) from L2 into a ring of two slots
//   warp 1              MMA issuer, its loop warp-uniform, one elected lane at the instruction (tcgen05.mma, M = 128, N = 128 per hidden block)
//   warps 4-19          network warps (four threads per row): per 128-neuron block of a hidden layer: accumulator -> bias, ReLU, BF16
//                       -> next layer's operand; z -> a scratch tile in global memory
//   warps 20-27         env warps: the next tile's state rows as BF16 (layer-1 operand) and, with the record's observation, as FP16
//                       parts; take the head outputs out of TMEM, select the action, read z back and finish the step (tanh, Philox
//                       noise, reward, done, record, reset or new state, counters), four rows x eight 16-byte pieces per instruction
// The env warps work on tile i while the network warps and the tensor pipe are already on tile i + 1.
//
// Per tile the tensor pipe runs ten accumulator blocks that alternate between two 128-column accumulators:
//   layer 1 (4 blocks, A operand = X in shared memory), z (one block), layer 2 (4 blocks, A operand = h1 in tensor
//   memory), head (16 columns).  The epilogue of one block overlaps the MMAs of the next.
// z = A s keeps FP32 accuracy on the FP16 tensor path: state and matrix are each split into a high and a low FP16 part
// (power-of-two scaled so the low parts stay normal numbers), z = hi*hi + lo*hi + hi*lo with FP32 accumulation: 24
// instructions of K = 16, relative error about 2^-22 per term (the dropped lo*lo term and the low parts' rounding).
// Tensor memory (512 columns): [0, H/2) h1 as packed BF16 pairs; [256, 384) and [384, 512) the two accumulators.
// Shared memory: X (BF16 state tile, 32 KB) | U (128 KB: the FP16 high and low parts of the state tile in its first 64 KB
// until z is done, then h2, the head's A operand) | ring (64 KB) | barriers.
// Code size counts here: five roles execute five different programs at once, and with everything unrolled the kernel no longer fitted
// the instruction cache -- the issuing lane, which runs each line of its program once or a few times per tile, then took 446 cycles per
// MMA of the z product (64 on the tensor pipe) fetching instructions from L2.  So loops are unrolled only as far as their latency asks.
// Every wait is bounded: on a timeout the block raises an abort flag, records an error, waits for its copies and matrix instructions in
// flight, frees its TMEM and leaves.
#include <cstddef>

#include <cuda_fp16.h>

#include "tj_internal.h"
#include "tj_tc.cuh"

namespace tj {

namespace {

constexpr int PA_M = 128;                  // rows per tile
constexpr int PA_D = 128;                  // observation / state width this kernel is built for
constexpr int PA_NB = 128;                 // neurons per accumulator block
constexpr int PA_KC = 128;                 // K elements per weight chunk (128 x 128 x 2 bytes = 32 KB)
constexpr int PA_W_BYTES = PA_NB * PA_KC * 2;              // bytes of a hidden-layer weight chunk, and of one env-matrix part
constexpr int PA_STAGE_BYTES = PA_W_BYTES;
constexpr int PA_STAGES = 65536 / PA_STAGE_BYTES;
constexpr int PA_X_BYTES = PA_M * PA_D * 2;
constexpr int PA_U_BYTES = 131072;
constexpr int PA_NET_WARPS = 16, PA_ENV_WARPS = 8;   // one barrier arrival each
constexpr int PA_ENV0 = 4 + PA_NET_WARPS;  // warps 0-3: producer, MMA issuer, two idle; then network, then env
constexpr int PA_THREADS = 32 * (PA_ENV0 + PA_ENV_WARPS);
constexpr uint32_t PA_COL_HB = 0, PA_COL_ACC0 = 256, PA_COL_ACC1 = 384;
constexpr int PA_N3 = 16;                  // head width on the tensor cores
constexpr int PA_MAX_GRID = 192;           // thread blocks the z scratch is sized for
constexpr float PA_S_SCALE = 256.0f;       // state values are split after this scaling (|s| < 1.2: far below FP16's range)

struct PaSmem {
  uint64_t full[PA_STAGES], empty[PA_STAGES];
  uint64_t x_ready;        // env -> MMA: X holds the tile's BF16 rows
  uint64_t u_ready;        // env -> MMA: U holds the tile's FP16 high / low parts
  uint64_t acc_full[2];    // MMA -> network: an accumulator block is complete
  uint64_t acc_empty[2];   // network -> MMA: it has been drained (and its result stored)
  uint64_t head_full;      // MMA -> env and network: head outputs complete; U may be rewritten
  uint64_t env_taken;      // env -> MMA: head outputs are in registers
  uint64_t z_stored;       // network -> env: z of the tile is in the scratch tile
  uint64_t act_ready;      // env: the rows' actions are in shared memory
  uint64_t settled;        // after a timeout: the matrix instructions are over
  alignas(16) float bias[PA_NET_WARPS][32];   // per network warp: the biases of the columns it drains next
  uint8_t act[2][PA_M];    // by tile parity
  uint32_t tmem_base, copies;   // copies: bulk copies queued so far
  int abort_flag;
};

static_assert(offsetof(PaSmem, bias) % 16 == 0 && sizeof(PaSmem) <= 227 * 1024 - PA_X_BYTES - PA_U_BYTES - PA_STAGES * PA_STAGE_BYTES - 64, "layout");

// loads that stay where they are written: the compiler moves ordinary ones down to their uses
__device__ __forceinline__ float4 load_f4_cg(const float* p) {
  float4 v;
  asm volatile("ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ float4 load_f4_nc(const float* p) {
  float4 v;
  asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ float load_f1(const float* p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

__global__ void __launch_bounds__(PA_THREADS, 1) actor_tc_pipelined_kernel(const TcMlpParams p) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  constexpr int D = PA_D;
  const int H = p.H;
  uint8_t* xbuf = smem_raw;
  uint8_t* ubuf = xbuf + PA_X_BYTES;
  uint8_t* ring = ubuf + PA_U_BYTES;
  PaSmem* ctl = reinterpret_cast<PaSmem*>(ring + PA_STAGES * PA_STAGE_BYTES);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n_tiles = (p.n + PA_M - 1) / PA_M;
  // this block's work: its tiles once per step, step by step (a tile stays with its block, so a step needs nothing from another)
  const int my_tiles = (n_tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x, n_work = my_tiles * p.env.n_steps;
  const int n_hb = H / PA_NB;            // 128-neuron blocks per hidden layer
  // Thread blocks walk the neuron blocks of a layer in rotated order, so that at any moment they stream different
  // parts of the weights from L2 (the arithmetic per neuron is unchanged)
  const int rot = (int)(blockIdx.x % (unsigned)n_hb);
  const int n_kc2 = H / PA_KC;           // K chunks of a layer-2 block (a layer-1 block has one)

  if (tid == 0) {
    for (int s = 0; s < PA_STAGES; ++s) { mbar_init(&ctl->full[s], 1); mbar_init(&ctl->empty[s], 1); }
    mbar_init(&ctl->x_ready, PA_ENV_WARPS);
    mbar_init(&ctl->u_ready, PA_ENV_WARPS);
    mbar_init(&ctl->acc_full[0], 1);
    mbar_init(&ctl->acc_full[1], 1);
    mbar_init(&ctl->acc_empty[0], PA_NET_WARPS);
    mbar_init(&ctl->acc_empty[1], PA_NET_WARPS);
    mbar_init(&ctl->head_full, 1);
    mbar_init(&ctl->env_taken, PA_ENV_WARPS);
    mbar_init(&ctl->z_stored, PA_NET_WARPS);
    mbar_init(&ctl->act_ready, 4);
    mbar_init(&ctl->settled, 1);
    ctl->copies = 0;
    ctl->abort_flag = 0;
  }
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&ctl->tmem_base)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = ctl->tmem_base;
  chain_begin();
  volatile int* abort_flag = &ctl->abort_flag;
  const TcEnvParams& ev = p.env;

  if (warp < 4) {
    // registers: 896 threads x 72 at launch = 64,512; 128 x 56 + 512 x 56 + 256 x 112 = 64,512 after the changes
    asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
    if (warp == 0 && lane == 0) {
      // ---------------------------------------------------------------- producer
      // order per tile (the order the MMA issuer consumes): layer 1 (one chunk per block), env matrix (high part, low
      // part), layer 2 (H/128 chunks per block), head
      uint32_t it = 0;
      // every block re-reads the same chunks each tile while state rows and records stream through L2 once: the chunks
      // are fetched with an evict-last policy, the streams are written with evict-first stores
      const unsigned long long keep_policy = l2_evict_last_policy();
      const uint32_t head_bytes = (uint32_t)PA_N3 * H * 2;
      const int n1 = n_hb, n2 = n_hb * n_kc2;
      for (int v = 0; v < n_work && !*abort_flag; ++v) {
        for (int c = 0; c < n1 + 2 + n2 + 1; ++c, ++it) {
          const uint8_t* src;
          uint32_t bytes = PA_W_BYTES;
          if (c < n1) src = reinterpret_cast<const uint8_t*>(p.wtc) + (size_t)((c + rot) % n_hb) * PA_W_BYTES;
          else if (c < n1 + 2) src = reinterpret_cast<const uint8_t*>(ev.lgA16) + (size_t)(c - n1) * PA_W_BYTES;
          else if (c < n1 + 2 + n2) {
            const int idx = c - n1 - 2;
            src = reinterpret_cast<const uint8_t*>(p.wtc) + (size_t)(n1 + ((idx / n_kc2 + rot) % n_hb) * n_kc2 + idx % n_kc2) * PA_W_BYTES;
          }
          else { src = reinterpret_cast<const uint8_t*>(p.wtc) + (size_t)(n1 + n2) * PA_W_BYTES; bytes = head_bytes; }
          const int s = it % PA_STAGES;
          if (!tc_wait(&ctl->empty[s], ((it / PA_STAGES) & 1) ^ 1, abort_flag)) goto done;
          mbar_expect_tx(&ctl->full[s], bytes);
          bulk_copy_g2s_keep(ring + (size_t)s * PA_STAGE_BYTES, src, bytes, &ctl->full[s], keep_policy);
          ctl->copies = it + 1;
        }
      }
    } else if (warp == 1) {
      const uint32_t leader = elect_one();
      // ---------------------------------------------------------------- MMA issuer
      // Accumulator uses of a tile: u = 0 .. n_hb-1 layer 1, n_hb z, n_hb+1 .. 2 n_hb layer 2, 2 n_hb + 1 head; use u
      // writes accumulator u & 1 (the count per tile is even, so the pattern repeats).  The network warps drain every use
      // but the head (acc_empty), the env warps take the head (env_taken).
      uint32_t it = 0, tiles = 0, nwait0 = 0, nwait1 = 0;
      const uint32_t idesc_h = make_idesc(PA_NB), idesc16 = make_idesc(PA_N3), idesc_z = make_idesc_f16(D);
      // descriptors as (low, high) words: the high word is fixed per operand shape, the low word steps by 16 per K = 16
      const uint32_t x_lo = desc_lo(smem_addr(xbuf), 128u), u_lo = desc_lo(smem_addr(ubuf), 128u);
      const uint32_t ulo_lo = desc_lo(smem_addr(ubuf) + (uint32_t)PA_X_BYTES, 128u);
      const uint32_t ring_lo = desc_lo(smem_addr(ring), 128u);
      const uint32_t hi_k128 = desc_hi(2048u);                       // operands 128 K-elements wide (X, U, weight chunks)
      const uint32_t hi_head = desc_hi((uint32_t)(H / 8) * 128u);    // operands H K-elements wide (h2, head weights)
      // before use u may overwrite its accumulator, the previous use of that accumulator must have been read out
      auto acquire = [&](int u) -> bool {
        if (u == 0) return true;      // accumulator 0: its last drain was awaited before the previous tile's head
        if (u == 1) return tiles == 0 || tc_wait_warp(&ctl->env_taken, (tiles - 1) & 1, abort_flag);
        return (u & 1) ? tc_wait_warp(&ctl->acc_empty[1], (nwait1++) & 1, abort_flag) : tc_wait_warp(&ctl->acc_empty[0], (nwait0++) & 1, abort_flag);
      };
      for (; tiles < (uint32_t)n_work; ++tiles) {
        if (!tc_wait_warp(&ctl->x_ready, tiles & 1, abort_flag)) goto done;
        // layer 1: one chunk per 128-neuron block; A operand = X in shared memory
        for (int b = 0; b < n_hb; ++b, ++it) {
          const int u = b;
          if (!acquire(u)) goto done;
          const uint32_t acc = tmem + ((u & 1) ? PA_COL_ACC1 : PA_COL_ACC0);
          const uint32_t s = it % PA_STAGES;
          if (!tc_wait_warp(&ctl->full[s], (it / PA_STAGES) & 1, abort_flag)) goto done;
          tc_fence_after();
          const uint32_t b_lo = ring_lo + s * (PA_STAGE_BYTES / 16);
#pragma unroll 4
          for (int j = 0; j < PA_KC / 16; ++j) umma_ss(acc, x_lo + j * 16u, hi_k128, b_lo + j * 16u, hi_k128, idesc_h, j != 0, leader);
          umma_commit(&ctl->empty[s], leader);
          umma_commit((u & 1) ? &ctl->acc_full[1] : &ctl->acc_full[0], leader);
        }
        // z = A s from the FP16 parts: (s_hi, A_hi) + (s_lo, A_hi) with the first chunk, (s_hi, A_lo) with the second
        {
          const int u = n_hb;
          if (!tc_wait_warp(&ctl->u_ready, tiles & 1, abort_flag)) goto done;
          if (!acquire(u)) goto done;
          const uint32_t acc = tmem + ((u & 1) ? PA_COL_ACC1 : PA_COL_ACC0);
          for (int part = 0; part < 2; ++part, ++it) {
            const uint32_t s = it % PA_STAGES;
            if (!tc_wait_warp(&ctl->full[s], (it / PA_STAGES) & 1, abort_flag)) goto done;
            tc_fence_after();
            const uint32_t b_lo = ring_lo + s * (PA_STAGE_BYTES / 16);
#pragma unroll 2
            for (int j = 0; j < D / 16; ++j) {
              umma_ss(acc, u_lo + j * 16u, hi_k128, b_lo + j * 16u, hi_k128, idesc_z, (part | j) != 0, leader);
              if (part == 0) umma_ss(acc, ulo_lo + j * 16u, hi_k128, b_lo + j * 16u, hi_k128, idesc_z, 1u, leader);
            }
            umma_commit(&ctl->empty[s], leader);
          }
          umma_commit((u & 1) ? &ctl->acc_full[1] : &ctl->acc_full[0], leader);
        }
        // layer 2: per block H / PA_KC chunks; A operand = h1 in tensor memory (8 columns per K = 16); the drain of the last
        // layer-1 block (awaited by the first block here) completes h1
        for (int b = 0; b < n_hb; ++b) {
          const int u = n_hb + 1 + b;
          if (!acquire(u)) goto done;
          const uint32_t acc = tmem + ((u & 1) ? PA_COL_ACC1 : PA_COL_ACC0);
          for (int c = 0; c < n_kc2; ++c, ++it) {
            const uint32_t s = it % PA_STAGES;
            if (!tc_wait_warp(&ctl->full[s], (it / PA_STAGES) & 1, abort_flag)) goto done;
            tc_fence_after();
            const uint32_t b_lo = ring_lo + s * (PA_STAGE_BYTES / 16);
            const uint32_t a_col = tmem + PA_COL_HB + (uint32_t)(c * (PA_KC / 2));
#pragma unroll 4
            for (int j = 0; j < PA_KC / 16; ++j) umma_ts(acc, a_col + (uint32_t)(j * 8), b_lo + j * 16u, hi_k128, idesc_h, (c | j) != 0, leader);
            umma_commit(&ctl->empty[s], leader);
          }
          umma_commit((u & 1) ? &ctl->acc_full[1] : &ctl->acc_full[0], leader);
        }
        // head: 16 outputs, K = H, A operand = h2 in shared memory; accumulator 1.  Both remaining drains complete h2.
        {
          if (!acquire(2 * n_hb + 1)) goto done;
          if (!tc_wait_warp(&ctl->acc_empty[0], (nwait0++) & 1, abort_flag)) goto done;
          const uint32_t s = it % PA_STAGES;
          if (!tc_wait_warp(&ctl->full[s], (it / PA_STAGES) & 1, abort_flag)) goto done;
          tc_fence_after();
          const uint32_t b_lo = ring_lo + s * (PA_STAGE_BYTES / 16);
#pragma unroll 4
          for (int j = 0; j < H / 16; ++j) umma_ss(tmem + PA_COL_ACC1, u_lo + j * 16u, hi_head, b_lo + j * 16u, hi_head, idesc16, j != 0, leader);
          umma_commit(&ctl->empty[s], leader);
          umma_commit(&ctl->head_full, leader);
          ++it;
        }
      }
    }
  } else if (warp < PA_ENV0) {
    // ------------------------------------------------------------------ network warps
    asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
    const int q = warp & 3;                       // TMEM lane quarter this warp may access
    const int hsel = (warp - 4) >> 2;             // which quarter of a block's columns
    const int r = q * 32 + lane;                  // row of the tile = TMEM lane
    const uint32_t t_lane = tmem + ((uint32_t)(q * 32) << 16);
    uint32_t tiles = 0, nfull0 = 0, nfull1 = 0;
    // Biases go through a shared-memory row of this warp, loaded one use ahead: 28 KB of L1 hold little beside 227 KB of shared memory, so
    // eight loads between accumulator and operand cost an L2 round trip in every drain
    float* bias_row = ctl->bias[warp - 4];
    int b = rot;                                  // neuron block of the next use that has one
    float bias_next = __ldg(p.b1 + b * PA_NB + hsel * 32 + lane);
    for (; tiles < (uint32_t)n_work; ++tiles) {
      for (int u = 0; u <= 2 * n_hb; ++u) {
        const int buf = u & 1;
        const int layer = u < n_hb ? 0 : 1, c0 = b * PA_NB + hsel * 32;   // first of this thread's 32 columns
        if (u != n_hb) {
          __syncwarp();
          bias_row[lane] = bias_next;
          b = b + 1 == n_hb ? 0 : b + 1;
          bias_next = __ldg((u + 1 < n_hb || u == 2 * n_hb ? p.b1 : p.b2) + b * PA_NB + hsel * 32 + lane);
        }
        if (!tc_wait_elect(buf ? &ctl->acc_full[1] : &ctl->acc_full[0], (buf ? nfull1++ : nfull0++) & 1, abort_flag)) goto done;
        tc_fence_after();
        const uint32_t t_acc = t_lane + (buf ? PA_COL_ACC1 : PA_COL_ACC0) + (uint32_t)(hsel * 32);
        if (u == n_hb) {
          // z: this thread's 32 components go to the block's scratch tile, where the env warps pick them up
          uint32_t v[32];
          tmem_ld16(t_acc, v);
          tmem_ld16(t_acc + 16u, v + 16);
          tmem_ld_wait();
          tc_fence_before();
          // scratch tile [k/4][row][4]: a warp's 32 rows are contiguous
          float* zs = ev.z_scratch + ((size_t)blockIdx.x * 2 + (tiles & 1)) * (PA_M * D);
#pragma unroll
          for (int i = 0; i < 8; ++i)
            *reinterpret_cast<uint4*>(zs + ((size_t)(hsel * 8 + i) * PA_M + r) * 4) = make_uint4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
          mbar_arrive_warp(&ctl->acc_empty[buf]);
          mbar_arrive_warp(&ctl->z_stored);
          continue;
        }
        uint32_t v[32], o[16];
        tmem_ld16(t_acc, v);
        tmem_ld16(t_acc + 16u, v + 16);
        tmem_ld_wait();
#pragma unroll
        for (int j4 = 0; j4 < 8; ++j4) {
          const float4 bb = *reinterpret_cast<const float4*>(bias_row + 4 * j4);
          o[2 * j4] = pack_bf16x2_relu(__uint_as_float(v[4 * j4]) + bb.x, __uint_as_float(v[4 * j4 + 1]) + bb.y);
          o[2 * j4 + 1] = pack_bf16x2_relu(__uint_as_float(v[4 * j4 + 2]) + bb.z, __uint_as_float(v[4 * j4 + 3]) + bb.w);
        }
        if (layer == 0) {
          tmem_st16(t_lane + PA_COL_HB + (uint32_t)(c0 / 2), o);
        } else {
          uint8_t* dst = ubuf + ((size_t)(r >> 3) * (H / 8)) * 128 + (r & 7) * 16 + (size_t)(c0 / 8) * 128;
#pragma unroll
          for (int g = 0; g < 4; ++g)
            *reinterpret_cast<uint4*>(dst + (size_t)g * 128) = make_uint4(o[4 * g], o[4 * g + 1], o[4 * g + 2], o[4 * g + 3]);
        }
        if (layer == 0) tmem_st_wait();
        else fence_async_smem();
        tc_fence_before();
        mbar_arrive_warp(&ctl->acc_empty[buf]);
      }
    }
  } else {
    // ------------------------------------------------------------------ env warps
    asm volatile("setmaxnreg.inc.sync.aligned.u32 112;");
    const int ew = warp - PA_ENV0;                 // 0..7; the first four also read the head outputs (one TMEM quarter each)
    const int e_r4 = lane >> 3, e_kq = lane & 7;   // four rows x eight 16-byte pieces per warp instruction, four pieces per lane and row
    uint32_t tiles = 0;
    // this lane's pieces of a tile's row groups g and g + 1, all in flight at once
    auto load_rows = [&](int tile, int g, float4 (&v)[2][4]) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const long long row = (long long)tile * PA_M + ew * 16 + (g + h) * 4 + e_r4;
        const float* xr = p.x + (size_t)(row < p.n ? row : 0) * D;
#pragma unroll
        for (int i = 0; i < 4; ++i)
          v[h][i] = row < p.n ? __ldcg(reinterpret_cast<const float4*>(xr + (e_kq + 8 * i) * 4)) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    };
    // BF16 rows of a tile -> X (layer-1 A operand)
    auto convert_x = [&](int tile) {
#pragma unroll 1
      for (int g = 0; g < 4; g += 2) {
        float4 v[2][4];
        load_rows(tile, g, v);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int rr = ew * 16 + (g + h) * 4 + e_r4;
          uint8_t* dx = xbuf + ((size_t)(rr >> 3) * (D / 8)) * 128 + (rr & 7) * 16;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int k4 = e_kq + 8 * i;
            *reinterpret_cast<uint2*>(dx + (size_t)(k4 >> 1) * 128 + (k4 & 1) * 8) =
                make_uint2(pack_bf16x2(v[h][i].x, v[h][i].y), pack_bf16x2(v[h][i].z, v[h][i].w));
          }
        }
      }
      fence_async_smem();
      mbar_arrive_warp(&ctl->x_ready);
    };
    // FP16 high / low parts of a tile's scaled rows -> U (A operand of z = A s); the FP32 row is the record's observation
    auto convert_u = [&](int tile, uint32_t block) {
#pragma unroll 1
      for (int g = 0; g < 4; g += 2) {
        float4 v[2][4];
        load_rows(tile, g, v);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int rr = ew * 16 + (g + h) * 4 + e_r4;
          const long long row = (long long)tile * PA_M + rr;
          const bool live = row < p.n;
          uint8_t* dhi = ubuf + ((size_t)(rr >> 3) * (D / 8)) * 128 + (rr & 7) * 16;
          uint8_t* dlo = dhi + PA_X_BYTES;
          float* rec = ev.ring + ((unsigned long long)block * (uint32_t)p.n + (unsigned long long)(live ? row : 0)) * ev.rec_words;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int k4 = e_kq + 8 * i;
            const float4 sv = v[h][i];
            // high part: the scaled value cut to 11 significant bits (exact in FP16); low part: the exact remainder, rounded
            float4 s4, hi, lo;
            s4.x = sv.x * PA_S_SCALE; s4.y = sv.y * PA_S_SCALE; s4.z = sv.z * PA_S_SCALE; s4.w = sv.w * PA_S_SCALE;
            hi.x = __uint_as_float(__float_as_uint(s4.x) & 0xFFFFE000u); lo.x = s4.x - hi.x;
            hi.y = __uint_as_float(__float_as_uint(s4.y) & 0xFFFFE000u); lo.y = s4.y - hi.y;
            hi.z = __uint_as_float(__float_as_uint(s4.z) & 0xFFFFE000u); lo.z = s4.z - hi.z;
            hi.w = __uint_as_float(__float_as_uint(s4.w) & 0xFFFFE000u); lo.w = s4.w - hi.w;
            const size_t off = (size_t)(k4 >> 1) * 128 + (k4 & 1) * 8;
            *reinterpret_cast<uint2*>(dhi + off) = make_uint2(pack_f16x2(hi.x, hi.y), pack_f16x2(hi.z, hi.w));
            *reinterpret_cast<uint2*>(dlo + off) = make_uint2(pack_f16x2(lo.x, lo.y), pack_f16x2(lo.z, lo.w));
            if (live) __stcs(reinterpret_cast<float4*>(rec + k4 * 4), sv);
          }
        }
      }
      fence_async_smem();
      mbar_arrive_warp(&ctl->u_ready);
    };
    unsigned long long n_episodes = 0;
    double ret_sum = 0.0;
    const float zc = ev.z_to_t;                    // accumulator -> 2 log2(e) * z
    // the first round has no tile to finish, it only converts: one copy of the conversion's code (see the note on code size above)
    bool warm = false;
    // the next piece of work is another tile (its last step is done) unless this block has only one
    const bool several = my_tiles > 1;
    int tile = 0, next_tile = blockIdx.x;
    // ring blocks (of one step's records each) and step numbers of both
    uint32_t block = 0, next_block = ev.block0, step = 0, next_step = 0;
    for (int v = -1; v < n_work; ++v) {
      const bool more = v + 1 < n_work, early = more && (several || !warm);
      // layer 1 and z of this tile are complete, so X is free: the next tile's rows go in while layer 2 runs
      if (warm && !tc_wait_elect(&ctl->z_stored, tiles & 1, abort_flag)) goto done;
      if (early) {
        convert_x(next_tile);
        // pull the rows of the tile after the next towards L2
        const long long prow = (long long)(next_tile + (int)gridDim.x) * PA_M + ew * 16 + (lane >> 1);
        if (prow < p.n) {
          const float* xn = p.x + (size_t)prow * D + (lane & 1) * 64;
          prefetch_l2(xn);
          prefetch_l2(xn + 32);
        }
      }
      if (!warm) {
      } else if (ew < 4) {
        const int r = ew * 32 + lane;              // row of the tile = TMEM lane
        const long long row = (long long)tile * PA_M + r;
        if (!tc_wait_elect(&ctl->head_full, tiles & 1, abort_flag)) goto done;
        tc_fence_after();
        uint32_t qraw[16];
        tmem_ld16(tmem + ((uint32_t)(ew * 32) << 16) + PA_COL_ACC1, qraw);
        tmem_ld_wait();
        tc_fence_before();
        mbar_arrive_warp(&ctl->env_taken);
        // epsilon-greedy on this row: explore iff x0 < threshold, else the first maximum
        float qv[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) qv[j] = __uint_as_float(qraw[j]) + (j < p.Aout ? __ldg(p.b3 + j) : 0.f);
        if (row < p.n && p.out) {
          float* o = p.out + ((size_t)step * p.n + (size_t)row) * p.Aout;
#pragma unroll
          for (int j = 0; j < 16; ++j)
            if (j < p.Aout) o[j] = qv[j];
        }
        const uint4 w = stream_words(ev.seed, STREAM_ACTION, 0, (uint32_t)row, ev.t + step);
        int best = 0;
        float qb = qv[0];
#pragma unroll
        for (int j = 1; j < 16; ++j)
          if (j < ev.A && qv[j] > qb) { qb = qv[j]; best = j; }
        ctl->act[tiles & 1][r] = ((unsigned long long)w.x < ev.explore_thr) ? (uint8_t)__umulhi(w.y, (uint32_t)ev.A) : (uint8_t)best;
        mbar_arrive_warp(&ctl->act_ready);
      } else {
        mbar_arrive_warp(&ctl->env_taken);         // this warp has finished the previous tile
        if (!tc_wait_elect(&ctl->head_full, tiles & 1, abort_flag)) goto done;
      }
      // the head of this tile is complete, so U is free: the next tile's FP16 parts go in before this tile's env step -- or, where
      // the next piece of work is this tile again, both conversions after it
#pragma unroll 1
      for (int pass = 0; pass < 2; ++pass) {
        if ((pass == 0) == (early || !more)) {
          if (more) {
            if (!early) convert_x(next_tile);
            convert_u(next_tile, next_block);
          }
          continue;
        }
        if (!warm) continue;
        if (!tc_wait_elect(&ctl->act_ready, tiles & 1, abort_flag)) goto done;
        const float* zs = ev.z_scratch + ((size_t)blockIdx.x * 2 + (tiles & 1)) * (PA_M * D);
#pragma unroll 1
        for (int g = 0; g < 4; ++g) {
          const int rr = ew * 16 + g * 4 + e_r4;
          const long long row = (long long)tile * PA_M + rr;
          const bool live = row < p.n;
          const int action = ctl->act[tiles & 1][rr];
          float* rec = ev.ring + ((unsigned long long)block * (uint32_t)p.n + (unsigned long long)(live ? row : 0)) * ev.rec_words;
          const int ep0 = __float_as_int(load_f1(reinterpret_cast<const float*>(ev.ep_step) + (live ? row : 0)));
          const float ret0 = load_f1(ev.ep_return + (live ? row : 0));
          const float* Ba = ev.lgB_t + (size_t)action * D;     // B[a] times 2 log2(e)
          // s' = tanh(z + B[a]) + noise; piece k4 = components 4 k4 .. 4 k4 + 3 = one Philox block
          // z, B's row and the counters are on their way while the noise, which needs none of them, is made (a row group took 6,900 cycles
          // with every load behind the instructions that its use follows, 6,000 now)
          float4 zz[4], bb[4], sn[4];
          float3 n01[4], n23[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            zz[i] = load_f4_cg(zs + ((size_t)(e_kq + 8 * i) * PA_M + rr) * 4);
            bb[i] = load_f4_nc(Ba + 4 * (e_kq + 8 * i));
          }
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const uint4 w = stream_words(ev.seed, STREAM_NOISE, (uint32_t)(e_kq + 8 * i), (uint32_t)row, ev.t + step);
            n01[i] = box_muller_scaled(w.x, w.y, ev.noise_std);
            n23[i] = box_muller_scaled(w.z, w.w, ev.noise_std);
          }
          float sq = 0.f;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int k4 = e_kq + 8 * i;
            float4 o;
            o.x = fmaf(n01[i].x, n01[i].y, tanh_from_t(fmaf(zz[i].x, zc, bb[i].x)));
            o.y = fmaf(n01[i].x, n01[i].z, tanh_from_t(fmaf(zz[i].y, zc, bb[i].y)));
            o.z = fmaf(n23[i].x, n23[i].y, tanh_from_t(fmaf(zz[i].z, zc, bb[i].z)));
            o.w = fmaf(n23[i].x, n23[i].z, tanh_from_t(fmaf(zz[i].w, zc, bb[i].w)));
            sq = fmaf(o.x, o.x, sq); sq = fmaf(o.y, o.y, sq); sq = fmaf(o.z, o.z, sq); sq = fmaf(o.w, o.w, sq);
            sn[i] = o;
            if (live) __stcs(reinterpret_cast<float4*>(rec + D + 4 * k4), o);
          }
          // the eight lanes of a row add their partial squared norms (same order in every lane)
          sq += __shfl_xor_sync(0xffffffffu, sq, 1);
          sq += __shfl_xor_sync(0xffffffffu, sq, 2);
          sq += __shfl_xor_sync(0xffffffffu, sq, 4);
          if (live) {
            const float rew = -sq / (float)D;
            int ep = ep0 + 1;
            float ep_ret = ret0 + rew;
            const int done = (sqrtf(sq) > ev.done_norm || ep >= ev.max_ep) ? 1 : 0;
            float* st = ev.state + (size_t)row * D;
            if (done) {
              ep_ret = 0.f;
              ep = 0;
#pragma unroll 1
              for (int i = 0; i < 4; ++i) {
                const int k4 = e_kq + 8 * i;
                const uint4 w = stream_words(ev.seed, STREAM_RESET, (uint32_t)k4, (uint32_t)row, ev.t + step);
                *reinterpret_cast<float4*>(st + 4 * k4) = make_float4(uniform_range(w.x, -0.1f, 0.2f), uniform_range(w.y, -0.1f, 0.2f),
                                                                      uniform_range(w.z, -0.1f, 0.2f), uniform_range(w.w, -0.1f, 0.2f));
              }
            } else {
#pragma unroll
              for (int i = 0; i < 4; ++i) *reinterpret_cast<float4*>(st + 4 * (e_kq + 8 * i)) = sn[i];
            }
            if (e_kq == 0) {
              *reinterpret_cast<float4*>(rec + 2 * D) =
                  make_float4(__int_as_float(action), rew, __int_as_float(done), __int_as_float(ev.version));
              if (done) {
                n_episodes += 1;
                ret_sum += (double)(ret0 + rew);
              }
              ev.ep_step[row] = ep;
              ev.ep_return[row] = ep_ret;
            }
          }
        }
      }
      tiles += warm;
      warm = true;
      __syncwarp();                                // a row's step counters, written by one lane, are read by eight in the next step
      tile = next_tile; block = next_block; step = next_step;
      next_tile += gridDim.x;
      if (next_tile >= n_tiles) {
        next_tile = blockIdx.x;
        ++next_step;
        if (++next_block == ev.n_blocks) next_block = 0;
      }
    }
    // episode statistics: one atomic pair per warp
    {
      unsigned long long n = n_episodes;
      double rs = ret_sum;
      for (int o = 16; o > 0; o >>= 1) {
        n += __shfl_down_sync(0xffffffffu, n, o);
        rs += __shfl_down_sync(0xffffffffu, rs, o);
      }
      if (lane == 0 && n) {
        atomicAdd(&ev.stats->episodes, n);
        atomicAdd(&ev.stats->return_sum, rs);
      }
      if (blockIdx.x == 0 && tid == PA_ENV0 * 32) {
        uint32_t b = ev.block0;
        for (int i = 0; i < ev.n_steps; ++i) {
          ev.block_ver[b] = ev.version;
          if (++b == ev.n_blocks) b = 0;
        }
      }
    }
  }
done:
  __syncthreads();
  if (ctl->abort_flag) {
    if (tid == 0) atomicExch(p.error, 2ull);
    tc_settle(&ctl->settled, warp == 1, ctl->full, PA_STAGES, ctl->copies);
    __syncthreads();
  }
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
  }
}

// The env matrix A [128][128] scaled by `scale` (a power of two) as two FP16 chunks, high parts then low parts, each in the
// layout of a weight chunk (row = component of z, column = component of s); B [n_actions][128] times 2 log2(e).
__global__ void pack_env_f16_kernel(const float* __restrict__ A, const float* __restrict__ B, float scale, int n_b,
                                    uint16_t* __restrict__ dst, float* __restrict__ b_t) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < PA_D * PA_D) {
    const int core = i / 64, in_core = i % 64;
    const int rg = core / (PA_D / 8), kg = core % (PA_D / 8);
    const int n = rg * 8 + in_core / 8, k = kg * 8 + in_core % 8;
    const float v = A[(size_t)n * PA_D + k] * scale;
    const __half hi = __float2half_rn(v);
    const __half lo = __float2half_rn(v - __half2float(hi));
    dst[i] = __half_as_ushort(hi);
    dst[PA_D * PA_D + i] = __half_as_ushort(lo);
  }
  if (i < n_b) b_t[i] = B[i] * 2.88539008177792681472f;
}

}  // namespace

bool tc_pipelined_supported(int D, int H, int A) {
  return D == PA_D && H >= PA_NB && H <= 512 && H % PA_NB == 0 && A >= 1 && A <= PA_N3;
}

size_t tc_pipelined_scratch_floats() { return (size_t)PA_MAX_GRID * 2 * PA_M * PA_D; }
size_t tc_pipelined_env_halfs() { return (size_t)2 * PA_D * PA_D; }
float tc_pipelined_state_scale() { return PA_S_SCALE; }

cudaError_t launch_pack_pipelined_env(const float* A, const float* B, float scale, int n_actions, uint16_t* dst, float* b_t,
                                      cudaStream_t s) {
  const int n = PA_D * PA_D > n_actions * PA_D ? PA_D * PA_D : n_actions * PA_D;
  pack_env_f16_kernel<<<(n + 255) / 256, 256, 0, s>>>(A, B, scale, n_actions * PA_D, dst, b_t);
  return cudaGetLastError();
}

cudaError_t launch_actor_tc_pipelined(const TcMlpParams& p, int sm_count, cudaStream_t s) {
  if (p.n <= 0) return cudaSuccess;
  if (!tc_pipelined_supported(p.D, p.H, p.Aout) || !p.env.fused) return cudaErrorInvalidConfiguration;
  const size_t smem = (size_t)PA_X_BYTES + PA_U_BYTES + (size_t)PA_STAGES * PA_STAGE_BYTES + sizeof(PaSmem) + 64;
  const int n_tiles = (p.n + PA_M - 1) / PA_M;
  int grid = n_tiles < sm_count ? n_tiles : sm_count;
  if (grid > PA_MAX_GRID) grid = PA_MAX_GRID;
  if (!p.env.z_scratch || !p.env.lgA16 || !p.env.lgB_t) return cudaErrorInvalidValue;
  return launch_chained(actor_tc_pipelined_kernel, grid, PA_THREADS, smem, s, p);
}

}  // namespace tj
