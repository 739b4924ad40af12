// Parameter publish (dependency I, learner -> actor): one launch turns the blob
//   [W1 HxD, b1 H, W2 HxH, b2 H, W3 AxH, b3 A (, Wv H, bv 1)]
// into every layout that the context's kernels read:
//   - the FP32 layout, each matrix transposed to [in][out padded to 4] (rounded to bfloat16 where the context asks for it);
//   - BF16 contexts: the two tensor-core kernels' chunk streams (K-major core matrices of 8 rows x 16 bytes);
//   - split-operand contexts: W2 as FP16 high and low parts in that kernel's chunk stream, scaled by a power of two.
//
// A block takes one tile of 32 neurons x KT inputs of W1 or W2 through shared memory: read once along the inputs, written
// once per layout, each time in runs of at least 64 contiguous bytes (one kernel per layout, thread per element, read the
// blob with a stride of a row and once per layout: 11.7 us in three launches for 128-512-512-16, 17 us in two for the split
// parts of 6-256-256-3).  Bound by launch and memory latency: the largest blob is 1.4 MB.
#include <cuda_fp16.h>

#include "tj_async.cuh"
#include "tj_internal.h"

namespace tj {

namespace {

__device__ __forceinline__ uint32_t bf16_bits_rne(float x) {
  const uint32_t u = __float_as_uint(x);
  if ((u & 0x7F800000u) == 0x7F800000u) return u >> 16;
  return (u + 0x7FFFu + ((u >> 16) & 1u)) >> 16;
}

// element (row, k) of an operand part of `kc` columns in the core-matrix layout, in halfs; k a multiple of 8
__device__ __forceinline__ size_t core_offset(int row, int k, int kc) {
  return ((size_t)(row >> 3) * (kc >> 3) + (k >> 3)) * 64 + (size_t)(row & 7) * 8;
}

// NT threads; SPLIT: split-operand context, launched as clusters of eight blocks.  Cluster 0 owns W2: each of its blocks
// reads an eighth into shared memory, they agree on the largest |entry| (a scan of the whole matrix by every block took 14 us), then
// pack what they hold (7.3 us with a second read of it).
template <int NT, bool SPLIT>
__global__ void __launch_bounds__(NT) publish_kernel(const PublishParams p) {
  chain_begin();
  chain_next();
  constexpr int KT = NT / 8;                      // inputs per tile
  extern __shared__ float pub_sm[];               // one tile [32][KT + 1], or a cluster-0 block's tiles of W2
  __shared__ float red[NT / 32];
  __shared__ float cluster_max;
  const int D = p.L.D, H = p.L.H, A = p.L.A, Hp = p.L.Hp, Ap = p.L.Ap, tid = threadIdx.x;
  const float* W1 = p.blob;
  const float* b1 = W1 + (size_t)H * D;
  const float* W2 = b1 + H;
  const float* b2 = W2 + (size_t)H * H;
  const float* W3 = b2 + H;
  const float* b3 = W3 + (size_t)A * H;
  const float* Wv = b3 + A;
  const float* bv = Wv + H;
  const int row_tiles = (Hp + 31) / 32, k_tiles1 = (D + KT - 1) / KT, k_tiles2 = (H + KT - 1) / KT;
  const int n1 = row_tiles * k_tiles1, n2 = row_tiles * k_tiles2;

  // tile t of W (H x K) -> shared memory; returns this thread's largest |entry|
  auto load_tile = [&](float (*tile)[KT + 1], const float* W, int K, int t) {
    const int n0 = (t % row_tiles) * 32, k0 = (t / row_tiles) * KT;
    float m = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = tid / KT + i * 8, c = tid % KT;
      const float v = n0 + r < H && k0 + c < K ? W[(size_t)(n0 + r) * K + k0 + c] : 0.f;
      tile[r][c] = v;
      m = fmaxf(m, fabsf(v));
    }
    return m;
  };
  // the tile in shared memory -> every layout
  auto write_tile = [&](const float (*tile)[KT + 1], int K, int t, float* dst, int layer, float split_scale) {
    const int n0 = (t % row_tiles) * 32, k0 = (t / row_tiles) * KT;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int n = n0 + (tid & 31), k = k0 + (tid >> 5) + i * (NT / 32);
      if (n < Hp && k < K) {
        float v = tile[tid & 31][k - k0];
        if (p.bf16) v = __uint_as_float(bf16_bits_rne(v) << 16);
        dst[(size_t)k * Hp + n] = v;
      }
    }
    // core-matrix layouts: a thread packs eight inputs of one neuron (16 bytes); consecutive threads the eight rows of a core
    // matrix, then the next eight inputs
    if (tid < 32 * (KT / 8)) {
      const int r = ((tid / KT) << 3) + (tid & 7), kk = ((tid >> 3) % (KT / 8)) * 8, n = n0 + r, k = k0 + kk;
      if (n < H && k < K) {
        if (SPLIT) {
          if (layer == 1) {
            uint32_t hi[4], lo[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const float v0 = tile[r][kk + 2 * i] * split_scale, v1 = tile[r][kk + 2 * i + 1] * split_scale;
              const __half h0 = __float2half_rn(v0), h1 = __float2half_rn(v1);
              const __half l0 = __float2half_rn(v0 - __half2float(h0)), l1 = __float2half_rn(v1 - __half2float(h1));
              hi[i] = (uint32_t)__half_as_ushort(h0) | ((uint32_t)__half_as_ushort(h1) << 16);
              lo[i] = (uint32_t)__half_as_ushort(l0) | ((uint32_t)__half_as_ushort(l1) << 16);
            }
            uint16_t* d = p.split + (size_t)(2 * (k / 32)) * (H * 32) + core_offset(n, k % 32, 32);
            *reinterpret_cast<uint4*>(d) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
            *reinterpret_cast<uint4*>(d + (size_t)H * 32) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
          }
        } else if (p.tc) {
          uint32_t o[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) o[i] = bf16_bits_rne(tile[r][kk + 2 * i]) | (bf16_bits_rne(tile[r][kk + 2 * i + 1]) << 16);
          const uint4 o4 = make_uint4(o[0], o[1], o[2], o[3]);
          const size_t base = layer == 0 ? 0 : (size_t)H * D;
          const int NB = H > 256 ? H / 2 : H;      // neurons per chunk of the general kernel's stream, 32 inputs each
          *reinterpret_cast<uint4*>(p.tc + base + ((size_t)(n / NB) * (K / 32) + k / 32) * ((size_t)NB * 32) + core_offset(n % NB, k % 32, 32)) = o4;
          if (p.tc_pipe)                           // chunks of 128 neurons x 128 inputs
            *reinterpret_cast<uint4*>(p.tc_pipe + base + ((size_t)(n / 128) * (K / 128) + k / 128) * (128 * 128) + core_offset(n % 128, k % 128, 128)) = o4;
        }
      }
    }
  };

  float (*tile)[KT + 1] = reinterpret_cast<float (*)[KT + 1]>(pub_sm);
  int job = blockIdx.x;
  if (SPLIT) {
    if (job < 8) {                                 // cluster 0: the hidden x hidden matrix, every block's share read once
      float m = 0.f;
      for (int t = job, i = 0; t < n2; t += 8, ++i) m = fmaxf(m, load_tile(tile + 32 * i, W2, H, t));
      for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
      if ((tid & 31) == 0) red[tid >> 5] = m;
      __syncthreads();
      if (tid < 32) {
        m = tid < NT / 32 ? red[tid] : 0.f;
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (tid == 0) cluster_max = m;
      }
      cluster_sync_all();
      if (tid < 32) {
        m = tid < 8 ? cluster_load_f32(&cluster_max, tid) : 0.f;
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (tid == 0) red[0] = m;
      }
      cluster_sync_all();                          // nobody leaves while a peer reads its shared memory
      m = red[0];
      // largest entry into [1024, 2048): far inside FP16's range, low parts of all but the tiniest entries normal
      int e = 0;
      if (m > 0.f && isfinite(m)) e = 10 - (int)floorf(log2f(m));
      e = e < -24 ? -24 : (e > 24 ? 24 : e);
      const float sc = exp2f((float)e);
      if (job == 0 && tid == 0) {
        p.split_scale[0] = sc;
        p.split_scale[1] = 1.0f / (sc * p.split_h_scale);
      }
      for (int t = job, i = 0; t < n2; t += 8, ++i) write_tile(tile + 32 * i, H, t, p.dst + p.L.off_W2t, 1, sc);
      return;
    }
    job -= 8;
  }
  if (job < n1 || (!SPLIT && job < n1 + n2)) {
    const int layer = job < n1 ? 0 : 1, t = job - layer * n1, K = layer ? H : D;
    load_tile(tile, layer ? W2 : W1, K, t);
    __syncthreads();
    write_tile(tile, K, t, p.dst + (layer ? p.L.off_W2t : p.L.off_W1t), layer, 0.f);
    return;
  }
  job -= n1 + (SPLIT ? 0 : n2);
  // biases and the head, element by element
  int i = job * NT + tid;
  if (i < 2 * Hp) {
    const int n = i < Hp ? i : i - Hp;
    p.dst[(i < Hp ? p.L.off_b1 : p.L.off_b2) + n] = n < H ? (i < Hp ? b1 : b2)[n] : 0.f;
    return;
  }
  i -= 2 * Hp;
  if (i < H * Ap) {
    const int k = i % H, n = i / H;
    float v = n < A ? W3[(size_t)n * H + k] : (p.value_head && n == A ? Wv[k] : 0.f);
    if (p.bf16) v = __uint_as_float(bf16_bits_rne(v) << 16);
    p.dst[p.L.off_W3t + (size_t)k * Ap + n] = v;
    return;
  }
  i -= H * Ap;
  if (i < Ap) {
    p.dst[p.L.off_b3 + i] = i < A ? b3[i] : (p.value_head && i == A ? bv[0] : 0.f);
    return;
  }
  i -= Ap;
  if (p.tc && i < 16 * H) {                        // head of the tensor-core streams: 16 rows x H columns
    const int k = i % H, n = i / H;
    const float v = n < A ? W3[(size_t)n * H + k] : (p.value_head && n == A ? Wv[k] : 0.f);
    const size_t o = (size_t)H * D + (size_t)H * H + core_offset(n, k & ~7, H) + (k & 7);
    p.tc[o] = (uint16_t)bf16_bits_rne(v);
    if (p.tc_pipe) p.tc_pipe[o] = (uint16_t)bf16_bits_rne(v);
  }
}

}  // namespace

cudaError_t launch_publish(const PublishParams& p, cudaStream_t s) {
  const WeightLayout& L = p.L;
  const bool split = p.split != nullptr;
  const int NT = split ? 1024 : 256, KT = NT / 8, row_tiles = (L.Hp + 31) / 32;
  const int n1 = row_tiles * ((L.D + KT - 1) / KT), n2 = row_tiles * ((L.H + KT - 1) / KT);
  const int rest = 2 * L.Hp + L.H * L.Ap + L.Ap + (p.tc ? 16 * L.H : 0), n_rest = (rest + NT - 1) / NT;
  const size_t tile_bytes = (size_t)32 * (KT + 1) * sizeof(float);
  if (!split) return launch_chained(publish_kernel<256, false>, n1 + n2 + n_rest, 256, tile_bytes, s, p);
  const size_t smem = tile_bytes * ((n2 + 7) / 8);       // 33 KB at most (hidden 256)
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at[2];
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 8; at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3((8 + n1 + n_rest + 7) / 8 * 8);
  cfg.blockDim = dim3(1024);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, publish_kernel<1024, true>, p);
}

}  // namespace tj
