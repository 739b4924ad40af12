// Learner update (Algorithm 1: theta <- theta + alpha * delta * grad V(s; theta)) as one minibatch semi-gradient step on
// the mean Huber loss of the TD error, FP32, on parameter blobs in the publish layout
// [W1 H x D, b1, W2 H x H, b2, W3 A x H, b3] (row-major out x in):
//   forward   h1, h2 of the online network kept, q = Q(s, a; theta), q' = max_a Q(s', a; theta_target),
//             delta = r + gamma (1 - done) q' - q, g = -clip(delta, -kappa, kappa) / n  (= dL/dq)
//   backward  dh2 = g W3[a] (h2 > 0), dh1 = (W2^T dh2) (h1 > 0)
//   update    W3[a] -= lr sum_j g_j h2_j, W2 -= lr dh2^T h1, W1 -= lr dh1^T x, biases likewise
// Every sum runs in a fixed order that depends on the shapes alone, so a step is reproducible bit for bit.
#include "tj_async.cuh"
#include "tj_internal.h"
#include "tj_fma.cuh"
#include "tj_tc.cuh"

namespace tj {

namespace {

constexpr int SG_ROWS = 16;       // minibatch rows per loss partial

// ---------------------------------------------------------------------------------------------------------------------
// Wide networks and large minibatches: the layers as tiled FP32 matrix products.  C[m][n] = epi(sum_k A[m][k] Bop[k][n]): A row-major
// M x K.  B_KN false: B is N x K row-major (a weight matrix as the forward pass uses it, Bop = B^T); true: B is K x N row-major (the
// same matrix in the backward pass).
// 64 x 64 tile per block (32 rows where that leaves SMs idle), 32 k per step in one of two stages.  Two groups of 128 threads take
// alternate halves of each step, a thread 8 x 4 outputs (4 x 4 in the 32-row tile) with two rows per instruction, and add their sums
// at the end: a fixed order.  An update has few tiles per SM, so what bounds a tile is latency: one group of four warps with
// 16 k per step waited for shared and global memory two cycles of three (dh1 of
// 4,096 x 256 outputs, K = 256: 23.6 us then, 17.9 now; W2's gradient 28.5 and 19.2; the FMA rate alone allows 7.3).
constexpr int GM_BN = 64, GM_BK = 32, GM_THREADS = 256;
template <int BM>
constexpr int GM_STAGE = GM_BK * (BM + 4 + GM_BN + 4);   // floats of one of the two stages

// acc (RM x 4, two rows per entry) += over K rows of As (RM values) and Bs (4 values), the next row's operands on their way meanwhile
template <int RM, int K, int LDA, int LDB>
__device__ __forceinline__ void multiply_step(const float* As, const float* Bs, f32x2 (&acc)[RM / 2][4]) {
  f32x2 av[2][RM / 2];
  float4 bq[2];
  auto load = [&](int k, f32x2 (&a)[RM / 2], float4& b) {
    if constexpr (RM == 2) {
      a[0] = *reinterpret_cast<const f32x2*>(As + k * LDA);
    } else {
#pragma unroll
      for (int i = 0; i < RM / 4; ++i) {
        const ulonglong2 v = ld_pairs(As + k * LDA + i * 4);
        a[i * 2] = v.x; a[i * 2 + 1] = v.y;
      }
    }
    b = *reinterpret_cast<const float4*>(Bs + k * LDB);
  };
  load(0, av[0], bq[0]);
#pragma unroll
  for (int k = 0; k < K; ++k) {
    if (k + 1 < K) load(k + 1, av[(k + 1) & 1], bq[(k + 1) & 1]);
    const float4 b = bq[k & 1];
    const f32x2 bv[4] = {dup2(b.x), dup2(b.y), dup2(b.z), dup2(b.w)};
#pragma unroll
    for (int i = 0; i < RM / 2; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) fma2(acc[i][j], av[k & 1][i], bv[j]);
  }
}

// four consecutive floats of a row from column c (zero beyond the matrix): a 16-byte load where the row allows it
__device__ __forceinline__ float4 load_row4(const float* base, int ld, int row, int n_rows, int c, int n_cols, bool vec) {
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (row < n_rows && c < n_cols) {
    const float* src = base + (size_t)row * ld + c;
    if (vec && c + 3 < n_cols) {
      v = __ldg(reinterpret_cast<const float4*>(src));
    } else {
      v.x = __ldg(src);
      if (c + 1 < n_cols) v.y = __ldg(src + 1);
      if (c + 2 < n_cols) v.z = __ldg(src + 2);
      if (c + 3 < n_cols) v.w = __ldg(src + 3);
    }
  }
  return v;
}

// One BM x 64 tile over k in [k_begin, k_end).  load_a(r, k) gives A[r][k .. k+3] (A_KM: A[r .. r+3][k]) with r counted from the tile's
// first row, load_b likewise (B_KN: four columns of row k).  This thread's share of the result is out[RM / 2][4]: rows `row0` .. and
// columns `col0` .. of the tile.
// CHAIN: the fixed rounding order of tj_fma.cuh instead, acc = first; acc = fma(A, B, acc) for k = 0, 1, 2, ...  The two groups then
// take half of the rows each over the whole of every step (a third more operand loads per FMA).
template <int BM, bool A_KM, bool B_KN, bool CHAIN, class LoadA, class LoadB>
__device__ __forceinline__ void tile_product(LoadA load_a, LoadB load_b, int k_begin, int k_end, float* sm, const float (&first)[4],
                                             float (&out)[BM / 16][4], int& row0, int& col0) {
  constexpr int RM = CHAIN ? BM / 16 : BM / 8, LDA = BM + 4, LDB = GM_BN + 4, NA = BM * GM_BK / 4 / GM_THREADS,
                NB = GM_BN * GM_BK / 4 / GM_THREADS;
  const int tid = threadIdx.x, kg = tid >> 7, ty = (tid & 127) >> 4, tx = tid & 15;
  row0 = ty * (BM / 8) + kg * (BM / 16);
  col0 = tx * 4;
  f32x2 acc[RM / 2][4];
#pragma unroll
  for (int i = 0; i < RM / 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = CHAIN ? dup2(first[j]) : 0ull;
  // the next step's operands travel from global memory to registers while this one is multiplied.  Piece i of a row-major operand:
  // four k of a row, four pieces (64 bytes) of eight rows per warp; of a k-major one: four columns of row k
  auto piece_r = [](int i, int rows) { return (i >> 2) % rows; };
  auto piece_k = [](int i, int rows) { return (i & 3) * 4 + 16 * (i / (4 * rows)); };
  float4 ra[NA], rb[NB];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int u = 0; u < NA; ++u) {
      const int i = tid + u * GM_THREADS;
      ra[u] = A_KM ? load_a((i % (BM / 4)) * 4, k0 + i / (BM / 4)) : load_a(piece_r(i, BM), k0 + piece_k(i, BM));
    }
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      const int i = tid + u * GM_THREADS;
      rb[u] = B_KN ? load_b((i % 16) * 4, k0 + i / 16) : load_b(piece_r(i, GM_BN), k0 + piece_k(i, GM_BN));
    }
  };
  fetch(k_begin);
  int stage = 0;
#pragma unroll 1
  for (int k0 = k_begin; k0 < k_end; k0 += GM_BK, stage ^= 1) {
    // two stages: whoever writes one has passed the barrier after which nobody reads it
    float* As = sm + stage * GM_STAGE<BM>;
    float* Bs = As + GM_BK * LDA;
    auto put = [](float* dst, int ld, bool km, int r, int k, const float4 v) {
      if (km) {
        *reinterpret_cast<float4*>(dst + k * ld + r) = v;
      } else {
        dst[k * ld + r] = v.x; dst[(k + 1) * ld + r] = v.y; dst[(k + 2) * ld + r] = v.z; dst[(k + 3) * ld + r] = v.w;
      }
    };
#pragma unroll
    for (int u = 0; u < NA; ++u) {
      const int i = tid + u * GM_THREADS;
      if (A_KM) put(As, LDA, true, (i % (BM / 4)) * 4, i / (BM / 4), ra[u]);
      else put(As, LDA, false, piece_r(i, BM), piece_k(i, BM), ra[u]);
    }
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      const int i = tid + u * GM_THREADS;
      if (B_KN) put(Bs, LDB, true, (i % 16) * 4, i / 16, rb[u]);
      else put(Bs, LDB, false, piece_r(i, GM_BN), piece_k(i, GM_BN), rb[u]);
    }
    __syncthreads();
    if (k0 + GM_BK < k_end) fetch(k0 + GM_BK);
    if constexpr (CHAIN) multiply_step<RM, GM_BK, LDA, LDB>(As + row0, Bs + tx * 4, acc);
    else multiply_step<RM, GM_BK / 2, LDA, LDB>(As + kg * (GM_BK / 2) * LDA + ty * RM, Bs + kg * (GM_BK / 2) * LDB + tx * 4, acc);
  }
  if constexpr (CHAIN) {
#pragma unroll
    for (int i = 0; i < RM / 2; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float2 v = halves(acc[i][j]);
        out[2 * i][j] = v.x;
        out[2 * i + 1][j] = v.y;
      }
    return;
  }
  // the groups swap halves of their rows: group 0 finishes the first RM / 2, group 1 the others
  __syncthreads();
  f32x2* mine = reinterpret_cast<f32x2*>(sm) + kg * RM * 128 + (tid & 127);
  const f32x2* theirs = reinterpret_cast<const f32x2*>(sm) + (kg ^ 1) * RM * 128 + (tid & 127);
#pragma unroll
  for (int i = 0; i < RM / 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) mine[(i * 4 + j) * 128] = kg ? acc[i][j] : acc[RM / 4 + i][j];
  __syncthreads();
#pragma unroll
  for (int i = 0; i < RM / 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float2 a = halves(kg ? acc[RM / 4 + i][j] : acc[i][j]), b = halves(theirs[(i * 4 + j) * 128]);
      out[2 * i][j] = a.x + b.x;
      out[2 * i + 1][j] = a.y + b.y;
    }
}

// four consecutive outputs of a row, a 16-byte store where the row allows it
__device__ __forceinline__ void store_row4(float* dst, const float (&v)[4], int left, bool vec) {
  if (vec && left >= 4) {
    *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (j < left) dst[j] = v[j];
  }
}

template <bool B_KN, int EPI, int BM>
__device__ __forceinline__ void sg_gemm_body(const float* __restrict__ A, int lda, const float* __restrict__ B, int ldb,
                                             float* __restrict__ C, int ldc, int M, int N, int K,
                                             const float* __restrict__ bias, const float* __restrict__ mask, int ldm) {
  __shared__ __align__(16) float sm[2 * GM_STAGE<BM>];
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * GM_BN;
  const bool vecA = (lda & 3) == 0 && (reinterpret_cast<uintptr_t>(A) & 15) == 0;
  const bool vecB = (ldb & 3) == 0 && (reinterpret_cast<uintptr_t>(B) & 15) == 0;
  float bv[4] = {0.f, 0.f, 0.f, 0.f};
  auto load_bias = [&](int c) {
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (c + j < N) bv[j] = __ldg(bias + c + j);
  };
  if (EPI == GM_CHAIN_RELU) load_bias(n0 + (int)(threadIdx.x & 15) * 4);
  float out[BM / 16][4];
  int row0, col0;
  tile_product<BM, false, B_KN, EPI == GM_CHAIN_RELU>([&](int r, int k) { return load_row4(A, lda, m0 + r, M, k, K, vecA); },
                                [&](int c, int k) {
                                  return B_KN ? load_row4(B, ldb, k, K, n0 + c, N, vecB) : load_row4(B, ldb, n0 + c, N, k, K, vecB);
                                },
                                0, K, sm, bv, out, row0, col0);
  const int n = n0 + col0;
  if (n >= N) return;
  const bool vecC = (ldc & 3) == 0 && (reinterpret_cast<uintptr_t>(C) & 15) == 0;
  const bool vecM = EPI == GM_MASK && (ldm & 3) == 0 && (reinterpret_cast<uintptr_t>(mask) & 15) == 0;
  if (EPI == GM_BIAS_RELU || EPI == GM_BIAS) load_bias(n);
#pragma unroll
  for (int i = 0; i < BM / 16; ++i) {
    const int m = m0 + row0 + i;
    if (m >= M) break;
    if (EPI == GM_MASK) {
      const float4 h = load_row4(mask, ldm, m, M, n, N, vecM);
      out[i][0] = h.x > 0.f ? out[i][0] : 0.f; out[i][1] = h.y > 0.f ? out[i][1] : 0.f;
      out[i][2] = h.z > 0.f ? out[i][2] : 0.f; out[i][3] = h.w > 0.f ? out[i][3] : 0.f;
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        out[i][j] = EPI == GM_CHAIN_RELU ? relu1(out[i][j]) : (EPI == GM_BIAS_RELU ? fmaxf(out[i][j] + bv[j], 0.f) : out[i][j] + bv[j]);
    }
    store_row4(C + (size_t)m * ldc + n, out[i], N - n, vecC);
  }
}

// one product, or the same product for two operand sets of one shape (the two networks): blockIdx.z picks the set
struct GemmPair { const float* A[2]; const float* B[2]; float* C[2]; const float* bias[2]; };
template <bool B_KN, int EPI, int BM>
__global__ void __launch_bounds__(GM_THREADS) sg_gemm_kernel(const GemmPair pr, int lda, int ldb, int ldc, int M, int N, int K,
                                                             const float* __restrict__ mask, int ldm) {
  chain_begin();
  const bool z = blockIdx.z != 0;
  sg_gemm_body<B_KN, EPI, BM>(z ? pr.A[1] : pr.A[0], lda, z ? pr.B[1] : pr.B[0], ldb, z ? pr.C[1] : pr.C[0], ldc, M, N, K,
                              z ? pr.bias[1] : pr.bias[0], mask, ldm);
}

// The heads of both networks for wide hidden layers: out[row][a] = bias[a] + sum_k h[row][k] W[a][k], a < A <= 16, H a
// multiple of 128.  A 32-row FMA tile pads the few outputs to 64 columns and pays a block barrier per 16 k; here a warp takes
// four rows at a time: lane l reads the 16-byte pieces l, l + 32, ... of the rows (coalesced), multiplies them with the head's
// weights (in shared memory, laid out so that consecutive lanes read consecutive 16-byte words) into 16 partial outputs per row, and
// the 16 x 32 partials of a row are summed by a fixed halving exchange (16 shuffles).  blockIdx.y picks the network.  Row by row the
// weights' way out of shared memory was the bound (2 x 8,192 rows x 512: 26.4 us, 18.3 with four rows per read of them).
constexpr int HD_ROWS = 64, HD_R = 4;   // rows per block: eight per warp, four at a time
__global__ void __launch_bounds__(256) sg_heads_kernel(const GemmPair pr, int n_rows, int H, int A, int ldc) {
  extern __shared__ __align__(16) float4 hd_w[];       // [(j * 4 + kk) * 4 + aq][lane]: W[aq * 4 .. + 3][4 (32 j + lane) + kk]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool z = blockIdx.y != 0;
  const float* __restrict__ W = z ? pr.B[1] : pr.B[0];
  const float* __restrict__ hrows = z ? pr.A[1] : pr.A[0];
  const float* __restrict__ bias = z ? pr.bias[1] : pr.bias[0];
  float* __restrict__ out = z ? pr.C[1] : pr.C[0];
  const int nj = H / 128;
  chain_begin();
  // row a of the head, four columns per thread, into component a % 4 of its four words
  const bool vecW = (reinterpret_cast<uintptr_t>(W) & 15) == 0;
  for (int i = tid; i < 16 * 32 * nj; i += blockDim.x) {
    const int a = i / (32 * nj), q = i % (32 * nj);
    float4 w = make_float4(0.f, 0.f, 0.f, 0.f);
    if (a < A) {
      const float* src = W + (size_t)a * H + 4 * q;
      w = vecW ? __ldg(reinterpret_cast<const float4*>(src)) : make_float4(__ldg(src), __ldg(src + 1), __ldg(src + 2), __ldg(src + 3));
    }
    float* d = reinterpret_cast<float*>(hd_w + ((q >> 5) * 16 + (a >> 2)) * 32 + (q & 31)) + (a & 3);
    d[0] = w.x; d[4 * 128] = w.y; d[8 * 128] = w.z; d[12 * 128] = w.w;
  }
  __syncthreads();
  const int a_mine = ((lane >> 4) & 1) * 8 + ((lane >> 3) & 1) * 4 + ((lane >> 2) & 1) * 2 + ((lane >> 1) & 1);
  const float b_mine = a_mine < A ? bias[a_mine] : 0.f;
#pragma unroll 1
  for (int r = warp * HD_R; r < HD_ROWS; r += 8 * HD_R) {
    const int row = blockIdx.x * HD_ROWS + r;
    if (row >= n_rows) break;
    f32x2 v2[HD_R][8];
#pragma unroll
    for (int q = 0; q < HD_R; ++q)
#pragma unroll
      for (int i = 0; i < 8; ++i) v2[q][i] = 0ull;
    auto piece = [&](int q, int j) {                       // a row beyond the last reads the last one again and is not stored
      const int rq = row + q < n_rows ? row + q : n_rows - 1;
      return __ldg(reinterpret_cast<const float4*>(hrows + (size_t)rq * H) + 32 * j + lane);
    };
    float4 x[HD_R];
#pragma unroll
    for (int q = 0; q < HD_R; ++q) x[q] = piece(q, 0);
#pragma unroll 1
    for (int j = 0; j < nj; ++j) {
      float4 xn[HD_R];
#pragma unroll
      for (int q = 0; q < HD_R; ++q) xn[q] = piece(q, j + 1 < nj ? j + 1 : j);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        f32x2 xs[HD_R];
#pragma unroll
        for (int q = 0; q < HD_R; ++q) xs[q] = dup2(kk == 0 ? x[q].x : kk == 1 ? x[q].y : kk == 2 ? x[q].z : x[q].w);
#pragma unroll
        for (int aq = 0; aq < 4; ++aq) {
          const ulonglong2 w = ld_pairs(reinterpret_cast<const float*>(hd_w + ((j * 4 + kk) * 4 + aq) * 32 + lane));
#pragma unroll
          for (int q = 0; q < HD_R; ++q) {
            fma2(v2[q][2 * aq], xs[q], w.x);
            fma2(v2[q][2 * aq + 1], xs[q], w.y);
          }
        }
      }
#pragma unroll
      for (int q = 0; q < HD_R; ++q) x[q] = xn[q];
    }
#pragma unroll
    for (int q = 0; q < HD_R; ++q) {
      float v[16];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float2 h = halves(v2[q][i]);
        v[2 * i] = h.x;
        v[2 * i + 1] = h.y;
      }
      // halving exchange: after the step with distance d a lane keeps the half of its values that its bit d selects
#define TJ_HD_STEP(D, CNT)                                                                     \
      {                                                                                           \
        const bool upper = (lane & (D)) != 0;                                                     \
        _Pragma("unroll") for (int i = 0; i < (CNT); ++i) {                                       \
          const float keep = upper ? v[i + (CNT)] : v[i], send = upper ? v[i] : v[i + (CNT)];    \
          v[i] = keep + __shfl_xor_sync(0xffffffffu, send, (D));                                 \
        }                                                                                         \
      }
      TJ_HD_STEP(16, 8)
      TJ_HD_STEP(8, 4)
      TJ_HD_STEP(4, 2)
      TJ_HD_STEP(2, 1)
#undef TJ_HD_STEP
      const float total = v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
      if (row + q < n_rows && (lane & 1) == 0 && a_mine < A) out[(size_t)(row + q) * ldc + a_mine] = total + b_mine;
    }
  }
}

// Tile height: 64 rows if that gives every SM a block, else 32 (a product that has too few tiles even so is bound by its chain
// of k-steps).
template <bool B_KN, int EPI>
cudaError_t sg_gemm(const SgdParams& p, const GemmPair& pr, int sets, int lda, int ldb, int ldc, int M, int N, int K, const float* mask, int ldm,
                    cudaStream_t s) {
  const int cols = (N + GM_BN - 1) / GM_BN, sms = p.sm_count > 0 ? p.sm_count : 148;
  ++*p.launches;
  auto go = [&](auto kernel, int bm) {
    return launch_chained(kernel, dim3(cols, (M + bm - 1) / bm, sets), GM_THREADS, 0, s, pr, lda, ldb, ldc, M, N, K, mask, ldm);
  };
  if ((long long)cols * ((M + 63) / 64) * sets >= sms) return go(sg_gemm_kernel<B_KN, EPI, 64>, 64);
  return go(sg_gemm_kernel<B_KN, EPI, 32>, 32);
}

// ---------------------------------------------------------------------------------------------------------------------
// The same product on the tensor cores, FP32-faithful: every operand is split into a TF32 high part (the top 19 bits) and
// the remainder, and C accumulates A_hi B_hi + A_lo B_hi + A_hi B_lo in FP32 (the dropped A_lo B_lo term is 2^-22 of the
// product, and the tensor core reads each remainder with 11 significant bits: another 2^-22 each).  A: M x K row-major, B: N x K row-major (a weight matrix as the forward pass uses it), K a multiple of 4, rows
// 16-byte aligned.  One 128 x 128 tile per block, accumulator in tensor memory (128 columns); per step of 16 k the
// threads split the step's operands into one of two shared-memory stages (K-major core matrices of 8 rows x 16 bytes)
// while the tensor core works on the other, and the operands of the following TG_PF steps are on their way from global
// memory to registers.  65 KB of shared memory: two blocks per SM cover each other's waits.
constexpr int TG_M = 128, TG_N = 128, TG_K = 16, TG_THREADS = 256, TG_PF = 3;
constexpr int TG_OPER_BYTES = TG_M * TG_K * 4;            // one operand part of one stage: 8 KB
constexpr int TG_STAGE_BYTES = 4 * TG_OPER_BYTES;         // A_hi | A_lo | B_hi | B_lo
constexpr int TG_SMEM_BYTES = 2 * TG_STAGE_BYTES + 1024;  // + alignment slack

template <int EPI>
__global__ void __launch_bounds__(TG_THREADS, 2) sg_gemm_tc_kernel(const float* __restrict__ A, int lda, const float* __restrict__ B,
                                                                   int ldb, float* __restrict__ C, int ldc, int M, int N, int K,
                                                                   const float* __restrict__ bias, const float* __restrict__ mask,
                                                                   int ldm, const UpdateWatch watch) {
  extern __shared__ uint8_t tg_raw[];
  uint8_t* stage0 = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(tg_raw) + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t done[2];
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = blockIdx.y * TG_M, n0 = blockIdx.x * TG_N;
  if (tid == 0) {
    mbar_init(&done[0], 1);
    mbar_init(&done[1], 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tmem_base)), "r"(128u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;
  chain_begin();

  // loader mapping: a warp instruction covers eight rows x four 16-byte pieces (64 contiguous bytes per row); warp w
  // owns rows 16 w .. 16 w + 15 of both operands' tiles, a thread two pieces of each
  static_assert(TG_K == 16, "the loader maps four 16-byte pieces to a row");
  const int r8 = lane >> 2, kq = lane & 3;
  // TG_PF register sets: the operands of the next TG_PF steps are in flight from global memory at any time
  float4 ra[TG_PF][2], rb[TG_PF][2];
  auto fetch = [&](int k0, float4 (&fa)[2], float4 (&fb)[2]) {
    const int k = k0 + kq * 4;
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      const int rr = warp * 16 + g * 8 + r8;
      fa[g] = (m0 + rr < M && k < K) ? __ldg(reinterpret_cast<const float4*>(A + (size_t)(m0 + rr) * lda + k)) : make_float4(0.f, 0.f, 0.f, 0.f);
      fb[g] = (n0 + rr < N && k < K) ? __ldg(reinterpret_cast<const float4*>(B + (size_t)(n0 + rr) * ldb + k)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  auto split_store = [](uint8_t* hi_dst, uint8_t* lo_dst, const float4 v) {
    float4 hi, lo;
    hi.x = __uint_as_float(__float_as_uint(v.x) & 0xFFFFE000u); lo.x = v.x - hi.x;
    hi.y = __uint_as_float(__float_as_uint(v.y) & 0xFFFFE000u); lo.y = v.y - hi.y;
    hi.z = __uint_as_float(__float_as_uint(v.z) & 0xFFFFE000u); lo.z = v.z - hi.z;
    hi.w = __uint_as_float(__float_as_uint(v.w) & 0xFFFFE000u); lo.w = v.w - hi.w;
    *reinterpret_cast<float4*>(hi_dst) = hi;
    *reinterpret_cast<float4*>(lo_dst) = lo;
  };
  const int nk = (K + TG_K - 1) / TG_K;
  const uint32_t idesc = make_idesc_tf32(TG_N);
  constexpr uint32_t SBO = (TG_K / 4) * 128u;     // eight rows further: one row group of K/4 core matrices
  bool ok = true;
  int issued = 0;                                 // steps whose products the tensor core has been given
  // one step: registers -> split -> stage i & 1, the tensor core's products on it, the load of step i + TG_PF.  Returns
  // false (for every thread alike) when a wait ran out.
  auto step = [&](int i, float4 (&fa)[2], float4 (&fb)[2]) -> bool {
    const int s = i & 1;
    uint8_t* st = stage0 + (size_t)s * TG_STAGE_BYTES;
    // the tensor core must be done with this stage (its use two steps ago).  One warp polls the barrier, the others
    // sleep at the block barrier: polls from every warp would take shared-memory cycles from the tensor core, whose
    // TF32 operand reads (8 KB per instruction) already need most of them
    if (i >= 2) {
      if (warp == 1) ok = tc_wait_elect(&done[s], (uint32_t)(((i >> 1) - 1) & 1), &abort_flag);
      if (__syncthreads_or(!ok)) return false;
    }
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      const int rr = warp * 16 + g * 8 + r8;
      const size_t off = (size_t)(rr >> 3) * SBO + (size_t)(rr & 7) * 16 + (size_t)kq * 128;
      split_store(st + off, st + TG_OPER_BYTES + off, fa[g]);
      split_store(st + 2 * TG_OPER_BYTES + off, st + 3 * TG_OPER_BYTES + off, fb[g]);
    }
    fence_async_smem();
    __syncthreads();
    if (tid == 0) {
      tc_fence_after();
      const uint32_t a_hi = smem_addr(st), a_lo = a_hi + TG_OPER_BYTES, b_hi = a_hi + 2 * TG_OPER_BYTES, b_lo = a_hi + 3 * TG_OPER_BYTES;
#pragma unroll
      for (int j = 0; j < TG_K / 8; ++j) {
        const uint32_t o = (uint32_t)j * 256u;
        umma_tf32(tmem, make_desc(a_hi + o, 128u, SBO), make_desc(b_hi + o, 128u, SBO), idesc, (i | j) != 0, 1u);
        umma_tf32(tmem, make_desc(a_lo + o, 128u, SBO), make_desc(b_hi + o, 128u, SBO), idesc, true, 1u);
        umma_tf32(tmem, make_desc(a_hi + o, 128u, SBO), make_desc(b_lo + o, 128u, SBO), idesc, true, 1u);
      }
      umma_commit(&done[s], 1u);
    }
    issued = i + 1;
    if (i + TG_PF < nk) fetch((i + TG_PF) * TG_K, fa, fb);
    return true;
  };
#pragma unroll
  for (int pf = 0; pf < TG_PF; ++pf)
    if (pf < nk) fetch(pf * TG_K, ra[pf], rb[pf]);
  bool running = true;
  for (int i = 0; i < nk && running; i += TG_PF) {
#pragma unroll
    for (int pf = 0; pf < TG_PF; ++pf)
      if (running && i + pf < nk) running = step(i + pf, ra[pf], rb[pf]);
  }
  // every product is complete once the last commit has arrived (a commit covers all earlier ones of its thread)
  if (running && warp == 1) ok = tc_wait_elect(&done[(nk - 1) & 1], (uint32_t)(((nk - 1) >> 1) & 1), &abort_flag);
  ok = !__syncthreads_or(!ok || !running);
  if (ok) {
    tc_fence_after();
    const int q = warp & 3, hsel = warp >> 2;      // TMEM lane quarter of this warp, column half
    const int m = m0 + q * 32 + lane;
    const uint32_t t_acc = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(hsel * 64);
    uint32_t v[64];
#pragma unroll
    for (int g = 0; g < 4; ++g) tmem_ld16(t_acc + (uint32_t)(g * 16), v + 16 * g);
    tmem_ld_wait();
    if (m < M) {
      const bool vec = (ldc & 3) == 0 && (reinterpret_cast<uintptr_t>(C) & 15) == 0;
#pragma unroll
      for (int c4 = 0; c4 < 16; ++c4) {
        const int n = n0 + hsel * 64 + c4 * 4;
        if (n >= N) break;
        float o[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float x = __uint_as_float(v[c4 * 4 + j]);
          if (n + j < N) {
            if (EPI == GM_BIAS_RELU) x = fmaxf(x + __ldg(bias + n + j), 0.f);
            else if (EPI == GM_BIAS) x = x + __ldg(bias + n + j);
            else x = __ldg(mask + (size_t)m * ldm + n + j) > 0.f ? x : 0.f;
          }
          o[j] = x;
        }
        float* dst = C + (size_t)m * ldc + n;
        if (vec && n + 3 < N) {
          *reinterpret_cast<float4*>(dst) = make_float4(o[0], o[1], o[2], o[3]);
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (n + j < N) dst[j] = o[j];
        }
      }
    }
  } else if (tid == 0) {
    update_failed(watch);
    for (int i = issued > 2 ? issued - 2 : 0; i < issued; ++i) mbar_settle(&done[i & 1], (uint32_t)((i >> 1) & 1));
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(128u) : "memory");
}

// dst[c][r] = src[r][c] for an n x n matrix (32 x 32 tiles through shared memory, both sides coalesced)
__global__ void __launch_bounds__(256) sg_transpose_kernel(const float* __restrict__ src, float* __restrict__ dst, int n) {
  chain_begin();
  __shared__ float tile[32][33];
  const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int i = ty; i < 32; i += 8)
    if (r0 + i < n && c0 + tx < n) tile[i][tx] = src[(size_t)(r0 + i) * n + c0 + tx];
  __syncthreads();
  for (int i = ty; i < 32; i += 8)
    if (c0 + i < n && r0 + tx < n) dst[(size_t)(c0 + i) * n + r0 + tx] = tile[tx][i];
}

// Shapes the tensor-core product takes: 16-byte rows on both operands and enough 128 x 128 tiles to occupy most SMs (with
// fewer, the FMA tiles spread the work over more blocks and finish sooner).  The 96 were measured against 128 x 64 FMA tiles; against
// the present ones the line lies higher.  Whole tj_sgd_step, us, on the tensor cores / FMA tiles: 32 inputs, hidden 384: 96 tiles
// 203 / 177, 192 336 / 322, 384 657 / 618, 768 1,117 / 1,217; 4 inputs, hidden 256: 64 tiles 123 / 86, 128 150 / 147, 256 253 / 270,
// 512 520 / 559; 32 inputs, hidden 700: 384 tiles 961 / 1,002.
static bool tc_gemm_ok(const float* A, int lda, const float* B, int ldb, int M, int N, int K) {
  const long long tiles = (long long)((M + TG_M - 1) / TG_M) * ((N + TG_N - 1) / TG_N);
  return (K & 3) == 0 && (lda & 3) == 0 && (ldb & 3) == 0 && (reinterpret_cast<uintptr_t>(A) & 15) == 0 &&
         (reinterpret_cast<uintptr_t>(B) & 15) == 0 && K >= 32 && tiles >= 96;
}

// forward-layout products (B is N x K) of both sets: tensor cores where the shape allows, the FMA tiles otherwise
template <int EPI>
cudaError_t sg_layer(const SgdParams& p, const GemmPair& pr, int sets, int lda, int ldb, int ldc, int M, int N, int K, const float* mask, int ldm,
                     cudaStream_t s) {
  bool tc = N >= 128;
  for (int z = 0; z < sets; ++z) tc = tc && tc_gemm_ok(pr.A[z], lda, pr.B[z], ldb, M, N, K);
  if (!tc) return sg_gemm<false, EPI>(p, pr, sets, lda, ldb, ldc, M, N, K, mask, ldm, s);
  for (int z = 0; z < sets; ++z) {
    ++*p.launches;
    const cudaError_t e = launch_chained<1024>(sg_gemm_tc_kernel<EPI>, dim3((N + TG_N - 1) / TG_N, (M + TG_M - 1) / TG_M), TG_THREADS, TG_SMEM_BYTES, s, pr.A[z],
                                         lda, pr.B[z], ldb, pr.C[z], ldc, M, N, K, pr.bias[z], mask, ldm, p.watch);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Heads, loss, its gradient at the outputs and dh2 for at most four outputs, a warp per minibatch row: the row of h2 (and of the target
// network's) against the few head rows, summed by shuffles; then dh2[i] = sum_a g[a] W3[a][i] (+ g[A] Wv[i]) where h2[i] > 0, the row
// still in L1.  Bound by reading h2 twice and writing dh2 (as a 32-row product tile per head, a loss kernel and a product with K = A
// this was four launches and 37 us for 4,096 rows x 256 units).  Loss partials per SG_ROWS rows.
template <bool PPO>
__global__ void __launch_bounds__(32 * SG_ROWS) sgd_rows_kernel(const SgdParams p, const float* t2) {
  __shared__ float part[5][SG_ROWS];
  chain_begin();
  const int H = p.H, D = p.D, A = p.A, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float *W3 = p.theta + (size_t)H * D + H + (size_t)H * H + H, *b3 = W3 + (size_t)A * H, *Wv = b3 + A;
  const float *T3 = p.theta_target + (size_t)H * D + H + (size_t)H * H + H, *tb3 = T3 + (size_t)A * H;
  {
    const int r = warp, j = blockIdx.x * SG_ROWS + r;
    float l[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
    if (j < p.n) {
      const float* h = p.h2 + (size_t)j * H;
      const float* t = PPO ? h : t2 + (size_t)j * H;
      const int act0 = p.act[j], act = act0 < 0 ? 0 : (act0 >= A ? A - 1 : act0);
      const float s0 = PPO ? p.logp_old[j] : p.rew[j], s1 = PPO ? p.adv[j] : 0.f, s2 = PPO ? p.ret[j] : 0.f;
      const int dn = PPO ? 0 : p.done[j];
      float q[4] = {0.f, 0.f, 0.f, 0.f}, qt[4] = {0.f, 0.f, 0.f, 0.f};
      for (int i = lane; i < H; i += 32) {
        const float x = h[i], y = PPO ? 0.f : t[i];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          if (a < A) {
            q[a] = fmaf(x, __ldg(W3 + a * H + i), q[a]);
            if (!PPO) qt[a] = fmaf(y, __ldg(T3 + a * H + i), qt[a]);
          } else if (PPO && a == A) {
            q[a] = fmaf(x, __ldg(Wv + i), q[a]);
          }
        }
      }
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        for (int o = 16; o > 0; o >>= 1) {
          q[a] += __shfl_xor_sync(0xffffffffu, q[a], o);
          if (!PPO) qt[a] += __shfl_xor_sync(0xffffffffu, qt[a], o);
        }
        if (a < A) {
          q[a] += __ldg(b3 + a);
          if (!PPO) qt[a] += __ldg(tb3 + a);
        } else if (PPO && a == A) {
          q[a] += __ldg(Wv + H);
        }
      }
      float g[4] = {0.f, 0.f, 0.f, 0.f};
      if (PPO) {
        float lmax = q[0];
#pragma unroll
        for (int a = 1; a < 4; ++a)
          if (a < A) lmax = fmaxf(lmax, q[a]);
        float Z = 0.f, ent = 0.f, logp = 0.f, val = 0.f;
#pragma unroll
        for (int a = 0; a < 4; ++a)
          if (a < A) Z += expf(q[a] - lmax);
        const float logZ = lmax + logf(Z);
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          if (a < A) {
            const float lp = q[a] - logZ;
            ent -= expf(lp) * lp;
            if (a == act) logp = lp;
          } else if (a == A) {
            val = q[a];
          }
        }
        const float ratio = expf(logp - s0);
        const float rc = fminf(fmaxf(ratio, 1.f - p.clip_eps), 1.f + p.clip_eps);
        const float t1 = ratio * s1, t3 = rc * s1;
        const bool unclipped = t1 <= t3;
        const float dv = val - s2, inv_n = 1.f / (float)p.n, g_logp = unclipped ? -s1 * ratio : 0.f;
        l[1] = -(unclipped ? t1 : t3);
        l[2] = 0.5f * dv * dv;
        l[3] = ent;
        l[4] = unclipped ? 0.f : 1.f;
        l[0] = l[1] + p.c_v * l[2] - p.c_e * l[3];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          if (a < A) {
            const float lp = q[a] - logZ, pi = expf(lp);
            const float dlogp = (a == act ? 1.f : 0.f) - pi, dent = -pi * (lp + ent);
            g[a] = (g_logp * dlogp - p.c_e * dent) * inv_n;
          } else if (a == A) {
            g[a] = p.c_v * dv * inv_n;
          }
        }
      } else {
        float qmax = qt[0], qs = 0.f;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          if (a > 0 && a < A) qmax = fmaxf(qmax, qt[a]);
          if (a == act) qs = q[a];
        }
        const float delta = s0 + p.gamma * (dn ? 0.f : 1.f) * qmax - qs, ad = fabsf(delta);
        l[0] = ad <= p.kappa ? 0.5f * delta * delta : p.kappa * (ad - 0.5f * p.kappa);
        const float gj = -fminf(fmaxf(delta, -p.kappa), p.kappa) / (float)p.n;
#pragma unroll
        for (int a = 0; a < 4; ++a) g[a] = a == act ? gj : 0.f;
      }
      if (lane == 0) {
        float* gr = p.g + (size_t)j * p.ldg;
#pragma unroll
        for (int a = 0; a < 4; ++a)
          if (a < p.ldg) gr[a] = g[a];
      }
      float* d = p.dh2 + (size_t)j * H;            // for the Q head t2 is this very row: every lane has read its entries above
      __syncwarp();
      for (int i = lane; i < H; i += 32) {
        float v = 0.f;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          if (a < A) v = fmaf(g[a], __ldg(W3 + a * H + i), v);
          else if (PPO && a == A) v = fmaf(g[a], __ldg(Wv + i), v);
        }
        d[i] = h[i] > 0.f ? v : 0.f;
      }
    }
    if (lane == 0)
#pragma unroll
      for (int k = 0; k < (PPO ? 5 : 1); ++k) part[k][r] = l[k];
  }
  __syncthreads();
  if (threadIdx.x < (PPO ? 5 : 1)) {
    float s = 0.f;
    for (int r = 0; r < SG_ROWS; ++r) s += part[threadIdx.x][r];
    if (PPO) p.stat_partial[(size_t)blockIdx.x * 5 + threadIdx.x] = s;
    else p.partial[blockIdx.x] = s;
  }
}

// TD error from both networks' second layers for at most four outputs, every sum in the order of td_kernel: lane a of a group of four
// sums output a of one (network, row) over k = 0, 1, 2, ..., with the block's rows of both layers and the heads' rows in shared memory;
// the loss partials cover the rows of one of td_kernel's tiles, added in row order.
struct TrLayout { int ldh, h, w3, q, hub, total; };       // row stride; offsets, floats: rows [2][rows], heads [2][4], outputs [2][rows][4]
__host__ __device__ inline TrLayout tr_layout(int H, int rows) {
  TrLayout L;
  L.ldh = 4 * (((H + 3) / 4) | 1);
  L.h = 0;
  L.w3 = 2 * rows * L.ldh;
  L.q = L.w3 + 8 * L.ldh;
  L.hub = L.q + 8 * rows;
  L.total = L.hub + rows;
  return L;
}
constexpr int TR_NT = 256;
__global__ void __launch_bounds__(TR_NT) td_rows_kernel(const TdParams p, const float* __restrict__ h2, const float* __restrict__ t2, int rows) {
  extern __shared__ __align__(16) float tr_sm[];
  chain_begin();
  const TrLayout L = tr_layout(p.H, rows);
  float* sm = tr_sm;
  const int tid = threadIdx.x, j0 = blockIdx.x * rows, here = min(rows, p.n - j0), H = p.H, Hq = 4 * ((H + 3) / 4);
  int act = 0, done = 0;
  float rew = 0.f;
  if (tid < here) { act = p.act[j0 + tid]; rew = p.rew[j0 + tid]; done = p.done[j0 + tid]; }
  // a warp per row: its units, then zeros up to a whole word, every copy of the block in flight at once (4,096 x 256: 10 us as a loop of
  // loads, 6 so; 2,048 x 200: 19 and 6).  Rows beyond the last are computed from what lies there and not used
  const bool vec = (H & 3) == 0 && (reinterpret_cast<uintptr_t>(h2) & 15) == 0 && (reinterpret_cast<uintptr_t>(t2) & 15) == 0;
  for (int s = tid >> 5; s < 2 * rows; s += TR_NT / 32) {
    const int net = s >= rows ? 1 : 0, r = s - net * rows, lane = tid & 31;
    if (r >= here) continue;
    const float* src = (net ? t2 : h2) + (size_t)(j0 + r) * H;
    float* dst = sm + L.h + s * L.ldh;
    if (vec) {
      for (int k = 4 * lane; k < H; k += 128) cp_async16(dst + k, src + k);
    } else {
      for (int k = lane; k < H; k += 32) cp_async4(dst + k, src + k);
      if (lane < Hq - H) dst[H + lane] = 0.f;
    }
  }
  cp_async_commit();
#pragma unroll 2
  for (int i = tid; i < 2 * Hq; i += TR_NT) {                    // W3 [H][4] as publish lays it out -> a row per output
    const int net = i >= Hq ? 1 : 0, k = i - net * Hq;
    float4 w = make_float4(0.f, 0.f, 0.f, 0.f);
    if (k < H) w = __ldg(reinterpret_cast<const float4*>((net ? p.Wtarget : p.Wonline) + p.off_W3t) + k);
    float* d = sm + L.w3 + net * 4 * L.ldh + k;
    d[0] = w.x; d[L.ldh] = w.y; d[2 * L.ldh] = w.z; d[3 * L.ldh] = w.w;
  }
  cp_async_wait<0>();
  __syncthreads();
  for (int g = tid; g < 8 * rows; g += TR_NT) {
    const int a = g & 3, s = g >> 2, net = s >= rows ? 1 : 0;
    sm[L.q + g] = fma_head<4>(__ldg((net ? p.Wtarget : p.Wonline) + p.off_b3 + a), sm + L.w3 + (net * 4 + a) * L.ldh, sm + L.h + s * L.ldh, Hq / 4);
  }
  __syncthreads();
  if (tid < here) {
    act = act < 0 ? 0 : (act >= p.A ? p.A - 1 : act);
    const float* qt = sm + L.q + 4 * (rows + tid);
    float qmax = qt[0];
    for (int i = 1; i < p.A; ++i) qmax = fmaxf(qmax, qt[i]);
    const float y = rew + p.gamma * (done ? 0.f : 1.f) * qmax;
    const float delta = y - sm[L.q + 4 * tid + act], ad = fabsf(delta);
    const float l = ad <= p.kappa ? 0.5f * delta * delta : p.kappa * (ad - 0.5f * p.kappa);
    if (p.td_out) p.td_out[j0 + tid] = delta;
    if (p.huber_out) p.huber_out[j0 + tid] = l;
    sm[L.hub + tid] = l;
  }
  __syncthreads();
  if (tid == 0) {
    float s = 0.f;
    for (int r = 0; r < here; ++r) s += sm[L.hub + r];
    p.partial[blockIdx.x] = s;
  }
}

// The same from Q values that other kernels computed, for more outputs: q (in) and g (out) share p.g ([n][A], a row is read before its
// own warp overwrites it), qt [n][A]; dh2 has one term per entry, the selected action's.  A row is a chain of round trips (action, its
// q, h2), so it loads what it can before the first of them: all of an h2 row in registers where 16-byte pieces of 512 units suffice
// (8,192 x 512: 6.6 us; 21 with scalar loads in the loop and two rows per warp).
__global__ void __launch_bounds__(32 * SG_ROWS) sgd_loss_kernel(const SgdParams p) {
  __shared__ float part[SG_ROWS];
  chain_begin();
  const int H = p.H, D = p.D, A = p.A, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, j = blockIdx.x * SG_ROWS + warp;
  const float* W3 = p.theta + (size_t)H * D + H + (size_t)H * H + H;
  float l = 0.f;
  if (j < p.n) {
    const float* h = p.h2 + (size_t)j * H;
    float* d = p.dh2 + (size_t)j * H;
    const bool in_regs = (H & 3) == 0 && H <= 512;
    float4 hv[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (in_regs && 4 * (lane + 32 * u) < H) hv[u] = *reinterpret_cast<const float4*>(h + 4 * (lane + 32 * u));
    const int act0 = p.act[j], act = act0 < 0 ? 0 : (act0 >= A ? A - 1 : act0);
    float* gr = p.g + (size_t)j * A;
    const float* tr = p.qt + (size_t)j * A;
    const float q_all = lane < A ? gr[lane] : 0.f, rew = p.rew[j];                // A <= 16 outputs
    const int dn = p.done[j];
    float qmax = lane < A ? tr[lane] : -INFINITY;
    for (int o = 16; o > 0; o >>= 1) qmax = fmaxf(qmax, __shfl_xor_sync(0xffffffffu, qmax, o));
    const float delta = rew + p.gamma * (dn ? 0.f : 1.f) * qmax - __shfl_sync(0xffffffffu, q_all, act), ad = fabsf(delta);
    l = ad <= p.kappa ? 0.5f * delta * delta : p.kappa * (ad - 0.5f * p.kappa);
    const float gj = -fminf(fmaxf(delta, -p.kappa), p.kappa) / (float)p.n;
    if (lane < A) gr[lane] = lane == act ? gj : 0.f;
    const float* w = W3 + (size_t)act * H;
    if (in_regs) {
      const bool vecW = (reinterpret_cast<uintptr_t>(w) & 15) == 0;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = 4 * (lane + 32 * u);
        if (i < H) {
          float4 wv;
          if (vecW) wv = __ldg(reinterpret_cast<const float4*>(w + i));
          else wv = make_float4(__ldg(w + i), __ldg(w + i + 1), __ldg(w + i + 2), __ldg(w + i + 3));
          *reinterpret_cast<float4*>(d + i) = make_float4(hv[u].x > 0.f ? gj * wv.x : 0.f, hv[u].y > 0.f ? gj * wv.y : 0.f,
                                                          hv[u].z > 0.f ? gj * wv.z : 0.f, hv[u].w > 0.f ? gj * wv.w : 0.f);
        }
      }
    } else {
      for (int i = lane; i < H; i += 32) d[i] = h[i] > 0.f ? gj * __ldg(w + i) : 0.f;
    }
  }
  if (lane == 0) part[warp] = l;
  __syncthreads();
  if (threadIdx.x == 0) {
    float s = 0.f;
    for (int r = 0; r < SG_ROWS; ++r) s += part[r];
    p.partial[blockIdx.x] = s;
  }
}

// out[k] = (sum over the blocks of partial k) / n, k = 0..4: a warp per statistic, a fixed tree
__global__ void __launch_bounds__(160) ppo_finish_kernel(const float* __restrict__ stat_partial, int n_blocks, int n, float* __restrict__ out) {
  chain_begin();
  chain_next();
  const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float s = 0.f;
  for (int b = lane; b < n_blocks; b += 32) s += stat_partial[(size_t)b * 5 + k];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) out[k] = s / (float)n;
}

// One gradient product of the update: C (M x N, at float offset `off` of the parameter blob) gets (Am rows)^T (Bm rows),
// a bias (Bm == nullptr) a column of ones.  Tiles of all products are numbered in one list: tile_begin is this product's
// first tile.
struct GradProduct {
  const float* Am;
  const float* Bm;
  int off, M, N, lda, ldb, tile_begin;
};
struct GradProducts {
  GradProduct g[8];
  int n, n_tiles;
};

constexpr int GP_TILE = 64;   // rows and columns of a gradient tile

// One tile of one gradient product over one range of minibatch rows
__device__ __forceinline__ void grad_tile(float* __restrict__ P, const GradProduct& d, int t, int count, int n_rows, int rows_per_range,
                                          float* __restrict__ sm) {
  const int M = d.M, N = d.N, lda = d.lda, ldb = d.ldb;
  const float* __restrict__ Am = d.Am;
  const float* __restrict__ Bm = d.Bm;
  const int tiles_n = (N + GP_TILE - 1) / GP_TILE;
  const int m0 = (t / tiles_n) * GP_TILE, n0 = (t % tiles_n) * GP_TILE;
  const int j_begin = blockIdx.y * rows_per_range;
  const int j_end = j_begin + rows_per_range < n_rows ? j_begin + rows_per_range : n_rows;
  const bool vecA = (lda & 3) == 0 && (reinterpret_cast<uintptr_t>(Am) & 15) == 0;
  const bool vecB = (ldb & 3) == 0 && (reinterpret_cast<uintptr_t>(Bm) & 15) == 0;
  const float none[4] = {0.f, 0.f, 0.f, 0.f};
  float out[GP_TILE / 16][4];
  int row0, col0;
  tile_product<GP_TILE, true, true, false>([&](int m, int j) { return load_row4(Am, lda, j, j_end, m0 + m, M, vecA); },
                                    [&](int c, int j) {
                                      if (Bm) return load_row4(Bm, ldb, j, j_end, n0 + c, N, vecB);
                                      return make_float4(j < j_end && n0 + c == 0 ? 1.f : 0.f, 0.f, 0.f, 0.f);   // a bias: one column of ones
                                    },
                                    j_begin, j_end, sm, none, out, row0, col0);
  const int n = n0 + col0;
  if (n >= N) return;
  float* dst = P + (size_t)blockIdx.y * count + d.off + n;
  const bool vec = (N & 3) == 0 && (reinterpret_cast<uintptr_t>(dst) & 15) == 0;
#pragma unroll
  for (int i = 0; i < GP_TILE / 16; ++i) {
    const int m = m0 + row0 + i;
    if (m < M) store_row4(dst + (size_t)m * N, out[i], N - n, vec);
  }
}

// The gradients of narrow operands (obs_dim <= 8, at most four outputs): W1, both hidden biases, the head and its biases.  As 64-column
// product tiles they were three of five tiles of an update and almost all padding.  Thread (s, n) sums neuron n of the block's 64
// over rows s, s + 4, ... of the range; the four sums meet in shared memory.
struct NarrowGrad {
  const float *dh1, *dh2, *h2, *g, *obs;
  int D, H, A, ldg, value_head, n_blocks;
};

__device__ __forceinline__ void grad_narrow_block(float* __restrict__ P, const NarrowGrad& d, int block, int j_begin, int j_end, float* sm) {
  const int n = block * 64 + (threadIdx.x & 63), s = threadIdx.x >> 6, H = d.H, D = d.D, A = d.A;
  float v[14];                                       // W1 [8] | b1 | b2 | head [4]
#pragma unroll
  for (int i = 0; i < 14; ++i) v[i] = 0.f;
  if (n < H) {
#pragma unroll 4
    for (int j = j_begin + s; j < j_end; j += 4) {
      const float d1 = d.dh1[(size_t)j * H + n], d2 = d.dh2[(size_t)j * H + n], h = d.h2[(size_t)j * H + n];
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (k < D) v[k] = fmaf(d1, __ldg(d.obs + (size_t)j * D + k), v[k]);
      v[8] += d1;
      v[9] += d2;
#pragma unroll
      for (int a = 0; a < 4; ++a)
        if (a < d.ldg) v[10 + a] = fmaf(h, __ldg(d.g + (size_t)j * d.ldg + a), v[10 + a]);
    }
  }
#pragma unroll
  for (int i = 0; i < 14; ++i) sm[(s * 14 + i) * 64 + (threadIdx.x & 63)] = v[i];
  __syncthreads();
  const int o_b1 = H * D, o_b2 = o_b1 + H + H * H, o_W3 = o_b2 + H, o_b3 = o_W3 + A * H;
  for (int i = threadIdx.x; i < 14 * 64; i += 256) {
    const int c = i >> 6, nn = block * 64 + (i & 63);
    const float t = (sm[i] + sm[i + 14 * 64]) + (sm[i + 2 * 14 * 64] + sm[i + 3 * 14 * 64]);
    if (nn >= H) continue;
    if (c < 8) {
      if (c < D) P[nn * D + c] = t;
    } else if (c < 10) {
      P[(c == 8 ? o_b1 : o_b2) + nn] = t;
    } else {
      const int a = c - 10;
      if (a < A) P[o_W3 + a * H + nn] = t;
      else if (d.value_head && a == A) P[o_b3 + A + nn] = t;
    }
  }
  if (block == 0 && threadIdx.x < 32 * 4) {          // output biases: a warp per output sums its column of g
    const int a = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (a < d.ldg) {
      float t = 0.f;
      for (int j = j_begin + lane; j < j_end; j += 32) t += __ldg(d.g + (size_t)j * d.ldg + a);
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      if (lane == 0) P[a < A ? o_b3 + a : o_b3 + A + H] = t;
    }
  }
}

// Every gradient product of one update in a single launch: thread block (tile, range) sums, over its range of minibatch
// rows, one 64 x 64 tile of one product and writes it to
// P[range][off + m * N + n] -- a partial gradient laid out like the parameter blob itself, `count` floats per range.
// No atomics: the apply kernel adds the ranges in order.
__global__ void __launch_bounds__(256) sgd_grad_partial_kernel(float* __restrict__ P, const GradProducts gp, const NarrowGrad narrow, int count,
                                                               int n_rows, int rows_per_range) {
  __shared__ __align__(16) float sm[2 * GM_STAGE<GP_TILE>];   // or 4 x 14 x 64 sums
  static_assert(4 * 14 * 64 <= 2 * GM_STAGE<GP_TILE>, "the narrow sums fit");
  chain_begin();
  if ((int)blockIdx.x >= gp.n_tiles) {
    const int j_begin = blockIdx.y * rows_per_range, j_end = min(j_begin + rows_per_range, n_rows);
    grad_narrow_block(P + (size_t)blockIdx.y * count, narrow, blockIdx.x - gp.n_tiles, j_begin, j_end, sm);
    return;
  }
  int q = 0;
  while (q + 1 < gp.n && (int)blockIdx.x >= gp.g[q + 1].tile_begin) ++q;
  const GradProduct& d = gp.g[q];
  const int t = blockIdx.x - d.tile_begin;
  grad_tile(P, d, t, count, n_rows, rows_per_range, sm);
}

// C[i] -= lr * (P[0][i] + P[1][i] + ...), the partial sums added in range order; nothing after a wait of the update that ran out
__global__ void sgd_apply_kernel(float* __restrict__ Cm, const float* __restrict__ P, int count, int n_ranges, float lr, const UpdateWatch watch) {
  chain_begin();
  chain_next();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const unsigned asked = update_ask(watch.failed, watch.number);
  float s = 0.f;
  if (i < count)
    for (int z = 0; z < n_ranges; ++z) s += P[(size_t)z * count + i];
  if (update_valid(watch.number, asked) && i < count) Cm[i] -= lr * s;
}

// the same gradient through Adam (Table 2's optimiser): m <- b1 m + (1-b1) g, v <- b2 v + (1-b2) g^2,
// theta <- theta - lr (m / c1) / (sqrt(v / c2) + eps) with the bias corrections c1 = 1 - b1^t, c2 = 1 - b2^t from the host
__global__ void sgd_apply_adam_kernel(float* __restrict__ Cm, float* __restrict__ m, float* __restrict__ v,
                                      const float* __restrict__ P, int count, int n_ranges, float lr, float beta1, float beta2,
                                      float eps, float c1, float c2, const UpdateWatch watch) {
  chain_begin();
  chain_next();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const unsigned asked = update_ask(watch.failed, watch.number);
  float g = 0.f;
  if (i < count)
    for (int z = 0; z < n_ranges; ++z) g += P[(size_t)z * count + i];
  if (!update_valid(watch.number, asked) || i >= count) return;
  const float mi = fmaf(beta1, m[i], (1.f - beta1) * g);
  const float vi = fmaf(beta2, v[i], (1.f - beta2) * g * g);
  m[i] = mi;
  v[i] = vi;
  Cm[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

}  // namespace

size_t sgd_partial_floats(int max_rows) {
  const size_t per16 = ((size_t)max_rows + SG_ROWS - 1) / SG_ROWS, fused = 5 * (size_t)SGD_FUSED_MAX_PARTS;
  return (per16 > fused ? per16 : fused) + 8;
}

// the partial gradients: one per row range of the layered path, or one per block of the fused kernel
size_t sgd_grad_partial_floats(int max_rows, int D, int H) {
  const size_t blob = (size_t)H * D + H + (size_t)H * H + H + 17 * (size_t)H + 17 + 3;
  size_t parts = SG_SPLITS;
  if (sgd_fused_ok(D, H, 1, 0)) {
    const size_t most = ((size_t)max_rows + 3) / 4;            // blocks of the fewest rows
    parts = most < SG_SPLITS ? SG_SPLITS : (most > SGD_FUSED_MAX_PARTS ? SGD_FUSED_MAX_PARTS : most);
  }
  return parts * blob;
}

size_t sgd_scratch_floats(int max_rows, int D, int H) {
  const size_t rows = ((size_t)max_rows + SG_ROWS - 1) / SG_ROWS * SG_ROWS;
  // h1, h2, dh1, dh2, g [rows][<= 16 actions + value], qt [rows][<= 16], loss partials, PPO's five per 16 rows, partial gradients of the whole
  // parameter blob (at most 16 actions and a value head); W2 transposed
  // + split copies of W1 (x 2 networks), W2 (x 2) and W2^T for the tensor-core products
  return 4 * rows * (size_t)H + rows * 33 + sgd_partial_floats(max_rows) + 5 * (rows / SG_ROWS) + 64 + (size_t)H * H + 4 /* UpdateWatch */ +
         sgd_grad_partial_floats(max_rows, D, H) + 2 * tc_pack_floats(H, D) + 3 * tc_pack_floats(H, H) + 64;
}

int sgd_partial_count(int n) { return (n + SG_ROWS - 1) / SG_ROWS; }

bool sgd_supported(int D, int H, int A) { return H >= 1 && D >= 1 && A >= 1 && A <= 16; }

namespace {
// wide layers with enough 128 x 256 tiles: the pre-split tensor-core products (both hidden layers must qualify)
bool use_tc2(const SgdParams& p) {
  return !p.value_head && p.n >= 512 && p.wpack && tc_gemm2_ok(p.obs, p.D, p.n, p.H, p.D) && tc_gemm2_ok(p.next_obs, p.D, p.n, p.H, p.D) &&
         tc_gemm2_ok(p.h1, p.H, p.n, p.H, p.H);
}

// dh1 = (dh2 W2) where h1 > 0, and every parameter update: C -= lr * (gradient rows)^T (input rows), a bias with a column of ones
cudaError_t backward_and_update(const SgdParams& p, float lr, const AdamParams* adam, cudaStream_t s) {
  const int D = p.D, H = p.H, A = p.A;
  const float* W2m = p.theta + (size_t)H * D + H;
  cudaError_t e;
  if (use_tc2(p)) {
    // W2^T was split with the other weight matrices at the start of the step
    TcGemmBatch b{};
    b.g[0] = TcGemm{p.dh2, H, p.wpack + 2 * tc_pack_floats(H, D) + 2 * tc_pack_floats(H, H), p.dh1, H, p.n, H, H, nullptr, p.h1, H};
    b.n = 1;
    ++*p.launches;
    e = launch_gemm_tc2(b, GM_MASK, p.watch, s);
  } else if (!p.value_head && H >= 128 && tc_gemm_ok(p.dh2, H, p.w2t, H, p.n, H, H)) {
    // the tensor-core product wants both operands K-major: dh1 = dh2 (W2^T)^T with W2^T written out first
    ++*p.launches;
    if ((e = launch_chained(sg_transpose_kernel, dim3((H + 31) / 32, (H + 31) / 32), 256, 0, s, W2m, p.w2t, H)) != cudaSuccess) return e;
    e = sg_layer<GM_MASK>(p, GemmPair{{p.dh2}, {p.w2t}, {p.dh1}, {nullptr}}, 1, H, H, H, p.n, H, H, p.h1, H, s);
  } else {
    e = sg_gemm<true, GM_MASK>(p, GemmPair{{p.dh2}, {W2m}, {p.dh1}, {nullptr}}, 1, H, H, H, p.n, H, H, p.h1, H, s);
  }
  if (e != cudaSuccess) return e;
  float* W1 = p.theta;
  float* b1 = W1 + (size_t)H * D;
  float* W2 = b1 + H;
  float* b2 = W2 + (size_t)H * H;
  float* W3 = b2 + H;
  float* b3 = W3 + (size_t)A * H;
  // the backward pass has read W2 and the heads; now the parameters may change: all products in one or two launches, then
  // one pass over the whole blob.  Products whose input width is a multiple of 128 go to the tensor cores (with their bias
  // gradient), the others to the FMA tiles.
  GradProducts gp{};
  auto add = [&](float* C, int M, int N, const float* Am, int lda, const float* Bm, int ldb) {
    GradProduct& d = gp.g[gp.n++];
    d.Am = Am;
    d.Bm = Bm;
    d.off = (int)(C - p.theta);
    d.M = M;
    d.N = N;
    d.lda = lda;
    d.ldb = ldb;
    d.tile_begin = gp.n_tiles;
    gp.n_tiles += ((M + GP_TILE - 1) / GP_TILE) * ((N + GP_TILE - 1) / GP_TILE);
  };
  TcWgradBatch tb{};
  const bool tc_grads = use_tc2(p);
  // one product and its bias: C [M][N] = G^T X, bias [M] = column sums of G
  auto product = [&](float* C, float* bias, int M, int N, const float* G, int ldg, const float* X, int ldx) {
    if (tc_grads && tc_wgrad_ok(N, p.n)) {
      TcWgrad& d = tb.g[tb.n++];
      d = TcWgrad{G, ldg, X, ldx, M, N, (int)(C - p.theta), (int)(bias - p.theta), tb.n_tiles};
      tb.n_tiles += tc_wgrad_tiles(M, N);
    } else {
      add(C, M, N, G, ldg, X, ldx);
      add(bias, M, 1, G, ldg, nullptr, 0);
    }
  };
  NarrowGrad narrow{};
  if (!tc_grads && D <= 8 && A + p.value_head <= 4) {
    add(W2, H, H, p.dh2, H, p.h1, H);
    narrow = NarrowGrad{p.dh1, p.dh2, p.h2, p.g, p.obs, D, H, A, p.ldg, p.value_head, (H + 63) / 64};
  } else {
    product(W1, b1, H, D, p.dh1, H, p.obs, D);
    product(W2, b2, H, H, p.dh2, H, p.h1, H);
    product(W3, b3, A, H, p.g, p.ldg, p.h2, H);    // no value head here: it comes with CartPole and Acrobot only
  }
  // row ranges: with tensor-core tiles about one thread block per SM in all (a block costs a fixed ~10 us beside its rows);
  // otherwise three per SM, but 128 rows or more per range
  const int sms = p.sm_count > 0 ? p.sm_count : 148;
  int n_ranges = tb.n_tiles > 0 ? sms / tb.n_tiles : 3 * sms / (gp.n_tiles + narrow.n_blocks);
  if (tb.n_tiles == 0 && n_ranges > (p.n + 127) / 128) n_ranges = (p.n + 127) / 128;
  if (n_ranges < 1) n_ranges = 1;
  if (n_ranges > SG_SPLITS) n_ranges = SG_SPLITS;
  const int rows_per_range = ((p.n + n_ranges - 1) / n_ranges + 31) / 32 * 32;
  n_ranges = (p.n + rows_per_range - 1) / rows_per_range;
  const int count = (int)(b3 + A - p.theta) + (p.value_head ? H + 1 : 0);
  *p.launches += (tb.n ? 1 : 0) + (gp.n_tiles + narrow.n_blocks > 0 ? 1 : 0) + 1;
  if (tb.n && (e = launch_wgrad_tc(tb, p.grad_partial, count, p.n, rows_per_range, n_ranges, p.watch, s)) != cudaSuccess) return e;
  if (gp.n_tiles + narrow.n_blocks > 0 &&
      (e = launch_chained(sgd_grad_partial_kernel, dim3(gp.n_tiles + narrow.n_blocks, n_ranges), 256, 0, s, p.grad_partial, gp, narrow, count, p.n,
                          rows_per_range)) != cudaSuccess)
    return e;
  if (adam)
    return launch_chained(sgd_apply_adam_kernel, (count + 255) / 256, 256, 0, s, p.theta, adam->m, adam->v, p.grad_partial, count, n_ranges, lr,
                          adam->beta1, adam->beta2, adam->eps, adam->c1, adam->c2, p.watch);
  return launch_chained(sgd_apply_kernel, (count + 255) / 256, 256, 0, s, p.theta, p.grad_partial, count, n_ranges, lr, p.watch);
}
}  // namespace

static cudaError_t sgd_step_layered(const SgdParams& p, float lr, const AdamParams* adam, cudaStream_t s) {
  const int n = p.n, D = p.D, H = p.H, A = p.A;
  const float *W1 = p.theta, *b1 = W1 + (size_t)H * D, *W2 = b1 + H, *b2 = W2 + (size_t)H * H, *W3 = b2 + H, *b3 = W3 + (size_t)A * H;
  const float *T1 = p.theta_target, *tb1 = T1 + (size_t)H * D, *T2 = tb1 + H, *tb2 = T2 + (size_t)H * H, *T3 = tb2 + H, *tb3 = T3 + (size_t)A * H;
  // online network: h1, h2 kept; target network: its activations borrow dh1 / dh2 (free until the backward pass)
  cudaError_t e;
  if (use_tc2(p)) {
    // both networks' weight matrices (and W2^T for the backward pass) split once, then each layer of both networks in one launch
    float* pk_W1 = p.wpack;
    float* pk_T1 = pk_W1 + tc_pack_floats(H, D);
    float* pk_W2 = pk_T1 + tc_pack_floats(H, D);
    float* pk_T2 = pk_W2 + tc_pack_floats(H, H);
    float* pk_W2t = pk_T2 + tc_pack_floats(H, H);
    TcPackJobs jobs{};
    jobs.j[jobs.n++] = TcPackJob{W1, D, 0, H, D, pk_W1};
    jobs.j[jobs.n++] = TcPackJob{T1, D, 0, H, D, pk_T1};
    jobs.j[jobs.n++] = TcPackJob{W2, H, 0, H, H, pk_W2};
    jobs.j[jobs.n++] = TcPackJob{T2, H, 0, H, H, pk_T2};
    jobs.j[jobs.n++] = TcPackJob{W2, H, 1, H, H, pk_W2t};
    if ((e = launch_pack_tf32_operands(jobs, s)) != cudaSuccess) return e;
    TcGemmBatch l1{};
    l1.g[0] = TcGemm{p.obs, D, pk_W1, p.h1, H, n, H, D, b1, nullptr, 0};
    l1.g[1] = TcGemm{p.next_obs, D, pk_T1, p.dh1, H, n, H, D, tb1, nullptr, 0};
    l1.n = 2;
    if ((e = launch_gemm_tc2(l1, GM_BIAS_RELU, p.watch, s)) != cudaSuccess) return e;
    TcGemmBatch l2{};
    l2.g[0] = TcGemm{p.h1, H, pk_W2, p.h2, H, n, H, H, b2, nullptr, 0};
    l2.g[1] = TcGemm{p.dh1, H, pk_T2, p.dh2, H, n, H, H, tb2, nullptr, 0};
    l2.n = 2;
    if ((e = launch_gemm_tc2(l2, GM_BIAS_RELU, p.watch, s)) != cudaSuccess) return e;
    *p.launches += 3;
  } else {
    const GemmPair l1{{p.obs, p.next_obs}, {W1, T1}, {p.h1, p.dh1}, {b1, tb1}}, l2{{p.h1, p.dh1}, {W2, T2}, {p.h2, p.dh2}, {b2, tb2}};
    if ((e = sg_layer<GM_BIAS_RELU>(p, l1, 2, D, D, H, n, H, D, nullptr, 0, s)) != cudaSuccess) return e;
    if ((e = sg_layer<GM_BIAS_RELU>(p, l2, 2, H, H, H, n, H, H, nullptr, 0, s)) != cudaSuccess) return e;
  }
  if (A <= 4) {
    ++*p.launches;
    if ((e = launch_chained(sgd_rows_kernel<false>, sgd_partial_count(n), 32 * SG_ROWS, 0, s, p, (const float*)p.dh2)) != cudaSuccess) return e;
    return backward_and_update(p, lr, adam, s);
  }
  // both heads in one launch: Q of the online network into g, of the target network into qt
  const GemmPair heads{{p.h2, p.dh2}, {W3, T3}, {p.g, p.qt}, {b3, tb3}};
  const size_t hd_smem = (size_t)H * 16 * sizeof(float);
  if (H % 128 == 0 && hd_smem <= 96 * 1024) {
    ++*p.launches;
    e = launch_chained(sg_heads_kernel, dim3((n + HD_ROWS - 1) / HD_ROWS, 2), 256, hd_smem, s, heads, n, H, A, A);
  } else {
    e = sg_gemm<false, GM_BIAS>(p, heads, 2, H, H, A, n, A, H, nullptr, 0, s);
  }
  if (e != cudaSuccess) return e;
  ++*p.launches;
  if ((e = launch_chained(sgd_loss_kernel, sgd_partial_count(n), 32 * SG_ROWS, 0, s, p)) != cudaSuccess) return e;
  return backward_and_update(p, lr, adam, s);
}

cudaError_t launch_sgd_step(const SgdParams& p, float lr, const AdamParams* adam, float* loss_out, cudaStream_t s) {
  if (sgd_fused_ok(p.D, p.H, p.A, 0)) {
    *p.launches += 2;
    return launch_sgd_fused(p, lr, adam, loss_out, s);
  }
  cudaError_t e = sgd_step_layered(p, lr, adam, s);
  if (e == cudaSuccess && loss_out) {
    ++*p.launches;
    e = launch_td_finish(p.partial, sgd_partial_count(p.n), p.n, loss_out, s, p.watch);
  }
  return e;
}

cudaError_t launch_td_layers(const TdParams& t, int sm_count, int* grid_out, cudaStream_t s) {
  int launches = 0;
  SgdParams p{};
  p.sm_count = sm_count;
  p.launches = &launches;
  const size_t nH = (size_t)t.n * t.H;
  float *h1 = t.layers, *h2 = h1 + nH, *t1 = h2 + nH, *t2 = t1 + nH;
  const float *W = t.Wonline, *T = t.Wtarget;
  const GemmPair l1{{t.obs, t.next_obs}, {W + t.off_W1t, T + t.off_W1t}, {h1, t1}, {W + t.off_b1, T + t.off_b1}};
  const GemmPair l2{{h1, t1}, {W + t.off_W2t, T + t.off_W2t}, {h2, t2}, {W + t.off_b2, T + t.off_b2}};
  cudaError_t e = sg_gemm<true, GM_CHAIN_RELU>(p, l1, 2, t.D, t.Hp, t.H, t.n, t.H, t.D, nullptr, 0, s);
  if (e == cudaSuccess) e = sg_gemm<true, GM_CHAIN_RELU>(p, l2, 2, t.H, t.Hp, t.H, t.n, t.H, t.H, nullptr, 0, s);
  const int rows = td_tile_rows(t.H);
  *grid_out = (t.n + rows - 1) / rows;
  if (e == cudaSuccess)
    e = launch_chained(td_rows_kernel, *grid_out, TR_NT, (size_t)tr_layout(t.H, rows).total * sizeof(float), s, t, (const float*)h2, (const float*)t2, rows);
  return e;
}

cudaError_t launch_ppo_step(const SgdParams& p, float lr, const AdamParams* adam, float* stats_out, cudaStream_t s) {
  if (sgd_fused_ok(p.D, p.H, p.A, 1)) {
    *p.launches += 2;
    return launch_sgd_fused(p, lr, adam, stats_out, s);
  }
  if (p.A > 3) return cudaErrorInvalidConfiguration;           // the segment environments have two or three actions
  const int n = p.n, D = p.D, H = p.H;
  const float *W1 = p.theta, *b1 = W1 + (size_t)H * D, *W2 = b1 + H, *b2 = W2 + (size_t)H * H;
  cudaError_t e;
  if ((e = sg_gemm<false, GM_BIAS_RELU>(p, GemmPair{{p.obs}, {W1}, {p.h1}, {b1}}, 1, D, D, H, n, H, D, nullptr, 0, s)) != cudaSuccess) return e;
  if ((e = sg_gemm<false, GM_BIAS_RELU>(p, GemmPair{{p.h1}, {W2}, {p.h2}, {b2}}, 1, H, H, H, n, H, H, nullptr, 0, s)) != cudaSuccess) return e;
  *p.launches += stats_out ? 2 : 1;
  if ((e = launch_chained(sgd_rows_kernel<true>, sgd_partial_count(n), 32 * SG_ROWS, 0, s, p, (const float*)nullptr)) != cudaSuccess) return e;
  if (stats_out && (e = launch_chained(ppo_finish_kernel, 1, 160, 0, s, (const float*)p.stat_partial, sgd_partial_count(n), n, stats_out)) != cudaSuccess)
    return e;
  return backward_and_update(p, lr, adam, s);
}

}  // namespace tj
