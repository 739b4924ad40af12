// FP32 layers in the fixed rounding order of tj_mlp.cuh -- acc = bias; acc = fma(Wt[k][n], x[k][e], acc) for k = 0, 1, 2, ... -- for
// tiles whose size is chosen at run time, two environments (or samples) per instruction: fma.rn.f32x2 rounds each half as fmaf
// does, costs one issue slot for two FMAs and so leaves slots for the operand loads.
//
// Activations are k-major, x[k][E] (E a multiple of four), weights [k][ldw].  A thread owns EPT rows x NPT neurons, both in quads: rows
// 4 eg .. 4 eg + 3 and, with EPT = 8, the same four of the tile's second half; neurons NPT ng ..  So a warp's loads are whole runs of 16-byte words or broadcasts.
#pragma once
#include <cuda_runtime.h>

namespace tj {

typedef unsigned long long f32x2;

__device__ __forceinline__ void fma2(f32x2& acc, f32x2 a, f32x2 b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b)); }
__device__ __forceinline__ f32x2 dup2(float x) {
  f32x2 d;
  asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(x));
  return d;
}
__device__ __forceinline__ float2 halves(f32x2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ ulonglong2 ld_pairs(const float* p) { return *reinterpret_cast<const ulonglong2*>(p); }

// Cycles per k measured for one block (ideal = E x width / 128): E 32, width 128: 4 x 2 on 512 threads 65, 8 x 2 on 256 57, 4 x 4 on
// 256 51, 8 x 4 on 128 49 (ideal 32); E 64, width 128: 8 x 4 82 (64); E 56, width 256: 8 x 4 201 (112).  The
// neuron groups run fastest over the lanes (eg fastest: 8 x 2 74, 4 x 2 81): the row operand is then a broadcast.
//
// a thread's share of a layer: row quad eg, neuron group ng; half = rows between its two row quads (EPT = 8)
struct FmaTile { int eg, ng, half; };

template <int EPT, int NPT>
struct FmaAcc { f32x2 v[NPT][EPT / 2]; };

template <int NPT>
__device__ __forceinline__ void fma_load_w(const float* w, float (&out)[NPT]) {
  if constexpr (NPT == 1) {
    out[0] = *w;
  } else if constexpr (NPT == 2) {
    const float2 a = *reinterpret_cast<const float2*>(w);
    out[0] = a.x; out[1] = a.y;
  } else {
    const float4 a = *reinterpret_cast<const float4*>(w);
    out[0] = a.x; out[1] = a.y; out[2] = a.z; out[3] = a.w;
  }
}

template <int EPT, int NPT>
__device__ __forceinline__ void fma_bias(FmaAcc<EPT, NPT>& acc, const float* b, const FmaTile& t) {
  float bv[NPT];
  fma_load_w<NPT>(b + NPT * t.ng, bv);
#pragma unroll
  for (int n = 0; n < NPT; ++n)
#pragma unroll
    for (int e = 0; e < EPT / 2; ++e) acc.v[n][e] = dup2(bv[n]);
}

// acc += over k in [0, K): W [k][ldw], x [k][E], both in shared memory
template <int EPT, int NPT, int UNROLL>
__device__ __forceinline__ void fma_accumulate(FmaAcc<EPT, NPT>& acc, const float* W, int ldw, const float* x, int E, int K, const FmaTile& t) {
  const float* wp = W + NPT * t.ng;
  const float* xp = x + 4 * t.eg;
#pragma unroll UNROLL
  for (int k = 0; k < K; ++k) {
    float w[NPT];
    fma_load_w<NPT>(wp, w);
    f32x2 xv[EPT / 2];
#pragma unroll
    for (int u = 0; u < EPT / 4; ++u) {
      const ulonglong2 a = ld_pairs(xp + u * t.half);
      xv[2 * u] = a.x; xv[2 * u + 1] = a.y;
    }
#pragma unroll
    for (int n = 0; n < NPT; ++n) {
      const f32x2 ww = dup2(w[n]);
#pragma unroll
      for (int e = 0; e < EPT / 2; ++e) fma2(acc.v[n][e], ww, xv[e]);
    }
    wp += ldw;
    xp += E;
  }
}

__device__ __forceinline__ float relu1(float v) { return v > 0.f ? v : 0.f; }

// relu(acc) -> y[n][E], the next layer's k-major operand
template <int EPT, int NPT>
__device__ __forceinline__ void fma_store_kmajor(const FmaAcc<EPT, NPT>& acc, float* y, int E, const FmaTile& t) {
#pragma unroll
  for (int n = 0; n < NPT; ++n) {
#pragma unroll
    for (int u = 0; u < EPT / 4; ++u) {
      const float2 a = halves(acc.v[n][2 * u]), b = halves(acc.v[n][2 * u + 1]);
      *reinterpret_cast<float4*>(y + (NPT * t.ng + n) * E + 4 * t.eg + u * t.half) = make_float4(relu1(a.x), relu1(a.y), relu1(b.x), relu1(b.y));
    }
  }
}

// relu(acc) -> y[e][ld], row-major for the head
template <int EPT, int NPT>
__device__ __forceinline__ void fma_store_rows(const FmaAcc<EPT, NPT>& acc, float* y, int ld, const FmaTile& t) {
#pragma unroll
  for (int e = 0; e < EPT; ++e) {
    float v[NPT];
#pragma unroll
    for (int n = 0; n < NPT; ++n) {
      const float2 h = halves(acc.v[n][e / 2]);
      v[n] = relu1(e & 1 ? h.y : h.x);
    }
    float* row = y + (4 * t.eg + (e & 3) + (e >> 2) * t.half) * ld + NPT * t.ng;
    if constexpr (NPT == 1) row[0] = v[0];
    else if constexpr (NPT == 2) *reinterpret_cast<float2*>(row) = make_float2(v[0], v[1]);
    else *reinterpret_cast<float4*>(row) = make_float4(v[0], v[1], v[2], v[3]);
  }
}

// one output of the narrow head: acc = b; acc = fma(w[k], h[k], acc) over a row of h (both 16-byte aligned, zero padded to 4)
template <int UNROLL>
__device__ __forceinline__ float fma_head(float acc, const float* w, const float* h, int K4) {
#pragma unroll UNROLL
  for (int k = 0; k < K4; ++k) {
    const float4 a = *reinterpret_cast<const float4*>(w + 4 * k), b = *reinterpret_cast<const float4*>(h + 4 * k);
    acc = fmaf(a.x, b.x, acc);
    acc = fmaf(a.y, b.y, acc);
    acc = fmaf(a.z, b.z, acc);
    acc = fmaf(a.w, b.w, acc);
  }
  return acc;
}

}  // namespace tj
