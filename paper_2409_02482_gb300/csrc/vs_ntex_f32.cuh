// Fused FP32 kernels of the neural texture (the default layers): encoding,
// both hidden layers and the output layer of a tile of texels in one kernel
// each way, the activations kept in shared memory, every product an FP32 FMA.
//
// What bounds them: the FP32 pipes.  A 16 x 2 -> 64 -> 64 -> 27 network is
// 16 kFLOP per texel forward and 44 kFLOP for the adjoint against 54 and
// 236 bytes of texels and gradients, so the floor is FMA issue (72 TFLOP/s
// measured for independent FMAs on 152 SMs).  The unfused layers moved
// every activation through L2 three to five times and waited at each
// launch's barrier-separated 16-deep slices.
//
// Layout.  A group of 4 warps owns a tile of 64 texels.  An activation is
// stored unit-major, [unit][kFS] with the texels contiguous, so that a
// product's A operand is two 16-byte loads of a thread's 8 texels and its
// outputs go back as 16-byte stores; kFS = 68 puts consecutive units 4 banks
// apart, which makes the weight gradients' loads (4 texels of 8 consecutive
// units) free of conflicts.  A thread computes 8 texels x 4 units (4 x 4 for
// 32-wide outputs): 3 16-byte loads per 32 FMAs.  The FMAs are paired
// (fma.rn.f32x2, texel pairs): 57 against 54 TFLOP/s for the scalar form of
// this loop; with the weights stored twice instead of paired by moves 48,
// the loads' bandwidth then being the limit.  Groups share the CTA's weights
// and drift apart, so one group's gathers overlap another's products.
//
// Every sum over inputs runs in unit order from zero with one rounding per
// term, bias added last, as in k_gemm_abt: the activations -- and with them
// the ReLU masks -- do not depend on the kernel that computed them.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace vsn {

constexpr int kFT = 64;    // texels of a group's tile
constexpr int kFS = 68;    // floats between units of an activation
constexpr int kFG = 128;   // threads of a group

__device__ __forceinline__ void group_sync(int group) {
  asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "r"(kFG) : "memory");
}

// Position of a thread inside its group.
struct Pos {
  int w, ty, tx;   // warp; texel quad; unit quad within the warp
};

__device__ __forceinline__ uint64_t pair(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 unpair(uint64_t v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// A thread's outputs of a product with N units: 8 texels x 4 units for
// N = 64 (warp w: units 16 w + 4 tx .., texels 4 ty .. and 32 + 4 ty ..), 4 x 4
// for N = 32 (units 16 (w & 1) + 4 tx .., texels 32 (w >> 1) + 4 ty ..).
template <int N>
struct Out {
  static constexpr int Q = N / 32;   // texel quads per thread
  uint64_t v[2 * Q][4];              // [texel pair][unit]
  __device__ __forceinline__ static int unit(Pos p) { return (N == 64 ? 16 * p.w : 16 * (p.w & 1)) + 4 * p.tx; }
  __device__ __forceinline__ static int texel(Pos p, int q) { return (N == 64 ? 32 * q : 32 * (p.w >> 1)) + 4 * p.ty; }
  // the 4 texels of quad q at unit j of the thread
  __device__ __forceinline__ float4 quad(int q, int j) const {
    const float2 a = unpair(v[2 * q][j]), b = unpair(v[2 * q + 1][j]);
    return make_float4(a.x, a.y, b.x, b.y);
  }
};

// O[texel, n] = sum_k A[k][texel] B[k][n], k ascending (K a multiple of 4).
template <int N>
__device__ __forceinline__ void product(const float* A, const float* B, int K, Pos p, Out<N>& o) {
  constexpr int Q = Out<N>::Q;
#pragma unroll
  for (int i = 0; i < 2 * Q; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) o.v[i][j] = 0ull;
  const float* a = A + Out<N>::texel(p, 0);
  const float* b = B + Out<N>::unit(p);
#pragma unroll 4
  for (int k = 0; k < K; ++k) {
    uint64_t x[2 * Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(a + k * kFS + 32 * q);
      x[2 * q] = t.x;
      x[2 * q + 1] = t.y;
    }
    const float4 bv = *reinterpret_cast<const float4*>(b + k * N);
    const uint64_t y[4] = {pair(bv.x, bv.x), pair(bv.y, bv.y), pair(bv.z, bv.z), pair(bv.w, bv.w)};
#pragma unroll
    for (int i = 0; i < 2 * Q; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) o.v[i][j] = fma2(x[i], y[j], o.v[i][j]);
  }
}

__device__ __forceinline__ float4 relu4(float4 v, float b) {
  return make_float4(fmaxf(v.x + b, 0.0f), fmaxf(v.y + b, 0.0f), fmaxf(v.z + b, 0.0f), fmaxf(v.w + b, 0.0f));
}
__device__ __forceinline__ float4 keep4(float4 v, int first, int count) {   // zero from texel `count` on
  return make_float4(first < count ? v.x : 0.0f, first + 1 < count ? v.y : 0.0f, first + 2 < count ? v.z : 0.0f,
                     first + 3 < count ? v.w : 0.0f);
}

// dst = relu(o + bias), zero for texels from `live` on.
template <int N>
__device__ __forceinline__ void store_relu(const Out<N>& o, const float* bias, Pos p, int live, float* dst) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int n = Out<N>::unit(p) + j;
    const float b = bias[n];
#pragma unroll
    for (int q = 0; q < Out<N>::Q; ++q) {
      const int t = Out<N>::texel(p, q);
      *reinterpret_cast<float4*>(dst + n * kFS + t) = keep4(relu4(o.quad(q, j), b), t, live);
    }
  }
}

// act = o where act > 0, else 0 (the ReLU's adjoint, in place of the
// activation); the thread's sums per unit are added to csum.
template <int N>
__device__ __forceinline__ void mask_in_place(const Out<N>& o, Pos p, float* act, float csum[4]) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int n = Out<N>::unit(p) + j;
#pragma unroll
    for (int q = 0; q < Out<N>::Q; ++q) {
      float4* h = reinterpret_cast<float4*>(act + n * kFS + Out<N>::texel(p, q));
      const float4 a = *h, v = o.quad(q, j);
      const float4 d = make_float4(a.x > 0.0f ? v.x : 0.0f, a.y > 0.0f ? v.y : 0.0f, a.z > 0.0f ? v.z : 0.0f,
                                   a.w > 0.0f ? v.w : 0.0f);
      *h = d;
      csum[j] += (d.x + d.y) + (d.z + d.w);
    }
  }
}

// Encoding of the group's 64 texels (texel n0 + i of the texture in column i
// of X, zero from `live` on): two threads per texel, half of the levels
// each.  Same corners, weights and sums as k_encode.
__device__ __forceinline__ void encode_tile(const Enc& e, const float* table, int W, int H, int n0, int live, float* X,
                                            int g) {
  const int i = g & 63;
  const int l0 = (g >> 6) ? (e.L + 1) / 2 : 0, l1 = (g >> 6) ? e.L : (e.L + 1) / 2;
  const int n = n0 + (i < live ? i : live - 1);
  const int ty = n / W, tx = n - ty * W;
  const WarpCorners wc(e, ty, H);
  if (e.F == 2) {   // four levels at a time: 16 rows of 8 bytes in flight
    const float2* t2 = reinterpret_cast<const float2*>(table);
    for (int lb = l0; lb < l1; lb += 4) {
      float2 v[4][4];
      float w[4][4];
#pragma unroll
      for (int d = 0; d < 4; ++d) {
        const int l = lb + d < l1 ? lb + d : lb;
        uint32_t rw[4];
        wc.at(e, l, tx, ty, W, H, rw, w[d]);
#pragma unroll
        for (int c = 0; c < 4; ++c) v[d][c] = __ldg(t2 + ((size_t)l << e.logT) + rw[c]);
      }
#pragma unroll
      for (int d = 0; d < 4; ++d) {
        if (lb + d >= l1) break;
        float a0 = 0.0f, a1 = 0.0f;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          a0 = fmaf(w[d][c], v[d][c].x, a0);
          a1 = fmaf(w[d][c], v[d][c].y, a1);
        }
        X[(2 * (lb + d)) * kFS + i] = i < live ? a0 : 0.0f;
        X[(2 * (lb + d) + 1) * kFS + i] = i < live ? a1 : 0.0f;
      }
    }
    return;
  }
  for (int l = l0; l < l1; ++l) {
    uint32_t rw[4];
    float w[4];
    wc.at(e, l, tx, ty, W, H, rw, w);
    const float* t = table + ((size_t)l << e.logT) * e.F;
    for (int f = 0; f < e.F; ++f) {
      float a = 0.0f;
#pragma unroll
      for (int c = 0; c < 4; ++c) a = fmaf(w[c], __ldg(t + (size_t)rw[c] * e.F + f), a);
      X[(l * e.F + f) * kFS + i] = i < live ? a : 0.0f;
    }
  }
}

// dst[k][n] = src[n][k] (n_rows x k_cols row-major), zero outside, K x N.
__device__ __forceinline__ void stage_t(float* dst, const float* src, int n_rows, int k_cols, int K, int N) {
  for (int i = threadIdx.x; i < K * N; i += blockDim.x) {
    const int k = i / N, n = i - k * N;
    dst[i] = (n < n_rows && k < k_cols) ? __ldg(src + (size_t)n * k_cols + k) : 0.0f;
  }
}
// dst[r][c] = src[r][c] (rows x cols row-major), zero outside, R x C.
__device__ __forceinline__ void stage_r(float* dst, const float* src, int rows, int cols, int R, int C) {
  for (int i = threadIdx.x; i < R * C; i += blockDim.x) {
    const int r = i / C, c = i - r * C;
    dst[i] = (r < rows && c < cols) ? __ldg(src + (size_t)r * cols + c) : 0.0f;
  }
}
__device__ __forceinline__ void stage_v(float* dst, const float* src, int n, int N) {
  for (int i = threadIdx.x; i < N; i += blockDim.x) dst[i] = i < n ? __ldg(src + i) : 0.0f;
}

// ----------------------------------------------------------------------------
// forward
// ----------------------------------------------------------------------------
struct F32FwdArgs {
  const float *table, *W0, *b0, *W1, *b1, *W2, *b2;
  void* texels;
  int W, H, N, C, hidden, LF, dtype, pitch, ch0;
  int vec;   // 4 consecutive channels can be stored at once
};

constexpr int kFwdGroups = 4;   // 16 warps per SM

// HP, LP, CP: hidden units, encoding values and outputs padded to 32 or 64.
__host__ __device__ constexpr int f32_fwd_floats(int HP, int LP, int CP) {
  return LP * HP + HP * HP + HP * CP + 2 * HP + CP + kFwdGroups * ((LP > HP ? LP : HP) + HP) * kFS;
}

// Two buffers per group alternate between a layer's inputs and outputs, so a
// layer costs one group barrier.
template <int HP, int LP, int CP>
__global__ void __launch_bounds__(kFwdGroups * kFG, 1) k_mlp_fwd_f32(const F32FwdArgs a, const __grid_constant__ Enc e) {
  extern __shared__ __align__(16) float fsm[];
  float* W0 = fsm;                  // [LP][HP]
  float* W1 = W0 + LP * HP;         // [HP][HP]
  float* W2 = W1 + HP * HP;         // [HP][CP]
  float* b0 = W2 + HP * CP;
  float* b1 = b0 + HP;
  float* b2 = b1 + HP;
  constexpr int BIG = LP > HP ? LP : HP;
  const int g = threadIdx.x & (kFG - 1), group = threadIdx.x / kFG;
  float* U = b2 + CP + group * (BIG + HP) * kFS;   // inputs, then the second hidden layer
  float* V = U + BIG * kFS;                        // the first hidden layer
  const Pos p{g >> 5, g & 7, (g >> 3) & 3};
  stage_t(W0, a.W0, a.hidden, a.LF, LP, HP);
  stage_t(W1, a.W1, a.hidden, a.hidden, HP, HP);
  stage_t(W2, a.W2, a.C, a.hidden, HP, CP);
  stage_v(b0, a.b0, a.hidden, HP);
  stage_v(b1, a.b1, a.hidden, HP);
  stage_v(b2, a.b2, a.C, CP);
  const int K0 = (a.LF + 3) & ~3;
  __syncthreads();
  const int tiles = (a.N + kFT - 1) / kFT;
  for (int tile = blockIdx.x + gridDim.x * group; tile < tiles; tile += gridDim.x * kFwdGroups) {
    const int n0 = tile * kFT, live = min(kFT, a.N - n0);
    encode_tile(e, a.table, a.W, a.H, n0, live, U, g);
    for (int k = a.LF + (g >> 6); k < K0; k += 2) U[k * kFS + (g & 63)] = 0.0f;
    group_sync(group);
    Out<HP> o;
    product<HP>(U, W0, K0, p, o);
    store_relu<HP>(o, b0, p, live, V);
    group_sync(group);
    product<HP>(V, W1, HP, p, o);
    store_relu<HP>(o, b1, p, live, U);
    group_sync(group);
    Out<CP> y;
    product<CP>(U, W2, HP, p, y);
    const int c0 = Out<CP>::unit(p);
    float4 r[Out<CP>::Q][4];   // [quad][channel], 4 texels each
#pragma unroll
    for (int q = 0; q < Out<CP>::Q; ++q)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float b = b2[c0 + j];
        const float4 v = y.quad(q, j);
        r[q][j] = make_float4(v.x + b, v.y + b, v.z + b, v.w + b);
      }
    if (c0 < a.C) {
#pragma unroll
      for (int q = 0; q < Out<CP>::Q; ++q)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int t = Out<CP>::texel(p, q) + i;
          if (t >= live) continue;
          auto at = [&](int j) {
            const float4& f = r[q][j];
            return i == 0 ? f.x : (i == 1 ? f.y : (i == 2 ? f.z : f.w));
          };
          const size_t off = (size_t)(n0 + t) * a.pitch + a.ch0 + c0;
          if (a.dtype == 1) {
            __half* d = reinterpret_cast<__half*>(a.texels) + off;
            if (a.vec && c0 + 4 <= a.C) {
              const __half2 h0 = __floats2half2_rn(at(0), at(1)), h1 = __floats2half2_rn(at(2), at(3));
              *reinterpret_cast<uint2*>(d) = make_uint2(*reinterpret_cast<const uint32_t*>(&h0),
                                                        *reinterpret_cast<const uint32_t*>(&h1));
            } else {
#pragma unroll
              for (int j = 0; j < 4; ++j)
                if (c0 + j < a.C) d[j] = __float2half_rn(at(j));
            }
          } else {
            float* d = reinterpret_cast<float*>(a.texels) + off;
            if (a.vec && c0 + 4 <= a.C) {
              *reinterpret_cast<float4*>(d) = make_float4(at(0), at(1), at(2), at(3));
            } else {
#pragma unroll
              for (int j = 0; j < 4; ++j)
                if (c0 + j < a.C) d[j] = at(j);
            }
          }
        }
    }
    group_sync(group);   // U is the next tile's input
  }
}

// ----------------------------------------------------------------------------
// adjoint
// ----------------------------------------------------------------------------
struct F32BwdArgs {
  const float *table, *W0, *b0, *W1, *b1, *W2;
  const float* grad;   // dL/d(texels) [N, pitch], channels ch0 .. ch0 + C
  float *dW0, *db0, *dW1, *db1, *dW2, *db2;
  float* dX;           // dL/d(encoding) of texels n0 .. n0 + count, level-major [L][count][F]
  int W, H, n0, count, C, hidden, LF, F, pitch, ch0;
  int vec;             // 4 consecutive channels of grad can be loaded at once
};

// acc[i][j] += sum over the tile's texels of D[n_i][t] X[k_j][t]: the weight
// gradient of a layer (D: its N output units' adjoints, X: its K inputs).
// The group's threads split the N x K matrix: 4 units n (8 apart) by KT
// inputs k (4 apart) each; four texels per step, so 4 + KT 16-byte loads
// feed 16 KT FMAs.
template <int N, int K>
struct Wgrad {
  static constexpr int PARTS = N == 64 ? 2 : 4;     // warps along k
  static constexpr int KT = K / (4 * PARTS);
  float acc[4][KT];
  __device__ __forceinline__ static int n_of(Pos p, int i) { return p.ty + 8 * i + (N == 64 ? 32 * (p.w & 1) : 0); }
  __device__ __forceinline__ static int k_of(Pos p, int j) {
    return p.tx + 4 * j + (K / PARTS) * (N == 64 ? p.w >> 1 : p.w);
  }
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < KT; ++j) acc[i][j] = 0.0f;
  }
  __device__ __forceinline__ void add(const float* D, const float* X, Pos p) {
    const float* d = D + n_of(p, 0) * kFS;
    const float* x = X + k_of(p, 0) * kFS;
#pragma unroll 1
    for (int t = 0; t < kFT; t += 4) {
      float4 dv[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) dv[i] = *reinterpret_cast<const float4*>(d + 8 * i * kFS + t);
#pragma unroll
      for (int j = 0; j < KT; ++j) {
        const float4 xv = *reinterpret_cast<const float4*>(x + 4 * j * kFS + t);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          acc[i][j] = fmaf(dv[i].x, xv.x, acc[i][j]);
          acc[i][j] = fmaf(dv[i].y, xv.y, acc[i][j]);
          acc[i][j] = fmaf(dv[i].z, xv.z, acc[i][j]);
          acc[i][j] = fmaf(dv[i].w, xv.w, acc[i][j]);
        }
      }
    }
  }
  __device__ __forceinline__ void flush(float* dW, Pos p, int rows, int cols) const {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < KT; ++j)
        if (n_of(p, i) < rows && k_of(p, j) < cols) atomicAdd(dW + (size_t)n_of(p, i) * cols + k_of(p, j), acc[i][j]);
  }
};

constexpr int kBwdCP = 32;   // outputs of the fused adjoint, padded

__host__ __device__ constexpr int f32_bwd_groups(int LP) { return LP == 32 ? 3 : 2; }
__host__ __device__ constexpr int f32_bwd_floats(int HP, int LP) {
  return 2 * LP * HP + 2 * HP * HP + kBwdCP * HP + 2 * HP + f32_bwd_groups(LP) * (LP + 2 * HP + kBwdCP) * kFS;
}

// Sum of v over the 8 lanes of a warp that share tx (the texel quads).
__device__ __forceinline__ float sum_ty(float v) {
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Per tile: the forward's hidden layers again, then the layers' adjoints,
// each written over the activation that it has just consumed (H2 becomes
// dH2, H1 becomes dH1), so that a group holds X, H1, H2 and dY: 52 KB, three
// groups per SM beside 57 KB of weights (both orders of W0 and W1).  The
// weight gradients stay in registers over the group's tiles (64 per thread)
// and are added to the gradient vector once at the end; dX goes to the
// workspace for k_table_grad.
template <int HP, int LP>
__global__ void __launch_bounds__(f32_bwd_groups(LP) * kFG, 1)
    k_mlp_bwd_f32(const F32BwdArgs a, const __grid_constant__ Enc e) {
  constexpr int G = f32_bwd_groups(LP);
  extern __shared__ __align__(16) float fsm[];
  float* W0 = fsm;                   // [LP][HP]  layer 0
  float* W1 = W0 + LP * HP;          // [HP][HP]  layer 1
  float* W2r = W1 + HP * HP;         // [CP][HP]  dH2 = dY W2
  float* W1r = W2r + kBwdCP * HP;    // [HP][HP]  dH1 = dH2 W1
  float* W0r = W1r + HP * HP;        // [HP][LP]  dX = dH1 W0
  float* b0 = W0r + HP * LP;
  float* b1 = b0 + HP;
  const int g = threadIdx.x & (kFG - 1), group = threadIdx.x / kFG;
  float* X = b1 + HP + group * (LP + 2 * HP + kBwdCP) * kFS;
  float* H1 = X + LP * kFS;
  float* H2 = H1 + HP * kFS;
  float* dY = H2 + HP * kFS;
  const Pos p{g >> 5, g & 7, (g >> 3) & 3};
  stage_t(W0, a.W0, a.hidden, a.LF, LP, HP);
  stage_t(W1, a.W1, a.hidden, a.hidden, HP, HP);
  stage_r(W2r, a.W2, a.C, a.hidden, kBwdCP, HP);
  stage_r(W1r, a.W1, a.hidden, a.hidden, HP, HP);
  stage_r(W0r, a.W0, a.hidden, a.LF, HP, LP);
  stage_v(b0, a.b0, a.hidden, HP);
  stage_v(b1, a.b1, a.hidden, HP);
  const int K0 = (a.LF + 3) & ~3, KC = (a.C + 3) & ~3;
  // inputs beyond LF and outputs beyond C are zero throughout
  for (int k = a.LF + (g >> 6); k < LP; k += 2) X[k * kFS + (g & 63)] = 0.0f;
  for (int c = a.C + (g >> 6); c < kBwdCP; c += 2) dY[c * kFS + (g & 63)] = 0.0f;
  __syncthreads();
  Wgrad<HP, HP> g1;
  Wgrad<kBwdCP, HP> g2;
  Wgrad<HP, LP> g0;
  g1.clear();
  g2.clear();
  g0.clear();
  float s1[4] = {0.f, 0.f, 0.f, 0.f}, s0[4] = {0.f, 0.f, 0.f, 0.f}, s2 = 0.0f;
  const int tiles = (a.count + kFT - 1) / kFT;
  for (int tile = blockIdx.x + gridDim.x * group; tile < tiles; tile += gridDim.x * G) {
    const int i0 = tile * kFT, live = min(kFT, a.count - i0);
    {   // dY: two threads per texel, half of the channels each
      const int i = g & 63;
      const float* src = a.grad + (size_t)(a.n0 + i0 + i) * a.pitch + a.ch0;
      if (a.vec) {
        for (int c = 4 * (g >> 6); c < a.C; c += 8) {
          float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
          if (i < live) {
            if (c + 4 <= a.C) v = __ldg(reinterpret_cast<const float4*>(src + c));
            else {
              v.x = __ldg(src + c);
              if (c + 1 < a.C) v.y = __ldg(src + c + 1);
              if (c + 2 < a.C) v.z = __ldg(src + c + 2);
            }
          }
          dY[c * kFS + i] = v.x;
          dY[(c + 1) * kFS + i] = v.y;
          dY[(c + 2) * kFS + i] = v.z;
          dY[(c + 3) * kFS + i] = v.w;
        }
      } else {
        for (int c = g >> 6; c < a.C; c += 2) dY[c * kFS + i] = i < live ? __ldg(src + c) : 0.0f;
      }
    }
    encode_tile(e, a.table, a.W, a.H, a.n0 + i0, live, X, g);
    group_sync(group);
    {
      Out<HP> o;
      product<HP>(X, W0, K0, p, o);
      store_relu<HP>(o, b0, p, live, H1);
      group_sync(group);
      product<HP>(H1, W1, HP, p, o);
      store_relu<HP>(o, b1, p, live, H2);
      group_sync(group);
    }
    // db2: four threads per output, 16 texels each
#pragma unroll
    for (int t = 0; t < 16; t += 4) {
      const float4 v = *reinterpret_cast<const float4*>(dY + (g >> 2) * kFS + 16 * (g & 3) + t);
      s2 += (v.x + v.y) + (v.z + v.w);
    }
    g2.add(dY, H2, p);
    {
      Out<HP> o;
      product<HP>(dY, W2r, KC, p, o);
      group_sync(group);   // everybody has read H2
      mask_in_place<HP>(o, p, H2, s1);
      group_sync(group);
    }
    g1.add(H2, H1, p);
    {
      Out<HP> o;
      product<HP>(H2, W1r, HP, p, o);
      group_sync(group);
      mask_in_place<HP>(o, p, H1, s0);
      group_sync(group);
    }
    g0.add(H1, X, p);
    {
      Out<LP> o;
      product<LP>(H1, W0r, HP, p, o);
      const int k0 = Out<LP>::unit(p);
#pragma unroll
      for (int q = 0; q < Out<LP>::Q; ++q) {
        const int t = Out<LP>::texel(p, q);
        if (a.F == 2 && (a.count & 1) == 0 && k0 + 4 <= a.LF && t + 4 <= live) {
          // 4 texels x 2 features of a level: 32 contiguous bytes
#pragma unroll
          for (int j = 0; j < 4; j += 2) {
            const float4 u = o.quad(q, j), v = o.quad(q, j + 1);
            float4* d = reinterpret_cast<float4*>(a.dX + ((size_t)((k0 + j) >> 1) * a.count + i0 + t) * 2);
            d[0] = make_float4(u.x, v.x, u.y, v.y);
            d[1] = make_float4(u.z, v.z, u.w, v.w);
          }
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if (k0 + j >= a.LF) continue;
            const int l = (k0 + j) / a.F, f = (k0 + j) - l * a.F;
            float* d = a.dX + ((size_t)l * a.count + i0 + t) * a.F + f;
            const float4 u = o.quad(q, j);
            if (t < live) d[0] = u.x;
            if (t + 1 < live) d[a.F] = u.y;
            if (t + 2 < live) d[2 * a.F] = u.z;
            if (t + 3 < live) d[3 * a.F] = u.w;
          }
        }
      }
    }
    group_sync(group);   // X, H1, H2 and dY are the next tile's
  }
  g2.flush(a.dW2, p, a.C, a.hidden);
  g1.flush(a.dW1, p, a.hidden, a.hidden);
  g0.flush(a.dW0, p, a.hidden, a.LF);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int n = Out<HP>::unit(p) + j;
    const float u = sum_ty(s1[j]), v = sum_ty(s0[j]);
    if (p.ty == 0 && n < a.hidden) {
      atomicAdd(a.db1 + n, u);
      atomicAdd(a.db0 + n, v);
    }
  }
  s2 += __shfl_xor_sync(0xffffffffu, s2, 1);
  s2 += __shfl_xor_sync(0xffffffffu, s2, 2);
  if ((g & 3) == 0 && (g >> 2) < a.C) atomicAdd(a.db2 + (g >> 2), s2);
}

}  // namespace vsn
