// Surrogate EOS: an ensemble of MLPs 2 -> 128 -> 128 -> 128 -> 2 (tanh) mapping
// normalised (rho, e) to normalised (P, T), trained on MD answers of this library,
// used as a gate in front of the MD path (queries on which the ensemble disagrees
// fall back to MD).
//
// Precision (BF16 weights, FP32 accumulation): weight matrices enter every product
// rounded to bfloat16; hidden activations h1..h3 and the error signals dz2, dz3 that
// feed tensor-core products are bfloat16; biases, pre-activations, outputs, gradients
// and the Adam state are FP32 (FP32 master weights).
//
// The 128x128 layers (forward Z = H W^T, backward dW = dZ^T H and dH = dZ W) run on the
// 5th-generation tensor cores (tcgen05.mma, bf16 x bf16 -> fp32 in tensor memory): fused
// kernels for inference and for the forward and backward pass of a training batch, one
// GEMM for the rest; the 2-wide layers and the elementwise steps run on the CUDA cores.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <random>
#include <string>
#include <vector>

#include "mdeos_host.h"

namespace mdeos {

constexpr int kH = 128;
// parameter offsets of one model: W1[128,2] b1 W2[128,128] b2 W3[128,128] b3 W4[2,128] b4[2]
constexpr int kOffW1 = 0, kOffB1 = kOffW1 + kH * 2, kOffW2 = kOffB1 + kH;
constexpr int kOffB2 = kOffW2 + kH * kH, kOffW3 = kOffB2 + kH, kOffB3 = kOffW3 + kH * kH;
constexpr int kOffW4 = kOffB3 + kH, kOffB4 = kOffW4 + 2 * kH, kNParam = kOffB4 + 2;

// ---------------------------------------------------------------------------
// C[z](m, n) = sum_k A[z](m, k) B[z](k, n): bf16 operands with arbitrary strides (in
// elements), fp32 result (bf16_gemm_tc_kernel below).
struct GemmArgs {
  const __nv_bfloat16* A;
  const __nv_bfloat16* B;
  float* C;
  int M, N, K;
  long long sa_m, sa_k, sa_z, sb_k, sb_n, sb_z, sc_m, sc_n, sc_z;
  // split of K over S CTAs per tile (kchunk elements of K each, a multiple of the
  // staged chunk): with S > 1 every CTA writes its partial tile to ws[s][z][m][n]
  // (dense), summed in the order s = 0, 1, ... by gemm_splitk_reduce
  int S, kchunk;
  float* ws;
  // a second batch of products of the same shape, z >= z2 of Z in all (z2 = Z: none)
  const __nv_bfloat16 *A2, *B2;
  float* C2;
  int z2, Z;
};

// ---------------------------------------------------------------------------
// elementwise parts; index layout [model][sample][unit]

// two FP32 values in one register pair; the packed instructions round each half as the
// scalar ones do
__device__ __forceinline__ uint64_t f2_pack(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void f2_unpack(uint64_t v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// tanh for the hidden layers, whose outputs are rounded to bf16 next (half an ulp:
// 2^-9 relative).  |x| >= 1/4: tanh|x| = 1 - 2 / (1 + e^{2|x|}) with e^{2|x|} =
// 2^{2|x| log2 e} from ex2.approx and the reciprocal from rcp.approx; |x| < 1/4, where
// that form cancels: the odd series x (1 - x^2/3 + 2x^4/15 - 17x^6/315), whose first
// omitted term is below 4e-7 relative there.  Relative error below 2e-6 everywhere
// (3.8e-7 with exact exp2 and division; the approximate instructions add at most ~5e-7,
// largest near |x| = 1/4), so a bf16 rounding differs from that of the exact tanh only
// within 2e-6 of a rounding boundary.  Saturates to +-1 for large |x|; NaN stays NaN.
// Two values at a time: the multiply-adds in packed form fill half the issue slots (the
// special-function results bound the rest).  |x| c = |x c| and x poly = copysign(|x| poly, x)
// exactly, so the absolute value is taken by the exponential and the small branch keeps its
// sign by itself.
__device__ __forceinline__ void tanh_act2(uint64_t x, float& t0, float& t1) {
  const uint64_t one = f2_pack(1.0f, 1.0f);
  float x0, x1, a0, a1, e0, e1, r0, r1, b0, b1, s0, s1;
  f2_unpack(x, x0, x1);
  f2_unpack(f2_mul(x, f2_pack(2.885390081777927f, 2.885390081777927f)), a0, a1);  // 2 log2(e)
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e0) : "f"(fabsf(a0)));
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e1) : "f"(fabsf(a1)));
  f2_unpack(f2_add(one, f2_pack(e0, e1)), e0, e1);
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0) : "f"(e0));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r1) : "f"(e1));
  f2_unpack(f2_fma(f2_pack(-2.0f, -2.0f), f2_pack(r0, r1), one), b0, b1);
  const uint64_t x2 = f2_mul(x, x);
  uint64_t p = f2_fma(x2, f2_pack(-17.0f / 315.0f, -17.0f / 315.0f), f2_pack(2.0f / 15.0f, 2.0f / 15.0f));
  p = f2_fma(x2, p, f2_pack(-1.0f / 3.0f, -1.0f / 3.0f));
  p = f2_fma(x2, p, one);
  f2_unpack(f2_mul(x, p), s0, s1);
  t0 = fabsf(x0) < 0.25f ? s0 : copysignf(b0, x0);
  t1 = fabsf(x1) < 0.25f ? s1 : copysignf(b1, x1);
}

__device__ __forceinline__ float tanh_act(float x) {
  float t0, t1;
  tanh_act2(f2_pack(x, x), t0, t1);
  return t0;
}

// refresh the bf16 weight copies from the FP32 master parameters
__global__ void mlp_cast_weights(const float* P, __nv_bfloat16* W1b, __nv_bfloat16* W2b,
                                 __nv_bfloat16* W3b, __nv_bfloat16* W4b, __nv_bfloat16* W2t,
                                 __nv_bfloat16* W3t, int E) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const long long n = (long long)E * kH * kH;
  if (i >= n) return;
  const int e = (int)(i / (kH * kH)), r = (int)(i % (kH * kH));
  const float* p = P + (long long)e * kNParam;
  W2b[i] = __float2bfloat16_rn(p[kOffW2 + r]);
  W3b[i] = __float2bfloat16_rn(p[kOffW3 + r]);
  const long long t = (long long)e * kH * kH + (r % kH) * kH + r / kH;  // transposed
  W2t[t] = W2b[i];
  W3t[t] = W3b[i];
  if (r < 2 * kH) {
    W1b[(long long)e * 2 * kH + r] = __float2bfloat16_rn(p[kOffW1 + r]);
    W4b[(long long)e * 2 * kH + r] = __float2bfloat16_rn(p[kOffW4 + r]);
  }
}

// h1 = bf16(tanh(W1 x + b1)); x [B][2] FP32 (normalised, shared by the models)
__global__ void mlp_layer1(const float* X, const float* P, const __nv_bfloat16* W1b,
                           __nv_bfloat16* H1, int B, int E) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= (long long)E * B * kH) return;
  const int j = (int)(i % kH), b = (int)((i / kH) % B), e = (int)(i / ((long long)B * kH));
  const float w0 = __bfloat162float(W1b[(long long)e * 2 * kH + 2 * j]);
  const float w1 = __bfloat162float(W1b[(long long)e * 2 * kH + 2 * j + 1]);
  const float z = X[2 * b] * w0 + X[2 * b + 1] * w1 + P[(long long)e * kNParam + kOffB1 + j];
  H1[i] = __float2bfloat16_rn(tanh_act(z));
}

// h = bf16(tanh(Z + b)) for layers 2 and 3
__global__ void mlp_bias_tanh(const float* Z, const float* P, int off_b, __nv_bfloat16* Hout,
                              int B, int E) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= (long long)E * B * kH) return;
  const int j = (int)(i % kH), e = (int)(i / ((long long)B * kH));
  Hout[i] = __float2bfloat16_rn(tanh_act(Z[i] + P[(long long)e * kNParam + off_b + j]));
}

// y = W4 h3 + b4 (FP32 accumulation)
__global__ void mlp_output(const __nv_bfloat16* H3, const float* P, const __nv_bfloat16* W4b,
                           float* Y, int B, int E) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= (long long)E * B * 2) return;
  const int o = (int)(i % 2), b = (int)((i / 2) % B), e = (int)(i / (2LL * B));
  const __nv_bfloat16* h = H3 + ((long long)e * B + b) * kH;
  const __nv_bfloat16* w = W4b + (long long)e * 2 * kH + o * kH;
  float y = 0.f;
  for (int j = 0; j < kH; ++j) y = fmaf(__bfloat162float(w[j]), __bfloat162float(h[j]), y);
  Y[i] = y + P[(long long)e * kNParam + kOffB4 + o];
}

template <int BYTES>
__device__ __forceinline__ void cp_async(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;"
               ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "n"(BYTES) : "memory");
}

// Gradients that are sums over the batch alone: dW4, db4 (from dy, h3), db3, db2, db1
// (columns of dz3, dz2, dz1) and dW1 (dz1, x).  Each is one FP32 sum over b = 0, 1, ...
// in order, a chain of B dependent additions (1 us at B = 512); with the loads in the
// chain it took 40 us per kernel, five kernels.  Here a CTA (32 columns of one model)
// copies kColRows rows of its operands at a time into a ring of kColStages in shared memory
// with cp.async, and four warps walk a sum each through them.  Part 0 has dW4, db3 and
// db4, part 1 has dW1, db2 and db1: the walk is bound by shared-memory loads (one or two per
// row and sum), so the eight sums of 32 columns go to two SMs.
constexpr int kColRows = 128, kColStages = 4;
struct ColStage {                     // part 0 / part 1
  float f[kColRows][32];              // - / dz1
  __nv_bfloat16 a[kColRows][32];      // dz3 / dz2
  __nv_bfloat16 h[kColRows][32];      // h3 / -
  float p[kColRows][2];               // dy / x
};
constexpr int kColSmem = kColStages * (int)sizeof(ColStage);

struct ColArgs {
  const float *dY, *dZ1, *X;
  const __nv_bfloat16 *H3, *dZ3, *dZ2;
  float* G;
  int B;
  const float* part;  // sums of squared errors of npart tiles
  int npart;
  float* loss;
};

__device__ __forceinline__ void column_grads(const ColArgs& a, int e, int block, int part,
                                             unsigned char* sm) {
  ColStage* st = reinterpret_cast<ColStage*>(sm);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int j0 = block * 32, j = j0 + lane, B = a.B;
  const long long r0 = (long long)e * B;  // the model's first row
  auto load = [&](int k) {                // chunk k of the batch, at most kColRows rows
    const int b0 = k * kColRows, rows = min(kColRows, B - b0);
    ColStage& s = st[k & (kColStages - 1)];
    const __nv_bfloat16* dz = part == 0 ? a.dZ3 : a.dZ2;
    for (int q = tid; q < rows * 4; q += 256) {  // bf16 rows: four 16-byte pieces
      const int r = q >> 2, c = (q & 3) * 8;
      const long long at = (r0 + b0 + r) * kH + j0 + c;
      cp_async<16>(&s.a[r][c], dz + at);
      if (part == 0) cp_async<16>(&s.h[r][c], a.H3 + at);
    }
    if (part != 0)
      for (int q = tid; q < rows * 8; q += 256)
        cp_async<16>(&s.f[q >> 3][(q & 7) * 4], a.dZ1 + (r0 + b0 + (q >> 3)) * kH + j0 + (q & 7) * 4);
    for (int q = tid; q < rows; q += 256)
      cp_async<8>(s.p[q], part == 0 ? a.dY + (r0 + b0 + q) * 2 : a.X + (long long)(b0 + q) * 2);
  };
  if (e == 0 && block == 0 && part == 0 && warp == 7 && lane == 0) {
    // in order (reproducible), the rounding errors of the sum added at its end (a sum that
    // has overflowed has none: its difference of infinities would make it a NaN)
    float l = 0.f, c = 0.f;
#pragma unroll 8
    for (int k = 0; k < a.npart; ++k) {
      const float t = a.part[k], n = l + t, d = n - l;
      c += (l - (n - d)) + (t - d);
      l = n;
    }
    *a.loss = isfinite(l) ? l + c : l;
  }
  const int nk = (B + kColRows - 1) / kColRows;
  for (int k = 0; k < kColStages - 1; ++k) {
    if (k < nk) load(k);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  float sum = 0.f;
  for (int k = 0; k < nk; ++k) {
    if (k + kColStages - 1 < nk) load(k + kColStages - 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_group %0;" ::"n"(kColStages - 1) : "memory");
    __syncthreads();
    const ColStage& s = st[k & (kColStages - 1)];
    const int rows = min(kColRows, B - k * kColRows);
    if (warp < 2) {  // dW4 / dW1
      if (part == 0) {
#pragma unroll 16
        for (int r = 0; r < rows; ++r) sum = fmaf(s.p[r][warp], __bfloat162float(s.h[r][lane]), sum);
      } else {
#pragma unroll 16
        for (int r = 0; r < rows; ++r) sum = fmaf(s.f[r][lane], s.p[r][warp], sum);
      }
    } else if (warp == 2) {  // db3 / db2
#pragma unroll 16
      for (int r = 0; r < rows; ++r) sum += __bfloat162float(s.a[r][lane]);
    } else if (warp == 3) {  // db4 / db1
      if (part == 0) {
#pragma unroll 16
        for (int r = 0; r < rows; ++r) sum += s.p[r][lane & 1];
      } else {
#pragma unroll 16
        for (int r = 0; r < rows; ++r) sum += s.f[r][lane];
      }
    }
    __syncthreads();  // the stage is filled again in the next turn
  }
  float* g = a.G + (long long)e * kNParam;
  if (warp < 2)
    g[part == 0 ? kOffW4 + warp * kH + j : kOffW1 + 2 * j + warp] = sum;
  else if (warp == 2)
    g[(part == 0 ? kOffB3 : kOffB2) + j] = sum;
  else if (warp == 3 && part != 0)
    g[kOffB1 + j] = sum;
  else if (warp == 3 && block == 0 && lane < 2)
    g[kOffB4 + lane] = sum;
}

// Adam (Kingma & Ba) on the FP32 master parameters; omb = 1 - beta and c = 1 - beta^t,
// each evaluated in FP64 on the host and rounded once.  The 128 x 128 weight gradients
// come as S partial tiles per model (ws[s][which][e][m][n], which 0: W3, 1: W2), added in
// the order s = 0, 1, ...; the bf16 copies (W2 and W3 also transposed, for the products
// with dZ) are refreshed with the parameter.
struct AdamArgs {
  float *P, *Mm, *Vv;
  const float *G, *ws;
  __nv_bfloat16 *W1b, *W2b, *W3b, *W4b, *W2t, *W3t;
  int E, S;
  float lr, b1, b2, omb1, omb2, eps, c1, c2;
};

__global__ void mlp_adam(AdamArgs a) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x, e = blockIdx.y;
  if (r >= kNParam) return;
  const long long i = (long long)e * kNParam + r;
  const bool w2 = r >= kOffW2 && r < kOffB2, w3 = r >= kOffW3 && r < kOffB3;
  float g;
  if ((w2 || w3) && a.S > 1) {
    const long long part = 2LL * a.E * kH * kH;
    const float* p = a.ws + ((long long)(w2 ? a.E : 0) + e) * kH * kH + (r - (w2 ? kOffW2 : kOffW3));
    g = p[0];
#pragma unroll 4
    for (int s = 1; s < a.S; ++s) g += p[s * part];
  } else {
    g = a.G[i];
  }
  const float m = a.b1 * a.Mm[i] + a.omb1 * g;
  const float v = a.b2 * a.Vv[i] + a.omb2 * g * g;
  a.Mm[i] = m;
  a.Vv[i] = v;
  const float p = a.P[i] - a.lr * (m / a.c1) / (sqrtf(v / a.c2) + a.eps);
  a.P[i] = p;
  const __nv_bfloat16 pb = __float2bfloat16_rn(p);
  if (w2 || w3) {
    const int q = r - (w2 ? kOffW2 : kOffW3);
    const long long at = (long long)e * kH * kH;
    (w2 ? a.W2b : a.W3b)[at + q] = pb;
    (w2 ? a.W2t : a.W3t)[at + (q % kH) * kH + q / kH] = pb;
  } else if (r < kOffB1) {
    a.W1b[(long long)e * 2 * kH + r] = pb;
  } else if (r >= kOffW4 && r < kOffB4) {
    a.W4b[(long long)e * 2 * kH + r - kOffW4] = pb;
  }
}

// normalise physical inputs (rho, e) -> x, per sample
__global__ void mlp_normalise(const double* Xp, float* X, int B, double m0, double m1, double s0,
                              double s1) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  X[2 * b] = (float)((Xp[2 * b] - m0) / s0);
  X[2 * b + 1] = (float)((Xp[2 * b + 1] - m1) / s1);
}

// ensemble mean and (population) standard deviation of the physical outputs; with
// p_asinh the networks predict asinh(P), mapped back by sinh before averaging; inv = 1 / E
// where E is a power of two, else 0
__global__ void mlp_ensemble(const float* Y, int B, int E, double ym0, double ym1, double ys0,
                             double ys1, int p_asinh, double inv, double* mean,
                             double* sd) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= B * 2) return;
  const int o = i % 2;
  const double m = o ? ym1 : ym0, s = o ? ys1 : ys0;
  double a = 0.0, q = 0.0;
  for (int e = 0; e < E; ++e) {
    double y = (double)Y[(long long)e * B * 2 + i] * s + m;
    if (o == 0 && p_asinh) y = sinh(y);
    a += y;
    q += y * y;
  }
  // a power of two divides exactly as a product (a division is ten instructions of the
  // FP64 pipe, which bounds this kernel)
  if (inv > 0.0) {
    a *= inv;
    q *= inv;
  } else {
    a /= E;
    q /= E;
  }
  mean[i] = a;
  sd[i] = sqrt(fmax(q - a * a, 0.0));
}

// ---------------------------------------------------------------------------
// Fused inference on the 5th-generation tensor cores, in tiles of 128 samples of one
// model.  Layer 1 (2 -> 128) runs on the CUDA cores and writes h1 into shared memory;
// layers 2 and 3 are tcgen05.mma (M = N = 128, K = 128 in steps of 16, bf16 x bf16 ->
// fp32) with the accumulator in tensor memory (128 columns), completion signalled on
// an mbarrier; threads read their row back (tcgen05.ld, 32 columns at a time), add
// the bias, apply tanh and write the next operand into the same tile; the 128 -> 2
// output layer reads h3 back from shared memory.
//
// Operand layout in shared memory (no swizzle, K contiguous): 8 x 8 "core matrices"
// of 128 bytes; element (r, k) at (r / 8) * SBO + (k / 8) * LBO + (r % 8) * 16 +
// (k % 8) * 2 with LBO = 128 B (next core matrix along K) and SBO = 2048 B (next
// 8-row group).  Every address an MMA can form stays inside its 32 KB tile.

constexpr int kTcRows = 128;                   // samples per tile (TMEM lanes)
constexpr int kTcThreads = 256;                // two threads per row (column halves)
constexpr uint32_t kLbo = 128, kSbo = 2048;    // bytes
constexpr int kTcTile = kH * kH * 2;           // 32 KB per operand tile
// FP32 copies of the small parameters behind the tiles and the mbarrier: W1 as
// (w_c0, w_c1) pairs, b1, b2, b3, W4 (output-major), b4
constexpr int kTcSW1 = 0, kTcSB1 = kTcSW1 + 2 * kH, kTcSB2 = kTcSB1 + kH, kTcSB3 = kTcSB2 + kH;
constexpr int kTcSW4 = kTcSB3 + kH, kTcSB4 = kTcSW4 + 2 * kH, kTcSmall = kTcSB4 + 4;

__device__ __forceinline__ uint32_t tc_off(int r, int k) {
  return (uint32_t)((r >> 3) * kSbo + (k >> 3) * kLbo + (r & 7) * 16 + (k & 7) * 2);
}

// shared-memory matrix descriptor: start, LBO, SBO (all >> 4), version 1, no swizzle
__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr) {
  return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)((kLbo >> 4) & 0x3FFF) << 16) |
         ((uint64_t)((kSbo >> 4) & 0x3FFF) << 32) | (1ull << 46);
}

// instruction descriptor, kind::f16: D f32, A and B bf16, both K-major, N = M = 128
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kH >> 3) << 17) |
                            ((uint32_t)(kTcRows >> 4) << 24);

__device__ __forceinline__ void tc_mma(uint32_t tmem, uint64_t a, uint64_t b, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem), "l"(a), "l"(b), "r"(kIdesc), "r"(acc));
}

__device__ __forceinline__ void tc_commit(uint32_t mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
               ::"r"(mbar) : "memory");
}

__device__ __forceinline__ unsigned long long tc_clock_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

// wait on an mbarrier phase for at most ~1 s; false if it did not complete
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity) {
  unsigned long long t0 = 0;
  for (int it = 0; it < (1 << 24); ++it) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done) : "r"(mbar), "r"(parity) : "memory");
    if (done) return true;
    if ((it & 255) == 255) {
      const unsigned long long t = tc_clock_ns();
      if (t0 == 0) t0 = t;
      if (t - t0 > 1000000000ull) break;
    }
  }
  return false;
}

// 32 consecutive fp32 accumulator columns of this thread's TMEM lane
__device__ __forceinline__ void tc_ld32(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
      "%12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, "
      "%30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
        "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
        "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
}

// bf16(tanh(z + bias)) of 8 consecutive units, packed as one 16-byte core-matrix row
__device__ __forceinline__ uint4 tanh_pack8(const float* z, const float* bias) {
  uint4 pk;
  __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&pk);
#pragma unroll
  for (int j = 0; j < 8; j += 2) {
    float t0, t1;
    tanh_act2(f2_add(f2_pack(z[j], z[j + 1]), f2_pack(bias[j], bias[j + 1])), t0, t1);
    h[j >> 1] = __floats2bfloat162_rn(t0, t1);
  }
  return pk;
}

// Persistent: grid (CTAs per model, models), one CTA per SM.  The CTA stages its model's
// W2 and W3 once; its groups of 256 threads (up to kTcGroups, each with its own tile A, TMEM
// columns, mbarrier and named barrier) then take 128-input tiles independently.  Thread t
// of a group serves row m = t % 128 (TMEM lane m) and column half t / 128: warps w and w + 4
// read the same 32 lanes, columns 0-63 and 64-127.
//
// What bounds it is the 384 tanh per row: their issue slots (74 % of all, measured), and their
// special-function results (an exp2 at 32 and a reciprocal at 16 per clock and SM, measured:
// 9.2k cycles for two tiles).  A tile alternates between its product and its tanh, so other
// tiles have to fill the gaps: with two CTAs of 256 threads per SM, each with its own copy of
// the weights (101 KB), two tiles took 21.5k cycles; four groups around one copy (197 KB, all
// 512 TMEM columns) fill them (2^20 queries, normalising and averaging included: 1348 us
// before, 1104 now).
constexpr int kTcGroups = 4;
constexpr int infer_tc_smem(int groups) {
  return (2 + groups) * kTcTile + 1024 + 128 + kTcSmall * 4;
}

__device__ __forceinline__ void group_bar(int id) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(kTcThreads) : "memory");
}
__device__ __forceinline__ bool group_bar_and(int id, bool p) {
  int r;
  asm volatile(
      "{\n\t.reg .pred pi, po;\n\t"
      "setp.ne.s32 pi, %3, 0;\n\t"
      "bar.red.and.pred po, %1, %2, pi;\n\t"
      "selp.s32 %0, 1, 0, po;\n\t}"
      : "=r"(r) : "r"(id), "n"(kTcThreads), "r"((int)p) : "memory");
  return r != 0;
}

// GROUPS: a compile-time bound on the threads, so that one group, which has the SM to itself,
// has all the registers its chain of loads and products can use (64 a thread with four groups;
// 1000 queries, 4 models: 25.8 us so, 23.0 with 80).
template <int GROUPS>
__global__ void __launch_bounds__(GROUPS * kTcThreads, 1)
    mlp_infer_tc_kernel(const float* X, const float* P, const __nv_bfloat16* W1b,
                        const __nv_bfloat16* W2b, const __nv_bfloat16* W3b,
                        const __nv_bfloat16* W4b, float* Y, int B, int* err) {
  extern __shared__ __align__(1024) unsigned char tsm[];
  const uint32_t sbase = ((uint32_t)__cvta_generic_to_shared(tsm) + 1023u) & ~1023u;
  unsigned char* gbase = tsm + (sbase - (uint32_t)__cvta_generic_to_shared(tsm));
  constexpr int groups = GROUPS;
  const int e = blockIdx.y, tid = threadIdx.x % kTcThreads, grp = threadIdx.x / kTcThreads;
  const int warp = tid >> 5, bar = 1 + grp;
  const uint32_t sW2 = sbase, sW3 = sbase + kTcTile;
  const uint32_t sA = sbase + (uint32_t)(2 + grp) * kTcTile;
  unsigned char* gA = gbase + (2 + grp) * kTcTile;
  // behind the tiles: an mbarrier per group, the TMEM address, the small parameters
  const uint32_t sCtl = sbase + (uint32_t)(2 + groups) * kTcTile;
  unsigned char* gCtl = gbase + (2 + groups) * kTcTile;
  const uint32_t sMbar = sCtl + 8u * (uint32_t)grp, sTmem = sCtl + 64;
  const int m = tid & (kTcRows - 1), half = tid >> 7, c_lo = half * (kH / 2);
  const int ntiles = (B + kTcRows - 1) / kTcRows;
  const float* p = P + (long long)e * kNParam;
  float* sp = reinterpret_cast<float*>(gCtl + 128);  // small parameters
  for (int k = threadIdx.x; k < 2 * kH; k += blockDim.x) {  // the bf16-rounded weights, as FP32
    sp[kTcSW1 + k] = __bfloat162float(W1b[(long long)e * 2 * kH + k]);
    sp[kTcSW4 + k] = __bfloat162float(W4b[(long long)e * 2 * kH + k]);
  }
  for (int k = threadIdx.x; k < kH; k += blockDim.x) {
    sp[kTcSB1 + k] = p[kOffB1 + k];
    sp[kTcSB2 + k] = p[kOffB2 + k];
    sp[kTcSB3 + k] = p[kOffB3 + k];
  }
  if (threadIdx.x < 2) sp[kTcSB4 + threadIdx.x] = p[kOffB4 + threadIdx.x];
  const float* w4 = sp + kTcSW4 + half * kH;  // output unit = half
  // weights of this model into the canonical layout, 16 bytes at a time; consecutive
  // threads fill consecutive 16-byte rows of the core matrices (no bank conflicts)
  for (int q = threadIdx.x; q < kH * kH / 8; q += blockDim.x) {
    const int n = (q >> 7) * 8 + (q & 7), k = ((q >> 3) & 15) * 8;
    const uint4 a2 = *reinterpret_cast<const uint4*>(W2b + (long long)e * kH * kH + n * kH + k);
    const uint4 a3 = *reinterpret_cast<const uint4*>(W3b + (long long)e * kH * kH + n * kH + k);
    *reinterpret_cast<uint4*>(gbase + tc_off(n, k)) = a2;
    *reinterpret_cast<uint4*>(gbase + kTcTile + tc_off(n, k)) = a3;
  }
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sMbar) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // 128 TMEM columns per group (its 128 x 128 fp32 accumulator), a power of two in all
  constexpr uint32_t cols = groups * kH;
  if (threadIdx.x < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(sTmem), "r"(cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // weights -> tensor core
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(gCtl + 64);
  const uint32_t tacc = tmem + (uint32_t)(grp * kH);  // the group's accumulator
  // this thread's lane quarter (warp % 4) and column half
  const uint32_t tq = tacc + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c_lo;
  uint32_t commits = 0;  // MMA groups committed so far (mbarrier phase parity)
  bool ok = true;
  const int tstep = gridDim.x * groups;
  int tile = blockIdx.x + grp * gridDim.x;
  for (; tile < ntiles; tile += tstep) {
    const int b = tile * kTcRows + m;
    // layer 1 on the CUDA cores: this row's units c_lo .. c_lo + 63 -> tile A
    const float x0 = b < B ? X[2 * b] : 0.f, x1 = b < B ? X[2 * b + 1] : 0.f;
#pragma unroll 1
    for (int c = c_lo; c < c_lo + kH / 2; c += 8) {
      float z[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float2 w = *reinterpret_cast<const float2*>(sp + kTcSW1 + 2 * (c + j));
        z[j] = x0 * w.x + x1 * w.y;
      }
      *reinterpret_cast<uint4*>(gA + tc_off(m, c)) = tanh_pack8(z, sp + kTcSB1 + c);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // h1 -> tensor core
    group_bar(bar);
    for (int layer = 0; layer < 2; ++layer) {
      if (tid == 0) {
        const uint32_t sW = layer == 0 ? sW2 : sW3;
#pragma unroll
        for (int ks = 0; ks < kH / 16; ++ks)  // K step of 16 = two core matrices along K
          tc_mma(tacc, tc_desc(sA + ks * 2 * kLbo), tc_desc(sW + ks * 2 * kLbo), ks > 0);
        tc_commit(sMbar);
      }
      __syncwarp();
      const bool done = mbar_wait(sMbar, commits & 1u);
      ++commits;
      ok = group_bar_and(bar, done);  // the same decision in every thread of the group
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (!ok) break;
      // epilogue: h = bf16(tanh(z + b)) of this row's 64 units -> tile A (the MMA that
      // read it has completed): h2 feeds layer 3, h3 the output layer
      const float* bias = sp + (layer == 0 ? kTcSB2 : kTcSB3) + c_lo;
#pragma unroll 1
      for (int c0 = 0; c0 < kH / 2; c0 += 32) {
        float v[32];
        tc_ld32(tq + (uint32_t)c0, v);
#pragma unroll
        for (int j8 = 0; j8 < 32; j8 += 8)
          *reinterpret_cast<uint4*>(gA + tc_off(m, c_lo + c0 + j8)) =
              tanh_pack8(v + j8, bias + c0 + j8);
      }
      if (layer == 0) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      group_bar(bar);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    }
    if (!ok) break;
    // output unit `half` of row m: sum over the 128 units of h3 in order, FP32
    float y = 0.f;
#pragma unroll 1
    for (int c = 0; c < kH; c += 8) {
      const uint4 pk = *reinterpret_cast<const uint4*>(gA + tc_off(m, c));
      const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&pk);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float2 hf = __bfloat1622float2(h[j]);
        y = fmaf(w4[c + 2 * j], hf.x, y);
        y = fmaf(w4[c + 2 * j + 1], hf.y, y);
      }
    }
    if (b < B) Y[((long long)e * B + b) * 2 + half] = y + sp[kTcSB4 + half];
    group_bar(bar);  // tile A is rewritten by the next tile's layer 1
  }
  if (!ok) {  // NaN for this group's unfinished tiles; let MMAs in flight finish (bounded)
    if (tid == 0) atomicExch(err, 1);
    for (; tile < ntiles; tile += tstep) {
      const int b = tile * kTcRows + m;
      if (b < B) Y[((long long)e * B + b) * 2 + half] = __int_as_float(0x7fc00000);
    }
    mbar_wait(sMbar, (commits - 1u) & 1u);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  __syncwarp();
  if (threadIdx.x < 32)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols)
                 : "memory");
}

// ---------------------------------------------------------------------------
// Forward and backward pass of a training batch in one launch: grid (tiles of 128
// samples, models), the tiles, descriptors and thread roles of mlp_infer_tc_kernel.
//   Z2 = h1 W2^T, Z3 = h2 W3^T, y and dy from h3, dz3 = (dy W4)(1 - h3^2),
//   dh2 = dz3 W3, dz2 = dh2 (1 - h2^2), dh1 = dz2 W2, dz1 = dh1 (1 - h1^2).
// h1..h3, dz3, dz2 (bf16), dz1 and dy (FP32) go to device memory for the sums over the
// batch.  Products accumulate K in the same order of tcgen05.mma steps as
// bf16_gemm_tc_kernel's chunks, and every element is rounded where the layered form rounds it.
//
// A few CTAs walk one serial chain, so what bounds it is the latency of that chain.  All of
// it stays in shared memory, in five tiles of 32 KB: h1, W2, W3 and the transposes of W3 and
// W2.  h2 takes W2's place once its product is done, h3 W3's; dz3 and dz2 overwrite h3 and
// h2, and dz1 (FP32) the transposes.  The weights arrive by cp.async, W2 first.  A finished
// tile goes to device memory while the next product runs, 64 bytes of a row per lane group
// (a thread storing its own row touches 32 lines per store, and reading it back for the
// backward pass again).  Batch 512, 4 models: 27.5 us with the tiles stored and
// read back by rows, 21.4 now; with the sums and Adam a step of an epoch takes 46 us, host
// included (328 us with a launch per layer and product).
constexpr int kTrThreads = 512;    // four threads per row (column quarters)
constexpr int kTrCols = kH / 4;
constexpr int kTrSmem = 5 * kTcTile + 1024 + 64 + (kTcSmall + 4 * kTcRows + 8) * 4;

struct TrainArgs {
  const float *X, *T, *P;
  const __nv_bfloat16 *W1b, *W2b, *W3b, *W4b, *W2t, *W3t;
  __nv_bfloat16 *H1, *H2, *H3, *dZ3, *dZ2;
  float *dZ1, *dY, *part;
  int B;
  int* err;
};

// 16-byte unit u (0..2047) of a tile: eight lanes take eight rows of one core matrix (no bank
// conflicts), a warp 64 bytes of each of those rows
__device__ __forceinline__ void tile_unit(int u, int& r, int& c) {
  r = (u >> 7) * 8 + (u & 7);
  c = (((u >> 5) & 3) * 4 + ((u >> 3) & 3)) * 8;
}

// a tile's first `rows` rows to dst (rows of kH elements), by threads t of nt
__device__ __forceinline__ void store_tile(const unsigned char* tile, __nv_bfloat16* dst, int rows,
                                           int t, int nt) {
#pragma unroll 4
  for (int u = t; u < kTcRows * kH / 8; u += nt) {
    int r, c;
    tile_unit(u, r, c);
    if (r < rows)
      *reinterpret_cast<uint4*>(dst + (long long)r * kH + c) =
          *reinterpret_cast<const uint4*>(tile + tc_off(r, c));
  }
}

// dz = dh (1 - h^2) of eight units, h as packed bf16; returns bf16(dz) packed
__device__ __forceinline__ uint4 dtanh8(float* v, uint4 h) {
  const __nv_bfloat16* h8 = reinterpret_cast<const __nv_bfloat16*>(&h);
  uint4 out;
  __nv_bfloat16* o8 = reinterpret_cast<__nv_bfloat16*>(&out);
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const float x = __bfloat162float(h8[j]);
    v[j] = v[j] * (1.f - x * x);
    o8[j] = __float2bfloat16_rn(v[j]);
  }
  return out;
}

__global__ void __launch_bounds__(kTrThreads) mlp_train_tc_kernel(TrainArgs a) {
  extern __shared__ __align__(1024) unsigned char tsm[];
  const uint32_t sbase = ((uint32_t)__cvta_generic_to_shared(tsm) + 1023u) & ~1023u;
  unsigned char* gbase = tsm + (sbase - (uint32_t)__cvta_generic_to_shared(tsm));
  const uint32_t sMbar = sbase + 5 * kTcTile, sTmem = sMbar + 8;
  unsigned char *const g1 = gbase, *const g2 = gbase + kTcTile, *const g3 = gbase + 2 * kTcTile;
  const int e = blockIdx.y, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m = tid & (kTcRows - 1), quarter = tid >> 7, c_lo = quarter * kTrCols;
  const int B = a.B, b0 = blockIdx.x * kTcRows, b = b0 + m, rows = min(kTcRows, B - b0);
  const bool on = b < B;
  const long long row0 = ((long long)e * B + b0) * kH;  // the tile's first row in the model's arrays
  const float* p = a.P + (long long)e * kNParam;
  float* sp = reinterpret_cast<float*>(gbase + 5 * kTcTile + 64);  // small parameters
  float* sdy = sp + kTcSmall;                                       // dy
  float* ssq = sdy + 2 * kTcRows;                                   // squared errors
  float* spart = ssq + 2 * kTcRows;                                 // their sums by warp
  {  // the four operands, 16 bytes at a time into the canonical layout
    const __nv_bfloat16* w[4] = {a.W2b, a.W3b, a.W3t, a.W2t};
#pragma unroll
    for (int t = 0; t < 4; ++t) {
#pragma unroll
      for (int u = tid; u < kH * kH / 8; u += kTrThreads) {
        int n, k;
        tile_unit(u, n, k);
        cp_async<16>(gbase + (t + 1) * kTcTile + tc_off(n, k),
                     w[t] + (long long)e * kH * kH + n * kH + k);
      }
      if (t == 0) asm volatile("cp.async.commit_group;" ::: "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  for (int k = tid; k < 2 * kH; k += kTrThreads) {
    sp[kTcSW1 + k] = __bfloat162float(a.W1b[(long long)e * 2 * kH + k]);
    sp[kTcSW4 + k] = __bfloat162float(a.W4b[(long long)e * 2 * kH + k]);
  }
  for (int k = tid; k < kH; k += kTrThreads) {
    sp[kTcSB1 + k] = p[kOffB1 + k];
    sp[kTcSB2 + k] = p[kOffB2 + k];
    sp[kTcSB3 + k] = p[kOffB3 + k];
  }
  if (tid < 2) sp[kTcSB4 + tid] = p[kOffB4 + tid];
  const float x0 = on ? a.X[2 * b] : 0.f, x1 = on ? a.X[2 * b + 1] : 0.f;
  const float target = on && quarter < 2 ? a.T[2 * b + quarter] : 0.f;
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sMbar) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {  // 128 TMEM columns: the 128 x 128 fp32 accumulator
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(sTmem), "r"(kH) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(gbase + 5 * kTcTile + 8);
  const uint32_t tq = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c_lo;
  // accumulator = tile A times tile W (by number), once every thread has written its part
  // of tile A and its share of the weights has arrived
  const auto product = [&](int tA, int tW) {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // shared memory -> tensor core
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t sA = sbase + (uint32_t)tA * kTcTile, sW = sbase + (uint32_t)tW * kTcTile;
#pragma unroll
      for (int ks = 0; ks < kH / 16; ++ks)  // K step of 16 = two core matrices along K
        tc_mma(tmem, tc_desc(sA + ks * 2 * kLbo), tc_desc(sW + ks * 2 * kLbo), ks > 0);
      tc_commit(sMbar);
    }
    __syncwarp();
  };
  // the product's end, the same answer in every thread; false: the wait ran out
  int layer = 0;
  const auto finished = [&]() {
    const bool done = mbar_wait(sMbar, (uint32_t)layer & 1u);
    const bool ok = __syncthreads_and(done) != 0;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (ok) ++layer;
    return ok;
  };
  // h = bf16(tanh(z + b)) of this row's 32 units
  const auto hidden = [&](unsigned char* tile, const float* bias) {
    float v[32];
    tc_ld32(tq, v);
#pragma unroll
    for (int j = 0; j < 32; j += 8)
      *reinterpret_cast<uint4*>(tile + tc_off(m, c_lo + j)) = tanh_pack8(v + j, bias + c_lo + j);
  };
  // layer 1 on the CUDA cores
#pragma unroll 1
  for (int c = c_lo; c < c_lo + kTrCols; c += 8) {
    float z[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float2 w = *reinterpret_cast<const float2*>(sp + kTcSW1 + 2 * (c + j));
      z[j] = x0 * w.x + x1 * w.y;
    }
    *reinterpret_cast<uint4*>(g1 + tc_off(m, c)) = tanh_pack8(z, sp + kTcSB1 + c);
  }
  asm volatile("cp.async.wait_group 1;" ::: "memory");  // W2
  product(0, 1);
  store_tile(g1, a.H1 + row0, rows, tid, kTrThreads);
  bool ok = finished();
  if (ok) {
    hidden(g2, sp + kTcSB2);
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    product(1, 2);
    store_tile(g2, a.H2 + row0, rows, tid, kTrThreads);
    ok = finished();
  }
  if (ok) {
    hidden(g3, sp + kTcSB3);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();  // h3 is complete
    if (quarter < 2) {  // output unit = quarter
      const float* w4 = sp + kTcSW4 + quarter * kH;
      float y = 0.f;
#pragma unroll 4
      for (int c = 0; c < kH; c += 8) {
        const uint4 pk = *reinterpret_cast<const uint4*>(g3 + tc_off(m, c));
        const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&pk);
        const float4 wa = *reinterpret_cast<const float4*>(w4 + c);
        const float4 wb = *reinterpret_cast<const float4*>(w4 + c + 4);
        const float w[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float2 hf = __bfloat1622float2(h[j]);
          y = fmaf(w[2 * j], hf.x, y);
          y = fmaf(w[2 * j + 1], hf.y, y);
        }
      }
      y += sp[kTcSB4 + quarter];
      const float d = on ? y - target : 0.f;
      const float dyv = d / (float)B;  // 2 (y - t) / (2 B)
      if (on) a.dY[((long long)e * B + b) * 2 + quarter] = dyv;
      sdy[2 * m + quarter] = dyv;
      ssq[2 * m + quarter] = d * d;
    } else {
      store_tile(g3, a.H3 + row0, rows, tid - kTrThreads / 2, kTrThreads / 2);
    }
    __syncthreads();  // dy of both outputs; h3 has been read
    const float dy0 = sdy[2 * m], dy1 = sdy[2 * m + 1];
#pragma unroll 1
    for (int c = c_lo; c < c_lo + kTrCols; c += 8) {
      float v[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = dy0 * sp[kTcSW4 + c + j] + dy1 * sp[kTcSW4 + kH + c + j];
      uint4* h = reinterpret_cast<uint4*>(g3 + tc_off(m, c));
      *h = dtanh8(v, *h);
    }
    product(2, 3);
    // squared errors in sample order: sums of 32 by shuffles, of 256 in warp order; the
    // tiles' sums are added in order by mlp_batch_sums
    if (warp < 2 * kTcRows / 32) {
      float l = ssq[tid];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
      if (lane == 0) spart[warp] = l;
    }
    store_tile(g3, a.dZ3 + row0, rows, tid, kTrThreads);
    ok = finished();
    if (tid == 0) {
      float t = 0.f;
      for (int w = 0; w < 2 * kTcRows / 32; ++w) t += spart[w];
      a.part[(long long)e * gridDim.x + blockIdx.x] = t;
    }
  }
  if (ok) {
    float v[32];
    tc_ld32(tq, v);
#pragma unroll
    for (int j = 0; j < 32; j += 8) {
      uint4* h = reinterpret_cast<uint4*>(g2 + tc_off(m, c_lo + j));
      *h = dtanh8(v + j, *h);
    }
    product(1, 4);
    store_tile(g2, a.dZ2 + row0, rows, tid, kTrThreads);
    ok = finished();
  }
  if (ok) {
    // dz1 by rows of 512 B, their 16-byte units swapped by row (no bank conflicts), where
    // the transposes were
    float4* z1 = reinterpret_cast<float4*>(gbase + 3 * kTcTile);
    float v[32];
    tc_ld32(tq, v);
#pragma unroll
    for (int j = 0; j < 32; j += 8) {
      dtanh8(v + j, *reinterpret_cast<const uint4*>(g1 + tc_off(m, c_lo + j)));
      const int c = (c_lo + j) >> 2;
      z1[m * 32 + (c ^ (m & 7))] = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
      z1[m * 32 + ((c + 1) ^ (m & 7))] = make_float4(v[j + 4], v[j + 5], v[j + 6], v[j + 7]);
    }
    __syncthreads();
    float4* out = reinterpret_cast<float4*>(a.dZ1 + row0);
#pragma unroll 4
    for (int u = tid; u < kTcRows * 32; u += kTrThreads) {
      const int r = u >> 5, c = u & 31;
      if (r < rows) out[(long long)r * 32 + c] = z1[r * 32 + (c ^ (r & 7))];
    }
  } else {  // the tile's later outputs stay unwritten; let the MMAs in flight finish (bounded)
    if (tid == 0) atomicExch(a.err, 1);
    asm volatile("cp.async.wait_all;" ::: "memory");
    mbar_wait(sMbar, (uint32_t)layer & 1u);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  __syncwarp();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kH)
                 : "memory");
}

// ---------------------------------------------------------------------------
// The training products on the 5th-generation tensor cores: C[z](m, n) =
// sum_k A[z](m, k) B[z](k, n) with arbitrary strides (GemmArgs), one 128 x 128 tile of
// C per CTA with the fp32 accumulator in
// tensor memory.  K runs in chunks of 64, in two pairs of tiles in turn: 128 threads stage A's
// 128 x 64, the other 128 B's (128 columns of C) x 64 elements into the canonical no-swizzle
// K-major layout (8 x 8 core matrices of 128 B: element (r, k) at (r / 8) * 1024 + (k / 8) *
// 128 + (r % 8) * 16 + (k % 8) * 2; zero outside the matrices), one thread issues four
// tcgen05.mma of K = 16 and commits to the pair's mbarrier.  Every thread waits for a pair's
// last product (at most ~1 s, then the error flag is set and the tile is left unwritten)
// before it is filled again.  Epilogue: the accumulator goes through shared memory, so that a
// warp stores rows of C (a thread storing its own row touches 32 lines per store).

constexpr int kGK = 64;                   // K per staged chunk
constexpr uint32_t kGSbo = 1024;          // bytes between 8-row groups of a chunk
constexpr int kGTile = kTcRows * kGK * 2; // 16 KB per operand chunk

__device__ __forceinline__ uint32_t gk_off(int r, int k) {
  return (uint32_t)((r >> 3) * kGSbo + (k >> 3) * kLbo + (r & 7) * 16 + (k & 7) * 2);
}

__device__ __forceinline__ uint64_t gk_desc(uint32_t saddr) {
  return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)((kLbo >> 4) & 0x3FFF) << 16) |
         ((uint64_t)((kGSbo >> 4) & 0x3FFF) << 32) | (1ull << 46);
}

// One K chunk of an operand whose K runs along memory rows and whose row index is
// contiguous (16-byte aligned, in eights): thread t takes the 8 x 8 block (rows 8 (t % 16),
// K 8 (t / 16)), eight 16-byte loads along the rows, and transposes it in registers into
// eight core-matrix rows.  Element loads of the same chunk took 15 us per chunk.
__device__ __forceinline__ void stage_blocks(unsigned char* tile, const __nv_bfloat16* A, int row0,
                                             int rows, long long s_k, int k0, int kend, int t) {
  const int r = (t & 15) * 8, c = (t >> 4) * 8;
  uint4 v[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    v[u] = make_uint4(0u, 0u, 0u, 0u);
    if (row0 + r < rows && k0 + c + u < kend)
      v[u] = *reinterpret_cast<const uint4*>(A + (long long)(k0 + c + u) * s_k + row0 + r);
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    uint32_t w[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint4 lo = v[2 * u], hi = v[2 * u + 1];
      const uint32_t a = i < 2 ? lo.x : i < 4 ? lo.y : i < 6 ? lo.z : lo.w;
      const uint32_t b = i < 2 ? hi.x : i < 4 ? hi.y : i < 6 ? hi.z : hi.w;
      w[u] = __byte_perm(a, b, (i & 1) ? 0x7632 : 0x5410);
    }
    *reinterpret_cast<uint4*>(tile + gk_off(r + i, c)) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// one K chunk of an operand whose K runs along memory rows: thread r stages row r (its
// neighbours' elements are adjacent, so every load is coalesced), all loads of half a
// chunk in flight before eight elements at a time are stored as one core-matrix row
__device__ __forceinline__ void stage_strided(unsigned char* tile, const __nv_bfloat16* A, int row,
                                              int rows, long long s_row, long long s_k, int k0,
                                              int kend, int r) {
  const unsigned short* p = reinterpret_cast<const unsigned short*>(A) + (long long)row * s_row;
#pragma unroll 1
  for (int h = 0; h < kGK; h += kGK / 2) {
    uint32_t v[kGK / 4];
#pragma unroll
    for (int u = 0; u < kGK / 4; ++u) {
      const int k = k0 + h + 2 * u;
      const uint32_t lo = (row < rows && k < kend) ? p[(long long)k * s_k] : 0u;
      const uint32_t hi = (row < rows && k + 1 < kend) ? p[(long long)(k + 1) * s_k] : 0u;
      v[u] = lo | (hi << 16);
    }
#pragma unroll
    for (int c = 0; c < kGK / 2; c += 8)
      *reinterpret_cast<uint4*>(tile + gk_off(r, h + c)) =
          make_uint4(v[c / 2], v[c / 2 + 1], v[c / 2 + 2], v[c / 2 + 3]);
  }
}

constexpr int kGThreads = 256;
constexpr int kGSmem = 4 * kGTile + 1024;

__device__ __forceinline__ void gemm_tile(const GemmArgs& g, int bx, int by, int bz,
                                          unsigned char* raw, int* err) {
  __shared__ __align__(8) unsigned long long s_mbar[2];
  __shared__ uint32_t s_tmem;
  const uint32_t sbase = ((uint32_t)__cvta_generic_to_shared(raw) + 1023u) & ~1023u;
  unsigned char* gsm = raw + (sbase - (uint32_t)__cvta_generic_to_shared(raw));
  const int z = bz / g.S, sk = bz - z * g.S;
  const int m0 = by * kTcRows, n0 = bx * kH;
  const int kbeg = sk * g.kchunk, kend = min(g.K, kbeg + g.kchunk);  // this CTA's part of K
  const bool two = z >= g.z2;
  const int zi = two ? z - g.z2 : z;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t mbar = (uint32_t)__cvta_generic_to_shared(&s_mbar[0]);
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mbar) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mbar + 8) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {  // 128 TMEM columns: the 128 x 128 fp32 accumulator
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"((uint32_t)__cvta_generic_to_shared(&s_tmem)), "r"(kH) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(&s_tmem);
  // the operand this thread stages: rows o0 .. of `rows`, element (r, k) at O[r so_r + k so_k]
  const bool isB = tid >= kTcRows;
  const int t = tid & (kTcRows - 1);
  const __nv_bfloat16* O = isB ? (two ? g.B2 : g.B) + (long long)zi * g.sb_z
                               : (two ? g.A2 : g.A) + (long long)zi * g.sa_z;
  const int o0 = isB ? n0 : m0, orows = isB ? g.N : g.M;
  const long long so_r = isB ? g.sb_n : g.sa_m, so_k = isB ? g.sb_k : g.sa_k;
  // contiguous along K (and 16-byte aligned rows): eight elements per load, one core-matrix
  // row per store; contiguous along the rows, in aligned eights: 8 x 8 blocks; otherwise
  // element by element with the row index running fastest across the threads
  const bool al = ((uintptr_t)O & 15) == 0;
  const bool vec_k = so_k == 1 && (so_r & 7) == 0 && al && (g.K & 7) == 0;
  const bool blk = so_r == 1 && (so_k & 7) == 0 && al && (orows & 7) == 0;
  int nk = 0;  // chunks issued
  bool ok = true;
  for (int k0 = kbeg; k0 < kend; k0 += kGK, ++nk) {
    const int buf = nk & 1;
    if (nk >= 2) {  // the pair's last product
      const bool done = mbar_wait(mbar + 8 * buf, (uint32_t)((nk >> 1) - 1) & 1u);
      ok = __syncthreads_and(done) != 0;  // the same decision in every thread
      if (!ok) break;
    }
    unsigned char* tile = gsm + (2 * buf + (isB ? 1 : 0)) * kGTile;
    if (vec_k) {
#pragma unroll
      for (int c = 0; c < kGK; c += 8) {
        const int k = k0 + c;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (o0 + t < orows && k < kend)
          v = *reinterpret_cast<const uint4*>(O + (long long)(o0 + t) * so_r + k);
        *reinterpret_cast<uint4*>(tile + gk_off(t, c)) = v;
      }
    } else if (blk) {
      stage_blocks(tile, O, o0, orows, so_k, k0, kend, t);
    } else {
      stage_strided(tile, O, o0 + t, orows, so_r, so_k, k0, kend, t);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // tiles -> tensor core
    __syncthreads();
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t sA = sbase + (uint32_t)(2 * buf) * kGTile, sB = sA + kGTile;
#pragma unroll
      for (int ks = 0; ks < kGK / 16; ++ks)  // K step of 16 = two core matrices along K
        tc_mma(tmem, gk_desc(sA + ks * 2 * kLbo), gk_desc(sB + ks * 2 * kLbo),
               (k0 > kbeg || ks > 0) ? 1u : 0u);
      tc_commit(mbar + 8 * buf);
    }
    __syncwarp();
  }
  if (nk > 0) {  // the last commit covers every product before it
    const bool done = mbar_wait(mbar + 8 * ((nk - 1) & 1), (uint32_t)((nk - 1) >> 1) & 1u);
    ok = (__syncthreads_and(done) != 0) && ok;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  }
  if (ok) {
    // rows of 512 B in shared memory (no product reads it any more), their 16-byte units
    // swapped by row: warps w and w + 4 take TMEM lanes 32 (w % 4) .., 64 columns each
    float4* cs = reinterpret_cast<float4*>(gsm);
    const int r = (warp & 3) * 32 + lane;
    const uint32_t tl = tmem + ((uint32_t)((warp & 3) * 32) << 16);
#pragma unroll 1
    for (int c0 = (warp >> 2) * 64; c0 < (warp >> 2) * 64 + 64; c0 += 32) {
      float v[32];
      tc_ld32(tl + (uint32_t)c0, v);
#pragma unroll
      for (int j = 0; j < 8; ++j)
        cs[r * 32 + (((c0 >> 2) + j) ^ (r & 7))] =
            make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
    }
    __syncthreads();
    float* C = g.S > 1 ? g.ws + ((long long)sk * g.Z + z) * g.M * g.N
                       : (two ? g.C2 : g.C) + (long long)zi * g.sc_z;
    const long long cm = g.S > 1 ? g.N : g.sc_m, cn = g.S > 1 ? 1 : g.sc_n;
    const bool vec = cn == 1 && (cm & 3) == 0 && ((uintptr_t)C & 15) == 0;  // 16-byte stores
#pragma unroll 4
    for (int u = tid; u < kTcRows * 32; u += kGThreads) {
      const int i = u >> 5, q = u & 31, m = m0 + i, n = n0 + 4 * q;
      if (m >= g.M || n >= g.N) continue;
      const float4 x = cs[i * 32 + (q ^ (i & 7))];
      float* c = C + (long long)m * cm + (long long)n * cn;
      if (vec && n + 4 <= g.N) {
        *reinterpret_cast<float4*>(c) = x;
      } else {
        c[0] = x.x;
        if (n + 1 < g.N) c[cn] = x.y;
        if (n + 2 < g.N) c[2 * cn] = x.z;
        if (n + 3 < g.N) c[3 * cn] = x.w;
      }
    }
  } else if (tid == 0) {  // leave the tile unwritten (the wait above was the MMAs' last chance)
    atomicExch(err, 1);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  __syncwarp();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kH)
                 : "memory");
}

__global__ void __launch_bounds__(kGThreads) bf16_gemm_tc_kernel(GemmArgs g, int* err) {
  extern __shared__ __align__(1024) unsigned char tsm[];
  gemm_tile(g, blockIdx.x, blockIdx.y, blockIdx.z, tsm, err);
}

// Everything of a training batch that is a sum over its samples, in one launch: CTAs
// 0 .. 2 (kH / 32) E - 1 the column sums (the longer ones), the others the 128 x 128 weight
// gradients of both products.  Independent of one another and too few to fill the GPU, one
// after the other they took 9.4 + 18.1 us; together they take 9.7 (batch 512, 4 models).
constexpr int kSumSmem = kColSmem > kGSmem ? kColSmem : kGSmem;
__global__ void __launch_bounds__(kGThreads) mlp_batch_sums(ColArgs c, GemmArgs g, int ncol,
                                                            int* err) {
  extern __shared__ __align__(1024) unsigned char tsm[];
  const int i = blockIdx.x;
  if (i < ncol)
    column_grads(c, i / (2 * (kH / 32)), (i >> 1) & (kH / 32 - 1), i & 1, tsm);
  else
    gemm_tile(g, 0, 0, i - ncol, tsm, err);
}

// C[z](m, n) = sum over s = 0, 1, ..., S - 1 of the partial tiles ws[s][z][m][n]; C2 for z >= z2
__global__ void gemm_splitk_reduce(const float* ws, float* C, float* C2, int z2, int M, int N,
                                   int Z, int S, long long sc_m, long long sc_n, long long sc_z) {
  const long long per = (long long)M * N, all = per * Z;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < all;
       i += (long long)gridDim.x * blockDim.x) {
    const int z = (int)(i / per);
    const long long r = i - z * per;
    const int m = (int)(r / N), n = (int)(r - (long long)m * N);
    float acc = ws[i];
    for (int s = 1; s < S; ++s) acc += ws[s * all + i];
    (z < z2 ? C + z * sc_z : C2 + (z - z2) * sc_z)[m * sc_m + n * sc_n] = acc;
  }
}

// tanh_act2 of elements 2 i and 2 i + 1, one in each half
__global__ void debug_tanh_kernel(const float* x, float* y, int n) {
  const long long i = 2 * (blockIdx.x * (long long)blockDim.x + threadIdx.x);
  if (i >= n) return;
  float t0, t1;
  tanh_act2(f2_pack(x[i], x[i + 1 < n ? i + 1 : i]), t0, t1);
  y[i] = t0;
  if (i + 1 < n) y[i + 1] = t1;
}

}  // namespace mdeos

using namespace mdeos;

// batches of a training segment (see mdeos_surrogate_train), and its samples where the batches
// are large: whole batches, at least one
constexpr int kSegBatches = 16;
constexpr int kSegRows = 1 << 16;
static int train_seg(int batch) { return std::max(1, std::min(kSegBatches, kSegRows / batch)); }

// Staging of the calls on host arrays, one pinned and one device block that come and go with the
// surrogate, so that a call allocates nothing (a cudaFree in it could wait for whatever else
// runs on the device; in blocks of their own they took mdeos_surrogate_create to 0.99 ms, 0.91 so).
// predict: two slots of kIoRows queries, or max_batch if that is fewer (inputs 16 B; outputs a
// head with the error word, mean and sd 16 B each, 8 B per model) and one device block of
// outputs.  Training: two segments of samples (16 B each) and their batches' losses.
constexpr int kIoRows = 1 << 15;
constexpr size_t kIoHead = 256;
struct Staging {
  char *host = nullptr, *dev = nullptr;
  char *h_in[2], *h_out[2], *d_out;
  float *h_seg[2], *d_seg[2], *h_loss, *d_loss;  // losses [2][kSegBatches]
  cudaEvent_t io_done[2] = {nullptr, nullptr}, seg_done[2] = {nullptr, nullptr};
  cudaError_t allocate(int max_batch, int E) {
    const auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
    const size_t rows = (size_t)std::min(max_batch, kIoRows);
    const size_t in = up(rows * 16), out = up(kIoHead + rows * (32 + 8 * (size_t)E));
    // the longest segment of any batch size
    const size_t seg = up(16 * (size_t)std::max(max_batch, std::min(kSegRows, kSegBatches * max_batch)));
    const size_t loss = up(2 * kSegBatches * 4);
    cudaError_t e = cudaMallocHost((void**)&host, 2 * (in + out + seg) + loss);
    if (e == cudaSuccess) e = cudaMalloc((void**)&dev, out + 2 * seg + loss);
    if (e != cudaSuccess) return e;
    char *h = host, *d = dev;
    d_out = d;
    d += out;
    for (int k = 0; k < 2; ++k) {
      h_in[k] = h;
      h_out[k] = h + in;
      h_seg[k] = (float*)(h + in + out);
      h += in + out + seg;
      d_seg[k] = (float*)d;
      d += seg;
      e = cudaEventCreateWithFlags(&io_done[k], cudaEventDisableTiming);
      if (e == cudaSuccess) e = cudaEventCreateWithFlags(&seg_done[k], cudaEventDisableTiming);
      if (e != cudaSuccess) return e;
    }
    h_loss = (float*)h;
    d_loss = (float*)d;
    return e;
  }
  void release() {
    for (int k = 0; k < 2; ++k) {
      if (io_done[k]) cudaEventDestroy(io_done[k]);
      if (seg_done[k]) cudaEventDestroy(seg_done[k]);
    }
    if (host) cudaFreeHost(host);
    if (dev) cudaFree(dev);
  }
};

struct mdeos_surrogate {
  mdeos_handle* h = nullptr;
  int E = 4, maxB = 0;
  double norm[8] = {0, 0, 1, 1, 0, 0, 1, 1};  // x mean(2), x std(2), y mean(2), y std(2)
  int p_asinh = 0;  // 1: the networks learn asinh(P) (norm[4], norm[6] in those units)
  long long step = 0;
  float *P = nullptr, *G = nullptr, *Mm = nullptr, *Vv = nullptr;
  __nv_bfloat16 *W1b = nullptr, *W2b = nullptr, *W3b = nullptr, *W4b = nullptr;
  __nv_bfloat16 *W2t = nullptr, *W3t = nullptr;  // transposed, for the products with dZ
  __nv_bfloat16 *H1 = nullptr, *H2 = nullptr, *H3 = nullptr, *dZb = nullptr;
  float *Z = nullptr, *dZf = nullptr, *X = nullptr, *T = nullptr, *Y = nullptr, *dY = nullptr;
  float* loss = nullptr;
  double* Xp = nullptr;
  int* err = nullptr;  // set by the fused kernel when an MMA wait ran out
  float* ws = nullptr;  // partial tiles of the products whose K is split
  long long ws_elems = 0;
  int infer_path = MDEOS_SURROGATE_INFER_TC;
  Staging io;
  bool tc_ready = false, train_ready = false;
  int nsm = 1;
  std::vector<void*> allocs;
  // misfit map: RMS relative pressure residual of the ensemble mean per cell of a
  // bins x bins grid over the inputs it was fitted on (infinite: too few samples)
  int mis_bins = 0;
  double mis_lo[2] = {0, 0}, mis_hi[2] = {1, 1};
  std::vector<double> mis;
  double mis_threshold = INFINITY;  // gate: reject above this (infinite: map not used)
};

#define SCK(call)                                                                      \
  do {                                                                                 \
    cudaError_t e_ = (call);                                                           \
    if (e_ != cudaSuccess)                                                             \
      return set_error(MDEOS_ECUDA, std::string(#call ": ") + cudaGetErrorString(e_)); \
  } while (0)

constexpr int kMaxSplitK = 16;  // most CTAs one tile's K is split over

// the training products: tcgen05 tiles of 128 x 128 (bf16_gemm_tc_kernel); a tensor-core
// wait that ran out sets *err (device int) and leaves its tile unwritten.  Products with
// few tiles and a long K (the weight gradients, K = batch) split K over up to
// kMaxSplitK CTAs per tile, at least two chunks each, when the workspace ws (ws_elems
// floats) holds the partial tiles; the partials are summed in a fixed order, so every
// result is the same from run to run.
//
// gemm_plan fixes the split; a second batch (A2, B2 -> C2, same shape and strides) may share
// the launch and does not change it.
static GemmArgs gemm_plan(float* ws, long long ws_elems, const __nv_bfloat16* A,
                          const __nv_bfloat16* B, float* C, int M, int N, int K, long long sa_m,
                          long long sa_k, long long sa_z, long long sb_k, long long sb_n,
                          long long sb_z, long long sc_m, long long sc_n, long long sc_z, int Z,
                          const __nv_bfloat16* A2 = nullptr, const __nv_bfloat16* B2 = nullptr,
                          float* C2 = nullptr) {
  const int tiles = ((N + kH - 1) / kH) * ((M + kTcRows - 1) / kTcRows) * Z;
  const int nch = (K + kGK - 1) / kGK;
  const int Zall = A2 != nullptr ? 2 * Z : Z;
  int S = 1, per = nch;
  if (ws && tiles < 64 && nch >= 4) {
    const int s0 = std::min(nch / 2, kMaxSplitK);
    per = (nch + s0 - 1) / s0;
    S = (nch + per - 1) / per;  // every split holds at least one chunk
    if ((long long)S * Zall * M * N > ws_elems) S = 1, per = nch;
  }
  return GemmArgs{A, B, C, M, N, K, sa_m, sa_k, sa_z, sb_k, sb_n, sb_z, sc_m, sc_n, sc_z,
                  S, per * kGK, S > 1 ? ws : nullptr, A2, B2, C2, Z, Zall};
}

// the partial tiles of a split summed into C (and C2)
static cudaError_t gemm_reduce(const GemmArgs& g, cudaStream_t st) {
  if (g.S > 1) {
    const long long all = (long long)g.Z * g.M * g.N;
    gemm_splitk_reduce<<<(int)std::min<long long>((all + 255) / 256, 1024), 256, 0, st>>>(
        g.ws, g.C, g.C2, g.z2, g.M, g.N, g.Z, g.S, g.sc_m, g.sc_n, g.sc_z);
  }
  return cudaGetLastError();
}

static cudaError_t gemm(cudaStream_t st, int* err, float* ws, long long ws_elems,
                        const __nv_bfloat16* A, const __nv_bfloat16* B, float* C, int M, int N,
                        int K, long long sa_m, long long sa_k, long long sa_z, long long sb_k,
                        long long sb_n, long long sb_z, long long sc_m, long long sc_n,
                        long long sc_z, int Z) {
  const GemmArgs g = gemm_plan(ws, ws_elems, A, B, C, M, N, K, sa_m, sa_k, sa_z, sb_k, sb_n, sb_z,
                               sc_m, sc_n, sc_z, Z);
  cudaError_t e = cudaFuncSetAttribute(bf16_gemm_tc_kernel,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, kGSmem);
  if (e != cudaSuccess) return e;
  dim3 grid((N + kH - 1) / kH, (M + kTcRows - 1) / kTcRows, Z * g.S);
  bf16_gemm_tc_kernel<<<grid, kGThreads, kGSmem, st>>>(g, err);
  return gemm_reduce(g, st);
}

static int nblk(long long n, int t = 256) { return (int)((n + t - 1) / t); }

// layered forward of all models on s->X (B samples): H1..H3, and the outputs into Y
static cudaError_t forward(mdeos_surrogate* s, int B, float* Y, cudaStream_t st) {
  const int E = s->E;
  const long long EB = (long long)E * B;
  const long long sz = (long long)B * kH;
  cudaError_t e;
  mlp_layer1<<<nblk(EB * kH), 256, 0, st>>>(s->X, s->P, s->W1b, s->H1, B, E);
  // Z2 = H1 W2^T: A(m=b, k=j) = H1[b][j], B(k=j, n=o) = W2[o][j]
  e = gemm(st, s->err, s->ws, s->ws_elems, s->H1, s->W2b, s->Z, B, kH, kH, kH, 1, sz, 1, kH, kH * kH, kH, 1, sz, E);
  if (e != cudaSuccess) return e;
  mlp_bias_tanh<<<nblk(EB * kH), 256, 0, st>>>(s->Z, s->P, kOffB2, s->H2, B, E);
  e = gemm(st, s->err, s->ws, s->ws_elems, s->H2, s->W3b, s->Z, B, kH, kH, kH, 1, sz, 1, kH, kH * kH, kH, 1, sz, E);
  if (e != cudaSuccess) return e;
  mlp_bias_tanh<<<nblk(EB * kH), 256, 0, st>>>(s->Z, s->P, kOffB3, s->H3, B, E);
  mlp_output<<<nblk(EB * 2), 256, 0, st>>>(s->H3, s->P, s->W4b, Y, B, E);
  return cudaGetLastError();
}

// Gradients of the mean-squared error of one batch (X, T: device float[B][2]) in two
// launches: the fused forward and backward pass per 128 samples, the sums over the batch.
// With `splits` the two 128 x 128 weight gradients are left as *splits partial tiles in
// s->ws for mlp_adam (one split: in s->G), else they are added into s->G.
static cudaError_t gradients(mdeos_surrogate* s, const float* X, const float* T, int B, float* loss,
                             int* splits, cudaStream_t st) {
  const int E = s->E;
  const long long sz = (long long)B * kH;
  if (!s->train_ready) {
    cudaError_t e = cudaFuncSetAttribute(mlp_train_tc_kernel,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, kTrSmem);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(mlp_batch_sums, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               kSumSmem);
    if (e != cudaSuccess) return e;
    s->train_ready = true;
  }
  __nv_bfloat16* dZ2 = reinterpret_cast<__nv_bfloat16*>(s->Z);  // Z itself is not used here
  TrainArgs a{X, T, s->P, s->W1b, s->W2b, s->W3b, s->W4b, s->W2t, s->W3t,
              s->H1, s->H2, s->H3, s->dZb, dZ2, s->dZf, s->dY, s->Y, B, s->err};
  dim3 grid((B + kTcRows - 1) / kTcRows, E);
  mlp_train_tc_kernel<<<grid, kTrThreads, kTrSmem, st>>>(a);
  // dW3 = dZ3^T H2: A(m=o, k=b) = dZ3[b][o], B(k=b, n=j) = H2[b][j]; dW2 = dZ2^T H1 alike
  const GemmArgs g = gemm_plan(s->ws, s->ws_elems, s->dZb, s->H2, s->G + kOffW3, kH, kH, B, 1, kH,
                               sz, kH, 1, sz, kH, 1, kNParam, E, dZ2, s->H1, s->G + kOffW2);
  // the tiles' squared errors go through Y, which only inference uses
  const ColArgs c{s->dY, s->dZf, X, s->H3, s->dZb, dZ2, s->G, B, s->Y, (int)(grid.x * grid.y), loss};
  const int ncol = 2 * (kH / 32) * E;
  mlp_batch_sums<<<ncol + g.Z * g.S, kGThreads, kSumSmem, st>>>(c, g, ncol, s->err);
  count_launch(s->h, 2);
  if (splits) {
    *splits = g.S;
    return cudaGetLastError();
  }
  if (g.S > 1) count_launch(s->h, 1);
  return gemm_reduce(g, st);
}

static cudaError_t cast_weights(mdeos_surrogate* s, cudaStream_t st) {
  mlp_cast_weights<<<nblk((long long)s->E * kH * kH), 256, 0, st>>>(s->P, s->W1b, s->W2b, s->W3b,
                                                                    s->W4b, s->W2t, s->W3t, s->E);
  return cudaGetLastError();
}

extern "C" mdeos_status mdeos_surrogate_destroy(mdeos_surrogate* s);

extern "C" mdeos_status mdeos_surrogate_create(mdeos_handle* h, int32_t n_models, int32_t max_batch,
                                               uint64_t seed, mdeos_surrogate** out) {
  if (!h || !out || n_models < 1 || n_models > 16 || max_batch < 1 || max_batch > (1 << 22))
    return set_error(MDEOS_EINVAL, "bad surrogate_create arguments");
  *out = nullptr;
  mdeos_surrogate* s = new mdeos_surrogate();
  s->h = h;
  s->E = n_models;
  s->maxB = max_batch;
  const int E = n_models;
  const long long EB = (long long)E * max_batch;
  cudaError_t e = cudaSetDevice(handle_device(h));
  auto dalloc = [&](void** p, size_t bytes) {
    if (e == cudaSuccess) e = cudaMalloc(p, bytes);
    if (e == cudaSuccess) e = cudaMemset(*p, 0, bytes);
    if (e == cudaSuccess) s->allocs.push_back(*p);
  };
  const size_t np = (size_t)E * kNParam;
  dalloc((void**)&s->P, np * 4);
  dalloc((void**)&s->G, np * 4);
  dalloc((void**)&s->Mm, np * 4);
  dalloc((void**)&s->Vv, np * 4);
  dalloc((void**)&s->W1b, (size_t)E * 2 * kH * 2);
  dalloc((void**)&s->W2b, (size_t)E * kH * kH * 2);
  dalloc((void**)&s->W3b, (size_t)E * kH * kH * 2);
  dalloc((void**)&s->W4b, (size_t)E * 2 * kH * 2);
  dalloc((void**)&s->W2t, (size_t)E * kH * kH * 2);
  dalloc((void**)&s->W3t, (size_t)E * kH * kH * 2);
  dalloc((void**)&s->H1, EB * kH * 2);
  dalloc((void**)&s->H2, EB * kH * 2);
  dalloc((void**)&s->H3, EB * kH * 2);
  dalloc((void**)&s->dZb, EB * kH * 2);
  dalloc((void**)&s->Z, EB * kH * 4);
  dalloc((void**)&s->dZf, EB * kH * 4);
  dalloc((void**)&s->X, (size_t)max_batch * 2 * 4);
  dalloc((void**)&s->T, (size_t)max_batch * 2 * 4);
  dalloc((void**)&s->Y, EB * 2 * 4);
  dalloc((void**)&s->dY, EB * 2 * 4);
  dalloc((void**)&s->loss, 256);
  dalloc((void**)&s->Xp, (size_t)max_batch * 2 * 8);
  dalloc((void**)&s->err, 256);
  s->ws_elems = 2LL * kMaxSplitK * E * kH * kH;  // two products' partial tiles
  dalloc((void**)&s->ws, (size_t)s->ws_elems * 4);
  if (e == cudaSuccess) e = s->io.allocate(max_batch, E);
  if (e != cudaSuccess) {
    mdeos_surrogate_destroy(s);
    return set_error(MDEOS_ECUDA, std::string("surrogate_create: ") + cudaGetErrorString(e));
  }
  // Glorot-uniform weights, zero biases
  std::vector<float> p(np, 0.f);
  std::mt19937_64 rng(seed);
  std::uniform_real_distribution<double> u(-1.0, 1.0);
  for (int m = 0; m < E; ++m) {
    float* q = p.data() + (size_t)m * kNParam;
    const double l1 = std::sqrt(6.0 / (kH + 2)), l2 = std::sqrt(6.0 / (2 * kH));
    for (int i = 0; i < 2 * kH; ++i) q[kOffW1 + i] = (float)(l1 * u(rng));
    for (int i = 0; i < kH * kH; ++i) q[kOffW2 + i] = (float)(l2 * u(rng));
    for (int i = 0; i < kH * kH; ++i) q[kOffW3 + i] = (float)(l2 * u(rng));
    for (int i = 0; i < 2 * kH; ++i) q[kOffW4 + i] = (float)(l1 * u(rng));
  }
  cudaStream_t st = handle_stream(h);
  e = cudaMemcpyAsync(s->P, p.data(), np * 4, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cast_weights(s, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) {
    mdeos_surrogate_destroy(s);
    return set_error(MDEOS_ECUDA, std::string("surrogate init: ") + cudaGetErrorString(e));
  }
  *out = s;
  return MDEOS_OK;
}

extern "C" mdeos_status mdeos_surrogate_set_params(mdeos_surrogate* s, const float* params,
                                                   const double* norm) {
  if (!s) return set_error(MDEOS_EINVAL, "surrogate is NULL");
  cudaStream_t st = handle_stream(s->h);
  SCK(cudaSetDevice(handle_device(s->h)));
  if (params) {
    const size_t np = (size_t)s->E * kNParam;
    SCK(cudaMemcpyAsync(s->P, params, np * 4, cudaMemcpyHostToDevice, st));
    SCK(cudaMemsetAsync(s->Mm, 0, np * 4, st));
    SCK(cudaMemsetAsync(s->Vv, 0, np * 4, st));
    s->step = 0;
    SCK(cast_weights(s, st));
  }
  if (norm) std::memcpy(s->norm, norm, sizeof(s->norm));
  SCK(cudaStreamSynchronize(st));
  return MDEOS_OK;
}

extern "C" mdeos_status mdeos_surrogate_get_params(mdeos_surrogate* s, float* params, double* norm) {
  if (!s) return set_error(MDEOS_EINVAL, "surrogate is NULL");
  SCK(cudaSetDevice(handle_device(s->h)));
  cudaStream_t st = handle_stream(s->h);
  if (params)
    SCK(cudaMemcpyAsync(params, s->P, (size_t)s->E * kNParam * 4, cudaMemcpyDeviceToHost, st));
  SCK(cudaStreamSynchronize(st));
  if (norm) std::memcpy(norm, s->norm, sizeof(s->norm));
  return MDEOS_OK;
}

// the tensor-core error flag of the surrogate's kernels: read and cleared (synchronous)
static mdeos_status take_tc_error(mdeos_surrogate* s, cudaStream_t st) {
  int err = 0;
  SCK(cudaMemcpyAsync(&err, s->err, 4, cudaMemcpyDeviceToHost, st));
  SCK(cudaMemsetAsync(s->err, 0, 4, st));
  SCK(cudaStreamSynchronize(st));
  if (err) return set_error(MDEOS_ETIMEDOUT, "surrogate: a tensor-core wait ran out");
  return MDEOS_OK;
}

// normalised inputs/targets of n samples into s->X / s->T (host FP64 in)
static mdeos_status load_batch(mdeos_surrogate* s, const double* xp, const double* yp, int n,
                               cudaStream_t st) {
  std::vector<float> x(2 * (size_t)n), t;
  for (int b = 0; b < n; ++b)
    for (int c = 0; c < 2; ++c)
      x[2 * b + c] = (float)((xp[2 * b + c] - s->norm[c]) / s->norm[2 + c]);
  SCK(cudaMemcpyAsync(s->X, x.data(), x.size() * 4, cudaMemcpyHostToDevice, st));
  if (yp) {
    t.resize(2 * (size_t)n);
    for (int b = 0; b < n; ++b)
      for (int c = 0; c < 2; ++c) {
        const double y = (c == 0 && s->p_asinh) ? std::asinh(yp[2 * b]) : yp[2 * b + c];
        t[2 * b + c] = (float)((y - s->norm[4 + c]) / s->norm[6 + c]);
      }
    SCK(cudaMemcpyAsync(s->T, t.data(), t.size() * 4, cudaMemcpyHostToDevice, st));
  }
  SCK(cudaStreamSynchronize(st));  // the host vectors go out of scope
  return MDEOS_OK;
}

extern "C" mdeos_status mdeos_surrogate_grads(mdeos_surrogate* s, const double* x, const double* y,
                                              int32_t n, float* grads, double* loss) {
  if (!s || !x || !y || n < 1 || n > s->maxB) return set_error(MDEOS_EINVAL, "bad grads arguments");
  SCK(cudaSetDevice(handle_device(s->h)));
  cudaStream_t st = handle_stream(s->h);
  mdeos_status ms = load_batch(s, x, y, n, st);
  if (ms != MDEOS_OK) return ms;
  SCK(gradients(s, s->X, s->T, n, s->loss, nullptr, st));
  if (grads)
    SCK(cudaMemcpyAsync(grads, s->G, (size_t)s->E * kNParam * 4, cudaMemcpyDeviceToHost, st));
  float l = 0.f;
  SCK(cudaMemcpyAsync(&l, s->loss, 4, cudaMemcpyDeviceToHost, st));
  SCK(cudaStreamSynchronize(st));
  if (loss) *loss = (double)l / (2.0 * n * s->E);
  return take_tc_error(s, st);
}

extern "C" mdeos_status mdeos_surrogate_train(mdeos_surrogate* s, const double* x, const double* y,
                                              int32_t n, int32_t epochs, int32_t batch, double lr,
                                              uint64_t seed, int32_t set_norm, double* loss_out) {
  if (!s || !x || !y || n < 1 || epochs < 0 || batch < 1 || batch > s->maxB || !(lr > 0))
    return set_error(MDEOS_EINVAL, "bad train arguments");
  if (set_norm) {  // normalisers from the training data: mean and standard deviation
    for (int c = 0; c < 4; ++c) {
      const double* a = c < 2 ? x : y;
      const int col = c % 2;
      const bool as = c == 2 && s->p_asinh;  // pressure learned as asinh(P)
      auto val = [&](int i) { return as ? std::asinh(a[2 * i + col]) : a[2 * i + col]; };
      double m = 0.0, q = 0.0;
      for (int i = 0; i < n; ++i) m += val(i);
      m /= n;
      for (int i = 0; i < n; ++i) q += (val(i) - m) * (val(i) - m);
      const double sdv = std::sqrt(q / n);
      s->norm[(c < 2 ? 0 : 4) + col] = m;
      s->norm[(c < 2 ? 2 : 6) + col] = sdv > 0 ? sdv : 1.0;
    }
  }
  SCK(cudaSetDevice(handle_device(s->h)));
  cudaStream_t st = handle_stream(s->h);
  std::mt19937_64 rng(seed);
  std::vector<int> perm(n);
  for (int i = 0; i < n; ++i) perm[i] = i;
  // The batches go to the device in segments of up to kSegBatches (two pinned buffers in
  // turn, so a segment is gathered and normalised while the one before trains), and their
  // losses come back with them.
  const int nbat = n / batch;  // full batches only
  const int seg = train_seg(batch);
  Staging& io = s->io;
  const float b1 = 0.9f, b2 = 0.999f;
  for (int ep = 0; ep < epochs; ++ep) {
    std::shuffle(perm.begin(), perm.end(), rng);
    double lsum = 0.0;
    int held[2] = {0, 0};  // batches of the segment in flight in each buffer
    // the losses of buffer t's segment, once it is done
    auto collect = [&](int t) -> cudaError_t {
      if (held[t] == 0) return cudaSuccess;
      const cudaError_t e = cudaEventSynchronize(io.seg_done[t]);
      for (int k = 0; k < held[t]; ++k)
        lsum += (double)io.h_loss[t * kSegBatches + k] / (2.0 * batch * s->E);
      held[t] = 0;
      return e;
    };
    int turn = 0;
    for (int b0 = 0; b0 < nbat; b0 += seg, turn ^= 1) {
      const int nb = std::min(seg, nbat - b0);
      const size_t rows = (size_t)nb * batch;
      SCK(collect(turn));
      float* hx = io.h_seg[turn];
      float* ht = hx + 2 * rows;
      for (size_t k = 0; k < rows; ++k) {
        const size_t i = (size_t)perm[(size_t)b0 * batch + k];
        for (int c = 0; c < 2; ++c) {
          const double t = (c == 0 && s->p_asinh) ? std::asinh(y[2 * i]) : y[2 * i + c];
          hx[2 * k + c] = (float)((x[2 * i + c] - s->norm[c]) / s->norm[2 + c]);
          ht[2 * k + c] = (float)((t - s->norm[4 + c]) / s->norm[6 + c]);
        }
      }
      float* dx = io.d_seg[turn];
      float* dl = io.d_loss + turn * kSegBatches;
      SCK(cudaMemcpyAsync(dx, hx, rows * 16, cudaMemcpyHostToDevice, st));
      for (int k = 0; k < nb; ++k) {
        const float* bx = dx + 2 * (size_t)k * batch;
        int S = 1;
        SCK(gradients(s, bx, bx + 2 * rows, batch, dl + k, &S, st));
        ++s->step;
        AdamArgs a{s->P, s->Mm, s->Vv, s->G, s->ws, s->W1b, s->W2b, s->W3b, s->W4b, s->W2t, s->W3t,
                   s->E, S, (float)lr, b1, b2, (float)(1.0 - 0.9), (float)(1.0 - 0.999), 1e-8f,
                   (float)(1.0 - std::pow(0.9, (double)s->step)),
                   (float)(1.0 - std::pow(0.999, (double)s->step))};
        mlp_adam<<<dim3(nblk(kNParam), s->E), 256, 0, st>>>(a);
        SCK(cudaGetLastError());
        count_launch(s->h, 1);
      }
      SCK(cudaMemcpyAsync(io.h_loss + turn * kSegBatches, dl, (size_t)nb * 4,
                          cudaMemcpyDeviceToHost, st));
      SCK(cudaEventRecord(io.seg_done[turn], st));
      held[turn] = nb;
    }
    SCK(collect(turn));  // the older segment first: the losses add up in batch order
    SCK(collect(turn ^ 1));
    if (loss_out) loss_out[ep] = nbat ? lsum / nbat : 0.0;
  }
  return take_tc_error(s, st);
}

static_assert(kTcGroups == 4, "infer_tc_fn");
using InferKernel = void (*)(const float*, const float*, const __nv_bfloat16*, const __nv_bfloat16*,
                             const __nv_bfloat16*, const __nv_bfloat16*, float*, int, int*);
static InferKernel infer_tc_fn(int groups) {
  return groups == 1 ? mlp_infer_tc_kernel<1>
                     : (groups == 2 ? mlp_infer_tc_kernel<2> : mlp_infer_tc_kernel<4>);
}

// inference of B <= maxB inputs (device FP64 [B][2]) -> per-model s->Y and the ensemble
// mean / sd (device FP64 [B][2]) on stream st
static cudaError_t infer(mdeos_surrogate* s, const double* dx, int B, double* dmean, double* dsd,
                         float* dY, int path, cudaStream_t st) {
  mlp_normalise<<<nblk(B), 256, 0, st>>>(dx, s->X, B, s->norm[0], s->norm[1], s->norm[2],
                                         s->norm[3]);
  cudaError_t e;
  if (path == MDEOS_SURROGATE_INFER_MMA) {
    e = forward(s, B, dY, st);
    count_launch(s->h, 8);  // six of the layers (K = 128 is not split)
  } else {
    if (!s->tc_ready) {
      for (int g = 1; g <= kTcGroups; g *= 2) {
        e = cudaFuncSetAttribute(infer_tc_fn(g), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 infer_tc_smem(g));
        if (e != cudaSuccess) return e;
      }
      int dev = 0;
      e = cudaGetDevice(&dev);
      if (e == cudaSuccess) e = cudaDeviceGetAttribute(&s->nsm, cudaDevAttrMultiProcessorCount, dev);
      if (e != cudaSuccess) return e;
      s->tc_ready = true;
    }
    // one CTA per SM and model share; as many groups (tiles at a time) per CTA as keep
    // every CTA's groups busy: few tiles spread over more SMs first
    const int tiles = (B + kTcRows - 1) / kTcRows;
    const int per_model = std::max(1, std::min(tiles, s->nsm / s->E));
    int groups = 1;
    while (groups < kTcGroups && tiles > per_model * groups) groups *= 2;
    dim3 grid(per_model, s->E);
    infer_tc_fn(groups)<<<grid, groups * kTcThreads, infer_tc_smem(groups), st>>>(
        s->X, s->P, s->W1b, s->W2b, s->W3b, s->W4b, dY, B, s->err);
    e = cudaGetLastError();
    count_launch(s->h, 3);
  }
  if (e != cudaSuccess) return e;
  mlp_ensemble<<<nblk(2 * B), 256, 0, st>>>(dY, B, s->E, s->norm[4], s->norm[5], s->norm[6],
                                            s->norm[7], s->p_asinh,
                                            (s->E & (s->E - 1)) == 0 ? 1.0 / s->E : 0.0, dmean, dsd);
  return cudaGetLastError();
}

extern "C" mdeos_status mdeos_surrogate_set_output_transform(mdeos_surrogate* s, int32_t mode) {
  if (!s || (mode != MDEOS_SURROGATE_P_LINEAR && mode != MDEOS_SURROGATE_P_ASINH))
    return set_error(MDEOS_EINVAL, "bad output transform");
  s->p_asinh = mode == MDEOS_SURROGATE_P_ASINH ? 1 : 0;
  return MDEOS_OK;
}

extern "C" mdeos_status mdeos_surrogate_set_infer_path(mdeos_surrogate* s, int32_t path) {
  if (!s || (path != MDEOS_SURROGATE_INFER_TC && path != MDEOS_SURROGATE_INFER_MMA))
    return set_error(MDEOS_EINVAL, "bad inference path");
  s->infer_path = path;
  return MDEOS_OK;
}

extern "C" mdeos_status mdeos_surrogate_infer_device(mdeos_surrogate* s, const double* d_x,
                                                     int32_t n, double* d_mean, double* d_sd,
                                                     void* stream) {
  if (!s || (n > 0 && (!d_x || !d_mean || !d_sd)) || n < 0)
    return set_error(MDEOS_EINVAL, "bad infer_device arguments");
  SCK(cudaSetDevice(handle_device(s->h)));
  cudaStream_t st = stream ? (cudaStream_t)stream : handle_stream(s->h);
  for (int off = 0; off < n; off += s->maxB) {
    const int B = std::min(s->maxB, n - off);
    SCK(infer(s, d_x + 2 * (size_t)off, B, d_mean + 2 * (size_t)off, d_sd + 2 * (size_t)off, s->Y,
              s->infer_path, st));
  }
  return MDEOS_OK;
}

extern "C" mdeos_status mdeos_surrogate_predict(mdeos_surrogate* s, const double* x, int32_t n,
                                                double* mean, double* sd, float* per_model) {
  if (!s || !x || n < 0) return set_error(MDEOS_EINVAL, "bad predict arguments");
  SCK(cudaSetDevice(handle_device(s->h)));
  cudaStream_t st = handle_stream(s->h);
  // One copy in and one out per piece, through pinned memory: the piece's mean, sd and per-model
  // outputs and the error word share a device block.  (Copies to and from pageable memory are
  // waited for one by one: eight of them took half of a 2000-query call, 123 us; it takes 67
  // now.  Into arrays that the device has not written before they are far slower: 2^18 queries,
  // one model, 7.2 ms.)  Two slots in turn: the host copies one piece's arrays while the device
  // works on the other's.
  const int chunk = std::min(s->maxB, kIoRows);
  int err = 0;
  int held[2] = {0, 0}, first[2] = {0, 0};  // queries of the piece in flight in each slot
  auto collect = [&](int t) -> cudaError_t {
    const int B = held[t], off = first[t];
    if (B == 0) return cudaSuccess;
    held[t] = 0;
    const cudaError_t e = cudaEventSynchronize(s->io.io_done[t]);
    if (e != cudaSuccess) return e;
    const size_t ob = (size_t)B * 16;
    const char* h = s->io.h_out[t];
    if (mean) std::memcpy(mean + 2 * (size_t)off, h + kIoHead, ob);
    if (sd) std::memcpy(sd + 2 * (size_t)off, h + kIoHead + ob, ob);
    if (per_model)
      for (int m = 0; m < s->E; ++m)
        std::memcpy(per_model + ((size_t)m * n + off) * 2, h + kIoHead + 2 * ob + (size_t)m * B * 8,
                    (size_t)B * 8);
    err |= *reinterpret_cast<const int*>(h);
    return cudaSuccess;
  };
  const auto run = [&]() -> cudaError_t {
    cudaError_t e = cudaSuccess;
    for (int off = 0, t = 0; off < n && e == cudaSuccess; off += chunk, t ^= 1) {
      if ((e = collect(t)) != cudaSuccess) break;
      const int B = std::min(chunk, n - off);
      const size_t ob = (size_t)B * 16, yb = per_model ? (size_t)s->E * B * 8 : 0;
      char* d = s->io.d_out;
      std::memcpy(s->io.h_in[t], x + 2 * (size_t)off, ob);
      e = cudaMemcpyAsync(s->Xp, s->io.h_in[t], ob, cudaMemcpyHostToDevice, st);
      if (e == cudaSuccess)
        e = infer(s, s->Xp, B, (double*)(d + kIoHead), (double*)(d + kIoHead + ob),
                  (float*)(d + kIoHead + 2 * ob), s->infer_path, st);
      if (e == cudaSuccess) e = cudaMemcpyAsync(d, s->err, 4, cudaMemcpyDeviceToDevice, st);
      if (e == cudaSuccess)
        e = cudaMemcpyAsync(s->io.h_out[t], d, kIoHead + 2 * ob + yb, cudaMemcpyDeviceToHost, st);
      if (e == cudaSuccess) e = cudaEventRecord(s->io.io_done[t], st);
      if (e != cudaSuccess) break;
      held[t] = B;
      first[t] = off;
    }
    for (int t = 0; t < 2 && e == cudaSuccess; ++t) e = collect(t);
    if (e != cudaSuccess) cudaStreamSynchronize(st);  // nothing still uses the slots
    return e;
  };
  SCK(run());
  if (err) {
    SCK(cudaMemsetAsync(s->err, 0, 4, st));
    SCK(cudaStreamSynchronize(st));
    return set_error(MDEOS_ETIMEDOUT, "surrogate: a tensor-core wait ran out");
  }
  return MDEOS_OK;
}

// Surrogate answer where the ensemble agrees (sd_P <= threshold * max(|P|, 1)),
// the MD path (requests evaluated with natoms = md_natoms) elsewhere.
// cell of the misfit grid holding input (rho, e); -1 outside the fitted range
static int misfit_cell(const mdeos_surrogate* s, double rho, double e) {
  if (s->mis_bins < 1) return -1;
  const double in[2] = {rho, e};
  int c[2];
  for (int k = 0; k < 2; ++k) {
    const double t = (in[k] - s->mis_lo[k]) / (s->mis_hi[k] - s->mis_lo[k]);
    if (!(t >= 0.0 && t <= 1.0)) return -1;
    c[k] = std::min((int)(t * s->mis_bins), s->mis_bins - 1);
  }
  return c[0] * s->mis_bins + c[1];
}

static double misfit_at(const mdeos_surrogate* s, double rho, double e) {
  const int c = misfit_cell(s, rho, e);
  return c < 0 ? INFINITY : s->mis[c];
}

extern "C" mdeos_status mdeos_surrogate_fit_misfit(mdeos_surrogate* s, const double* x,
                                                   const double* y, int32_t n, int32_t bins,
                                                   int32_t min_count) {
  if (!s || !x || !y || n < 1 || bins < 1 || bins > 1024 || min_count < 1)
    return set_error(MDEOS_EINVAL, "bad fit_misfit arguments");
  std::vector<double> mean(2 * (size_t)n), sd(2 * (size_t)n);
  mdeos_status ms = mdeos_surrogate_predict(s, x, n, mean.data(), sd.data(), nullptr);
  if (ms != MDEOS_OK) return ms;
  for (int k = 0; k < 2; ++k) {
    s->mis_lo[k] = INFINITY;
    s->mis_hi[k] = -INFINITY;
    for (int i = 0; i < n; ++i) {
      s->mis_lo[k] = std::min(s->mis_lo[k], x[2 * i + k]);
      s->mis_hi[k] = std::max(s->mis_hi[k], x[2 * i + k]);
    }
    if (!(s->mis_hi[k] > s->mis_lo[k])) s->mis_hi[k] = s->mis_lo[k] + 1.0;
  }
  s->mis_bins = bins;
  std::vector<double> sum((size_t)bins * bins, 0.0);
  std::vector<int> cnt((size_t)bins * bins, 0);
  for (int i = 0; i < n; ++i) {
    const int c = misfit_cell(s, x[2 * i], x[2 * i + 1]);
    if (c < 0) continue;
    const double r = (mean[2 * i] - y[2 * i]) / std::max(std::fabs(y[2 * i]), 1.0);
    sum[c] += r * r;
    ++cnt[c];
  }
  s->mis.assign((size_t)bins * bins, INFINITY);
  for (size_t c = 0; c < s->mis.size(); ++c)
    if (cnt[c] >= min_count) s->mis[c] = std::sqrt(sum[c] / cnt[c]);
  return MDEOS_OK;
}

extern "C" mdeos_status mdeos_surrogate_misfit(const mdeos_surrogate* s, const double* x,
                                               int32_t n, double* out) {
  if (!s || !x || !out || n < 0) return set_error(MDEOS_EINVAL, "bad misfit arguments");
  if (s->mis_bins < 1) return set_error(MDEOS_EINVAL, "no misfit map fitted");
  for (int i = 0; i < n; ++i) out[i] = misfit_at(s, x[2 * i], x[2 * i + 1]);
  return MDEOS_OK;
}

extern "C" mdeos_status mdeos_surrogate_set_misfit_threshold(mdeos_surrogate* s,
                                                             double threshold) {
  if (!s || !(threshold >= 0.0)) return set_error(MDEOS_EINVAL, "bad misfit threshold");
  if (std::isfinite(threshold) && s->mis_bins < 1)
    return set_error(MDEOS_EINVAL, "no misfit map fitted");
  s->mis_threshold = threshold;
  return MDEOS_OK;
}

extern "C" mdeos_status mdeos_surrogate_gated_eval(mdeos_surrogate* s, const mdeos_request* reqs,
                                                   int32_t n, double threshold, int32_t md_natoms,
                                                   mdeos_result* out, int32_t* used_md) {
  if (!s || !reqs || !out || n < 0 || !(threshold >= 0))
    return set_error(MDEOS_EINVAL, "bad gated_eval arguments");
  std::vector<double> x(2 * (size_t)n), mean(2 * (size_t)n), sd(2 * (size_t)n);
  for (int i = 0; i < n; ++i) {
    x[2 * i] = reqs[i].rho;
    x[2 * i + 1] = reqs[i].e;
  }
  mdeos_status ms = mdeos_surrogate_predict(s, x.data(), n, mean.data(), sd.data(), nullptr);
  if (ms != MDEOS_OK) return ms;
  std::vector<mdeos_request> md;
  std::vector<int> idx;
  for (int i = 0; i < n; ++i) {
    const bool ok = sd[2 * i] <= threshold * std::max(std::fabs(mean[2 * i]), 1.0) &&
                    (reqs[i].flags & MDEOS_REQ_TEMPERATURE) == 0 &&
                    (!std::isfinite(s->mis_threshold) ||
                     misfit_at(s, reqs[i].rho, reqs[i].e) <= s->mis_threshold);
    if (used_md) used_md[i] = ok ? 0 : 1;
    if (ok) {
      mdeos_result& r = out[i];
      std::memset(&r, 0, sizeof(r));
      r.P = mean[2 * i];
      r.T = mean[2 * i + 1];
      r.P_se = sd[2 * i];
      r.T_se = sd[2 * i + 1];
      r.sigma[0] = r.sigma[1] = r.sigma[2] = r.P;
      r.element_id = reqs[i].element_id;
      r.natoms = 0;
      r.status = MDEOS_OK;
      r.path = -2;  // answered by the surrogate
    } else {
      mdeos_request q = reqs[i];
      if (md_natoms > 0) q.natoms = md_natoms;
      md.push_back(q);
      idx.push_back(i);
    }
  }
  if (!md.empty()) {
    uint64_t t = 0;
    ms = mdeos_submit(s->h, md.data(), (int)md.size(), &t);
    if (ms != MDEOS_OK) return ms;
    std::vector<mdeos_result> r(md.size());
    ms = mdeos_poll(s->h, t, r.data(), -1);
    if (ms != MDEOS_OK) return ms;
    for (size_t k = 0; k < md.size(); ++k) out[idx[k]] = r[k];
  }
  return MDEOS_OK;
}

extern "C" mdeos_status mdeos_surrogate_destroy(mdeos_surrogate* s) {
  if (!s) return MDEOS_OK;
  if (s->h) {
    cudaSetDevice(handle_device(s->h));
    cudaStreamSynchronize(handle_stream(s->h));
  }
  s->io.release();
  for (void* p : s->allocs) cudaFree(p);
  delete s;
  return MDEOS_OK;
}

extern "C" mdeos_status mdeos_debug_gemm_bf16(const uint16_t* A, const uint16_t* B, float* C,
                                              int32_t M, int32_t N, int32_t K, int64_t sa_m,
                                              int64_t sa_k, int64_t sb_k, int64_t sb_n,
                                              int64_t sc_m, int64_t sc_n, void* stream) {
  if (!A || !B || !C || M < 1 || N < 1 || K < 1)
    return set_error(MDEOS_EINVAL, "bad gemm arguments");
  cudaStream_t st = (cudaStream_t)stream;
  int* err = nullptr;
  float* ws = nullptr;
  const long long ws_elems = (long long)kMaxSplitK * M * N;
  SCK(cudaMallocAsync(&err, sizeof(int), st));
  SCK(cudaMemsetAsync(err, 0, sizeof(int), st));
  SCK(cudaMallocAsync(&ws, (size_t)ws_elems * 4, st));
  cudaError_t e = gemm(st, err, ws, ws_elems, reinterpret_cast<const __nv_bfloat16*>(A),
                       reinterpret_cast<const __nv_bfloat16*>(B), C, M, N, K, sa_m, sa_k, 0, sb_k,
                       sb_n, 0, sc_m, sc_n, 0, 1);
  int herr = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFreeAsync(err, st);
  cudaFreeAsync(ws, st);
  if (e != cudaSuccess) return set_error(MDEOS_ECUDA, cudaGetErrorString(e));
  if (herr) return set_error(MDEOS_ETIMEDOUT, "gemm: a tensor-core wait ran out");
  return MDEOS_OK;
}

extern "C" mdeos_status mdeos_debug_tanh(const float* x, float* y, int32_t n, void* stream) {
  if (!x || !y || n < 1) return set_error(MDEOS_EINVAL, "bad tanh arguments");
  cudaStream_t st = (cudaStream_t)stream;
  debug_tanh_kernel<<<(n - 1) / 512 + 1, 256, 0, st>>>(x, y, n);
  SCK(cudaGetLastError());
  SCK(cudaStreamSynchronize(st));
  return MDEOS_OK;
}
