// Learned per-cell cost and initial-step model: BF16 tensor-core GEMMs with FP32
// accumulation (mma.sync m16n8k16), GELU MLP forward/backward, Adam on FP32
// master weights, and the predictions the scheduler consumes.
//
// The paper has no learned component: DLBFoam balances measured per-process cost
// (Methodology, "DLBFoam: Dynamic load balancing"; Results, Fig. 4). Here the
// integrator's own per-cell logs (substeps, first accepted step) train a model
// that orders the work queue heaviest-first and seeds each cell's first step.

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <random>
#include <string>
#include <vector>

#include "chem.h"
#include "chem_capi_internal.h"
#include "chem_fixed.cuh"
#include "chem_mlp.h"
#include "chem_mlp_internal.h"

namespace {

constexpr int kH = 128;      // hidden width
typedef __nv_bfloat16 bf16;

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float z) {
  return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * 0.39894228040143268f * expf(-0.5f * z * z);
}

// ---------------------------------------------------------------------------
// features: x = [T/1000, ln p, ln(Y_k + 1e-20)], optionally standardised
// ---------------------------------------------------------------------------
__device__ __forceinline__ double feature(const double* T, const double* p, const double* Y, int K, int64_t c,
                                          int d) {
  if (d == 0) return T[c] * 1e-3;
  if (d == 1) return log(p[c]);
  return log(Y[(size_t)c * K + (d - 2)] + 1e-20);
}

__global__ void k_feature_stats(const double* T, const double* p, const double* Y, int K, int64_t n,
                                double* sums /* [2 D] */) {
  extern __shared__ double sh[];
  const int D = K + 2;
  for (int i = threadIdx.x; i < 2 * D; i += blockDim.x) sh[i] = 0.0;
  __syncthreads();
  for (int64_t r = blockIdx.x; r < n; r += gridDim.x)
    for (int d = threadIdx.x; d < D; d += blockDim.x) {
      const double x = feature(T, p, Y, K, r, d);
      sh[d] += x;
      sh[D + d] += x * x;
    }
  __syncthreads();
  for (int i = threadIdx.x; i < 2 * D; i += blockDim.x) atomicAdd(&sums[i], sh[i]);
}

__global__ void k_target_stats(const int32_t* sub, const double* hf, int64_t n, double* sums /* [4] */) {
  double a = 0, a2 = 0, b = 0, b2 = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double t0 = log(fmax((double)sub[i], 1.0)), t1 = log(fmax(hf[i], 1e-300));
    a += t0;
    a2 += t0 * t0;
    b += t1;
    b2 += t1 * t1;
  }
  for (int o = 16; o; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    a2 += __shfl_xor_sync(0xffffffffu, a2, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
    b2 += __shfl_xor_sync(0xffffffffu, b2, o);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&sums[0], a);
    atomicAdd(&sums[1], a2);
    atomicAdd(&sums[2], b);
    atomicAdd(&sums[3], b2);
  }
}

// ---------------------------------------------------------------------------
// forward pass (and backward pass) of a batch in one kernel
//
// Everything between the features and the results stays in shared memory and registers; the
// weights are loaded once per CTA. A layer is computed 32 columns at a time, so that the code
// of its product and its GELUs (16 a lane) exists once: with all 128 columns in registers it
// was 64 KB long, twice the instruction cache, at 128 registers a thread.
// Prediction: each warp takes 16 rows through the model on its own. Training: a CTA takes 64
// rows, four warps to 16 of them, each with 32 columns of every layer, so that the dependent
// layers are short and an SM has 16 warps although a minibatch is one tile per SM.
//
// Four kernels per pass with one FP64 logarithm and division per feature took 527 us for
// 65,536 rows of 54 species and were bound by the FP64 pipe (3.5 M logarithms of some 25
// operations at 19 cycles per warp and SM: 180 us) and by element-wise strided operand
// loads; this kernel takes 47 us. It is bound by issue and dependent instructions (0.56 warp
// instructions per cycle and scheduler): half of its 7,800 instructions per 16 rows are the
// 256 x 16 GELUs' erff. The gradient of 8,192 rows took 332 us in 17 launches, with two passes
// over the activations in global memory per layer, copies and an allocation; now 61 us, of
// which this kernel has 31 (one tile per SM: the layers' chain) and the reduction 6.
// ---------------------------------------------------------------------------
struct MlpP {
  const double *T, *p, *Y;
  const int* perm;  // row order of a training epoch (null: as given)
  int64_t row0, n;  // rows [row0, row0 + n) of that order
  int K, D, Dp;     // species, features, features rounded up to 16
  const float* norm;  // mu_x[D], sd_x[D], mu_t[2], sd_t[2]
  const bf16* wb;     // BF16 weights
  const float* w;     // FP32 weights (biases)
  int64_t ob1, oW2, ob2, oW3, ob3, nw;
  // prediction
  float zmax;  // > 0: rows with a standardised feature beyond +-zmax get a NaN initial step
  float *ln_cost, *ln_h0, *cost;
  double* h0;
  // training
  const int32_t* sub;
  const double* hf;
  float inv_B;
  float* part;  // [CTAs][part_stride]: gradient in the order of the weights, then the loss
  int64_t part_stride;
};

constexpr int kLd = kH + 8;  // row length of the 128-wide tiles (rows 16 bytes off in banks: no conflicts)
constexpr int kPredictWarps = 16, kTrainWarps = 16, kTrainRows = 64;
constexpr size_t kMaxSmemMlp = 232448;
constexpr int kFeatureBatch = 14;                // loads in flight per lane
constexpr int kListed = 32 + 32 * kFeatureBatch;  // features a warp may have listed

struct MlpSmem {  // byte offsets
  int W2, norm, vec, X, H1, H2, dZ2, dZ1, head, total;
};
// rows: of the CTA's tiles
__host__ __device__ inline MlpSmem mlp_smem(int Dp, int rows, bool train) {
  MlpSmem o;
  const int ld1 = Dp + 8, tile = rows * kLd * 2;
  o.W2 = kH * ld1 * 2;
  o.norm = o.W2 + kH * kLd * 2;
  o.vec = o.norm + Dp * 8;
  o.X = o.vec + 4 * kH * 4;
  o.H1 = o.X + rows * ld1 * 2;
  o.H2 = o.H1 + tile;
  o.dZ2 = o.H2 + (train ? tile : 0);
  o.dZ1 = o.dZ2 + (train ? tile : 0);
  o.head = o.dZ1 + (train ? tile : 0);
  o.total = o.head + (train ? rows * 13 * 4 : 0);
  return o;
}

__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldsm(uint32_t (&r)[4], const bf16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((uint32_t)__cvta_generic_to_shared(p)) : "memory");
}
__device__ __forceinline__ void ldsm_t(uint32_t (&r)[4], const bf16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((uint32_t)__cvta_generic_to_shared(p)) : "memory");
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}

// acc[16 rows][32 columns] += A B over ksteps x 16: A [row][k], B stored [column][k], or with
// BT [k][column]
template <bool BT>
__device__ __forceinline__ void product(float (&acc)[4][4], const bf16* A, int lda, const bf16* B, int ldb, int ksteps,
                                        int lane) {
  A += (lane & 15) * lda + (lane >> 4) * 8;
  B += BT ? (lane & 15) * ldb + (lane >> 4) * 8 : ((lane & 7) + ((lane >> 4) << 3)) * ldb + ((lane >> 3) & 1) * 8;
  const int kb = BT ? 16 * ldb : 16, nb = BT ? 16 : 16 * ldb;
#pragma unroll 4
  for (int k = 0; k < ksteps; ++k) {
    uint32_t a[4], b[2][4];
    ldsm(a, A + k * 16);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (BT) ldsm_t(b[h], B + k * kb + h * nb);
      else ldsm(b[h], B + k * kb + h * nb);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      mma_bf16(acc[2 * h], a, b[h][0], b[h][1]);
      mma_bf16(acc[2 * h + 1], a, b[h][2], b[h][3]);
    }
  }
}

// The feature's standardised value z in FP32 arithmetic from the leading bits of v, with a
// bound e on its distance from the FP64 result rounded to FP32; false where the arithmetic
// does not cover v (negative, beyond FP32's range, not finite).
// ln s = E ln 2 + ln 2 log2(m), m in [0.707, 1.414): __log2f is within 2^-22 there, E ln 2 - mu
// is one rounding with the upper bits of ln 2, the truncated bits of v and the rounded 1e-20
// shift s by under 2.4e-7: 4.8e-7 + 1.2e-7 |t| in all, taken as 8e-7 + 4e-7 |t|.
enum { FEAT_Y, FEAT_P, FEAT_T };
template <int KIND>
__device__ __forceinline__ bool feature_fast(double v, float2 norm, float* z, float* e) {
  const int hi = __double2hiint(v);
  const int fe = (hi >> 20) - 896;
  float s = __int_as_float((fe << 23) | ((hi & 0xfffff) << 3) | (int)((unsigned)__double2loint(v) >> 29));
  bool ok = hi >= 0 && fe < 255;
  if (KIND == FEAT_Y) s = (fe > 0 ? s : 0.0f) + 1e-20f;
  else ok = ok && fe > 0;
  float t, et;
  if (KIND == FEAT_T) {
    t = fmaf(s, 1e-3f, -norm.x);
    et = fmaf(s, 2.5e-10f, 8e-7f);
  } else {
    const int b = __float_as_int(s);
    const int E = (b - 0x3f3504f3) >> 23;
    const float Ef = __int_as_float(0x4b400000 + E) - 12582912.0f;  // E as a float
    const float l = __log2f(__int_as_float(b - (E << 23)));
    t = fmaf(Ef, 0.693145751953125f, -norm.x) + fmaf(Ef, 1.42860682e-6f, 0.693147182f * l);
    et = 8e-7f;
  }
  *z = t * norm.y;
  *e = fmaf(fmaf(fabsf(t), 4e-7f, et), fabsf(norm.y), 3.2e-7f * fabsf(*z));
  return ok && fabsf(*z) > 1e-30f && fabsf(*z) < 1e30f;
}

// Whether every value in [z - e, z + e] rounds to the same BF16 and lies on one side of zmax
// (zmax 0: none); the bounds are formed from z's two parts.
__device__ __forceinline__ bool feature_settled(float z, float zl, float e, float zmax) {
  const uint32_t h = pack_bf16(z + (zl - e), z + (zl + e));
  return !((h ^ (h >> 16)) & 0xffffu) && !(zmax > 0.0f && fabsf(fabsf(z) - zmax) <= fabsf(zl) + e);
}

// The same with the logarithm in 64-bit fixed point (52 fractional bits, within 2^-51): the
// quotient to twice FP32's precision, z + zl, with a bound e on its error.
__device__ __forceinline__ bool feature_fixed(double s, float mu, float sd, float* z, float* zl, float* e) {
  const int ex = __double2hiint(s) >> 20;
  if (ex < 1 || ex >= 2047 || !(fabsf(mu) < 512.0f)) return false;  // also negative s
  const long long t = chem::fx_log(s, 52) - chem::fx_from_double((double)mu);
  const float th = (float)t, inv = 1.0f / sd;
  const float tl = (float)(t - (long long)th);
  constexpr float kUnit = 2.220446049250313e-16f;  // 2^-52
  const float q = th * inv;
  *z = q * kUnit;
  *zl = (fmaf(-q, sd, th) + tl) * inv * kUnit;
  *e = fmaf(fabsf(*z), 1e-12f, fmaf(fabsf(mu), 2.0f, 3.0f) * kUnit * fabsf(inv));  // with the formula's own rounding
  return fabsf(*z) > 1e-18f && fabsf(*z) < 1e18f;
}

// A warp's R x D feature tile (BF16); rows beyond nr are zero. The BF16 value is that of the
// FP64 formula: where the FP32 value's error bound reaches across a rounding boundary (or
// across zmax), some one element in 500 and a pressure that is the same everywhere, the
// element is put on a list, and the warp goes through those side by side: in fixed point,
// and where even that does not settle the rounding, by the formula itself. (By the formula
// for all of the list, its 66 FP64 instructions per warp took a quarter of the kernel's time.)
// Returns the rows beyond zmax.
template <bool TRAIN, int R>
__device__ __forceinline__ uint32_t feature_tile(const MlpP& p, bf16* X, int ld, const float2* norm, uint16_t* list,
                                                 int64_t r0, int nr, int lane) {
  const int K = p.K, EY = R * K;
  const uint32_t inv_k = (1u << 20) / (uint32_t)K + 1;  // e / K for e < 16 K, K < 256
  const int64_t mine = p.row0 + r0 + ((lane & (R - 1)) < nr ? lane & (R - 1) : 0);
  const int64_t src = TRAIN && p.perm ? (int64_t)p.perm[mine] : mine;
  uint32_t far = 0;
  int cnt = 0;
  auto put = [&](int r, int d, float z) {
    X[r * ld + d] = __float2bfloat16(z);
    if (p.zmax > 0.0f && !(fabsf(z) <= p.zmax)) far |= 1u << r;
  };
  auto listed = [&]() {
    __syncwarp();
    for (int i0 = 0; i0 < cnt; i0 += 32) {
      const int c = list[min(i0 + lane, cnt - 1)];
      const int q = c - EY;
      const int r = q >= 0 ? q & (R - 1) : (int)((uint32_t)c * inv_k >> 20);
      const int d = q >= 0 ? q / R : c - r * K + 2;
      const int64_t row = __shfl_sync(0xffffffffu, src, r);
      const float mu = p.norm[d], sd = p.norm[p.D + d];
      float z = 0.0f, zl = 0.0f, e = 0.0f;
      bool ok = d > 0 && feature_fixed(d == 1 ? p.p[row] : p.Y[(size_t)row * K + (d - 2)] + 1e-20, mu, sd, &z, &zl, &e);
      ok = ok && feature_settled(z, zl, e, p.zmax);
      z += zl;
      if (!ok) z = (float)((feature(p.T, p.p, p.Y, K, row, d) - mu) / sd);
      put(r, d, z);
    }
    __syncwarp();
    cnt = 0;
  };
  auto take = [&](int code, int r, int d, bool valid, bool ok, float z, float e) {
    const bool slow = valid && (!ok || !feature_settled(z, 0.0f, e, p.zmax));
    if (valid && !slow) put(r, d, z);
    const uint32_t m = __ballot_sync(0xffffffffu, slow);
    if (m) {
      if (slow) list[cnt + __popc(m & ((1u << lane) - 1))] = (uint16_t)code;
      cnt += __popc(m);
    }
  };
  {
    const int r = lane & (R - 1), d = lane / R;  // lanes from 2 R on have no element
    const bool valid = d < 2 && r < nr;
    float z, e;
    bool ok;
    if (d == 0) ok = feature_fast<FEAT_T>(p.T[src], norm[0], &z, &e);
    else ok = feature_fast<FEAT_P>(p.p[src], norm[1], &z, &e);
    __syncwarp();
    if (d < 2 && !valid) X[r * ld + d] = __float2bfloat16(0.0f);
    take(EY + lane, r, d, valid, ok, z, e);
  }
  constexpr int U = R == 16 ? kFeatureBatch : 8;
#pragma unroll 1
  for (int e0 = 0; e0 < EY; e0 += 32 * U) {
    double v[U];
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const int i = e0 + j * 32 + lane;
      if (TRAIN) {
        const int r = (int)((uint32_t)min(i, EY - 1) * inv_k >> 20);
        const int64_t row = __shfl_sync(0xffffffffu, src, r);
        v[j] = i < EY && r < nr ? p.Y[(size_t)row * K + (i - r * K)] : 1.0;
      } else {
        v[j] = i < nr * K ? __ldcs(p.Y + (size_t)(p.row0 + r0) * K + i) : 1.0;
      }
    }
#pragma unroll
    for (int j = 0; j < U; ++j) {
      if (e0 + j * 32 >= EY) break;
      const int i = e0 + j * 32 + lane;
      const int r = (int)((uint32_t)min(i, EY - 1) * inv_k >> 20), k = min(i, EY - 1) - r * K;
      float z, e;
      const bool ok = feature_fast<FEAT_Y>(v[j], norm[2 + k], &z, &e);
      if (i < EY && r >= nr) X[r * ld + 2 + k] = __float2bfloat16(0.0f);
      take(i, r, 2 + k, i < EY && r < nr, ok, z, e);
    }
    if (cnt > 32 || (cnt > 0 && e0 + 32 * U >= EY)) listed();
  }
  __syncwarp();
  return __reduce_or_sync(0xffffffffu, far);
}

// out[o][i] (+)= sum over the CTA's 64 rows of A[row][o] B[row][i], o < 128, i < cols, in pieces
// of 16 x 32 dealt to the warps
__device__ __forceinline__ void weight_gradient(const bf16* A, const bf16* B, int ldb, int cols, int warp, int lane,
                                                bool add, float* out) {
  const int ar = (lane & 7) + ((lane >> 4) << 3), am = ((lane >> 3) & 1) * 8;
  const int br = lane & 15, bn = (lane >> 4) * 8;
  const int chunks = (cols + 31) / 32;
  const bool pairs = cols % 2 == 0;
#pragma unroll 1
  for (int u = warp; u < 8 * chunks; u += kTrainWarps) {
    const int o0 = (u & 7) * 16, c0 = (u >> 3) * 32;
    const bool second = c0 + 16 < cols;
    float acc[4][4] = {};
#pragma unroll
    for (int kt = 0; kt < kTrainRows / 16; ++kt) {
      uint32_t a[4], b[4];
      ldsm_t(a, A + (kt * 16 + ar) * kLd + o0 + am);
      ldsm_t(b, B + (kt * 16 + br) * ldb + c0 + bn);
      mma_bf16(acc[0], a, b[0], b[1]);
      mma_bf16(acc[1], a, b[2], b[3]);
      if (second) {
        ldsm_t(b, B + (kt * 16 + br) * ldb + c0 + 16 + bn);
        mma_bf16(acc[2], a, b[0], b[1]);
        mma_bf16(acc[3], a, b[2], b[3]);
      }
    }
#pragma unroll
    for (int nt = 0; nt < 4; ++nt)
#pragma unroll
      for (int q = 0; q < 4; q += 2) {
        const int i = c0 + nt * 8 + (lane & 3) * 2;
        float* w = out + (size_t)(o0 + (lane >> 2) + q * 4) * cols + i;
        if (pairs && i < cols) {
          float2* w2 = reinterpret_cast<float2*>(w);
          const float2 old = add ? *w2 : make_float2(0.0f, 0.0f);
          *w2 = make_float2(old.x + acc[nt][q], old.y + acc[nt][q + 1]);
        } else {
          if (i < cols) *w = add ? *w + acc[nt][q] : acc[nt][q];
          if (i + 1 < cols) w[1] = add ? w[1] + acc[nt][q + 1] : acc[nt][q + 1];
        }
      }
  }
}

template <bool TRAIN>
__global__ void __launch_bounds__((TRAIN ? kTrainWarps : kPredictWarps) * 32, 1) k_mlp(const MlpP p) {
  extern __shared__ __align__(16) unsigned char sm[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int NT = TRAIN ? kTrainWarps * 32 : blockDim.x, warps = NT / 32;
  const int rows = TRAIN ? kTrainRows : warps * 16;  // of the CTA's tiles
  const MlpSmem L = mlp_smem(p.Dp, rows, TRAIN);
  const int g = lane >> 2, t4 = lane & 3, ld1 = p.Dp + 8;
  bf16* W1 = reinterpret_cast<bf16*>(sm);
  bf16* W2 = reinterpret_cast<bf16*>(sm + L.W2);
  float2* norm = reinterpret_cast<float2*>(sm + L.norm);
  float* b1 = reinterpret_cast<float*>(sm + L.vec);
  float *b2 = b1 + kH, *w30 = b2 + kH, *w31 = w30 + kH;
  bf16* X = reinterpret_cast<bf16*>(sm + L.X);
  bf16* H1 = reinterpret_cast<bf16*>(sm + L.H1);
#pragma unroll 4
  for (int r = warp; r < kH; r += warps)
    for (int k = lane; k < p.Dp; k += 32) W1[r * ld1 + k] = k < p.D ? p.wb[r * p.D + k] : __float2bfloat16(0.0f);
#pragma unroll 4
  for (int i = tid; i < kH * kH / 8; i += NT)
    *reinterpret_cast<uint4*>(W2 + (i >> 4) * kLd + (i & 15) * 8) = reinterpret_cast<const uint4*>(p.wb + p.oW2)[i];
  for (int d = tid; d < p.D; d += NT) norm[d] = make_float2(p.norm[d], 1.0f / p.norm[p.D + d]);
  for (int i = tid; i < kH; i += NT) {
    b1[i] = p.w[p.ob1 + i];
    b2[i] = p.w[p.ob2 + i];
    w30[i] = __bfloat162float(p.wb[p.oW3 + i]);
    w31[i] = __bfloat162float(p.wb[p.oW3 + kH + i]);
  }
  for (int i = tid; i < rows * (p.Dp - p.D); i += NT) X[(i % rows) * ld1 + p.D + i / rows] = __float2bfloat16(0.0f);
  __syncthreads();
  const float b30 = p.w[p.ob3], b31 = p.w[p.ob3 + 1];
  const float* nt = p.norm + 2 * p.D;
  // a layer's 32 columns c0 .. c0 + 31 of the warp's 16 rows, as the lane's pairs of columns
  // c0 + 8 j + 2 t4 in rows g and g + 8: z = acc + bias, h = GELU(z) rounded, slope = GELU'(z)
  auto layer = [&](const bf16* A, int lda, const bf16* W, int ldw, int ksteps, const float* bias, int c0, bf16* H,
                   float (&slope)[4][4], float (&o)[4], bool head) {
    float acc[4][4] = {};
    product<false>(acc, A, lda, W + c0 * ldw, ldw, ksteps, lane);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int c = c0 + j * 8 + t4 * 2;
      const float2 b = *reinterpret_cast<const float2*>(bias + c);
#pragma unroll
      for (int q = 0; q < 4; q += 2) {
        const float z0 = acc[j][q] + b.x, z1 = acc[j][q + 1] + b.y;
        const __nv_bfloat162 hh = __floats2bfloat162_rn(gelu(z0), gelu(z1));
        if (TRAIN || !head) *reinterpret_cast<__nv_bfloat162*>(H + (g + q * 4) * kLd + c) = hh;
        if (TRAIN) {
          slope[j][q] = gelu_grad(z0);
          slope[j][q + 1] = gelu_grad(z1);
        }
        if (head) {
          const float2 f = __bfloat1622float2(hh);
          const float2 u0 = *reinterpret_cast<const float2*>(w30 + c), u1 = *reinterpret_cast<const float2*>(w31 + c);
          o[q] += f.x * u0.x + f.y * u0.y;
          o[q + 1] += f.x * u1.x + f.y * u1.y;
        }
      }
    }
  };
  if (!TRAIN) {
    X += warp * 16 * ld1;
    H1 += warp * 16 * kLd;
    const int64_t tiles = (p.n + 15) / 16;
#pragma unroll 1
    for (int64_t tile = (int64_t)warp * gridDim.x + blockIdx.x; tile < tiles; tile += (int64_t)gridDim.x * warps) {
      const int64_t r0 = tile * 16;
      const int nr = (int)min((int64_t)16, p.n - r0);
      const uint32_t far = feature_tile<false, 16>(p, X, ld1, norm, reinterpret_cast<uint16_t*>(H1), r0, nr, lane);
      float slope[4][4], o[4] = {};
#pragma unroll 1
      for (int c0 = 0; c0 < kH; c0 += 32) layer(X, ld1, W1, ld1, p.Dp / 16, b1, c0, H1, slope, o, false);
      __syncwarp();
#pragma unroll 1
      for (int c0 = 0; c0 < kH; c0 += 32) layer(H1, kLd, W2, kLd, kH / 16, b2, c0, H1, slope, o, true);
      // rows g (o[0], o[1]) and g + 8 (o[2], o[3])
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        o[q] += __shfl_xor_sync(0xffffffffu, o[q], 1);
        o[q] += __shfl_xor_sync(0xffffffffu, o[q], 2);
      }
      const int r = g + (t4 & 1) * 8;
      if (t4 < 2 && r < nr) {
        const float l0 = ((t4 ? o[2] : o[0]) + b30) * nt[2] + nt[0];
        const float l1 = ((t4 ? o[3] : o[1]) + b31) * nt[3] + nt[1];
        const int64_t q = p.row0 + r0 + r;
        if (p.ln_cost) p.ln_cost[q] = l0;
        if (p.ln_h0) p.ln_h0[q] = l1;
        if (p.cost) p.cost[q] = expf(fminf(l0, 80.0f));
        if (p.h0)
          p.h0[q] = far >> r & 1 ? __longlong_as_double(0x7ff8000000000000LL) : fmax(exp((double)l1), 1e-14);
      }
      __syncwarp();
    }
    return;
  }
  bf16* H2 = reinterpret_cast<bf16*>(sm + L.H2);
  bf16* dZ2 = reinterpret_cast<bf16*>(sm + L.dZ2);
  bf16* dZ1 = reinterpret_cast<bf16*>(sm + L.dZ1);
  float* po = reinterpret_cast<float*>(sm + L.head);  // [rows][4 column groups][2] outputs
  float* ts = po + 8 * kTrainRows;                     // [rows][2] standardised targets
  float* dc = ts + 2 * kTrainRows;                     // [rows][3] d0, d1, loss
  const int rt = warp >> 2, c0 = (warp & 3) * 32;      // the warp's 16 rows and 32 columns
  bool add = false;
#pragma unroll 1
  for (int64_t base = (int64_t)blockIdx.x * kTrainRows; base < p.n; base += (int64_t)gridDim.x * kTrainRows) {
    constexpr int R = kTrainRows / kTrainWarps;  // rows of features per warp
    {
      const int64_t r0 = base + warp * R;
      const int nr = (int)max((int64_t)0, min((int64_t)R, p.n - r0));
      feature_tile<true, R>(p, X + warp * R * ld1, ld1, norm, reinterpret_cast<uint16_t*>(H1) + warp * kListed,
                            nr ? r0 : 0, nr, lane);
    }
    if (warp < kTrainRows * 2 / 32) {  // one target a lane: rows' cost, then their first step
      const int r = tid >> 1, w = tid & 1;
      float v = 0.0f;
      if (base + r < p.n) {
        const int64_t q = p.row0 + base + r;
        const int64_t src = p.perm ? (int64_t)p.perm[q] : q;
        const double t = log(w == 0 ? fmax((double)p.sub[src], 1.0) : fmax(p.hf[src], 1e-300));
        v = (float)((t - nt[w]) / nt[2 + w]);
      }
      ts[tid] = v;
    }
    __syncthreads();
    float s1[4][4], s2[4][4], o[4] = {};
    layer(X + rt * 16 * ld1, ld1, W1, ld1, p.Dp / 16, b1, c0, H1 + rt * 16 * kLd, s1, o, false);
    __syncthreads();
    layer(H1 + rt * 16 * kLd, kLd, W2, kLd, kH / 16, b2, c0, H2 + rt * 16 * kLd, s2, o, true);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      o[q] += __shfl_xor_sync(0xffffffffu, o[q], 1);
      o[q] += __shfl_xor_sync(0xffffffffu, o[q], 2);
    }
    if (t4 < 2) {
      float* e = po + (rt * 16 + g + t4 * 8) * 8 + (warp & 3) * 2;
      e[0] = t4 ? o[2] : o[0];
      e[1] = t4 ? o[3] : o[1];
    }
    __syncthreads();
    float d[4];
#pragma unroll
    for (int q = 0; q < 4; q += 2) {
      const int r = rt * 16 + g + q * 4;
      const float4 ea = *reinterpret_cast<const float4*>(po + r * 8), eb = *reinterpret_cast<const float4*>(po + r * 8 + 4);
      const bool in = base + r < p.n;
      const float r0 = in ? ea.x + ea.z + eb.x + eb.z + b30 - ts[2 * r] : 0.0f;
      const float r1 = in ? ea.y + ea.w + eb.y + eb.w + b31 - ts[2 * r + 1] : 0.0f;
      d[q] = r0 * p.inv_B;
      d[q + 1] = r1 * p.inv_B;
      if ((warp & 3) == 0 && t4 == 0) {
        dc[r * 3] = d[q];
        dc[r * 3 + 1] = d[q + 1];
        dc[r * 3 + 2] = 0.5f * (r0 * r0 + r1 * r1) * p.inv_B;
      }
    }
    // dZ2, and dZ1 = (dZ2 W2) GELU'(Z1)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int c = c0 + j * 8 + t4 * 2;
      const float2 u0 = *reinterpret_cast<const float2*>(w30 + c), u1 = *reinterpret_cast<const float2*>(w31 + c);
#pragma unroll
      for (int q = 0; q < 4; q += 2)
        *reinterpret_cast<uint32_t*>(dZ2 + (rt * 16 + g + q * 4) * kLd + c) =
            pack_bf16((d[q] * u0.x + d[q + 1] * u1.x) * s2[j][q], (d[q] * u0.y + d[q + 1] * u1.y) * s2[j][q + 1]);
    }
    __syncthreads();
    {
      float acc[4][4] = {};
      product<true>(acc, dZ2 + rt * 16 * kLd, kLd, W2 + c0, kLd, kH / 16, lane);
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int q = 0; q < 4; q += 2)
          *reinterpret_cast<uint32_t*>(dZ1 + (rt * 16 + g + q * 4) * kLd + c0 + j * 8 + t4 * 2) =
              pack_bf16(acc[j][q] * s1[j][q], acc[j][q + 1] * s1[j][q + 1]);
    }
    __syncthreads();
    // the CTA's contribution to the gradient
    float* part = p.part + blockIdx.x * p.part_stride;
    weight_gradient(dZ2, H1, kLd, kH, warp, lane, add, part + p.oW2);
    weight_gradient(dZ1, X, ld1, p.D, warp, lane, add, part);
    {
      const int c = tid & (kH - 1), what = tid / kH;  // b1, b2, the rows of W3
      const bf16* z = what == 0 ? dZ1 : what == 1 ? dZ2 : H2;
      float s = 0.0f;
#pragma unroll 8
      for (int r = 0; r < kTrainRows; ++r)
        s = fmaf(what < 2 ? 1.0f : dc[r * 3 + (what & 1)], __bfloat162float(z[r * kLd + c]), s);
      float* w = part + (what == 0 ? p.ob1 : what == 1 ? p.ob2 : p.oW3 + (what & 1) * kH) + c;
      *w = add ? *w + s : s;
    }
    if (tid < 3) {  // b3's gradient and the loss
      float v = 0.0f;
      for (int r = 0; r < kTrainRows; ++r) v += dc[r * 3 + tid];
      float* w = part + p.ob3 + tid;
      *w = add ? *w + v : v;
    }
    add = true;
    __syncthreads();
  }
}

// out[j] = sum over the S partials of part[s][j] in a fixed order, j <= nw; entry nw is the loss.
// 128 entries a CTA, the partials dealt to eight groups of threads: all loads of a thread
// are independent.
__global__ void __launch_bounds__(1024) k_reduce(const float* part, int S, int64_t stride, int64_t nw, float* out,
                                                 float* loss) {
  __shared__ float sh[8][128];
  const int64_t j = (int64_t)blockIdx.x * 128 + threadIdx.x;
  float s = 0.0f;
  if (j <= nw) {
#pragma unroll 8
    for (int i = threadIdx.y; i < S; i += 8) s += part[i * stride + j];
  }
  sh[threadIdx.y][threadIdx.x] = s;
  __syncthreads();
  if (threadIdx.y == 0 && j <= nw) {
    for (int i = 1; i < 8; ++i) s += sh[i][threadIdx.x];
    if (j < nw) out[j] = s;
    else *loss = s;
  }
}

__global__ void k_adam(float* w, const float* g, float* m, float* v, bf16* wb, int64_t n, float lr, float b1,
                       float b2, float eps, float c1, float c2) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    w[i] = wi;
    wb[i] = __float2bfloat16(wi);
  }
}

__global__ void k_to_bf16(const float* w, bf16* wb, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    wb[i] = __float2bfloat16(w[i]);
}

}  // namespace

// ---------------------------------------------------------------------------
// model object
// ---------------------------------------------------------------------------
struct chem_mlp_s {
  int K = 0, D = 0;
  int64_t nw = 0;  // weight+bias floats
  int64_t oW1 = 0, ob1 = 0, oW2 = 0, ob2 = 0, oW3 = 0, ob3 = 0;
  float* w = nullptr;  // FP32 master [nw]
  float* g = nullptr;  // gradient [nw]
  float* m = nullptr;
  float* v = nullptr;
  bf16* wb = nullptr;  // BF16 copy [nw]
  float* norm = nullptr;          // device: mu_x[D], sd_x[D], mu_t[2], sd_t[2]
  std::vector<float> norm_h;      // host copy
  int64_t adam_t = 0;
  // kept between calls: the CTAs' partial gradients, the gradient and loss on the host
  float* part = nullptr;   // [num_sms][part_stride]
  float* host = nullptr;   // pinned, [nw + 1]
  int64_t part_stride = 0;
  int num_sms = 0;
  std::string err;
};

static chem_status mlp_cuda(chem_mlp m, cudaError_t e, const char* what) {
  if (e == cudaSuccess) return CHEM_OK;
  if (m) m->err = std::string(what) + ": " + cudaGetErrorString(e);
  return e == cudaErrorMemoryAllocation ? CHEM_ERR_OOM : CHEM_ERR_CUDA;
}

#define MLP_TRY(m, call)                                    \
  do {                                                      \
    chem_status s_ = mlp_cuda((m), (call), #call);          \
    if (s_ != CHEM_OK) return s_;                           \
  } while (0)

// what a gradient needs beside the weights; allocated with the first one
static chem_status mlp_train_scratch(chem_mlp m) {
  if (m->host) return CHEM_OK;
  if (!m->part) MLP_TRY(m, cudaMalloc(&m->part, m->num_sms * m->part_stride * sizeof(float)));
  MLP_TRY(m, cudaMallocHost(&m->host, (m->nw + 1) * sizeof(float)));
  return CHEM_OK;
}

extern "C" chem_status chem_mlp_create(int32_t n_species, uint64_t seed, chem_mlp* out) {
  if (!out || n_species < 1 || n_species > 255) return CHEM_ERR_INVALID_ARG;
  *out = nullptr;
  chem_mlp m = new chem_mlp_s();
  m->K = n_species;
  m->D = n_species + 2;
  const int D = m->D;
  m->oW1 = 0;
  m->ob1 = m->oW1 + (int64_t)kH * D;
  m->oW2 = m->ob1 + kH;
  m->ob2 = m->oW2 + (int64_t)kH * kH;
  m->oW3 = m->ob2 + kH;
  m->ob3 = m->oW3 + 2 * kH;
  m->nw = m->ob3 + 2;
  std::vector<float> w(m->nw);
  std::mt19937_64 rng(seed);
  std::uniform_real_distribution<double> U(-1.0, 1.0);
  auto fill = [&](int64_t o, int64_t cnt, int fan) {
    for (int64_t i = 0; i < cnt; ++i) w[o + i] = (float)(U(rng) / std::sqrt((double)fan));
  };
  fill(m->oW1, (int64_t)kH * D, D);
  fill(m->ob1, kH, D);
  fill(m->oW2, (int64_t)kH * kH, kH);
  fill(m->ob2, kH, kH);
  fill(m->oW3, 2 * kH, kH);
  fill(m->ob3, 2, kH);
  m->norm_h.assign(2 * D + 4, 0.0f);
  for (int d = 0; d < D; ++d) m->norm_h[D + d] = 1.0f;
  m->norm_h[2 * D + 2] = m->norm_h[2 * D + 3] = 1.0f;
  m->part_stride = (m->nw + 32) / 32 * 32;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&m->num_sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_mlp<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmemMlp);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_mlp<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmemMlp);
  if (e == cudaSuccess) e = cudaMalloc(&m->w, m->nw * 4);
  if (e == cudaSuccess) e = cudaMalloc(&m->g, m->nw * 4);
  if (e == cudaSuccess) e = cudaMalloc(&m->m, m->nw * 4);
  if (e == cudaSuccess) e = cudaMalloc(&m->v, m->nw * 4);
  if (e == cudaSuccess) e = cudaMalloc(&m->wb, m->nw * sizeof(bf16));
  if (e == cudaSuccess) e = cudaMalloc(&m->norm, m->norm_h.size() * 4);
  if (e == cudaSuccess) e = cudaMemcpy(m->w, w.data(), m->nw * 4, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(m->m, 0, m->nw * 4);
  if (e == cudaSuccess) e = cudaMemset(m->v, 0, m->nw * 4);
  if (e == cudaSuccess) e = cudaMemcpy(m->norm, m->norm_h.data(), m->norm_h.size() * 4, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    k_to_bf16<<<64, 256>>>(m->w, m->wb, m->nw);
    e = cudaDeviceSynchronize();
  }
  if (e != cudaSuccess) {
    chem_mlp_destroy(m);
    return e == cudaErrorMemoryAllocation ? CHEM_ERR_OOM : CHEM_ERR_CUDA;
  }
  *out = m;
  return CHEM_OK;
}

extern "C" chem_status chem_mlp_destroy(chem_mlp m) {
  if (!m) return CHEM_ERR_INVALID_ARG;
  cudaDeviceSynchronize();
  for (void* p : {(void*)m->w, (void*)m->g, (void*)m->m, (void*)m->v, (void*)m->wb, (void*)m->norm, (void*)m->part})
    if (p) cudaFree(p);
  if (m->host) cudaFreeHost(m->host);
  delete m;
  return CHEM_OK;
}

extern "C" chem_status chem_mlp_attach(chem_handle h, chem_mlp m) {
  if (!h) return CHEM_ERR_INVALID_ARG;
  if (m && m->K != h->K) {
    h->err = "chem_mlp_attach: model and mechanism disagree on the number of species";
    return CHEM_ERR_INVALID_ARG;
  }
  h->mlp = m;
  return CHEM_OK;
}

extern "C" chem_status chem_mlp_get_params(chem_mlp m, float* buf, int64_t* n_floats) {
  if (!m || !n_floats) return CHEM_ERR_INVALID_ARG;
  const int64_t nn = (int64_t)m->norm_h.size();
  *n_floats = nn + m->nw;
  if (!buf) return CHEM_OK;
  std::memcpy(buf, m->norm_h.data(), nn * 4);
  MLP_TRY(m, cudaMemcpy(buf + nn, m->w, m->nw * 4, cudaMemcpyDeviceToHost));
  return CHEM_OK;
}

extern "C" chem_status chem_mlp_set_params(chem_mlp m, const float* buf, int64_t n_floats) {
  if (!m || !buf) return CHEM_ERR_INVALID_ARG;
  const int64_t nn = (int64_t)m->norm_h.size();
  if (n_floats != nn + m->nw) {
    m->err = "chem_mlp_set_params: wrong length";
    return CHEM_ERR_INVALID_ARG;
  }
  std::memcpy(m->norm_h.data(), buf, nn * 4);
  MLP_TRY(m, cudaMemcpy(m->norm, buf, nn * 4, cudaMemcpyHostToDevice));
  MLP_TRY(m, cudaMemcpy(m->w, buf + nn, m->nw * 4, cudaMemcpyHostToDevice));
  k_to_bf16<<<64, 256>>>(m->w, m->wb, m->nw);
  MLP_TRY(m, cudaDeviceSynchronize());
  return CHEM_OK;
}

// ---------------------------------------------------------------------------
// building blocks
// ---------------------------------------------------------------------------
static MlpP mlp_args(chem_mlp m, int64_t n, const double* T, const double* p, const double* Y) {
  MlpP a{};
  a.T = T;
  a.p = p;
  a.Y = Y;
  a.n = n;
  a.K = m->K;
  a.D = m->D;
  a.Dp = (m->D + 15) / 16 * 16;
  a.norm = m->norm;
  a.wb = m->wb;
  a.w = m->w;
  a.ob1 = m->ob1;
  a.oW2 = m->oW2;
  a.ob2 = m->ob2;
  a.oW3 = m->oW3;
  a.ob3 = m->ob3;
  a.nw = m->nw;
  return a;
}

// gradient and loss of the rows of `a`
static chem_status fwd_bwd(chem_mlp m, MlpP a, cudaStream_t st, float* grad, float* loss) {
  a.inv_B = 1.0f / (float)a.n;
  a.part = m->part;
  a.part_stride = m->part_stride;
  const int grid = (int)std::min<int64_t>((a.n + kTrainRows - 1) / kTrainRows, m->num_sms);
  k_mlp<true><<<grid, kTrainWarps * 32, mlp_smem(a.Dp, kTrainRows, true).total, st>>>(a);
  k_reduce<<<(int)((m->nw + 128) / 128), dim3(128, 8), 0, st>>>(m->part, grid, m->part_stride, m->nw, grad, loss);
  return mlp_cuda(m, cudaGetLastError(), "mlp backward");
}

// Adam's bias corrections 1 - beta^t for the FP32 betas the kernel uses, evaluated in
// double and rounded once (1 - beta2^t in float loses ~1e-5 relative for small t).
static void adam_corrections(float b1, float b2, int64_t t, float* c1, float* c2) {
  *c1 = (float)(1.0 - std::pow((double)b1, (double)t));
  *c2 = (float)(1.0 - std::pow((double)b2, (double)t));
}

static chem_status set_normalisation(chem_mlp m, int64_t n, const double* T, const double* p, const double* Y,
                                     const int32_t* sub, const double* hf, cudaStream_t st) {
  const int D = m->D;
  double* sums = nullptr;
  MLP_TRY(m, cudaMalloc(&sums, (2 * D + 4) * sizeof(double)));
  cudaMemsetAsync(sums, 0, (2 * D + 4) * sizeof(double), st);
  const int grid = (int)std::min<int64_t>(n, 512);
  k_feature_stats<<<grid, 128, 2 * D * sizeof(double), st>>>(T, p, Y, m->K, n, sums);
  k_target_stats<<<(int)std::min<int64_t>((n + 255) / 256, 512), 256, 0, st>>>(sub, hf, n, sums + 2 * D);
  std::vector<double> h(2 * D + 4);
  cudaError_t e = cudaMemcpyAsync(h.data(), sums, h.size() * 8, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFree(sums);
  MLP_TRY(m, e);
  for (int d = 0; d < D; ++d) {
    const double mu = h[d] / n;
    const double var = std::max(h[D + d] / n - mu * mu, 0.0);
    m->norm_h[d] = (float)mu;
    m->norm_h[D + d] = (float)std::max(std::sqrt(var), 1e-3);
  }
  for (int t = 0; t < 2; ++t) {
    const double mu = h[2 * D + 2 * t] / n;
    const double var = std::max(h[2 * D + 2 * t + 1] / n - mu * mu, 0.0);
    m->norm_h[2 * D + t] = (float)mu;
    m->norm_h[2 * D + 2 + t] = (float)std::max(std::sqrt(var), 1e-3);
  }
  MLP_TRY(m, cudaMemcpyAsync(m->norm, m->norm_h.data(), m->norm_h.size() * 4, cudaMemcpyHostToDevice, st));
  MLP_TRY(m, cudaStreamSynchronize(st));
  return CHEM_OK;
}

extern "C" chem_status chem_mlp_train(chem_mlp m, int64_t n, const double* T, const double* p, const double* Y,
                                      const int32_t* substeps, const double* h_first, int32_t epochs,
                                      int32_t batch, double lr, uint64_t seed, float* loss_host, void* stream) {
  if (!m || n < 1 || !T || !p || !Y || !substeps || !h_first || epochs < 0 || batch < 32 || !(lr > 0.0))
    return CHEM_ERR_INVALID_ARG;
  if (n > 2147483647LL) return CHEM_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  chem_status s = set_normalisation(m, n, T, p, Y, substeps, h_first, st);
  if (s != CHEM_OK) return s;
  s = mlp_train_scratch(m);
  if (s != CHEM_OK) return s;
  int* perm_d = nullptr;
  float* loss_d = nullptr;
  MLP_TRY(m, cudaMalloc(&perm_d, (size_t)n * sizeof(int)));
  const int B = (int)std::min<int64_t>(batch, n);
  const int nb = (int)((n + B - 1) / B);
  MLP_TRY(m, cudaMalloc(&loss_d, (size_t)nb * sizeof(float)));
  MlpP a = mlp_args(m, 0, T, p, Y);
  a.sub = substeps;
  a.hf = h_first;
  a.perm = perm_d;
  std::vector<int> perm(n);
  std::mt19937_64 rng(seed);
  std::vector<float> batch_losses(nb);
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  for (int ep = 0; ep < epochs; ++ep) {
    for (int64_t i = 0; i < n; ++i) perm[i] = (int)i;
    std::shuffle(perm.begin(), perm.end(), rng);
    MLP_TRY(m, cudaMemcpyAsync(perm_d, perm.data(), n * sizeof(int), cudaMemcpyHostToDevice, st));
    for (int bi = 0; bi < nb; ++bi) {
      a.row0 = (int64_t)bi * B;
      a.n = std::min<int64_t>(B, n - a.row0);
      s = fwd_bwd(m, a, st, m->g, loss_d + bi);
      if (s != CHEM_OK) return s;
      ++m->adam_t;
      float c1, c2;
      adam_corrections(b1, b2, m->adam_t, &c1, &c2);
      k_adam<<<64, 256, 0, st>>>(m->w, m->g, m->m, m->v, m->wb, m->nw, (float)lr, b1, b2, eps, c1, c2);
    }
    // the host permutation buffer is reused next epoch: wait, and collect the batch losses
    MLP_TRY(m, cudaMemcpyAsync(batch_losses.data(), loss_d, nb * sizeof(float), cudaMemcpyDeviceToHost, st));
    MLP_TRY(m, cudaStreamSynchronize(st));
    if (loss_host) {
      double acc = 0.0;
      for (int bi = 0; bi < nb; ++bi) acc += batch_losses[bi];
      loss_host[ep] = (float)(acc / nb);
    }
  }
  MLP_TRY(m, cudaStreamSynchronize(st));
  cudaFree(perm_d);
  cudaFree(loss_d);
  return mlp_cuda(m, cudaGetLastError(), "chem_mlp_train");
}

extern "C" chem_status chem_mlp_gradient(chem_mlp m, int64_t n, const double* T, const double* p, const double* Y,
                                         const int32_t* substeps, const double* h_first, float* loss_host,
                                         float* grad_host, void* stream) {
  if (!m || n < 1 || n > 1 << 20 || !T || !p || !Y || !substeps || !h_first) return CHEM_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  chem_status s = mlp_train_scratch(m);
  if (s != CHEM_OK) return s;
  MlpP a = mlp_args(m, n, T, p, Y);
  a.sub = substeps;
  a.hf = h_first;
  // the reduction writes the result to the pinned buffer itself
  s = fwd_bwd(m, a, st, m->host, m->host + m->nw);
  if (s != CHEM_OK) return s;
  MLP_TRY(m, cudaStreamSynchronize(st));
  if (grad_host) std::memcpy(grad_host, m->host, m->nw * 4);
  if (loss_host) *loss_host = m->host[m->nw];
  return CHEM_OK;
}

extern "C" chem_status chem_mlp_apply_gradient(chem_mlp m, const float* grad_host, double lr, void* stream) {
  if (!m || !grad_host || !(lr > 0.0) || !std::isfinite(lr)) return CHEM_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  MLP_TRY(m, cudaMemcpyAsync(m->g, grad_host, m->nw * 4, cudaMemcpyHostToDevice, st));
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  ++m->adam_t;
  float c1, c2;
  adam_corrections(b1, b2, m->adam_t, &c1, &c2);
  k_adam<<<64, 256, 0, st>>>(m->w, m->g, m->m, m->v, m->wb, m->nw, (float)lr, b1, b2, eps, c1, c2);
  MLP_TRY(m, cudaGetLastError());
  MLP_TRY(m, cudaStreamSynchronize(st));
  return CHEM_OK;
}

// zmax > 0: cells with a standardised feature beyond +-zmax training standard
// deviations get a NaN initial step (the integrator then takes its heuristic).
static chem_status predict_into(chem_mlp m, int64_t n, const double* T, const double* p, const double* Y, float* ln_cost,
                                float* ln_h0, float* cost, double* h0, cudaStream_t st, float zmax = 0.0f) {
  MlpP a = mlp_args(m, n, T, p, Y);
  a.zmax = h0 ? zmax : 0.0f;
  a.ln_cost = ln_cost;
  a.ln_h0 = ln_h0;
  a.cost = cost;
  a.h0 = h0;
  // a CTA per SM, with no more warps than there are tiles of 16 rows for it or memory
  const int64_t tiles = (n + 15) / 16;
  const int grid = (int)std::min<int64_t>(tiles, m->num_sms);
  int warps = std::max(4, (int)std::min<int64_t>((tiles + grid - 1) / grid, kPredictWarps));
  while (mlp_smem(a.Dp, warps * 16, false).total > (int)kMaxSmemMlp) --warps;
  const size_t smem = mlp_smem(a.Dp, warps * 16, false).total;
  k_mlp<false><<<grid, warps * 32, smem, st>>>(a);
  return mlp_cuda(m, cudaGetLastError(), "chem_mlp_predict");
}

extern "C" chem_status chem_mlp_predict(chem_mlp m, int64_t n, const double* T, const double* p, const double* Y,
                                        float* ln_cost, float* ln_h0, void* stream) {
  if (!m || n < 0 || (n > 0 && (!T || !p || !Y))) return CHEM_ERR_INVALID_ARG;
  if (n == 0) return CHEM_OK;
  return predict_into(m, n, T, p, Y, ln_cost, ln_h0, nullptr, nullptr, static_cast<cudaStream_t>(stream));
}

// Scheduler hook: predicted cost (float, substeps) and initial step (double) per cell.
chem_status chem_internal_mlp_predict(chem_handle h, const double* T, const double* p, const double* Y, int64_t n,
                                      cudaStream_t st, const float** cost, const double** h0) {
  float* c = nullptr;
  double* hh = nullptr;
  chem_status s = chem_internal_learned_buffers(h, n, &c, &hh, nullptr);
  if (s != CHEM_OK) return s;
  s = predict_into(h->mlp, n, T, p, Y, nullptr, nullptr, c, h0 ? hh : nullptr, st,
                   (float)h->h0_range);
  if (s != CHEM_OK) {
    h->err = h->mlp->err;
    return s;
  }
  *cost = c;
  if (h0) *h0 = hh;
  return CHEM_OK;
}

void chem_internal_release_learned(chem_handle h) { h->mlp = nullptr; }
