// learned.cu -- learned per-row polynomial smoother: features, MLP inference
// and training kernels, and the two-grid error-reduction gradient that the
// training minimises.  The paper lists polynomial smoothers as future work
// (Sec. 5); the network and its training are this library's own.
//
// MLP: 16 -> 64 -> 64 -> 3, tanh, FP16 weights.  Inference runs the three
// layers on the tensor cores (mma.sync, FP16 operands with FP32 accumulation,
// activations as two FP16 parts); training keeps FP32 master weights on the
// CUDA cores.  Coefficients: c_q = omega_k (delta_q0 + o_q).  The weight
// gradients are deterministic fixed-order sums over rows.
#include <cmath>
#include <cstring>
#include <vector>

#include <cuda_fp16.h>

#include "amg_internal.cuh"

namespace amg {

constexpr int NF = 16, NH = 64, NO = 3;
constexpr int W1O = 0, B1O = NH * NF, W2O = B1O + NH, B2O = W2O + NH * NH, W3O = B2O + NH, B3O = W3O + NO * NH;
constexpr int NP = B3O + NO;
static_assert(NP == AMG_MLP_NPARAM, "parameter layout");

// ------------------------------------------------------------------ features
// Row i, d = |A_ii|, t_j = -A_ij / d (j != i):
//  0: 1   1: #off/8   2..9: eight largest |A_ij|/d descending   10: fraction of
//  off-diagonals with the sign of A_ii   11: (sum_j A_ij)/A_ii   12: level/4
//  13: min t_j   14: max t_j   15: sum |A_ij|/d.  Sums in CSR order by IEEE
//  additions, quotients as below: the FP32 features of a sequential evaluation.
//
// The FP64 pipe bounds it (a warp instruction takes 16 cycles of an SM), so an
// entry takes one quotient (|A_ij|/d = |t_j|) and two additions in FP64; what the
// features only compare (minimum, maximum, the eight largest) is compared after
// the rounding to FP32, which is monotone and gives the same FP32 features.  The
// eight largest stay in registers (a compare-exchange chain with static indices;
// an insertion with a moving index kept them in local memory).  A block reads its
// rows' entries through shared memory, where the threads' row-by-row order is
// free of the strided global accesses.  1024^2 FEM rows (7.3 M entries): 671 -> 240 us.

// v / d for d > 0 with r = RN(1/d): q = v r, then one residual correction
// q + (v - q d) r (Markstein, "Computation of elementary functions on the IBM RISC
// System/6000 processor", 1990).  With q within an ulp the result is the correctly
// rounded quotient.  q = RN(v r) can be 1.5 ulp off; then a quotient within 2^-51 of an
// ulp of a rounding boundary can come out as its FP64 neighbour, a difference of 2^-53
// in an FP32 feature's sums or before its rounding.  Outside a safe range of exponents
// the division is taken as is.
__device__ __forceinline__ bool quotient_safe(double d) { return d > 0x1p-400 && d < 0x1p400; }
__device__ __forceinline__ double quotient(double v, double d, double r, bool safe) {
  const int ev = (__double2hiint(v) >> 20) & 0x7ff;  // biased exponent
  if (safe && ev > 1023 - 400 && ev < 1023 + 400) {
    const double q = __dmul_rn(v, r);
    return __fma_rn(__fma_rn(-q, d, v), r, q);
  }
  if (safe && v == 0.0) return v;
  return __ddiv_rn(v, d);
}

constexpr int kFeatThreads = 128;
constexpr int kFeatStage = 2048;  // entries of a block's rows staged in shared memory

__global__ void __launch_bounds__(kFeatThreads) k_features(int32_t n, const int32_t *__restrict__ rp,
                                                           const int32_t *__restrict__ ci,
                                                           const double *__restrict__ val, int32_t level,
                                                           float *__restrict__ feat) {
  __shared__ double sv[kFeatStage];
  __shared__ int32_t sc[kFeatStage];
  __shared__ float sf[kFeatThreads * (NF + 1)];  // rows padded: no bank conflicts
  for (int32_t i0 = blockIdx.x * kFeatThreads; i0 < n; i0 += gridDim.x * kFeatThreads) {
    const int32_t rows = min(kFeatThreads, n - i0);
    const int32_t b0 = rp[i0], cnt = rp[i0 + rows] - b0;
    const bool staged = cnt <= kFeatStage;
    if (staged)
      for (int32_t p = threadIdx.x; p < cnt; p += kFeatThreads) {
        sv[p] = __ldcs(val + b0 + p);
        sc[p] = __ldcs(ci + b0 + p);
      }
    __syncthreads();
    const int32_t i = i0 + threadIdx.x;
    if (threadIdx.x < rows) {
      // entries p0 .. p1 - 1 of v_ and c_
      auto row = [&](const double *__restrict__ v_, const int32_t *__restrict__ c_, int32_t p0, int32_t p1) {
        double aii = 0.0;
        for (int32_t p = p0; p < p1; ++p)
          if (c_[p] == i) aii = v_[p];
        const double d = fabs(aii);
        const bool safe = quotient_safe(d);
        const double r = __drcp_rn(d);
        float top[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        double rowsum = 0.0, abssum = 0.0;
        float tmin = 0.0f, tmax = 0.0f;
        int32_t noff = 0, nsame = 0;
        for (int32_t p = p0; p < p1; ++p) {
          const double v = v_[p];
          rowsum = __dadd_rn(rowsum, v);
          if (c_[p] == i) continue;
          const double t = quotient(-v, d, r, safe);
          abssum = __dadd_rn(abssum, fabs(t));
          const float tf = (float)t;
          if (noff == 0 || tf < tmin) tmin = tf;
          if (noff == 0 || tf > tmax) tmax = tf;
          // the sign of v: that of -t, except that a zero has none
          if ((tf < 0.0f && aii > 0.0) || (tf > 0.0f && aii < 0.0) ||
              (tf == 0.0f && ((v > 0.0 && aii > 0.0) || (v < 0.0 && aii < 0.0))))
            nsame++;
          noff++;
          float a = fabsf(tf);
#pragma unroll
          for (int k = 0; k < 8; ++k) {  // keep the list descending: the smaller one moves on
            const float hi = fmaxf(top[k], a);
            a = fminf(top[k], a);
            top[k] = hi;
          }
        }
        float *f = sf + threadIdx.x * (NF + 1);
        f[0] = 1.0f;
        f[1] = (float)noff * 0.125f;  // exact, like level / 4; 24-bit integers' quotient rounds the same in FP32
#pragma unroll
        for (int k = 0; k < 8; ++k) f[2 + k] = top[k];
        f[10] = noff ? __fdiv_rn((float)nsame, (float)noff) : 0.0f;
        f[11] = (float)quotient(aii < 0.0 ? -rowsum : rowsum, d, r, safe);
        f[12] = (float)level * 0.25f;
        f[13] = tmin;
        f[14] = tmax;
        f[15] = (float)abssum;
      };
      if (staged) row(sv, sc, rp[i] - b0, rp[i + 1] - b0);
      else row(val, ci, rp[i], rp[i + 1]);
    }
    __syncthreads();
    for (int32_t q = threadIdx.x; q < rows * NF; q += kFeatThreads)
      feat[(size_t)i0 * NF + q] = sf[(q / NF) * (NF + 1) + q % NF];
    __syncthreads();
  }
}

// ------------------------------------------------------------------ MLP in FP32 (training)
// A block of 256 threads takes a tile of 64 rows through the network in shared
// memory: thread (tr, tu) holds 4 rows x 4 units (rows 4 tr + i, units tu + 16 j), so
// that 8 float4 loads feed 64 multiply-adds, where a thread per row read one weight
// per multiply-add and left most SMs idle on the few thousand rows of a training
// problem.  The sums keep the order of a sequential evaluation: bias first, then
// k = 0, 1, ... by fused multiply-adds.
constexpr int kTile = 64, kMlpThreads = 256;
constexpr int FS = NF + 4, HS = NH + 4;  // row strides in shared memory (float4 loads without bank conflicts)
struct MlpShared {
  float w1[NH * FS], w2[NH * HS], w3[NO * NH], b1[NH], b2[NH], b3[4];
  float feat[kTile * FS], dout[kTile * 4];
  float h1[kTile * HS], h2[kTile * HS], dz2[kTile * HS];
  // columns with a nonzero entry, as each warp saw its part of the tile: bit k of
  // feat[w] for feature k, bit v % 32 of dz2[w] for unit v (w % 2 = v / 32), bit u / 4 of
  // dz1[w][u % 4] for unit u
  struct {
    unsigned feat[kMlpThreads / 32], dz2[kMlpThreads / 32], dz1[kMlpThreads / 32][4];
  } nz;
};

__device__ __forceinline__ void mlp_load_weights(MlpShared &m, const float *__restrict__ w) {
  for (int k = threadIdx.x; k < NH * NF; k += kMlpThreads) m.w1[(k / NF) * FS + k % NF] = w[W1O + k];
  for (int k = threadIdx.x; k < NH * NH; k += kMlpThreads) m.w2[(k / NH) * HS + k % NH] = w[W2O + k];
  for (int k = threadIdx.x; k < NO * NH; k += kMlpThreads) m.w3[k] = w[W3O + k];
  for (int k = threadIdx.x; k < NH; k += kMlpThreads) {
    m.b1[k] = w[B1O + k];
    m.b2[k] = w[B2O + k];
  }
  if (threadIdx.x < NO) m.b3[threadIdx.x] = w[B3O + threadIdx.x];
}

// h = tanh(W x + b) for the tile: x rows of stride XS, W rows of stride XS, K inputs
template <int K, int XS>
__device__ __forceinline__ void mlp_layer(const float *x, const float *w, const float *b, float *h) {
  const int tu = threadIdx.x % 16, r0 = 4 * (threadIdx.x / 16);
  float z[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) z[i][j] = b[tu + 16 * j];
#pragma unroll 4
  for (int k = 0; k < K; k += 4) {
    float4 xv[4], wv[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) xv[i] = *reinterpret_cast<const float4 *>(x + (r0 + i) * XS + k);
#pragma unroll
    for (int j = 0; j < 4; ++j) wv[j] = *reinterpret_cast<const float4 *>(w + (tu + 16 * j) * XS + k);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        z[i][j] = fmaf(wv[j].x, xv[i].x, z[i][j]);
        z[i][j] = fmaf(wv[j].y, xv[i].y, z[i][j]);
        z[i][j] = fmaf(wv[j].z, xv[i].z, z[i][j]);
        z[i][j] = fmaf(wv[j].w, xv[i].w, z[i][j]);
      }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) h[(r0 + i) * HS + tu + 16 * j] = tanhf(z[i][j]);
}

// the tile's features (zero beyond the last row) and hidden activations
__device__ __forceinline__ void mlp_hidden(MlpShared &m, int32_t n, int32_t base, const float *__restrict__ feat) {
  bool nz = false;
  for (int q = threadIdx.x; q < kTile * NF; q += kMlpThreads) {  // a thread stays in its column
    const int32_t r = base + q / NF;
    const float f = r < n ? feat[(size_t)r * NF + q % NF] : 0.0f;
    nz |= f != 0.0f;
    m.feat[(q / NF) * FS + q % NF] = f;
  }
  const unsigned b = __ballot_sync(0xffffffffu, nz);
  if (threadIdx.x % 32 == 0) m.nz.feat[threadIdx.x / 32] = (b | b >> 16) & 0xffffu;
  __syncthreads();
  mlp_layer<NF, FS>(m.feat, m.w1, m.b1, m.h1);
  __syncthreads();
  mlp_layer<NH, HS>(m.h1, m.w2, m.b2, m.h2);
  __syncthreads();
}

// coefficients c_q = omega (delta_q0 + o_q), o = MLP(feat), omega per row
__global__ void __launch_bounds__(kMlpThreads) k_mlp_coef(int32_t n, const float *__restrict__ wg,
                                                          const float *__restrict__ feat,
                                                          const double *__restrict__ omega,
                                                          double *__restrict__ coef) {
  extern __shared__ __align__(16) unsigned char mlp_sm[];
  MlpShared &m = *reinterpret_cast<MlpShared *>(mlp_sm);
  mlp_load_weights(m, wg);
  for (int32_t base = blockIdx.x * kTile; base < n; base += gridDim.x * kTile) {
    mlp_hidden(m, n, base, feat);
    const int r = threadIdx.x / 4, q = threadIdx.x % 4;
    if (q < NO && base + r < n) {
      float o = m.b3[q];
      for (int v = 0; v < NH; ++v) o = fmaf(m.w3[q * NH + v], m.h2[r * HS + v], o);
      coef[3 * (size_t)(base + r) + q] = omega[base + r] * ((q == 0 ? 1.0 : 0.0) + (double)o);
    }
    __syncthreads();
  }
}

// Sum of products in twice the working precision (Ogita, Rump and Oishi, "Accurate
// sum and dot product", SIAM J. Sci. Comput. 26, 2005): the product and the sum each
// with their rounding error, the errors summed alongside.  The sums over rows are
// FP64 results; GB300 issues an FP64 multiply-add on 2 lanes of an SM a clock and
// this in 10 FP32 operations on 128, so the 64 terms of a tile are summed as a pair
// and the tiles in FP64.  Against the exact sum of the same FP32 terms its error is
// below 1e-13 of the sum of their magnitudes; the terms themselves carry FP32
// roundings, so that the gradient's error against a 64-bit network (1.0e-7 to
// 2.5e-7 for 1,024 to 40,000 FEM rows) is the same to seven digits as with FP64 sums.
//
// The error terms are exact while nothing overflows (an infinity or NaN stays in the
// pair to its end) and no product's error is subnormal: what a tile's 64 products can
// lose there is at most 64 x 2^-150, below 2^-48 of a sum of at least 2^-96.  A sum
// that is not finite or smaller than that, a parameter's own, is taken again in FP64
// (wide_sum), except for the usual case of a zero sum with a column of zeros.
struct Pair {
  float hi = 0.0f, lo = 0.0f;
  __device__ __forceinline__ void add_err(float p, float e) {
    const float s = __fadd_rn(hi, p), t = __fsub_rn(s, hi);
    const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, t)), __fsub_rn(p, t));
    hi = s;
    lo = __fadd_rn(lo, __fadd_rn(e, err));
  }
  __device__ __forceinline__ void mac(float a, float b) {
    const float p = __fmul_rn(a, b);
    add_err(p, __fmaf_rn(a, b, -p));
  }
  __device__ __forceinline__ void add(float a) { add_err(a, 0.0f); }
  __device__ __forceinline__ bool zero() const { return hi == 0.0f && lo == 0.0f; }
  __device__ __forceinline__ bool finite() const { return isfinite(hi) && isfinite(lo); }  // enough for add
  __device__ __forceinline__ bool sound() const { return fabsf(hi) >= 0x1p-96f && finite(); }
  __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};

// sum over the tile's rows of x y (y null: of x) in FP64; row strides sx, sy
__device__ __forceinline__ double wide_sum(const float *x, int sx, const float *y, int sy) {
  double s = 0.0;
#pragma unroll 1
  for (int r = 0; r < kTile; ++r) s = fma((double)x[r * sx], y ? (double)y[r * sy] : 1.0, s);
  return s;
}
__device__ __forceinline__ bool nz_feat(const MlpShared &m, int k) {
  unsigned b = 0;
#pragma unroll
  for (int w = 0; w < kMlpThreads / 32; ++w) b |= m.nz.feat[w];
  return b >> k & 1u;
}
__device__ __forceinline__ bool nz_dz2(const MlpShared &m, int v) {
  unsigned b = 0;
#pragma unroll
  for (int w = 0; w < kMlpThreads / 32; w += 2) b |= m.nz.dz2[w + v / 32];
  return b >> (v % 32) & 1u;
}
__device__ __forceinline__ bool nz_dz1(const MlpShared &m, int u) {
  unsigned b = 0;
#pragma unroll
  for (int w = 0; w < kMlpThreads / 32; ++w) b |= m.nz.dz1[w][u % 4];
  return b >> (u / 4) & 1u;
}

// the tile's weight gradients, added to the thread's sums: W2 (4 x 4 a thread), W1
// (4 a thread), then b1, b2, W3, b3 (one or two a thread)
constexpr int kMisc = 2 * NH + NO * NH + NO;  // 323
__device__ __forceinline__ void mlp_w2_sums(const MlpShared &m, double (&g2)[16]) {
  const int v0 = 4 * (threadIdx.x / 16), u0 = 4 * (threadIdx.x % 16);
  unsigned again = 0;  // sums to be taken in FP64
  Pair a[16];
  for (int r = 0; r < kTile; ++r) {
    const float4 d = *reinterpret_cast<const float4 *>(m.dz2 + r * HS + v0);
    const float4 h = *reinterpret_cast<const float4 *>(m.h1 + r * HS + u0);
    const float dv[4] = {d.x, d.y, d.z, d.w}, hv[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) a[4 * i + j].mac(dv[i], hv[j]);
  }
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    if (a[q].sound()) g2[q] += a[q].value();
    else if (!a[q].zero() || nz_dz2(m, v0 + q / 4)) again |= 1u << q;
  }
#pragma unroll 1
  for (; again; again &= again - 1) {
    const int k = __ffs(again) - 1;
    const double t = wide_sum(m.dz2 + v0 + k / 4, HS, m.h1 + u0 + k % 4, HS);
#pragma unroll
    for (int q = 0; q < 16; ++q)
      if (q == k) g2[q] += t;
  }
}
// dz1 is in m.h2's place by then; W3 and b3 come from m.h2 before (pass 0)
__device__ __forceinline__ void mlp_w1_sums(const MlpShared &m, double (&g1)[4]) {
  const int u = threadIdx.x / 4, k0 = 4 * (threadIdx.x % 4);
  unsigned again = 0;
  Pair a[4];
  for (int r = 0; r < kTile; ++r) {
    const float d = m.h2[r * HS + u];
    const float4 f = *reinterpret_cast<const float4 *>(m.feat + r * FS + k0);
    a[0].mac(d, f.x);
    a[1].mac(d, f.y);
    a[2].mac(d, f.z);
    a[3].mac(d, f.w);
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (a[q].sound()) g1[q] += a[q].value();
    else if (!a[q].zero() || (nz_feat(m, k0 + q) && nz_dz1(m, u))) again |= 1u << q;
  }
#pragma unroll 1
  for (; again; again &= again - 1) {
    const int k = __ffs(again) - 1;
    const double t = wide_sum(m.h2 + u, HS, m.feat + k0 + k, FS);
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (q == k) g1[q] += t;
  }
}
__device__ __forceinline__ void mlp_misc_sums(const MlpShared &m, int pass, double (&g)[2]) {
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int o = threadIdx.x + q * kMlpThreads;
    if (o >= kMisc || (o < NH) != (pass == 1)) continue;  // b1 needs dz1: the second pass
    const int w3 = o - 2 * NH;  // index into W3, then b3
    const float *x = o < NH ? m.h2 + o : (o < 2 * NH ? m.dz2 + o - NH : m.dout + (w3 < NO * NH ? w3 / NH : w3 - NO * NH));
    const float *y = o >= 2 * NH && w3 < NO * NH ? m.h2 + w3 % NH : nullptr;
    const int sx = o < 2 * NH ? HS : 4;
    Pair a;
    for (int r = 0; r < kTile; ++r) {
      if (y) a.mac(x[r * sx], y[r * HS]);
      else a.add(x[r * sx]);
    }
    g[q] += (y ? a.sound() : a.finite()) ? a.value() : wide_sum(x, sx, y, HS);
  }
}
__device__ __forceinline__ int misc_param(int o) {
  return o < NH ? B1O + o : (o < 2 * NH ? B2O + o - NH : (o < 2 * NH + NO * NH ? W3O + o - 2 * NH : B3O + o - 2 * NH - NO * NH));
}

// partial[block][parameter] = sum over the block's tiles of d<dout, MLP_w(feat)>/dw:
// dz2 = (W3^T dout) (1 - h2^2), dz1 = (W2^T dz2) (1 - h1^2), and the sums over rows
// of dz1 x feat, dz2 x h1, dout x h2 and of dz1, dz2, dout
__global__ void __launch_bounds__(kMlpThreads, 2) k_mlp_grad(int32_t n, const float *__restrict__ wg,
                                                          const float *__restrict__ feat,
                                                          const float *__restrict__ dout,
                                                          double *__restrict__ partial) {
  extern __shared__ __align__(16) unsigned char mlp_sm[];
  MlpShared &m = *reinterpret_cast<MlpShared *>(mlp_sm);
  mlp_load_weights(m, wg);
  double g2[16] = {0.0}, g1[4] = {0.0}, gm[2] = {0.0};
  for (int32_t base = blockIdx.x * kTile; base < n; base += gridDim.x * kTile) {
    {
      const int r = threadIdx.x / 4, q = threadIdx.x % 4;
      m.dout[threadIdx.x] = q < NO && base + r < n ? dout[(size_t)(base + r) * NO + q] : 0.0f;
    }
    mlp_hidden(m, n, base, feat);
    const int lane = threadIdx.x % 32, wid = threadIdx.x / 32;
    bool nz = false;
    for (int q = threadIdx.x; q < kTile * NH; q += kMlpThreads) {  // a thread stays in its column
      const int r = q / NH, v = q % NH;
      const float h2 = m.h2[r * HS + v];
      const float dh = m.w3[v] * m.dout[4 * r] + m.w3[NH + v] * m.dout[4 * r + 1] + m.w3[2 * NH + v] * m.dout[4 * r + 2];
      const float d = dh * (1.0f - h2 * h2);
      nz |= d != 0.0f;
      m.dz2[r * HS + v] = d;
    }
    const unsigned b2 = __ballot_sync(0xffffffffu, nz);
    if (lane == 0) m.nz.dz2[wid] = b2;
    __syncthreads();
    float dz1[4][4];
    const int u0 = 4 * (threadIdx.x % 16), r0 = 4 * (threadIdx.x / 16);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) dz1[i][j] = 0.0f;
#pragma unroll 4
    for (int v = 0; v < NH; ++v) {
      const float4 w = *reinterpret_cast<const float4 *>(m.w2 + v * HS + u0);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float d = m.dz2[(r0 + i) * HS + v];
        dz1[i][0] = fmaf(w.x, d, dz1[i][0]);
        dz1[i][1] = fmaf(w.y, d, dz1[i][1]);
        dz1[i][2] = fmaf(w.z, d, dz1[i][2]);
        dz1[i][3] = fmaf(w.w, d, dz1[i][3]);
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float h1 = m.h1[(r0 + i) * HS + u0 + j];
        dz1[i][j] *= 1.0f - h1 * h1;
      }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const unsigned b1 = __ballot_sync(0xffffffffu, dz1[0][j] != 0.0f || dz1[1][j] != 0.0f || dz1[2][j] != 0.0f ||
                                                         dz1[3][j] != 0.0f);
      if (lane == 0) m.nz.dz1[wid][j] = (b1 | b1 >> 16) & 0xffffu;
    }
    mlp_w2_sums(m, g2);
    mlp_misc_sums(m, 0, gm);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) m.h2[(r0 + i) * HS + u0 + j] = dz1[i][j];
    __syncthreads();
    mlp_w1_sums(m, g1);
    mlp_misc_sums(m, 1, gm);
    __syncthreads();
  }
  double *out = partial + (size_t)blockIdx.x * NP;
  const int v0 = 4 * (threadIdx.x / 16), u0 = 4 * (threadIdx.x % 16);
#pragma unroll
  for (int q = 0; q < 16; ++q) out[W2O + (v0 + q / 4) * NH + u0 + q % 4] = g2[q];
#pragma unroll
  for (int q = 0; q < 4; ++q) out[W1O + (threadIdx.x / 4) * NF + 4 * (threadIdx.x % 4) + q] = g1[q];
#pragma unroll
  for (int q = 0; q < 2; ++q)
    if (threadIdx.x + q * kMlpThreads < kMisc) out[misc_param(threadIdx.x + q * kMlpThreads)] = gm[q];
}

// sum of a parameter's partials over the blocks: 8 threads a parameter take
// interleaved blocks, then a fixed tree
__device__ __forceinline__ double sum_blocks(const double *__restrict__ partial, int nb, double (*sh)[33]) {
  const int k = blockIdx.x * 32 + threadIdx.x % 32, g = threadIdx.x / 32;
  double a = 0.0;
  if (k < NP)
    for (int c = g; c < nb; c += 8) a += partial[(size_t)c * NP + k];
  sh[g][threadIdx.x % 32] = a;
  __syncthreads();
  double t = 0.0;
  if (g == 0)
    for (int q = 0; q < 8; ++q) t += sh[q][threadIdx.x];
  return t;  // in the first 32 threads
}

__global__ void __launch_bounds__(256) k_grad_sum(const double *__restrict__ partial, int nb,
                                                  double *__restrict__ dst) {
  __shared__ double sh[8][33];
  const double g = sum_blocks(partial, nb, sh);
  const int k = blockIdx.x * 32 + threadIdx.x;
  if (threadIdx.x < 32 && k < NP) dst[k] = g;
}

// Adam step on the FP32 master weights (bias-corrected), gradient in FP64
__global__ void __launch_bounds__(256) k_grad_adam(const double *__restrict__ partial, int nb, float *__restrict__ w,
                                                   float *__restrict__ m, float *__restrict__ v, float lr, float b1,
                                                   float b2, float eps, int t) {
  __shared__ double sh[8][33];
  const double g = sum_blocks(partial, nb, sh);
  const int k = blockIdx.x * 32 + threadIdx.x;
  if (threadIdx.x >= 32 || k >= NP) return;
  const float c1 = 1.0f - powf(b1, (float)t), c2 = 1.0f - powf(b2, (float)t);
  const float gk = (float)g;
  m[k] = b1 * m[k] + (1.0f - b1) * gk;
  v[k] = b2 * v[k] + (1.0f - b2) * gk * gk;
  w[k] -= lr * (m[k] / c1) / (sqrtf(v[k] / c2) + eps);
}

// ------------------------------------------------------------------ MLP forward on tensor cores
// Inference with the FP16 weights as given: each warp takes 16 rows and runs the
// three layers as mma.sync m16n8k16 products (FP16 operands, FP32
// accumulation), the weights as B operands from shared memory.  An activation
// (FP32) enters as the sum of two FP16 parts, hi = fp16(h) and lo = fp16(h - hi),
// each multiplied by the exact FP16 weight and accumulated in FP32: about 22
// significant bits per product, so the outputs agree with the FP32 CUDA-core
// evaluation to FP32 rounding, where FP16 activations alone would lose three
// decimal digits.  The accumulator fragment of one layer (rows g, g+8; columns
// 2t, 2t+1 of each 8-column tile) is the A-operand fragment of the next, so the
// hidden activations never leave registers.  The weights lie in shared memory as the
// lanes' fragments, one 16-byte word for two k-tiles: read from their rows (128 bytes
// apart) the eight rows of a fragment met in the same banks.  2^20 rows: 166 -> 129 us;
// bound by issue (68 % of the slots, the tensor pipe active 32 % of the cycles).
__device__ __forceinline__ uint32_t pack_h2(__half x, __half y) {
  __half2 v = __halves2half2(x, y);
  return *reinterpret_cast<uint32_t *>(&v);
}
__device__ __forceinline__ void split_h2(float x, float y, uint32_t &hi, uint32_t &lo) {
  const __half2 h = __floats2half2_rn(x, y);
  const float2 f = __half22float2(h);
  const __half2 l = __floats2half2_rn(x - f.x, y - f.y);
  hi = *reinterpret_cast<const uint32_t *>(&h);
  lo = *reinterpret_cast<const uint32_t *>(&l);
}
// c += A (16x16, row) * B (16x8, col)
__device__ __forceinline__ void mma_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

constexpr int kTcWarps = 4;
__global__ void __launch_bounds__(32 * kTcWarps) k_mlp_forward_tc(int32_t n, const __half *__restrict__ wg,
                                                                  const float *__restrict__ feat,
                                                                  float *__restrict__ out) {
  // the B fragments of every lane, two k-tiles (layer 1: two n-tiles) per 16-byte word:
  // {b0, b1} of the first, {b0, b1} of the second
  __shared__ uint4 f1[NH / 16][32], f2[NH / 8][NH / 32][32], f3[NH / 32][32];
  __shared__ float2 bias[NH + 2];
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  {
    const int wid = threadIdx.x >> 5;
    auto wpair = [&](int idx) { return pack_h2(wg[idx], wg[idx + 1]); };
    for (int q = wid; q < NH / 16; q += kTcWarps) {
      const int at = W1O + (16 * q + g) * NF + 2 * t, at2 = at + 8 * NF;
      f1[q][lane] = make_uint4(wpair(at), wpair(at + 8), wpair(at2), wpair(at2 + 8));
    }
    for (int q = wid; q < NH / 8 * (NH / 32); q += kTcWarps) {
      const int at = W2O + (8 * (q >> 1) + g) * NH + 32 * (q & 1) + 2 * t;
      f2[q >> 1][q & 1][lane] = make_uint4(wpair(at), wpair(at + 8), wpair(at + 16), wpair(at + 24));
    }
    for (int q = wid; q < NH / 32; q += kTcWarps) {  // three outputs in an 8-column tile
      const int at = W3O + g * NH + 32 * q + 2 * t;
      f3[q][lane] = g < NO ? make_uint4(wpair(at), wpair(at + 8), wpair(at + 16), wpair(at + 24)) : make_uint4(0, 0, 0, 0);
    }
    for (int k = threadIdx.x; k < NH / 2; k += blockDim.x) {
      bias[k] = make_float2(__half2float(wg[B1O + 2 * k]), __half2float(wg[B1O + 2 * k + 1]));
      bias[NH / 2 + k] = make_float2(__half2float(wg[B2O + 2 * k]), __half2float(wg[B2O + 2 * k + 1]));
    }
    if (threadIdx.x == 0) {
      bias[NH] = make_float2(__half2float(wg[B3O]), __half2float(wg[B3O + 1]));
      bias[NH + 1] = make_float2(__half2float(wg[B3O + 2]), 0.0f);
    }
  }
  __syncthreads();
  for (int32_t tile = blockIdx.x * kTcWarps + (threadIdx.x >> 5); (int64_t)tile * 16 < n;
       tile += gridDim.x * kTcWarps) {
    const int32_t ra = tile * 16 + g, rb = ra + 8;
    // layer 1: A = features (16 x 16)
    uint32_t ah[4], al[4];
    {
      auto fv = [&](int32_t r, int k) { return r < n ? feat[(size_t)r * NF + k] : 0.0f; };
      split_h2(fv(ra, 2 * t), fv(ra, 2 * t + 1), ah[0], al[0]);
      split_h2(fv(rb, 2 * t), fv(rb, 2 * t + 1), ah[1], al[1]);
      split_h2(fv(ra, 2 * t + 8), fv(ra, 2 * t + 9), ah[2], al[2]);
      split_h2(fv(rb, 2 * t + 8), fv(rb, 2 * t + 9), ah[3], al[3]);
    }
    float c[8][4];
#pragma unroll
    for (int nt = 0; nt < 8; nt += 2) {
      const uint4 w = f1[nt / 2][lane];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const float2 bv = bias[4 * (nt + q) + t];
        c[nt + q][0] = c[nt + q][2] = bv.x;
        c[nt + q][1] = c[nt + q][3] = bv.y;
        mma_16816(c[nt + q], ah, q ? w.z : w.x, q ? w.w : w.y);
        mma_16816(c[nt + q], al, q ? w.z : w.x, q ? w.w : w.y);
      }
    }
    // tanh, then the accumulators as the A operand of the next layer (4 k-tiles)
    uint32_t hh[4][4], hl[4][4];
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      split_h2(tanhf(c[2 * kk][0]), tanhf(c[2 * kk][1]), hh[kk][0], hl[kk][0]);
      split_h2(tanhf(c[2 * kk][2]), tanhf(c[2 * kk][3]), hh[kk][1], hl[kk][1]);
      split_h2(tanhf(c[2 * kk + 1][0]), tanhf(c[2 * kk + 1][1]), hh[kk][2], hl[kk][2]);
      split_h2(tanhf(c[2 * kk + 1][2]), tanhf(c[2 * kk + 1][3]), hh[kk][3], hl[kk][3]);
    }
    // layer 2: 64 x 64
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      const float2 bv = bias[NH / 2 + 4 * nt + t];
      c[nt][0] = c[nt][2] = bv.x;
      c[nt][1] = c[nt][3] = bv.y;
#pragma unroll
      for (int kk = 0; kk < 4; kk += 2) {
        const uint4 w = f2[nt][kk / 2][lane];
        mma_16816(c[nt], hh[kk], w.x, w.y);
        mma_16816(c[nt], hl[kk], w.x, w.y);
        mma_16816(c[nt], hh[kk + 1], w.z, w.w);
        mma_16816(c[nt], hl[kk + 1], w.z, w.w);
      }
    }
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      split_h2(tanhf(c[2 * kk][0]), tanhf(c[2 * kk][1]), hh[kk][0], hl[kk][0]);
      split_h2(tanhf(c[2 * kk][2]), tanhf(c[2 * kk][3]), hh[kk][1], hl[kk][1]);
      split_h2(tanhf(c[2 * kk + 1][0]), tanhf(c[2 * kk + 1][1]), hh[kk][2], hl[kk][2]);
      split_h2(tanhf(c[2 * kk + 1][2]), tanhf(c[2 * kk + 1][3]), hh[kk][3], hl[kk][3]);
    }
    // layer 3: 3 outputs in the first 8-column tile (columns 3..7 zero)
    float o[4];
    const float2 bv = t < 2 ? bias[NH + t] : make_float2(0.0f, 0.0f);
    o[0] = o[2] = bv.x;
    o[1] = o[3] = bv.y;
#pragma unroll
    for (int kk = 0; kk < 4; kk += 2) {
      const uint4 w = f3[kk / 2][lane];
      mma_16816(o, hh[kk], w.x, w.y);
      mma_16816(o, hl[kk], w.x, w.y);
      mma_16816(o, hh[kk + 1], w.z, w.w);
      mma_16816(o, hl[kk + 1], w.z, w.w);
    }
    if (ra < n) {
      if (2 * t < NO) out[(size_t)ra * NO + 2 * t] = o[0];
      if (2 * t + 1 < NO) out[(size_t)ra * NO + 2 * t + 1] = o[1];
    }
    if (rb < n) {
      if (2 * t < NO) out[(size_t)rb * NO + 2 * t] = o[2];
      if (2 * t + 1 < NO) out[(size_t)rb * NO + 2 * t + 1] = o[3];
    }
  }
}

// c_q = omega (delta_q0 + o_q)
__global__ void k_coef_from_out(int32_t n, const float *__restrict__ out, double omega, double *__restrict__ coef) {
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < 3 * n; i += gridDim.x * blockDim.x)
    coef[i] = omega * ((i % 3 == 0 ? 1.0 : 0.0) + (double)out[i]);
}

// ------------------------------------------------------------------ two-grid loss
__device__ __forceinline__ uint64_t smix(uint64_t x) {
  uint64_t z = x + 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// The problems of one evaluation run in the same launches: blockIdx.y is the
// problem, blockIdx.z the error vector (up to kTgVecs at a time), the rows of all
// problems lie one after the other in the work arrays.  A training step over four
// problems and two vectors is 13 launches; one problem, vector and operation at a
// time was ~220 launches of 1-3 us on a few thousand rows each.
constexpr int kTgVecs = 4;
struct TgProblem {
  int32_t n, nc;
  int64_t off, offc;  // first row in the fine / coarse work arrays
  const int32_t *rp, *ci, *aptr, *amem, *agg;
  const double *val, *pw, *Ainv;
  double omega;
};
struct TgWork {  // [vector][all rows]
  double *e, *u0, *u1, *u2, *Ae, *rc, *xc, *dinv;
  double *part;  // [problem][vector][2][kTgParts]
  double *nrm0;  // [problem][vector]
  int64_t N, Nc;
};
constexpr int kTgParts = 1216;

__global__ void k_tg_inv_diag(const TgProblem *__restrict__ pr, TgWork w) {
  const TgProblem p = pr[blockIdx.y];
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < p.n; i += gridDim.x * blockDim.x) {
    double d = 0.0;
    for (int32_t q = p.rp[i]; q < p.rp[i + 1]; ++q)
      if (p.ci[q] == i) d = p.val[q];
    w.dinv[p.off + i] = 1.0 / d;
  }
}

// random error v: uniform in [-1, 1) from the splitmix64 counter (seed, v, i)
__global__ void k_tg_error(const TgProblem *__restrict__ pr, TgWork w, uint64_t seed, int v0) {
  const TgProblem p = pr[blockIdx.y];
  const uint64_t key = (seed + blockIdx.y) ^ ((uint64_t)(uint32_t)(v0 + blockIdx.z + 1) << 44);
  double *e = w.e + blockIdx.z * w.N + p.off;
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < p.n; i += gridDim.x * blockDim.x) {
    const uint64_t z = smix(key ^ (uint64_t)(uint32_t)i);
    e[i] = 2.0 * ((double)(z >> 11) * (1.0 / 9007199254740992.0)) - 1.0;
  }
}

__device__ __forceinline__ double tg_row(const TgProblem &p, int32_t i, const double *__restrict__ x) {
  double acc = 0.0;
  for (int32_t q = p.rp[i]; q < p.rp[i + 1]; ++q) acc += p.val[q] * x[p.ci[q]];
  return acc;
}

// block partial of one inner product
__device__ __forceinline__ void tg_part(double acc, double *part) {
  __shared__ double sh[8];
  acc = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int q = 0; q < 8; ++q) t += sh[q];
    *part = t;
  }
}
__device__ __forceinline__ double *tg_part_at(const TgWork &w, int which) {
  return w.part + (((int64_t)blockIdx.y * kTgVecs + blockIdx.z) * 2 + which) * kTgParts + blockIdx.x;
}

// Ae = A e.  FIRST: also u0 = D^-1 A e; the partial of e . Ae (nrm0; last: the numerator)
template <bool FIRST>
__global__ void __launch_bounds__(256) k_tg_energy(const TgProblem *__restrict__ pr, TgWork w) {
  const TgProblem p = pr[blockIdx.y];
  const int64_t o = blockIdx.z * w.N + p.off;
  double acc = 0.0;
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < p.n; i += gridDim.x * blockDim.x) {
    const double y = tg_row(p, i, w.e + o);
    if (FIRST) w.u0[o + i] = w.dinv[p.off + i] * y;
    else w.Ae[o + i] = y;
    acc += w.e[o + i] * y;
  }
  tg_part(acc, tg_part_at(w, FIRST ? 0 : 1));
}

// u1 = D^-1 A u0
__global__ void k_tg_u1(const TgProblem *__restrict__ pr, TgWork w) {
  const TgProblem p = pr[blockIdx.y];
  const int64_t o = blockIdx.z * w.N + p.off;
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < p.n; i += gridDim.x * blockDim.x)
    w.u1[o + i] = w.dinv[p.off + i] * tg_row(p, i, w.u0 + o);
}

// u2 = D^-1 A u1, e1 = e0 - sum_q c_q u_q (in place of e0)
__global__ void k_tg_smooth(const TgProblem *__restrict__ pr, TgWork w, const double *__restrict__ coef) {
  const TgProblem p = pr[blockIdx.y];
  const int64_t o = blockIdx.z * w.N + p.off;
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < p.n; i += gridDim.x * blockDim.x) {
    const double u2 = w.dinv[p.off + i] * tg_row(p, i, w.u1 + o);
    const double *c = coef + 3 * (p.off + i);
    w.u2[o + i] = u2;
    w.e[o + i] -= c[0] * w.u0[o + i] + c[1] * w.u1[o + i] + c[2] * u2;
  }
}

// Ae = A e1
__global__ void k_tg_product(const TgProblem *__restrict__ pr, TgWork w) {
  const TgProblem p = pr[blockIdx.y];
  const int64_t o = blockIdx.z * w.N + p.off;
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < p.n; i += gridDim.x * blockDim.x)
    w.Ae[o + i] = tg_row(p, i, w.e + o);
}

// coarse correction of the error: rc = P^T (A e1), xc = A_c^-1 rc, e2 = e1 - P xc
__global__ void k_tg_restrict(const TgProblem *__restrict__ pr, TgWork w) {
  const TgProblem p = pr[blockIdx.y];
  const double *r = w.Ae + blockIdx.z * w.N + p.off;
  for (int32_t I = blockIdx.x * blockDim.x + threadIdx.x; I < p.nc; I += gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int32_t m = p.aptr[I]; m < p.aptr[I + 1]; ++m) s += p.pw[p.amem[m]] * r[p.amem[m]];
    w.rc[blockIdx.z * w.Nc + p.offc + I] = s;
  }
}
// a warp per row, all vectors with the same entries of A_c^-1
__global__ void __launch_bounds__(256) k_tg_dense(const TgProblem *__restrict__ pr, TgWork w, int nv) {
  const TgProblem p = pr[blockIdx.y];
  const int lane = threadIdx.x & 31;
  for (int32_t i = blockIdx.x * 8 + (threadIdx.x >> 5); i < p.nc; i += gridDim.x * 8) {
    double s[kTgVecs] = {0.0};
    for (int32_t j = lane; j < p.nc; j += 32) {
      const double a = p.Ainv[(int64_t)i * p.nc + j];
#pragma unroll
      for (int v = 0; v < kTgVecs; ++v)
        if (v < nv) s[v] += a * w.rc[v * w.Nc + p.offc + j];
    }
#pragma unroll
    for (int v = 0; v < kTgVecs; ++v)
      if (v < nv) {
        const double t = warp_sum(s[v]);
        if (lane == 0) w.xc[v * w.Nc + p.offc + i] = t;
      }
  }
}
__global__ void k_tg_prolong(const TgProblem *__restrict__ pr, TgWork w) {
  const TgProblem p = pr[blockIdx.y];
  double *e = w.e + blockIdx.z * w.N + p.off;
  const double *xc = w.xc + blockIdx.z * w.Nc + p.offc;
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < p.n; i += gridDim.x * blockDim.x)
    e[i] -= p.pw[i] * xc[p.agg[i]];
}

// nrm0 = e0^T A e0 of every problem and vector, and *loss += scale sum (e2^T A e2) / nrm0 / nvec;
// one block, a warp per sum, then one thread in problem and vector order
__global__ void __launch_bounds__(1024) k_tg_fin(TgWork w, int np, int nv, int parts, int nvec, double scale,
                                                 double *loss) {
  __shared__ double num[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  double total = 0.0;
  for (int q0 = 0; q0 < np * nv; q0 += 16) {  // 16 (problem, vector) pairs a round, two sums each
    const int q = q0 + wid / 2, which = wid % 2;
    if (q < np * nv) {
      const double *part = w.part + ((int64_t)(q / nv * kTgVecs + q % nv) * 2 + which) * kTgParts;
      double s = 0.0;
      for (int j = lane; j < parts; j += 32) s += part[j];
      s = warp_sum(s);
      if (lane == 0) {
        num[wid] = s;
        if (which == 0) w.nrm0[q / nv * kTgVecs + q % nv] = s;
      }
    }
    __syncthreads();
    if (threadIdx.x == 0)
      for (int t = 0; t < 16 && q0 + t < np * nv; ++t) total += num[2 * t + 1] / num[2 * t] / nvec;
    __syncthreads();
  }
  if (threadIdx.x == 0) *loss += scale * total;
}

// dL/dc_q of row i: -sum_v (2 / (nrm0_v nvec)) (A e2_v)_i u_q,v,i; added to dcoef, or as
// dL/do_q = scale omega dL/dc_q into dout (once, with all vectors)
__global__ void k_tg_grad(const TgProblem *__restrict__ pr, TgWork w, int nv, int nvec, bool fresh,
                          double *__restrict__ dcoef, double scale, float *__restrict__ dout) {
  const TgProblem p = pr[blockIdx.y];
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < p.n; i += gridDim.x * blockDim.x) {
    const int64_t r = p.off + i;
    double d[3];
    for (int q = 0; q < 3; ++q) d[q] = fresh ? 0.0 : dcoef[3 * r + q];
    for (int v = 0; v < nv; ++v) {
      const double g = 2.0 / w.nrm0[blockIdx.y * kTgVecs + v] / nvec * w.Ae[v * w.N + r];
      d[0] -= g * w.u0[v * w.N + r];
      d[1] -= g * w.u1[v * w.N + r];
      d[2] -= g * w.u2[v * w.N + r];
    }
    for (int q = 0; q < 3; ++q) {
      if (dcoef) dcoef[3 * r + q] = d[q];
      if (dout) dout[3 * r + q] = (float)(scale * p.omega * d[q]);
    }
  }
}

__global__ void k_tg_omega_rows(const TgProblem *__restrict__ pr, double *__restrict__ omega) {
  const TgProblem p = pr[blockIdx.y];
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < p.n; i += gridDim.x * blockDim.x)
    omega[p.off + i] = p.omega;
}

// ------------------------------------------------------------------ host side
namespace {

inline int g256(int64_t n) { return grid_for(n, 256, 152 * 16); }

// the problems of an evaluation and its work arrays
struct TgSet {
  int np = 0, nv = 0, parts = 1;
  int64_t N = 0, Nc = 0;
  int32_t maxn = 0, maxnc = 0;
  DevBuf<TgProblem> prob;
  DevBuf<double> buf;
  TgWork w{};
  TgSet(Hierarchy *const *hs, int nh, int nvec, cudaStream_t s) : np(nh), nv(std::min(nvec, kTgVecs)) {
    std::vector<TgProblem> p(nh);
    for (int j = 0; j < nh; ++j) {
      const Hierarchy &h = *hs[j];
      if (h.L != 2) throw Error{AMG_ERR_BAD_INPUT, "two-grid loss needs a hierarchy with exactly two levels"};
      const Level &L = h.lev[0];
      p[j] = {L.n, h.lev[1].n, N, Nc, L.rp, L.ci, L.aptr, L.amem, L.agg, L.val, L.pw64, h.coarse_inv, L.omega};
      N += L.n;
      Nc += h.lev[1].n;
      maxn = std::max(maxn, L.n);
      maxnc = std::max(maxnc, h.lev[1].n);
    }
    parts = grid_for(maxn, 256, kTgParts);
    prob.resize(nh);
    AMG_CUDA(cudaMemcpyAsync(prob.p, p.data(), sizeof(TgProblem) * nh, cudaMemcpyHostToDevice, s));
    AMG_CUDA(cudaStreamSynchronize(s));  // p leaves scope
    buf.resize((size_t)N * (5 * nv + 1) + 2 * (size_t)Nc * nv + (size_t)nh * kTgVecs * (2 * kTgParts + 1));
    double *q = buf.p;
    auto take = [&](int64_t cnt) {
      double *r = q;
      q += cnt;
      return r;
    };
    w.N = N;
    w.Nc = Nc;
    w.e = take(N * nv);
    w.u0 = take(N * nv);
    w.u1 = take(N * nv);
    w.u2 = take(N * nv);
    w.Ae = take(N * nv);
    w.dinv = take(N);
    w.rc = take(Nc * nv);
    w.xc = take(Nc * nv);
    w.part = take((int64_t)nh * kTgVecs * 2 * kTgParts);
    w.nrm0 = take((int64_t)nh * kTgVecs);
    AMG_COUNT(), k_tg_inv_diag<<<rows(1), 256, 0, s>>>(prob.p, w);  // 1/A_ii in FP64
    AMG_LAUNCH_CHECK();
  }
  dim3 rows(int v) const { return dim3((unsigned)parts, (unsigned)np, (unsigned)v); }
};

// *loss += scale x the sum over the problems of the mean two-grid factor over nvec
// errors; its gradient into dcoef (N x 3) or dout (scaled by scale x omega).  With
// more than kTgVecs vectors the gradient is gathered in dcoef.
void tg_evaluate(TgSet &t, const double *coef, int nvec, uint64_t seed, double scale, double *loss, double *dcoef,
                 float *dout, cudaStream_t s) {
  for (int v0 = 0; v0 < nvec; v0 += kTgVecs) {
    const int nv = std::min(kTgVecs, nvec - v0);
    const dim3 g = t.rows(nv);
    const dim3 gc((unsigned)grid_for(t.maxnc, 256, kTgParts), (unsigned)t.np, (unsigned)nv);
    const dim3 gd((unsigned)grid_for(t.maxnc, 8, 152 * 16), (unsigned)t.np, 1);
    AMG_COUNT(), k_tg_error<<<g, 256, 0, s>>>(t.prob.p, t.w, seed, v0);
    AMG_COUNT(), k_tg_energy<true><<<g, 256, 0, s>>>(t.prob.p, t.w);
    AMG_COUNT(), k_tg_u1<<<g, 256, 0, s>>>(t.prob.p, t.w);
    AMG_COUNT(), k_tg_smooth<<<g, 256, 0, s>>>(t.prob.p, t.w, coef);
    AMG_COUNT(), k_tg_product<<<g, 256, 0, s>>>(t.prob.p, t.w);
    AMG_COUNT(), k_tg_restrict<<<gc, 256, 0, s>>>(t.prob.p, t.w);
    AMG_COUNT(), k_tg_dense<<<gd, 256, 0, s>>>(t.prob.p, t.w, nv);
    AMG_COUNT(), k_tg_prolong<<<g, 256, 0, s>>>(t.prob.p, t.w);
    AMG_COUNT(), k_tg_energy<false><<<g, 256, 0, s>>>(t.prob.p, t.w);
    AMG_COUNT(), k_tg_fin<<<1, 1024, 0, s>>>(t.w, t.np, nv, t.parts, nvec, scale, loss);
    if (dcoef || dout)
      AMG_COUNT(), k_tg_grad<<<t.rows(1), 256, 0, s>>>(t.prob.p, t.w, nv, nvec, v0 == 0, dcoef, scale,
                                                       v0 + nv >= nvec ? dout : nullptr);
  }
  AMG_LAUNCH_CHECK();
}

void mlp_smem(const void *kernel) {
  AMG_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(MlpShared)));
}
// blocks of the gradient kernel: two an SM; each leaves NP partial sums
inline int grad_blocks(int32_t n) { return grid_for(n, kTile, 152 * 2); }

}  // namespace

// Two-grid loss and gradient on a two-level hierarchy (device coef / dcoef);
// loss_dev receives the mean factor.
void twogrid_loss(Hierarchy &h, const double *coef, int nvec, uint64_t seed, double *loss_dev, double *dcoef,
                  cudaStream_t s) {
  Hierarchy *hp = &h;
  TgSet t(&hp, 1, nvec, s);
  AMG_CUDA(cudaMemsetAsync(loss_dev, 0, sizeof(double), s));
  tg_evaluate(t, coef, nvec, seed, 1.0, loss_dev, dcoef, nullptr, s);
}

void features(const Hierarchy &h, int level, float *feat_dev, cudaStream_t s) {
  const Level &L = h.lev[level];
  AMG_COUNT(), k_features<<<grid_for(L.n, kFeatThreads, 1 << 30), kFeatThreads, 0, s>>>(L.n, L.rp, L.ci, L.val, level,
                                                                                   feat_dev);
  AMG_LAUNCH_CHECK();
}

void mlp_forward_half(int32_t n, const uint16_t *w16_dev, const float *feat, float *out, cudaStream_t s) {
  if (n <= 0) return;
  const int blocks = grid_for(((int64_t)n + 15) / 16, kTcWarps, 152 * 20);  // four waves of resident blocks
  AMG_COUNT(), k_mlp_forward_tc<<<blocks, 32 * kTcWarps, 0, s>>>(n, reinterpret_cast<const __half *>(w16_dev), feat,
                                                                 out);
  AMG_LAUNCH_CHECK();
}

// dparam = d<dout, MLP_w(feat)>/dw  (FP32 weights, device)
void mlp_backward(int32_t n, const float *w, const float *feat, const float *dout, double *dparam, cudaStream_t s) {
  const int nb = grad_blocks(n);
  DevBuf<double> partial((size_t)nb * NP);
  mlp_smem((const void *)k_mlp_grad);
  AMG_COUNT(), k_mlp_grad<<<nb, kMlpThreads, sizeof(MlpShared), s>>>(n, w, feat, dout, partial.p);
  AMG_COUNT(), k_grad_sum<<<(NP + 31) / 32, 256, 0, s>>>(partial.p, nb, dparam);
  AMG_LAUNCH_CHECK();
}

// ------------------------------------------------------------------ fixed scratch
// MLP backward for callers that cannot allocate device memory: the work array
// (the blocks' weight-gradient sums, 1.4 MB) lives in one statically sized device
// array that every GPU loading this library holds until the process exits.  Rows
// per call are limited to kFixedMaxRows; calls that overlap on the GPU share the
// array and race.
constexpr int32_t kFixedMaxRows = 2048;
constexpr size_t kFixedBytes = (size_t)(kFixedMaxRows / kTile) * NP * sizeof(double);
static __device__ __align__(256) unsigned char g_fixed_scratch[kFixedBytes];

// Address of the array on the current device.  A host may not use the symbol
// itself as a device address, so every call asks the runtime for it with the
// device current: the lookup allocates nothing, the first one on a device loads
// the module that holds the array, and nothing cached can go stale when a
// context is reset and the array moves.
static void *fixed_scratch_address() {
  void *p = nullptr;
  const cudaError_t e = cudaGetSymbolAddress(&p, g_fixed_scratch);
  if (e != cudaSuccess)
    throw Error{AMG_ERR_CUDA, std::string("cudaGetSymbolAddress(fixed scratch): ") + cudaGetErrorString(e)};
  return p;
}

size_t fixed_scratch_bytes() { return kFixedBytes; }
int32_t fixed_scratch_max_rows() { return kFixedMaxRows; }

void mlp_backward_fixed(int32_t n, const float *w, const float *feat, const float *dout, double *dparam,
                        cudaStream_t s) {
  if (n < 0 || n > kFixedMaxRows)
    throw Error{AMG_ERR_BAD_INPUT, "amg_mlp_backward_noalloc: n = " + std::to_string(n) + " rows exceeds the " +
                                       std::to_string(kFixedMaxRows) + "-row limit of its fixed scratch"};
  // every scratch word read below is written first in the same call
  double *partial = static_cast<double *>(fixed_scratch_address());
  const int nb = grad_blocks(n);
  mlp_smem((const void *)k_mlp_grad);
  k_mlp_grad<<<nb, kMlpThreads, sizeof(MlpShared), s>>>(n, w, feat, dout, partial);
  k_grad_sum<<<(NP + 31) / 32, 256, 0, s>>>(partial, nb, dparam);
  AMG_LAUNCH_CHECK();
}

// The network is trained on the two-grid factor of level 0 and installed there;
// coarser levels keep damped Jacobi.
void apply_learned(Hierarchy &h, const uint16_t *w16_dev, cudaStream_t s) {
  for (int k = 0; k < std::min(h.L - 1, 1); ++k) {
    Level &L = h.lev[k];
    DevBuf<float> feat((size_t)L.n * NF), out((size_t)L.n * NO);
    DevBuf<double> coef((size_t)L.n * 3);
    features(h, k, feat.p, s);
    mlp_forward_half(L.n, w16_dev, feat.p, out.p, s);
    AMG_COUNT(), k_coef_from_out<<<g256(3 * (int64_t)L.n), 256, 0, s>>>(L.n, out.p, L.omega, coef.p);
    AMG_LAUNCH_CHECK();
    set_poly(h, k, coef.p, s);
  }
  h.p.smoother = 1;
  h.graph_kind = -1;
}

// Adam training of the MLP on the level-0 two-grid factor of each hierarchy
void train_smoother(Hierarchy *const *hs, int nh, int steps, double lr, int nvec, uint64_t seed, float *w_host,
                    double *loss_hist, cudaStream_t s) {
  TgSet t(hs, nh, nvec, s);
  const int nb = grad_blocks((int32_t)std::min<int64_t>(t.N, INT32_MAX));
  if (3 * t.N > INT32_MAX) throw Error{AMG_ERR_BAD_INPUT, "too many training rows"};
  const int32_t N = (int32_t)t.N;
  DevBuf<float> w(NP), m(NP), v(NP), feat((size_t)N * NF), dout((size_t)N * NO);
  DevBuf<double> loss(steps + 1), omega(N), coef((size_t)N * 3), partial((size_t)nb * NP);
  DevBuf<double> dcoef(nvec > kTgVecs ? (size_t)N * 3 : 1);
  AMG_CUDA(cudaMemcpyAsync(w.p, w_host, sizeof(float) * NP, cudaMemcpyHostToDevice, s));
  AMG_CUDA(cudaMemsetAsync(m.p, 0, sizeof(float) * NP, s));
  AMG_CUDA(cudaMemsetAsync(v.p, 0, sizeof(float) * NP, s));
  AMG_CUDA(cudaMemsetAsync(loss.p, 0, sizeof(double) * (steps + 1), s));
  AMG_COUNT(), k_tg_omega_rows<<<t.rows(1), 256, 0, s>>>(t.prob.p, omega.p);
  int64_t off = 0;
  for (int j = 0; j < nh; ++j) {
    features(*hs[j], 0, feat.p + off * NF, s);
    off += hs[j]->lev[0].n;
  }
  mlp_smem((const void *)k_mlp_coef);
  mlp_smem((const void *)k_mlp_grad);
  for (int q = 1; q <= steps; ++q) {
    AMG_COUNT(), k_mlp_coef<<<nb, kMlpThreads, sizeof(MlpShared), s>>>(N, w.p, feat.p, omega.p, coef.p);
    tg_evaluate(t, coef.p, nvec, seed + (uint64_t)q * 1000003ull, 1.0 / nh, loss.p + q - 1,
                nvec > kTgVecs ? dcoef.p : nullptr, dout.p, s);
    AMG_COUNT(), k_mlp_grad<<<nb, kMlpThreads, sizeof(MlpShared), s>>>(N, w.p, feat.p, dout.p, partial.p);
    AMG_COUNT(), k_grad_adam<<<(NP + 31) / 32, 256, 0, s>>>(partial.p, nb, w.p, m.p, v.p, (float)lr, 0.9f, 0.999f,
                                                          1e-8f, q);
    AMG_LAUNCH_CHECK();
  }
  if (loss_hist && steps > 0)
    AMG_CUDA(cudaMemcpyAsync(loss_hist, loss.p, sizeof(double) * steps, cudaMemcpyDeviceToHost, s));
  AMG_CUDA(cudaMemcpyAsync(w_host, w.p, sizeof(float) * NP, cudaMemcpyDeviceToHost, s));
  AMG_CUDA(cudaStreamSynchronize(s));
}

}  // namespace amg
