// solve.cu -- solve phase of the aggregation AMG method on the GPU.
//
// Preconditioner: Alg. 5 (K-cycle) on levels k < kcycle_levels and Alg. 4
// (V-cycle) below (Sec. 2.2), one damped-Jacobi pre- and post-smoothing step
// per level visit (Eq. damped Jacobi), piecewise-constant restriction (a
// segmented sum over aggregates) and prolongation (a gather), and the exact
// coarsest solve as a dense matrix-vector product with the inverse formed at
// setup.  Outer iteration: flexible CG (Sec. 2.2) in FP64.
//
// Data-dependent control stays on the device.  The branch of Alg. 5
// (||r~|| <= t ||r||) is written to a per-level predicate by the kernel that forms
// r~; every kernel of the second inner step reads the predicate and returns
// at once when the step is not taken.  The Krylov scalars live in device
// memory, so an outer iteration is a fixed sequence of launches that can be
// captured once as a CUDA graph and replayed.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <type_traits>

#include "amg_internal.cuh"

namespace amg {

// ============================================================== kernels
constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;

template <class VT>
struct SellArgs {
  int32_t n, nslices;
  const int64_t *sptr;
  const int32_t *scol;
  const void *sval;
  const int4 *spair;   // FP32 values: entries as {column, value} pairs (scol / sval null)
  const float *sdiag;  // split diagonal (reduced precision), else null
  const unsigned char *live;  // batch: 0 for slices whose systems all stopped (skipped); else null
  const VT *x;    // SpMV input
  VT *out;        // output vector
  const VT *rhs;  // right-hand side (residual epilogues)
  const VT *xin;  // the iterate that the last Horner step updates
  // fused inner products with left operand s = x (dot_y: the output): ND = 2:
  // {s.out, s.u1}, ND = 3: {s.out, s.u1, s.u2}, ND = 5: {x.out, x.u1, out.out, out.u1,
  // u1.u1}, ND = 1: {out.q64}; the blocks' sums to partials
  const VT *u1, *u2;
  const double *q64;
  int dot_y;
  double *partials;
  const int *pred;
  // polynomial smoother operands
  const VT *dinv;     // 1 / A_ii
  const VT *coef;     // n x 3 per-row coefficients c_0, c_1, c_2
  const VT *p0, *p1;  // earlier polynomial terms
  const VT *res;      // residual the Horner steps add back
  VT *out2;           // second output
};

// epilogues of the SELL kernel (y = A x):
//   E_Y            out = y
//   E_RESID        out = rhs - y
//   E_DSCALE       out = D^-1 y                               polynomial pre-smoother, term 1
//   E_POLYPRE      out = c0 p0 + c1 p1 + c2 D^-1 y            polynomial pre-smoother, sum
//   E_RESID_POLY   out = rhs - y, out2 = D^-1 (c2 out)        post-smoother: residual, Horner start
//   E_HORNER       out = D^-1 y + D^-1 (c1 res)               Horner middle step
//   E_HORNER_LAST  out = xin + D^-1 y + D^-1 (c0 res)         Horner last step, update
enum Epi { E_Y = 0, E_RESID = 1, E_DSCALE = 3, E_POLYPRE = 4, E_RESID_POLY = 5, E_HORNER = 6,
           E_HORNER_LAST = 7 };

template <class MV> __device__ __forceinline__ MV ld_stream(const MV *p) { return __ldcs(p); }
// FP32 matrices are stored as {column, value} pairs (Level::spair); BF16
// matrices keep separate column and value arrays with a lane's entries 2j and
// 2j+1 adjacent in each (one 8-byte column load, one 4-byte value load)
template <class MV> constexpr bool kPairs = std::is_same<MV, float>::value;
template <class MV> constexpr bool kHalfPairs = std::is_same<MV, __nv_bfloat16>::value;

// ---- inner products
// A kernel with inner products stores its blocks' sums, and every block of the kernel
// that needs the totals adds them up itself, in the same fixed order (sum_partials_of):
// the sums over the grid are no launch, no ticket and no trip of a last block through
// fence, atomic, partials and scalars, which added ~3.5 us to each of 12 kernels of an
// iteration (1.5-2 us now, in the kernel that reads them: 128^3 step 16.9 -> 16.5 ms,
// FEM 1024^2 solve 28.3 -> 26.1, learned 501^2 8.0 -> 7.0, 700^2 re-setup + solve 35.4 ->
// 32.3).  What the host or a predicate of later launches needs (the end of an
// outer iteration) is still formed by the last block (grid_totals).
// GB300 issues an FP64 warp instruction every 16 cycles an SM, so the reductions
// count them: the block's values go through shared memory and one warp per product
// adds 8 values a lane and 5 shuffles (12 warp instructions a product, against 45
// with a shuffle tree in each of the 8 warps).

// the block's sums of ND inner products to partials[k kRedBlocks + block].  `step`:
// only the threads of every step-th warp hold a value.  Every thread calls it.
template <int ND>
__device__ __forceinline__ void store_dots(const double (&acc)[ND], int step, double *partials) {
  __shared__ double sh[ND][kThreads];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < ND; ++k) sh[k][threadIdx.x] = acc[k];
  __syncthreads();
  if (wid < ND) {
    double v = sh[wid][lane];
    for (int q = step; q < kWarps; q += step) v += sh[wid][q * 32 + lane];
    v = warp_sum(v);
    if (lane == 0) partials[wid * kRedBlocks + blockIdx.x] = v;
  }
}

// kernels that add up a product's partials run at most two blocks of kSumThreads an SM:
// fewer blocks read the same partials, and each row's loads overlap the sums once
constexpr int kSumThreads = 512;
constexpr int kSumWarps = kSumThreads / 32;
inline int sum_grid(int64_t n) { return grid_for(n, kSumThreads, 304); }

// tot[k] = sum of the nb partials of product k, the same bits in every block; valid in
// thread 0 (up to lane 7 of warp 0, all lanes for few partials).  Every thread of the block calls it.  An FP64 addition takes ~60
// cycles to its result: up to 128 partials warp 0 sums alone (four loads a lane, all
// products side by side), more are shared among the block's warps.
template <int ND>
__device__ __forceinline__ void sum_partials_of(const double *partials, int nb, double (&tot)[ND]) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  constexpr int kAhead = 4;
  auto four = [&](int k, int j0, int stride) {
    double v[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u)
      v[u] = j0 + u * stride < nb ? __ldcg(partials + k * kRedBlocks + j0 + u * stride) : 0.0;
    return (v[0] + v[1]) + (v[2] + v[3]);
  };
  if (nb <= 32 * kAhead) {
    if (wid == 0) {
#pragma unroll
      for (int k = 0; k < ND; ++k) tot[k] = four(k, lane, 32);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < ND; ++k) tot[k] += __shfl_xor_sync(0xffffffffu, tot[k], o);
    }
    return;
  }
  constexpr int kPer = ND == 1 ? 8 : (ND == 2 ? 8 : (ND == 3 ? 4 : 3));  // warps per product
  static_assert(kPer * ND <= kSumWarps, "");
  __shared__ double sh[ND][8];
  const int k = wid / kPer, sub = wid % kPer;
  if (k < ND) {
    double t = 0.0;
    for (int j0 = sub * 32 + lane; j0 < nb; j0 += kAhead * kPer * 32) t += four(k, j0, kPer * 32);
    t = warp_sum(t);
    if (lane == 0) sh[k][sub] = t;
  }
  __syncthreads();
  if (wid == 0) {
#pragma unroll
    for (int q = 0; q < ND; ++q) tot[q] = lane < kPer ? sh[q][lane] : 0.0;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1)
#pragma unroll
      for (int q = 0; q < ND; ++q) tot[q] += __shfl_xor_sync(0xffffffffu, tot[q], o);
  }
}

// rows [r0, r1) of this block: equal contiguous shares, so that every SM has the same
// number of load batches
__device__ __forceinline__ void block_rows(int32_t n, int32_t &r0, int32_t &r1) {
  const int32_t share = (n + gridDim.x - 1) / gridDim.x, up = (share + 31) & ~31;
  r0 = (int32_t)min((int64_t)n, (int64_t)blockIdx.x * up);
  r1 = (int32_t)min((int64_t)n, (int64_t)r0 + up);
}

// totals of ND inner products over the grid; true in thread 0 of the last block
// only, with the totals in tot.  `step`: only the threads of every step-th warp
// hold a value.  Every thread of the block calls it, all blocks of the grid.
template <int ND, int T = kThreads>  // T threads a block
__device__ __forceinline__ bool grid_totals(const double (&acc)[ND], int step, double *partials, unsigned *ticket,
                                            double (&tot)[ND]) {
  __shared__ double sh[ND][T];
  __shared__ double tot_sh[ND];
  __shared__ bool last;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < ND; ++k) sh[k][threadIdx.x] = acc[k];
  __syncthreads();
  if (wid < ND) {
    double v = sh[wid][lane];
    for (int q = step; q < T / 32; q += step) v += sh[wid][q * 32 + lane];
    v = warp_sum(v);
    if (lane == 0) {
      if (gridDim.x == 1) {
        tot_sh[wid] = v;
      } else {
        partials[wid * kRedBlocks + blockIdx.x] = v;
        __threadfence();
      }
    }
  }
  __syncthreads();
  if (gridDim.x > 1) {
    if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return false;
    __threadfence();
#pragma unroll
    for (int k = 0; k < ND; ++k) {
      double v[kRedBlocks / T + 1];
#pragma unroll
      for (int u = 0; u <= kRedBlocks / T; ++u) {
        const int j = threadIdx.x + u * T;
        v[u] = j < (int)gridDim.x ? __ldcg(partials + k * kRedBlocks + j) : 0.0;
      }
      double t = v[0];
#pragma unroll
      for (int u = 1; u <= kRedBlocks / T; ++u)
        if (u * T < (int)gridDim.x) t += v[u];
      sh[k][threadIdx.x] = t;
    }
    __syncthreads();
    if (wid < ND) {
      double v = sh[wid][lane];
      for (int q = 1; q < T / 32 && q * 32 < (int)gridDim.x; ++q) v += sh[wid][q * 32 + lane];
      v = warp_sum(v);
      if (lane == 0) tot_sh[wid] = v;
    }
    __syncthreads();
  }
  if (threadIdx.x != 0) return false;
  if (gridDim.x > 1) *ticket = 0;
#pragma unroll
  for (int k = 0; k < ND; ++k) tot[k] = tot_sh[k];
  return true;
}

// per-block partial sums of one inner product -> partials[block] (no finish)
__device__ __forceinline__ void block_store_dot(double a, double *partials) {
  __shared__ double sh[kThreads];
  const int lane = threadIdx.x & 31;
  sh[threadIdx.x] = a;
  __syncthreads();
  if (threadIdx.x < 32) {
    double v = sh[lane];
#pragma unroll
    for (int q = 1; q < kWarps; ++q) v += sh[q * 32 + lane];
    v = warp_sum(v);
    if (lane == 0) partials[blockIdx.x] = v;
  }
}

// batch: live[sl] = 1 when some system with rows in slice sl still iterates.
// Rows of a stopped system are only ever read by that system, so its work can
// be skipped; a restarted system starts again from its recomputed residual.
// blockIdx.y is the level.
struct LiveArgs {
  int32_t n[kMaxLevels], nslices[kMaxLevels];
  const int32_t *sys[kMaxLevels];
  unsigned char *live[kMaxLevels];
};
__global__ void k_slice_live(const __grid_constant__ LiveArgs a, const int *bact) {
  pdl_trigger();
  pdl_wait();
  const int k = blockIdx.y;
  const int32_t n = a.n[k];
  const int32_t *__restrict__ sys = a.sys[k];
  for (int32_t sl = blockIdx.x * blockDim.x + threadIdx.x; sl < a.nslices[k]; sl += gridDim.x * blockDim.x) {
    unsigned char v = 0;
    for (int32_t q = sys[sl * 32]; q <= sys[min(sl * 32 + 31, n - 1)]; ++q)
      if (bact[q]) {
        v = 1;
        break;
      }
    a.live[k][sl] = v;
  }
}

// Resident blocks per SM of k_sell: FP32 vectors fit in 40 registers (6 blocks
// of 256 threads), FP64 vectors need 64 (4 blocks).
template <class VT>
constexpr int sell_min_blocks() { return sizeof(VT) == 4 ? 6 : 4; }

// ND: inner products that the launch fuses (compiled only where used, so that the
// plain SpMV does not hold their accumulators in registers)
// GATE: a batch's launch, skipping slices whose systems have all stopped
// (compiled only into the batch instantiations)
// With fused inner products: FP32 vectors need more than the 40 registers of six
// resident blocks (they spilled there), four blocks of 64; FP64 vectors hold ten
// entries and the row's operands in 80 registers, three blocks.  Ten entries: an FEM
// slice has nine with the diagonal, which took two steps of eight.
template <class VT>
constexpr int dot_blocks() { return sizeof(VT) == 4 ? 4 : 3; }
template <class VT, int ND>
constexpr int sell_launch_blocks() { return ND ? dot_blocks<VT>() : sell_min_blocks<VT>(); }

// The row's own operands of the epilogue EPI and of the inner products.  They are
// loaded with the first gathers: behind them, each was one more trip to L2 or HBM in
// the chain of a slice (ops_ahead; not where the registers do not reach: the
// polynomial's steps of several operands).
template <class VT, int EPI, int ND>
constexpr bool ops_ahead() { return EPI <= 1 || (sizeof(VT) == 4 && ND > 0); }
template <class VT>
struct RowOps {
  VT rhs, dinv, c0, c1, c2, p0, p1, res, xin, s, u1, u2;
  double q;
};
template <class VT, int EPI, int ND>
__device__ __forceinline__ RowOps<VT> load_row_ops(const SellArgs<VT> &a, int32_t row) {
  RowOps<VT> o;
  if constexpr (EPI == E_RESID || EPI == E_RESID_POLY) o.rhs = a.rhs[row];
  if constexpr (EPI >= E_DSCALE) o.dinv = a.dinv[row];
  if constexpr (EPI == E_POLYPRE || EPI == E_HORNER_LAST) o.c0 = a.coef[3 * row];
  if constexpr (EPI == E_POLYPRE || EPI == E_HORNER) o.c1 = a.coef[3 * row + 1];
  if constexpr (EPI == E_POLYPRE || EPI == E_RESID_POLY) o.c2 = a.coef[3 * row + 2];
  if constexpr (EPI == E_POLYPRE) {
    o.p0 = a.p0[row];
    o.p1 = a.p1[row];
  }
  if constexpr (EPI == E_HORNER || EPI == E_HORNER_LAST) o.res = a.res[row];
  if constexpr (EPI == E_HORNER_LAST) o.xin = a.xin[row];
  if constexpr (ND == 1) o.q = a.q64[row];
  if constexpr (ND >= 2) {
    o.s = a.x[row];
    o.u1 = a.u1[row];
  }
  if constexpr (ND == 3) o.u2 = a.u2[row];
  return o;
}

// row `row` of the epilogue EPI with the row's product y, and the launch's inner products
template <class VT, int EPI, int ND>
__device__ __forceinline__ void sell_epilogue(const SellArgs<VT> &a, int32_t row, VT y, const RowOps<VT> &w,
                                              double (&acc)[ND ? ND : 1]) {
  VT o;
  if (EPI == E_Y) o = y;
  else if (EPI == E_RESID) o = w.rhs - y;
  else if (EPI == E_DSCALE) o = w.dinv * y;
  else if (EPI == E_POLYPRE) o = w.c0 * w.p0 + w.c1 * w.p1 + w.c2 * (w.dinv * y);
  else if (EPI == E_RESID_POLY) {
    o = w.rhs - y;
    a.out2[row] = w.dinv * (w.c2 * o);
  } else if (EPI == E_HORNER)
    o = w.dinv * y + w.dinv * (w.c1 * w.res);
  else
    o = w.xin + (w.dinv * y + w.dinv * (w.c0 * w.res));
  a.out[row] = o;
  if constexpr (ND == 1) {
    acc[0] += (double)o * w.q;
  } else if constexpr (ND >= 2) {
    const double oy = (double)o, sv = ND != 5 && a.dot_y ? oy : (double)w.s, u1 = (double)w.u1;
    acc[0] += sv * oy;
    acc[1] += sv * u1;
    if constexpr (ND == 3) acc[2] += sv * (double)w.u2;
    if constexpr (ND == 5) {
      acc[2] += oy * oy;
      acc[3] += oy * u1;
      acc[4] += u1 * u1;
    }
  }
}

// y = A x over SELL-32, one warp per slice, one lane per row
template <class MV, class VT, int EPI, int ND, bool GATE>
__global__ void __launch_bounds__(kThreads, sell_launch_blocks<VT, ND>()) k_sell(SellArgs<VT> a) {
  pdl_trigger();
  const int lane = threadIdx.x & 31;
  const MV *__restrict__ sval = static_cast<const MV *>(a.sval);
  double acc[ND ? ND : 1] = {0.0};
  // U entries of a row per step: 6 with FP32 vectors (a 7-point row without its
  // split-off diagonal in one step, at 40 registers), 8 with FP64
  constexpr int U = sizeof(VT) == 4 ? 6 : (ND == 2 ? 10 : 8);
  bool first = true, run = true, live = true;
  constexpr bool kOpsAhead = ops_ahead<VT, EPI, ND>();
  // FP32 vectors at 64 registers wait for the predecessor after the first slice's
  // matrix loads have gone out; at 40 registers, and with FP64 vectors, that spills
  constexpr bool kAhead = sizeof(VT) == 4 && ND > 0;
  if constexpr (!kAhead) {
    pdl_wait();
    if (a.pred && *a.pred == 0) return;
    first = false;
  }
  auto enter = [&](int32_t sl) {
    if (!first) return;
    first = false;
    pdl_wait();
    run = !(a.pred && *a.pred == 0);
    if (GATE) live = sl < a.nslices && a.live[sl];
  };
  for (int32_t sl = blockIdx.x * kWarps + (threadIdx.x >> 5); sl < a.nslices; sl += gridDim.x * kWarps) {
    if (GATE && !first) {
      live = a.live[sl];
      if (!live) continue;
    }
    const int32_t row = sl * 32 + lane;
    VT y = VT(0), dg = VT(0), xr = VT(0);
    RowOps<VT> own;
    const bool diag = !std::is_same<MV, double>::value && a.sdiag != nullptr && row < a.n;
    const int64_t base = a.sptr[sl];
    const int32_t width = (int32_t)((a.sptr[sl + 1] - base) >> 5);
    // the split diagonal (FP32 / BF16 values only) is loaded right behind the first
    // step's matrix loads and x_row with the gathers, so that their latency overlaps
    if constexpr (kPairs<MV> || kHalfPairs<MV>) {
      // FP32 values: a lane's entries 2j and 2j+1 come in one 16-byte load;
      // BF16 values: their columns in one 8-byte load and their values in one
      // 4-byte load (widths are even, U is even).  FULL: all U entries exist
      static_assert(U % 2 == 0, "pairs need an even step");
      const int4 *__restrict__ pp = a.spair + (base >> 1) + lane;
      const int2 *__restrict__ cp2 = reinterpret_cast<const int2 *>(a.scol + base) + lane;
      const __nv_bfloat162 *__restrict__ vp2 = reinterpret_cast<const __nv_bfloat162 *>(sval + base) + lane;
      auto step = [&](int32_t e, auto full, auto size) {
        constexpr bool FULL = decltype(full)::value;
        constexpr int S = decltype(size)::value;  // entries of this step
        int32_t c[S];
        float v[S];
#pragma unroll
        for (int q = 0; q < S; q += 2) {
          if (FULL || e + q < width) {
            if constexpr (kPairs<MV>) {
              const int4 pr = ld_stream(pp + 16 * (e + q));
              c[q] = pr.x;
              v[q] = __int_as_float(pr.y);
              c[q + 1] = pr.z;
              v[q + 1] = __int_as_float(pr.w);
            } else {
              const int2 cc = ld_stream(cp2 + 16 * (e + q));
              const float2 vv = __bfloat1622float2(ld_stream(vp2 + 16 * (e + q)));
              c[q] = cc.x;
              c[q + 1] = cc.y;
              v[q] = vv.x;
              v[q + 1] = vv.y;
            }
          }
        }
        if (e == 0) {
          if (diag) dg = (VT)ld_stream(a.sdiag + row);
          enter(sl);
          if (diag) xr = a.x[row];
          if (kOpsAhead) own = load_row_ops<VT, EPI, ND>(a, min(row, a.n - 1));
        }
        VT xv[S];
#pragma unroll
        for (int q = 0; q < S; ++q)
          if (FULL || e + q < width) xv[q] = a.x[c[q]];
#pragma unroll
        for (int q = 0; q < S; ++q)
          if (FULL || e + q < width) y += v[q] * xv[q];
      };
      // a slice of U or U + 2 entries a row (a 7-point row, a P1 FEM row) takes
      // one step without predicates, whose loads all go out before the first gather
      using UStep = std::integral_constant<int, U>;
      using U2Step = std::integral_constant<int, U + 2>;
      if (width == U) {
        step(0, std::true_type{}, UStep{});
      } else if (width == U + 2) {
        step(0, std::true_type{}, U2Step{});
      } else {
        for (int32_t e = 0; e < width; e += U) step(e, std::false_type{}, UStep{});
      }
    } else {
      const int32_t *__restrict__ cp = a.scol + base + lane;
      const MV *__restrict__ vp = sval + base + lane;
      for (int32_t e = 0; e < width; e += U) {
        int32_t c[U];
        MV v[U];
#pragma unroll
        for (int q = 0; q < U; ++q) {
          if (e + q < width) {
            c[q] = ld_stream(cp + 32 * (e + q));
            v[q] = ld_stream(vp + 32 * (e + q));
          }
        }
        if (e == 0) {
          enter(sl);
          if (kOpsAhead) own = load_row_ops<VT, EPI, ND>(a, min(row, a.n - 1));
        }
        VT xv[U];
#pragma unroll
        for (int q = 0; q < U; ++q)
          if (e + q < width) xv[q] = a.x[c[q]];
#pragma unroll
        for (int q = 0; q < U; ++q)
          if (e + q < width) y += to_acc(v[q], VT(0)) * xv[q];
      }
    }
    enter(sl);  // a slice without entries has not waited yet
    if (!run) return;
    if (GATE && !live) continue;
    if (!kOpsAhead || width == 0) own = load_row_ops<VT, EPI, ND>(a, min(row, a.n - 1));
    if (diag) {
      if (width == 0) {  // a row without off-diagonal entries
        dg = (VT)a.sdiag[row];
        xr = a.x[row];
      }
      y += dg * xr;
    }
    if (row < a.n) sell_epilogue<VT, EPI, ND>(a, row, y, own, acc);
  }
  enter(a.nslices);  // a warp without a slice
  if (!run) return;
  if constexpr (ND > 0) store_dots<ND>(acc, 1, a.partials);
}

// The product on a small level (at most kSmallSlices slices): 2^wl warps share a
// slice, warp q taking its entries q, q + 2^wl, ... (pairs of entries for FP32 and
// BF16 values), and meet in shared memory in warp order.  Such a level leaves most
// of the GPU idle and lives in L2, so its time is one warp's chain of dependent
// loads: splitting the rows shortens the chain to one step whose matrix loads all
// go out before the wait for the predecessor.
template <class MV, class VT, int EPI, int ND, bool GATE>
__global__ void __launch_bounds__(kThreads) k_sell_small(SellArgs<VT> a, int wl) {
  pdl_trigger();
  __shared__ VT sh[kWarps][32];
  constexpr int U = 8;  // entries of a warp per step
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int wps = 1 << wl, sub = wid & (wps - 1), spb = kWarps >> wl;
  const MV *__restrict__ sval = static_cast<const MV *>(a.sval);
  double acc[ND ? ND : 1] = {0.0};
  bool first = true;
  for (int32_t s0 = blockIdx.x * spb; s0 < a.nslices; s0 += gridDim.x * spb) {
    const int32_t sl = s0 + (wid >> wl);
    const bool in = sl < a.nslices;
    const int32_t row = sl * 32 + lane;
    const bool mine = sub == 0 && in && row < a.n;  // this thread finishes the row
    const int64_t base = in ? a.sptr[sl] : 0;
    const int32_t width = in ? (int32_t)((a.sptr[sl + 1] - base) >> 5) : 0;
    VT dg = VT(0);
    if (!std::is_same<MV, double>::value && mine && a.sdiag) dg = (VT)a.sdiag[row];
    VT y = VT(0);
    auto step = [&](int32_t e0, auto &&between) {
      int32_t c[U];
      VT v[U];
      if constexpr (kPairs<MV> || kHalfPairs<MV>) {
        const int4 *__restrict__ pp = a.spair + (base >> 1) + lane;
        const int2 *__restrict__ cp2 = reinterpret_cast<const int2 *>(a.scol + base) + lane;
        const __nv_bfloat162 *__restrict__ vp2 = reinterpret_cast<const __nv_bfloat162 *>(sval + base) + lane;
#pragma unroll
        for (int q = 0; q < U; q += 2) {
          const int32_t pr = (e0 >> 1) + sub + (q >> 1) * wps;  // this warp's next pair
          c[q] = c[q + 1] = -1;
          if (2 * pr < width) {
            if constexpr (kPairs<MV>) {
              const int4 p4 = __ldg(pp + 32 * pr);
              c[q] = p4.x;
              v[q] = __int_as_float(p4.y);
              c[q + 1] = p4.z;
              v[q + 1] = __int_as_float(p4.w);
            } else {
              const int2 cc = __ldg(cp2 + 32 * pr);
              const float2 vv = __bfloat1622float2(vp2[32 * pr]);
              c[q] = cc.x;
              c[q + 1] = cc.y;
              v[q] = vv.x;
              v[q + 1] = vv.y;
            }
          }
        }
      } else {
#pragma unroll
        for (int q = 0; q < U; ++q) {
          const int32_t e = e0 + sub + q * wps;
          c[q] = -1;
          if (e < width) {
            c[q] = __ldg(a.scol + base + 32 * (int64_t)e + lane);
            v[q] = to_acc(sval[base + 32 * (int64_t)e + lane], VT(0));
          }
        }
      }
      between();
      VT xv[U];
#pragma unroll
      for (int q = 0; q < U; ++q)
        if (c[q] >= 0) xv[q] = a.x[c[q]];
#pragma unroll
      for (int q = 0; q < U; ++q)
        if (c[q] >= 0) y += v[q] * xv[q];
    };
    bool run = true;
    RowOps<VT> own;
    VT xr = VT(0);
    step(0, [&] {
      if (first) {
        first = false;
        pdl_wait();
        run = !(a.pred && *a.pred == 0);
      }
      if (mine) {
        if (!std::is_same<MV, double>::value && a.sdiag) xr = a.x[row];
        own = load_row_ops<VT, EPI, ND>(a, row);
      }
    });
    if (!run) return;  // the same in every thread of the grid
    const bool live = !GATE || (in && a.live[sl]);  // of a batch: a dead slice is not stored
    if (live)
      for (int32_t e0 = U * wps; e0 < width; e0 += U * wps) step(e0, [] {});
    if (wps > 1) {
      if (s0 != (int32_t)blockIdx.x * spb) __syncthreads();  // the last slice's sums have been read
      if (sub) sh[wid][lane] = y;
      __syncthreads();
      if (sub == 0)
        for (int q = 1; q < wps; ++q) y += sh[wid + q][lane];
    }
    if (mine && live) {
      if (!std::is_same<MV, double>::value && a.sdiag) y += dg * xr;
      sell_epilogue<VT, EPI, ND>(a, row, y, own, acc);
    }
  }
  if (first) {  // a block without a slice
    pdl_wait();
    if (a.pred && *a.pred == 0) return;
  }
  if constexpr (ND > 0) store_dots<ND>(acc, wps, a.partials);
}

// out = wd * rhs: damped Jacobi from a zero initial guess
template <class VT>
__global__ void k_scale(int32_t n, VT *out, const VT *__restrict__ wd, const VT *rhs, const int *pred,
                        const int32_t *__restrict__ sys, const int *bact) {
  pdl_trigger();
  const int32_t i0 = blockIdx.x * blockDim.x + threadIdx.x;
  VT w = i0 < n ? wd[i0] : VT(0);
  pdl_wait();
  if (pred && *pred == 0) return;
  for (int32_t i = i0; i < n; i += gridDim.x * blockDim.x) {
    if (i != i0) w = wd[i];
    if (!bact || bact[sys[i]]) out[i] = w * rhs[i];
  }
}

// r_{k+1}(I) = sum_{i in G_I} P(i, I) r_k(i); also the next level's smoothing start
// x0 = wd_{k+1} * r_{k+1} when that level smooths.  kRestrictLanes lanes share an
// aggregate (members t, t + 4, ... and a fixed shuffle tree); the members and
// weights of the first 16 are loaded before the wait, so that one gather is left
// behind it.  Aggregates hold ~5 to 11 rows, at most a few dozen.
constexpr int kRestrictLanes = 4;
constexpr int kRestrictAhead = 4;  // members a lane loads ahead
template <class VT>
struct Members {
  int32_t i[kRestrictAhead];
  VT p[kRestrictAhead];
  int32_t m0, m1;
  __device__ __forceinline__ void load(bool in, int32_t I, int t, const int32_t *__restrict__ aptr,
                                       const int32_t *__restrict__ amem, const VT *__restrict__ pwm) {
    m0 = in ? aptr[I] : 0;
    m1 = in ? aptr[I + 1] : 0;
#pragma unroll
    for (int u = 0; u < kRestrictAhead; ++u) {
      const int32_t m = m0 + t + u * kRestrictLanes;
      i[u] = -1;
      if (m < m1) {
        i[u] = amem[m];
        p[u] = pwm[m];
      }
    }
  }
  // sum over the members, the same in the aggregate's lanes
  __device__ __forceinline__ VT sum(int t, const int32_t *__restrict__ amem, const VT *__restrict__ pwm, const VT *r) {
    VT v[kRestrictAhead], s = VT(0);
#pragma unroll
    for (int u = 0; u < kRestrictAhead; ++u)
      if (i[u] >= 0) v[u] = r[i[u]];
#pragma unroll
    for (int u = 0; u < kRestrictAhead; ++u)
      if (i[u] >= 0) s += p[u] * v[u];
    for (int32_t m = m0 + t + kRestrictAhead * kRestrictLanes; m < m1; m += kRestrictLanes) s += pwm[m] * r[amem[m]];
#pragma unroll
    for (int o = kRestrictLanes / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
  }
};

template <class VT>
__global__ void __launch_bounds__(kThreads) k_restrict(int32_t nc, const int32_t *__restrict__ aptr,
                                                       const int32_t *__restrict__ amem, const VT *__restrict__ pwm,
                                                       const VT *r, VT *bc, const VT *__restrict__ wdc, VT *x0c,
                                                       const int *pred, const int32_t *__restrict__ sysc,
                                                       const int *bact) {
  pdl_trigger();
  const int t = threadIdx.x % kRestrictLanes;
  const int32_t per = gridDim.x * (kThreads / kRestrictLanes);
  const int32_t rounds = (nc + per - 1) / per;  // every lane of a warp runs the same rounds
  int32_t I = blockIdx.x * (kThreads / kRestrictLanes) + threadIdx.x / kRestrictLanes;
  for (int32_t q = 0; q < rounds; ++q, I += per) {
    const bool in = I < nc;
    Members<VT> mb;
    mb.load(in, I, t, aptr, amem, pwm);
    const VT w = in && wdc ? wdc[I] : VT(0);
    if (q == 0) {
      pdl_wait();
      if (pred && *pred == 0) return;
    }
    const VT s = mb.sum(t, amem, pwm, r);
    if (in && t == 0 && (!bact || bact[sysc[I]])) {
      bc[I] = s;
      if (wdc) x0c[I] = w * s;
    }
  }
}

// x_k += P_k x_{k+1}: a gather through the aggregate map
template <class VT>
__global__ void k_prolong(int32_t n, const int32_t *__restrict__ agg, const VT *__restrict__ pw, const VT *xc, VT *x,
                          const int *pred, const int32_t *__restrict__ sys, const int *bact) {
  pdl_trigger();
  const int32_t i0 = blockIdx.x * blockDim.x + threadIdx.x;
  int32_t g = i0 < n ? agg[i0] : 0;
  VT p = i0 < n ? pw[i0] : VT(0);
  pdl_wait();
  if (pred && *pred == 0) return;
  for (int32_t i = i0; i < n; i += gridDim.x * blockDim.x) {
    if (i != i0) {
      g = agg[i];
      p = pw[i];
    }
    if (!bact || bact[sys[i]]) x[i] += p * xc[g];
  }
}

// Post-smoothing after the coarse correction (Alg. 4/5): with x the iterate and r
// its residual before the correction,
//   out = x + P x_{k+1} + wd (r - (A P) x_{k+1}).
// A P has one entry per neighbouring aggregate (3-6 off the row's own, for 6-25 in
// a row of A) and gathers from the small vector x_{k+1}; the prolongation needs no
// launch of its own and A is not read again.
template <class VT>
struct PostArgs {
  int32_t n, nslices;
  const int64_t *ptr;
  const int4 *pair;    // FP32 vectors
  const int32_t *col;  // FP64 vectors
  const double *val;
  const VT *own, *pw, *wd;
  const int32_t *agg;
  const unsigned char *live;  // batch
  const VT *x, *r, *xc;
  VT *out;
  const double *q64;  // ND = 1: out . q64, the blocks' sums to partials
  double *partials;
  const int *pred;
};

// Resident blocks per SM, and the grid's wave: the row's operands, its first step's
// entries and their gathers all in flight at 80 (FP32) and 128 registers.  One block
// more an SM holds fewer (a solve of FEM 1024^2 in FP32 20.3 -> 20.7 ms, 90^3 in FP64
// 5.69 -> 6.30), 6 and 4 blocks 22.2 and 6.74 ms.
template <class VT>
constexpr int post_blocks() { return sizeof(VT) == 4 ? 3 : 2; }

template <class VT, int ND, bool GATE>
__global__ void __launch_bounds__(kThreads, post_blocks<VT>()) k_post(PostArgs<VT> a) {
  pdl_trigger();
  const int lane = threadIdx.x & 31;
  double acc[ND ? ND : 1] = {0.0};
  bool first = true, run = true;
  constexpr int U = 8;
  for (int32_t sl = blockIdx.x * kWarps + (threadIdx.x >> 5); sl < a.nslices; sl += gridDim.x * kWarps) {
    if (GATE && !first && !a.live[sl]) continue;
    const int32_t row = sl * 32 + lane;
    const int32_t rr = min(row, a.n - 1);
    const int64_t base = a.ptr[sl];
    const int32_t width = (int32_t)((a.ptr[sl + 1] - base) >> 5);
    const int32_t g = __ldcs(a.agg + rr);
    const VT own = __ldcs(a.own + rr), p = __ldcs(a.pw + rr), w = __ldcs(a.wd + rr);
    VT y = VT(0);
    auto step = [&](int32_t e, auto size, auto full, auto &&between) {
      constexpr int S = decltype(size)::value;
      constexpr bool FULL = decltype(full)::value;
      int32_t c[S];
      VT v[S];
      if constexpr (sizeof(VT) == 4) {
        const int4 *__restrict__ pp = a.pair + (base >> 1) + lane;
#pragma unroll
        for (int q = 0; q < S; q += 2)
          if (FULL || e + q < width) {
            const int4 p4 = ld_stream(pp + 16 * (e + q));
            c[q] = p4.x;
            v[q] = __int_as_float(p4.y);
            c[q + 1] = p4.z;
            v[q + 1] = __int_as_float(p4.w);
          }
      } else {
#pragma unroll
        for (int q = 0; q < S; ++q)
          if (FULL || e + q < width) {
            c[q] = ld_stream(a.col + base + 32 * (int64_t)(e + q) + lane);
            v[q] = ld_stream(a.val + base + 32 * (int64_t)(e + q) + lane);
          }
      }
      between();
      VT xv[S];
#pragma unroll
      for (int q = 0; q < S; ++q)
        if (FULL || e + q < width) xv[q] = a.xc[c[q]];
#pragma unroll
      for (int q = 0; q < S; ++q)
        if (FULL || e + q < width) y += v[q] * xv[q];
    };
    bool live = true;
    VT xg = VT(0), ri = VT(0), xi = VT(0);
    double qi = 0.0;
    auto enter = [&] {  // wait (first slice), then the row's own operands
      if (first) {
        first = false;
        pdl_wait();
        run = !(a.pred && *a.pred == 0);
        if (GATE) live = a.live[sl];
      }
      xg = a.xc[g];
      ri = a.r[rr];
      xi = a.x[rr];
      if constexpr (ND == 1) qi = a.q64[rr];
    };
    // widths 4 and 6, the neighbouring aggregates of a row of 5- and 7-point and P1
    // meshes (FP32: rounded up to even), take one step without predicates; all widths
    // by the predicated step: FEM 1024^2 20.27 -> 20.37 ms, 90^3 FP64 5.69 -> 5.73,
    // 97^3 BF16 58.7 -> 59.0, 700^2 19.56 -> 19.59
    using S4 = std::integral_constant<int, 4>;
    using S6 = std::integral_constant<int, 6>;
    using SU = std::integral_constant<int, U>;
    if (width == 4) step(0, S4{}, std::true_type{}, enter);
    else if (width == 6) step(0, S6{}, std::true_type{}, enter);
    else {
      step(0, SU{}, std::false_type{}, enter);
      for (int32_t e = U; e < width; e += U) step(e, SU{}, std::false_type{}, [] {});
    }
    if (!run) return;  // the same in every thread of the grid
    if (GATE && !live) continue;
    if (row < a.n) {
      const VT o = (xi + p * xg) + w * (ri - (own * xg + y));
      a.out[row] = o;
      if constexpr (ND == 1) acc[0] += (double)o * qi;
    }
  }
  if (first) {  // a warp without a slice
    pdl_wait();
    if (a.pred && *a.pred == 0) return;
  }
  if constexpr (ND > 0) store_dots<ND>(acc, 1, a.partials);
}

// exact coarsest solve x = A_L^-1 b (one warp per row, FP64 accumulation)
template <class VT>
__global__ void k_coarse(int32_t nL, const double *__restrict__ Ainv, const VT *b, VT *x, const int *pred) {
  pdl_wait_and_trigger();
  if (pred && *pred == 0) return;
  const int lane = threadIdx.x & 31;
  for (int32_t i = blockIdx.x * kWarps + (threadIdx.x >> 5); i < nL; i += gridDim.x * kWarps) {
    double s = 0.0;
    for (int32_t j = lane; j < nL; j += 32) s += Ainv[(int64_t)i * nL + j] * (double)b[j];
    s = warp_sum(s);
    if (lane == 0) x[i] = (VT)s;
  }
}

// restriction to the coarsest level and its exact solve in one launch: every
// block forms r_L = R r (as k_restrict does) in shared memory, then its warps
// take rows of x = A_L^-1 r_L.  The rows go round the blocks, one block an SM:
// an FP64 warp instruction takes 16 cycles of an SM, so the rows' dot products
// are spread over all of them.  The members of the first two passes of the
// restriction and a warp's first 256 entries of A_L^-1 are loaded before the wait.
constexpr int kFusedCoarseMax = 2048;
constexpr int kCoarseThreads = 512;
template <class VT>
__global__ void __launch_bounds__(kCoarseThreads, 1) k_restrict_coarse(
    int32_t nL, const int32_t *__restrict__ aptr, const int32_t *__restrict__ amem, const VT *__restrict__ pwm,
    const VT *r, const double *__restrict__ Ainv, VT *x, const int *pred) {
  __shared__ VT bsh[kFusedCoarseMax];
  pdl_trigger();
  constexpr int kPer = kCoarseThreads / kRestrictLanes;  // aggregates per pass
  const int t = threadIdx.x % kRestrictLanes, lane = threadIdx.x & 31;
  int32_t I = threadIdx.x / kRestrictLanes;
  Members<VT> m0, m1;
  m0.load(I < nL, I, t, aptr, amem, pwm);
  m1.load(I + kPer < nL, I + kPer, t, aptr, amem, pwm);
  int32_t i = blockIdx.x + gridDim.x * (threadIdx.x >> 5);
  double ar[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int32_t j = lane + 32 * u;
    ar[u] = i < nL && j < nL ? Ainv[(int64_t)i * nL + j] : 0.0;
  }
  pdl_wait();
  if (pred && *pred == 0) return;
  for (int32_t p = 0; p * kPer < nL; ++p, I += kPer) {
    if (p == 1) m0 = m1;
    if (p > 1) m0.load(I < nL, I, t, aptr, amem, pwm);
    const VT s = m0.sum(t, amem, pwm, r);
    if (t == 0 && I < nL) bsh[I] = s;
  }
  __syncthreads();
  for (bool ahead = true; i < nL; i += gridDim.x * (kCoarseThreads / 32), ahead = false) {
    double s = 0.0;
    if (ahead) {
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (32 * u < nL) s += ar[u] * (lane + 32 * u < nL ? (double)bsh[lane + 32 * u] : 0.0);
    }
    for (int32_t j = lane + (ahead ? 256 : 0); j < nL; j += 32) s += Ainv[(int64_t)i * nL + j] * (double)bsh[j];
    s = warp_sum(s);
    if (lane == 0) x[i] = (VT)s;
  }
}

// sum of the first nb partials of dot k, identical in every block
__device__ __forceinline__ double sum_partials(const double *part, int k, int nb) {
  __shared__ double sh[kWarps];
  __shared__ double result;
  double acc = 0.0;
  for (int j = threadIdx.x; j < nb; j += blockDim.x) acc += part[k * kRedBlocks + j];
  acc = warp_sum(acc);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x < 32) {
    double v = threadIdx.x < (int)(blockDim.x >> 5) ? sh[threadIdx.x] : 0.0;
    v = warp_sum(v);
    if (threadIdx.x == 0) result = v;
  }
  __syncthreads();
  return result;
}

// Vector kernels take kRows rows a thread and round, their loads issued before the
// first store: the compiler cannot move a load over a store that may alias, so a
// plain loop has one row's loads in flight (a batch's tiles, one block each: 116.3 ->
// 111.3 ms a pass of 40 systems with the tile sizes of build_tiles; the single-system
// kernels, a full wave of blocks, run the same either way).
constexpr int kRows = 4;
// kRows rows i, i + step, ... < end of r~ = r - s1 v, x0 = wd r~, ||r~||^2 and ||r||^2
template <class VT>
__device__ __forceinline__ void axpy_rt_rows(int32_t i, int32_t step, int32_t end, VT s1, const VT *r, const VT *v,
                                             VT *rt, const VT *__restrict__ wd, VT *x0, double (&acc)[2]) {
  VT rv[kRows], vv[kRows], wv[kRows];
#pragma unroll
  for (int u = 0; u < kRows; ++u) {
    const int32_t k = i + u * step;
    if (k < end) {
      rv[u] = r[k];
      vv[u] = v[k];
      wv[u] = wd[k];
    }
  }
#pragma unroll
  for (int u = 0; u < kRows; ++u) {
    const int32_t k = i + u * step;
    if (k < end) {
      const VT ti = rv[u] - s1 * vv[u];
      rt[k] = ti;
      x0[k] = wv[u] * ti;
      acc[0] += (double)ti * (double)ti;
      acc[1] += (double)rv[u] * (double)rv[u];
    }
  }
}

// r~ = r - (alpha_1/rho_1) v and the next smoothing start x0 = wd * r~, from the sums
// {c.v, c.r, v.v, v.r, r.r} of the product before (rho_1 and alpha_1: c.v and c.r, or
// v.v and v.r in the GMRES variant), and the test of Alg. 5: the second inner step runs
// iff the enclosing step runs and ||r~|| > t ||r||, with ||r~||^2 = r.r - 2 s v.r +
// s^2 v.v.  The subtraction keeps about 2^-50 of r.r, far below t^2 r.r for any
// threshold above kTestBySums; smaller ones take k_test on r~ itself.  A skipped
// enclosing step clears the flag.
constexpr double kTestBySums = 1e-4;
template <class VT>
__global__ void __launch_bounds__(kSumThreads) k_axpy_rt(int32_t n, const VT *r, const VT *v, VT *rt,
                                                         const VT *__restrict__ wd, VT *x0, double t, int gmres,
                                                         double *slots, int *flag, const double *part, int nb,
                                                         const int *pred) {
  __shared__ double s1_sh;
  pdl_trigger();
  pdl_wait();
  if (pred && *pred == 0) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *flag = 0;
    return;
  }
  int32_t r0, end;
  block_rows(n, r0, end);
  constexpr int32_t step = kSumThreads;
  const int32_t i0 = r0 + threadIdx.x;
  VT rv[kRows], vv[kRows], wv[kRows];
  auto load = [&](int32_t i) {
#pragma unroll
    for (int u = 0; u < kRows; ++u)
      if (i + u * step < end) {
        rv[u] = r[i + u * step];
        vv[u] = v[i + u * step];
        wv[u] = wd[i + u * step];
      }
  };
  load(i0);  // the first rows come with the partials
  double tot[5];
  sum_partials_of<5>(part, nb, tot);
  if (threadIdx.x == 0) {
    const double rho1 = gmres ? tot[2] : tot[0], a1 = gmres ? tot[3] : tot[1], s1 = a1 / rho1;
    s1_sh = s1;
    if (blockIdx.x == 0) {
      slots[S_RHO1] = rho1;
      slots[S_A1] = a1;
      slots[S_S1] = s1;
      if (t >= kTestBySums) {
        // an infinite ||r|| takes the first step of a finite length, as the comparison of
        // the norms does (rt2 is then no number)
        const double rt2 = (tot[4] - s1 * tot[3]) - s1 * (tot[3] - s1 * tot[2]);
        const bool second = isinf(tot[4]) ? !isfinite(s1) : !(rt2 <= t * t * tot[4]);
        *flag = second ? 1 : 0;
        if (second) slots[S_TAKEN] += 1.0;  // cycle trace
      }
    }
  }
  __syncthreads();
  const VT s1 = (VT)s1_sh;
  for (int32_t i = i0; i < end; i += kRows * step) {
    if (i != i0) load(i);
#pragma unroll
    for (int u = 0; u < kRows; ++u)
      if (i + u * step < end) {
        const VT ti = rv[u] - s1 * vv[u];
        rt[i + u * step] = ti;
        x0[i + u * step] = wv[u] * ti;
      }
  }
}

// the test of Alg. 5 on ||r~|| and ||r|| themselves (thresholds below kTestBySums)
template <class VT>
__global__ void __launch_bounds__(kThreads) k_test(int32_t n, const VT *r, const VT *rt, double t, double *slots,
                                                   int *flag, double *part, unsigned *ticket, const int *pred) {
  pdl_trigger();
  pdl_wait();
  if (pred && *pred == 0) return;
  double acc[2] = {0.0, 0.0}, tot[2];
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    acc[0] += (double)rt[i] * (double)rt[i];
    acc[1] += (double)r[i] * (double)r[i];
  }
  if (grid_totals<2>(acc, 1, part, ticket, tot)) {
    const bool second = !(sqrt(tot[0]) <= t * sqrt(tot[1]));
    *flag = second ? 1 : 0;
    if (second) slots[S_TAKEN] += 1.0;
  }
}

// x_{k+1} = (alpha1/rho1) c, or the two-step combination when it was taken: from the
// sums {beta, gamma, alpha_2} of the product w = A d (CG: d.w, d.v, d.r~; GMRES with w
// in place of d on the left), rho_2 = beta - gamma^2 / rho_1
template <class VT>
__global__ void __launch_bounds__(kSumThreads) k_combine(int32_t n, const VT *c, const VT *d, VT *x,
                                                         const double *slots, const int *flag, const double *part,
                                                         int nb, const int *pred) {
  __shared__ double w_sh[2];
  pdl_trigger();
  pdl_wait();
  if (pred && *pred == 0) return;
  const bool two = *flag != 0;
  int32_t r0, end;
  block_rows(n, r0, end);
  constexpr int32_t step = kSumThreads;
  const int32_t i0 = r0 + threadIdx.x;
  VT cv[kRows], dv[kRows];
  auto load = [&](int32_t i) {
#pragma unroll
    for (int u = 0; u < kRows; ++u)
      if (i + u * step < end) {
        cv[u] = c[i + u * step];
        dv[u] = two ? d[i + u * step] : VT(0);
      }
  };
  load(i0);
  if (two) {
    const double rho1 = slots[S_RHO1], s1 = slots[S_S1];
    double tot[3];
    sum_partials_of<3>(part, nb, tot);
    if (threadIdx.x == 0) {
      const double g1 = tot[1] / rho1, cd = tot[2] / (tot[0] - tot[1] * g1);
      w_sh[0] = s1 - g1 * cd;
      w_sh[1] = cd;
    }
  } else if (threadIdx.x == 0) {
    w_sh[0] = slots[S_S1];
    w_sh[1] = 0.0;
  }
  __syncthreads();
  const VT cc = (VT)w_sh[0], cd = (VT)w_sh[1];
  for (int32_t i = i0; i < end; i += kRows * step) {
    if (i != i0) load(i);
#pragma unroll
    for (int u = 0; u < kRows; ++u)
      if (i + u * step < end) x[i + u * step] = two ? cc * cv[u] + cd * dv[u] : cc * cv[u];
  }
}

// ---------------------------------------------------------------- outer FCG (FP64)
template <class VT>
__global__ void k_to_vt(int32_t n, const double *in, VT *__restrict__ out, const VT *__restrict__ wd,
                        VT *__restrict__ x0, const int *pred) {
  pdl_trigger();
  pdl_wait();
  if (pred && *pred == 0) return;
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const VT v = (VT)in[i];
    out[i] = v;
    x0[i] = wd[i] * v;
  }
}

// z = (double) zin
template <class VT>
__global__ void k_from_vt(int32_t n, const VT *zin, double *__restrict__ z, const int *pred) {
  pdl_trigger();
  pdl_wait();
  if (pred && *pred == 0) return;
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) z[i] = (double)zin[i];
}

// z^T q of the outer flexible CG where the cycle has no product to fuse it into (a
// hierarchy of one level)
template <class VT>
__global__ void __launch_bounds__(kThreads) k_dot_zq(int32_t n, const VT *z, const double *q, double *part,
                                                     const int *pred) {
  pdl_trigger();
  pdl_wait();
  if (pred && *pred == 0) return;
  double acc[1] = {0.0};
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    acc[0] += (double)z[i] * q[i];
  store_dots<1>(acc, 1, part);
}

// p = z + beta p, beta = -(z^T q_old) / (p_old^T q_old) from z^T q's partials (0 right
// after a restart); z in the cycle's vector type
template <class VT>
__global__ void __launch_bounds__(kSumThreads) k_fcg_p(int32_t n, const VT *z, double *p, double *slots,
                                                       const int *restart, const double *part, int nb,
                                                       const int *pred) {
  __shared__ double beta_sh;
  pdl_trigger();
  pdl_wait();
  if (pred && *pred == 0) return;
  const bool rs = *restart != 0;
  const double pq = slots[S_PQ];
  int32_t r0, end;
  block_rows(n, r0, end);
  const int32_t i0 = r0 + threadIdx.x;
  VT zv[kRows];
  double pv[kRows];
  auto load = [&](int32_t i) {
#pragma unroll
    for (int u = 0; u < kRows; ++u)
      if (i + u * kSumThreads < end) {
        zv[u] = z[i + u * kSumThreads];
        pv[u] = p[i + u * kSumThreads];
      }
  };
  load(i0);  // the first rows come with the partials
  double tot[1];
  sum_partials_of<1>(part, nb, tot);
  if (threadIdx.x == 0) {
    beta_sh = rs ? 0.0 : -tot[0] / pq;
    if (blockIdx.x == 0) slots[S_ZQ] = tot[0];
  }
  __syncthreads();
  const double beta = beta_sh;
  for (int32_t i = i0; i < end; i += kRows * kSumThreads) {
    if (i != i0) load(i);
#pragma unroll
    for (int u = 0; u < kRows; ++u)
      if (i + u * kSumThreads < end) p[i + u * kSumThreads] = rs ? (double)zv[u] : (double)zv[u] + beta * pv[u];
  }
}

struct FcgState {
  double *hist;
  int *it, *active, *restart, *status;
  volatile int *host;  // mapped pinned words: [0] iterations, [4] status
};

// kRows rows i, i + step, ... < end of the update of x and r, of the next
// preconditioner input rvt (nullable) and its smoothing start x0, and of ||r||^2
template <class VT>
struct FcgRows {
  double xv[kRows], rv[kRows], pv[kRows], qv[kRows];
  VT wv[kRows];
  __device__ __forceinline__ void load(int32_t i, int32_t step, int32_t end, const double *x, const double *r,
                                       const double *p, const double *q, const VT *__restrict__ wd) {
#pragma unroll
    for (int u = 0; u < kRows; ++u) {
      const int32_t k = i + u * step;
      if (k < end) {
        xv[u] = x[k];
        pv[u] = p[k];
        rv[u] = r[k];
        qv[u] = q[k];
        wv[u] = wd[k];
      }
    }
  }
  __device__ __forceinline__ void apply(int32_t i, int32_t step, int32_t end, double alpha, double *x, double *r,
                                        VT *rvt, VT *x0, double &acc) {
#pragma unroll
    for (int u = 0; u < kRows; ++u) {
      const int32_t k = i + u * step;
      if (k < end) {
        x[k] = xv[u] + alpha * pv[u];
        const double ri = rv[u] - alpha * qv[u];
        r[k] = ri;
        acc += ri * ri;
        const VT v = (VT)ri;
        if (rvt) rvt[k] = v;
        x0[k] = wv[u] * v;
      }
    }
  }
};

// alpha = p^T r / p^T q from the partials of the product q = A p;
// x += alpha p;  r -= alpha q;  the preconditioner input (in reduced precision
// also rounded to VT) and its smoothing start x0 = wd r.  The last block ends the
// outer iteration: relative residual into the history, iteration count,
// convergence / breakdown status (deactivates the following launches).
template <class VT>
__global__ void __launch_bounds__(kSumThreads, 2) k_fcg_update(int32_t n, double *x, double *r, const double *p,
                                                            const double *q, double *slots, const double *pq_part,
                                                            int nb, double *part, unsigned *ticket, VT *rvt,
                                                            const VT *__restrict__ wd, VT *x0, FcgState st,
                                                            const int *pred) {
  __shared__ double alpha_sh, pq_sh;
  pdl_trigger();
  pdl_wait();
  if (pred && *pred == 0) return;
  int32_t r0, end;
  block_rows(n, r0, end);
  const int32_t i0 = r0 + threadIdx.x;
  FcgRows<VT> rows;
  rows.load(i0, kSumThreads, end, x, r, p, q, wd);  // the first rows come with the partials
  {
    double tot[2];
    sum_partials_of<2>(pq_part, nb, tot);
    if (threadIdx.x == 0) {
      pq_sh = tot[0];
      alpha_sh = tot[1] / tot[0];
    }
    __syncthreads();
  }
  const double alpha = alpha_sh;
  double acc[1] = {0.0};
  for (int32_t i = i0; i < end; i += kRows * kSumThreads) {
    if (i != i0) rows.load(i, kSumThreads, end, x, r, p, q, wd);
    rows.apply(i, kSumThreads, end, alpha, x, r, rvt, x0, acc[0]);
  }
  double tot[1];
  if (grid_totals<1, kSumThreads>(acc, 1, part, ticket, tot)) {
    const double rel = sqrt(tot[0]) / sqrt(slots[S_NB2]);
    slots[S_PQ] = pq_sh;
    const int k = *st.it + 1;
    *st.it = k;
    st.hist[k] = rel;
    slots[S_RR] = tot[0];
    slots[S_REL] = rel;
    *st.restart = 0;
    int status = 0;
    if (!(pq_sh > 0.0)) status = AMG_ERR_BREAKDOWN;
    else if (!isfinite(rel)) status = AMG_ERR_NAN;
    else if (rel <= slots[S_TOL]) status = 1;  // updated residual converged: the host checks the true residual
    else if (k >= (int)slots[S_MAXIT]) status = AMG_ERR_NOT_CONVERGED;
    if (status != 0) {
      *st.status = status;
      *st.active = 0;
    }
    st.host[0] = k;
    __threadfence_system();
    st.host[4] = status;
    __threadfence_system();
  }
}

// block partial dot (generic)
__global__ void k_dot64(int32_t n, const double *a, const double *b, double *__restrict__ part, const int *pred) {
  pdl_wait_and_trigger();
  if (pred && *pred == 0) return;
  double acc = 0.0;
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) acc += a[i] * b[i];
  block_store_dot(acc, part);
}

__global__ void k_store_sum(const double *part, int nb, double *__restrict__ dst) {
  pdl_wait_and_trigger();
  const double v = sum_partials(part, 0, nb);
  if (threadIdx.x == 0) *dst = v;
}

// r = b - A x in FP64 (level-0 SELL with FP64 values), with ||r||^2 partials
__global__ void k_residual64(int32_t n, int32_t nslices, const int64_t *__restrict__ sptr,
                             const int32_t *__restrict__ scol, const double *__restrict__ sval,
                             const double *x, const double *b, double *__restrict__ r, double *__restrict__ part) {
  pdl_wait_and_trigger();
  const int lane = threadIdx.x & 31;
  double acc = 0.0;
  for (int32_t sl = blockIdx.x * kWarps + (threadIdx.x >> 5); sl < nslices; sl += gridDim.x * kWarps) {
    const int64_t base = sptr[sl];
    const int32_t width = (int32_t)((sptr[sl + 1] - base) >> 5);
    double y = 0.0;
    for (int32_t e = 0; e < width; ++e) {
      const int64_t at = base + 32 * e + lane;
      y += sval[at] * x[scol[at]];
    }
    const int32_t row = sl * 32 + lane;
    if (row < n) {
      const double ri = b[row] - y;
      r[row] = ri;
      acc += ri * ri;
    }
  }
  block_store_dot(acc, part);
}

// ---------------------------------------------------------------- outer FGMRES (FP64)
constexpr int kMaxRestart = 32;

// One Arnoldi step is the cycle, the product w = A z_j and four launches: the
// classical Gram-Schmidt coefficients (GS_DOT), the update and the coefficients of
// the reorthogonalisation (GS_AGAIN), its update with ||w|| and the Givens step
// (GS_LAST), and the next basis vector with the preconditioner's input.  The step
// number is a device word, so that one captured graph serves every step of a
// restart.  Bound by L2 up to a few 10^5 rows, by HBM beyond; what the separate
// sums, norm, scalar and conversion kernels cost was their launches' latency, and the
// host's wait for every step: 301^2 convection-diffusion in FP64, 19.1 -> 14.6 ms a solve.
struct FgArgs {
  int32_t n;
  int m;            // restart length (leading dimension of H)
  double *V, *Z;    // basis and preconditioned vectors, column by column
  double *w;        // A z_j
  const double *z;  // z_j, copied to Z by GS_DOT
  double *H, *fg;   // fg[0..m] = g, fg[m+1..2m] = cos, fg[2m+1..3m] = sin
  double *hc;       // coefficients of the running pass; hc[kMaxRestart + 1] = 1 / ||w||
  double *part;     // (kMaxRestart + 1) x kRedBlocks
  unsigned *ticket;
  int *step;        // j
  double *slots, *hist;
  int *it, *active, *status;
  volatile int *host;  // mapped pinned words: [0] iterations, [4] status
};
enum GsPass { GS_DOT = 0, GS_AGAIN = 1, GS_LAST = 2 };

// Givens rotations on column j of H (in shared memory), the residual estimate
// |g_{j+1}| / ||b|| into the history; deactivates the following steps when done
__device__ __forceinline__ void fg_givens(const FgArgs &a, int j, double *col, const double *cs, const double *sn,
                                          double nrm) {
  for (int l = 0; l < j; ++l) {
    const double p = col[l], q = col[l + 1];
    col[l] = cs[l] * p + sn[l] * q;
    col[l + 1] = -sn[l] * p + cs[l] * q;
  }
  const double p = col[j], den = sqrt(p * p + nrm * nrm), c = p / den, s = nrm / den;
  col[j] = den;
  a.fg[a.m + 1 + j] = c;
  a.fg[2 * a.m + 1 + j] = s;
  const double g = a.fg[j];
  a.fg[j + 1] = -s * g;
  a.fg[j] = c * g;
  a.hc[kMaxRestart + 1] = nrm != 0.0 ? 1.0 / nrm : 0.0;
  *a.step = j + 1;
  const int k = *a.it + 1;
  *a.it = k;
  const double rel = fabs(s * g) / sqrt(a.slots[S_NB2]);
  a.hist[k] = rel;
  a.slots[S_REL] = rel;
  int status = 0;
  if (!isfinite(rel)) status = AMG_ERR_NAN;
  else if (rel <= a.slots[S_TOL] || nrm == 0.0) status = 1;
  else if (k >= (int)a.slots[S_MAXIT]) status = AMG_ERR_NOT_CONVERGED;
  if (status != 0) {
    *a.status = status;
    *a.active = 0;
  }
  a.host[0] = k;
  __threadfence_system();
  a.host[4] = status;
  __threadfence_system();
}

// The columns go by eight: a thread keeps eight sums over its rows, the block's 256
// values of a column meet in one warp, and the last block sums the blocks' partials
// in block order (a warp holds up to four columns at a time).
template <int PASS>
__global__ void __launch_bounds__(kThreads) k_fg_gs(FgArgs a) {
  static_assert(kWarps == 8, "a warp per column of a group");
  __shared__ double sh[PASS == GS_LAST ? 1 : 8][kThreads];
  __shared__ double h[kMaxRestart + 1];
  __shared__ double cs[PASS == GS_LAST ? kMaxRestart : 1], sn[PASS == GS_LAST ? kMaxRestart : 1];
  __shared__ bool last;
  pdl_trigger();
  pdl_wait();
  if (*a.active == 0) return;
  const int j = *a.step, ncol = j + 1;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t n = a.n;
  const int32_t i0 = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
  double *w = a.w;
  const double *V = a.V;
  double norm2 = 0.0;
  if (PASS == GS_DOT) {
    for (int32_t i = i0; i < a.n; i += stride) a.Z[j * n + i] = a.z[i];
  } else {  // w -= sum_l h_l V_l
    if (threadIdx.x < ncol) h[threadIdx.x] = a.hc[threadIdx.x];
    __syncthreads();
    for (int32_t i = i0; i < a.n; i += stride) {
      double t = w[i];
      int l = 0;
      for (; l + 8 <= ncol; l += 8) {
        double v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = V[(l + q) * n + i];
#pragma unroll
        for (int q = 0; q < 8; ++q) t -= h[l + q] * v[q];
      }
      for (; l < ncol; ++l) t -= h[l] * V[l * n + i];
      w[i] = t;
      if (PASS == GS_LAST) norm2 += t * t;
    }
  }
  if constexpr (PASS == GS_LAST) {
    sh[0][threadIdx.x] = norm2;
    __syncthreads();
    if (wid == 0) {
      double v = sh[0][lane];
#pragma unroll
      for (int q = 1; q < kWarps; ++q) v += sh[0][q * 32 + lane];
      v = warp_sum(v);
      if (lane == 0) {
        a.part[blockIdx.x] = v;
        __threadfence();
      }
    }
  } else {
    for (int c0 = 0; c0 < ncol; c0 += 8) {
      double acc[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) acc[q] = 0.0;
      for (int32_t i = i0; i < a.n; i += stride) {
        const double wi = w[i];
        double v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = c0 + q < ncol ? V[(c0 + q) * n + i] : 0.0;
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (c0 + q < ncol) acc[q] += v[q] * wi;
      }
      __syncthreads();  // the previous group's sums have been read
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (c0 + q < ncol) sh[q][threadIdx.x] = acc[q];
      __syncthreads();
      if (c0 + wid < ncol) {
        double v = sh[wid][lane];
#pragma unroll
        for (int q = 1; q < kWarps; ++q) v += sh[wid][q * 32 + lane];
        v = warp_sum(v);
        if (lane == 0) {
          a.part[(c0 + wid) * kRedBlocks + blockIdx.x] = v;
          __threadfence();
        }
      }
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(a.ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  const int nb = gridDim.x;
  if constexpr (PASS != GS_LAST) {
    for (int c0 = wid; c0 < ncol; c0 += 4 * kWarps) {
      double v[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 2
      for (int b = lane; b < nb; b += 32)
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (c0 + u * kWarps < ncol) v[u] += __ldcg(a.part + (c0 + u * kWarps) * kRedBlocks + b);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int l = c0 + u * kWarps;
        if (l >= ncol) break;
        const double t = warp_sum(v[u]);
        if (lane == 0) {
          a.hc[l] = t;
          a.H[l * a.m + j] = PASS == GS_AGAIN ? a.H[l * a.m + j] + t : t;
        }
      }
    }
    if (threadIdx.x == 0) *a.ticket = 0;
  } else {
    double v = 0.0;
    for (int b = threadIdx.x; b < nb; b += kThreads) v += __ldcg(a.part + b);
    sh[0][threadIdx.x] = v;
    if (threadIdx.x < ncol) h[threadIdx.x] = a.H[threadIdx.x * a.m + j];
    if (threadIdx.x < j) {
      cs[threadIdx.x] = a.fg[a.m + 1 + threadIdx.x];
      sn[threadIdx.x] = a.fg[2 * a.m + 1 + threadIdx.x];
    }
    __syncthreads();
    if (wid == 0) {
      double t = sh[0][lane];
#pragma unroll
      for (int q = 1; q < kWarps; ++q) t += sh[0][q * 32 + lane];
      t = warp_sum(t);
      if (lane == 0) {
        *a.ticket = 0;
        fg_givens(a, j, h, cs, sn, sqrt(t));
      }
      __syncwarp();
      for (int l = lane; l < ncol; l += 32) a.H[l * a.m + j] = h[l];
    }
  }
}

// V_j = v * scale with the preconditioner's input and smoothing start.  START: V_0 =
// r / ||r||, g = (||r||, 0, ...); else V_j = w / ||w|| of the step just ended (the
// last step of a restart needs no next vector).
template <class VT, bool START>
__global__ void __launch_bounds__(kThreads) k_fg_basis(FgArgs a, const double *v, VT *in, const VT *__restrict__ wd,
                                                       VT *x0) {
  pdl_trigger();
  pdl_wait();
  int j = 0;
  double inv;
  if (START) {
    const double beta = sqrt(a.slots[S_RR]);
    if (blockIdx.x == 0) {
      for (int l = threadIdx.x; l <= a.m; l += blockDim.x) a.fg[l] = (l == 0) ? beta : 0.0;
      if (threadIdx.x == 0) *a.step = 0;
    }
    inv = beta != 0.0 ? 1.0 / beta : 0.0;
  } else {
    if (*a.active == 0) return;
    j = *a.step;
    if (j >= a.m) return;
    inv = a.hc[kMaxRestart + 1];
  }
  double *out = a.V + (int64_t)j * a.n;
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += gridDim.x * blockDim.x) {
    const double t = v[i] * inv;
    out[i] = t;
    in[i] = (VT)t;
    x0[i] = wd[i] * (VT)t;
  }
}

// x += sum_l y_l Z_l with y = H(0:j, 0:j)^-1 g, j the steps taken: every block solves
// the triangular system in its first warp (lane l holds row l; at most 32 rows)
__global__ void __launch_bounds__(kThreads) k_fg_xupdate(FgArgs a, double *__restrict__ x) {
  static_assert(kMaxRestart <= 32, "a lane per row");
  __shared__ double Hs[kMaxRestart][kMaxRestart + 1];
  __shared__ double y[kMaxRestart];
  pdl_trigger();
  pdl_wait();
  const int j = *a.step;
  for (int q = threadIdx.x; q < j * j; q += kThreads) Hs[q / j][q % j] = a.H[(q / j) * a.m + q % j];
  __syncthreads();
  if (threadIdx.x < 32) {
    const int l = threadIdx.x;
    double t = l < j ? a.fg[l] : 0.0;
    for (int q = j - 1; q >= 0; --q) {
      if (l == q) t /= Hs[q][q];
      const double yq = __shfl_sync(0xffffffffu, t, q);
      if (l < q) t -= Hs[l][q] * yq;
    }
    if (l < j) y[l] = t;
  }
  __syncthreads();
  const int64_t n = a.n;
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += gridDim.x * blockDim.x) {
    double t = x[i];
    int l = 0;
    for (; l + 8 <= j; l += 8) {
      double v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = a.Z[(l + q) * n + i];
#pragma unroll
      for (int q = 0; q < 8; ++q) t += y[l + q] * v[q];
    }
    for (; l < j; ++l) t += y[l] * a.Z[l * n + i];
    x[i] = t;
  }
}

// ---------------------------------------------------------------- batched systems
// Per-system scalars of the block-diagonal solve.  Inner products are
// segmented by system: every row tile lies inside one system; tile partials
// are summed per system in tile order (deterministic).

__global__ void k_sys_of(int32_t n, int32_t nsys, const int32_t *__restrict__ off, int32_t *__restrict__ sys) {
  pdl_wait_and_trigger();
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    int32_t lo = 0, hi = nsys - 1;
    while (lo < hi) {  // last system whose first row is <= i
      const int32_t mid = (lo + hi + 1) >> 1;
      if (off[mid] <= i) lo = mid; else hi = mid - 1;
    }
    sys[i] = lo;
  }
}

#define BS(slot, s) bslots[(int64_t)(slot)*nsys + (s)]

// per-system status of a batch while it runs: kIterating, kUpdatedConverged
// (the updated residual met tol; the true residual is checked next), then
// AMG_OK or a negative AMG_ERR_* code once the system has stopped
constexpr int kIterating = 2;
constexpr int kUpdatedConverged = 1;

// Per-system inner products and the scalars they lead to, in one launch: a block
// takes a row tile of one system, and the block that finishes a system's last tile
// sums the system's tiles in tile order and takes its scalar step.  Tiles of stopped
// systems are skipped (bact; null: all systems).  As separate launches the sums over
// tiles and the scalar steps were 21 of a pass's ~100 kernels.
enum BFin { BF_STORE = 0, BF_K1 = 1, BF_DECIDE = 2, BF_K3 = 3, BF_BETA = 4, BF_ALPHA = 5 };

struct SegArgs {
  int32_t ntiles, nsys;
  const int32_t *tile_row, *tile_sys, *sys_tile;
  const int *bact;
  double *tpart;  // 3 x ntiles
  int *ticket;    // nsys, 0 between launches
  double *bslots;
  int kind, slot0;  // BF_STORE: totals to slots slot0, slot0 + 1, ...
  int *flag;        // BF_K1 clears, BF_DECIDE sets the level's second-step flags (flag[nsys]: any)
  double t;         // BF_DECIDE
  const int *brs;   // BF_BETA: restart flags
};

constexpr int kSegThreads = 256;

__device__ __forceinline__ void run_bfin(const SegArgs &g, int32_t s, int nd, const double *tot) {
  double *bslots = g.bslots;
  const int32_t nsys = g.nsys;
  switch (g.kind) {
    case BF_STORE:
      for (int d = 0; d < nd; ++d) BS(g.slot0 + d, s) = tot[d];
      break;
    case BF_K1:  // Alg. 5 after v = A c: c^T v, c^T r
      BS(S_RHO1, s) = tot[0];
      BS(S_A1, s) = tot[1];
      BS(S_S1, s) = tot[1] / tot[0];
      break;
    case BF_DECIDE: {  // ||r~|| > t ||r|| (squared): this system needs the second inner step
      const bool second = !(tot[0] <= g.t * g.t * tot[1]);
      g.flag[s] = second ? 1 : 0;
      if (second) g.flag[nsys] = 1;
      break;
    }
    case BF_K3: {  // after w = A d: gamma = d^T v, beta = d^T w, alpha_2 = d^T r~
      const double gam = tot[0], g1 = gam / BS(S_RHO1, s), cd = tot[2] / (tot[1] - gam * g1);
      BS(S_CC, s) = BS(S_S1, s) - g1 * cd;
      BS(S_CD, s) = cd;
      break;
    }
    case BF_BETA:  // outer flexible CG: z^T q_old
      BS(S_ZQ, s) = tot[0];
      BS(S_BETA, s) = g.brs[s] ? 0.0 : -tot[0] / BS(S_PQ, s);
      break;
    default:  // p^T q, p^T r
      BS(S_PQ, s) = tot[0];
      BS(S_PR, s) = tot[1];
      BS(S_ALPHA, s) = tot[1] / tot[0];
  }
}

// the tile's sums; the block that completes system s runs its scalar step.  Every
// thread of the block calls it (tile t lies in system s).
template <int ND>
__device__ __forceinline__ void seg_finish(const double (&acc)[ND], const SegArgs &g, int32_t t, int32_t s) {
  __shared__ double sh[ND][kSegThreads];
  __shared__ double tot[ND];
  __shared__ bool last;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int32_t t0 = g.sys_tile[s], nt = g.sys_tile[s + 1] - t0;
#pragma unroll
  for (int k = 0; k < ND; ++k) sh[k][threadIdx.x] = acc[k];
  __syncthreads();
  if (wid < ND) {
    double v = sh[wid][lane];
#pragma unroll
    for (int q = 1; q < kSegThreads / 32; ++q) v += sh[wid][q * 32 + lane];
    v = warp_sum(v);
    if (lane == 0) {
      if (nt == 1) {
        tot[wid] = v;
      } else {
        g.tpart[(int64_t)wid * g.ntiles + t] = v;
        __threadfence();
      }
    }
  }
  __syncthreads();
  if (nt > 1) {
    if (threadIdx.x == 0) last = atomicAdd(g.ticket + s, 1) == nt - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    if (wid < ND) {
      const double *p = g.tpart + (int64_t)wid * g.ntiles + t0;
      double v = 0.0;
      for (int32_t q = lane; q < nt; q += 32) v += __ldcg(p + q);
      v = warp_sum(v);
      if (lane == 0) tot[wid] = v;
    }
    if (threadIdx.x == 0) g.ticket[s] = 0;
    __syncthreads();
  }
  if (threadIdx.x == 0) run_bfin(g, s, ND, tot);
}

// s . y0 (, s . y1, s . y2) of every system
template <class VS, class VY, int ND>
__global__ void __launch_bounds__(kSegThreads) k_segdot(SegArgs g, const VS *sv, const VY *y0, const VY *y1,
                                                        const VY *y2, const int *pred) {
  pdl_trigger();
  pdl_wait();
  if (g.kind == BF_K1 && blockIdx.x == 0 && threadIdx.x == 0) g.flag[g.nsys] = 0;  // also when the step is skipped
  if (pred && *pred == 0) return;
  for (int32_t t = blockIdx.x; t < g.ntiles; t += gridDim.x) {
    const int32_t s = g.tile_sys[t];
    if (g.bact && !g.bact[s]) continue;
    double acc[ND] = {0.0};
    const int32_t r1 = g.tile_row[t + 1];
#pragma unroll 4
    for (int32_t i = g.tile_row[t] + threadIdx.x; i < r1; i += kSegThreads) {
      const double x = (double)sv[i];
      acc[0] += x * (double)y0[i];
      if constexpr (ND > 1) acc[1] += x * (double)y1[i];
      if constexpr (ND > 2) acc[2] += x * (double)y2[i];
    }
    seg_finish<ND>(acc, g, t, s);
    __syncthreads();  // the shared sums are rewritten by the next tile
  }
}

// r~ = r - (alpha_1/rho_1) v and x0 = wd r~ per system, and the test of Alg. 5
template <class VT>
__global__ void __launch_bounds__(kSegThreads) k_baxpy_rt(SegArgs g, const VT *r, const VT *v, VT *rt,
                                                          const VT *__restrict__ wd, VT *x0, const int *pred) {
  pdl_trigger();
  pdl_wait();
  if (pred && *pred == 0) return;
  for (int32_t t = blockIdx.x; t < g.ntiles; t += gridDim.x) {
    const int32_t s = g.tile_sys[t];
    if (g.bact && !g.bact[s]) continue;
    const VT s1 = (VT)g.bslots[(int64_t)S_S1 * g.nsys + s];
    double acc[2] = {0.0, 0.0};
    const int32_t i1 = g.tile_row[t + 1];
    for (int32_t i = g.tile_row[t] + threadIdx.x; i < i1; i += kRows * kSegThreads)
      axpy_rt_rows<VT>(i, kSegThreads, i1, s1, r, v, rt, wd, x0, acc);
    seg_finish<2>(acc, g, t, s);
    __syncthreads();
  }
}

template <class VT>
__global__ void k_bcombine(int32_t n, const int32_t *__restrict__ sys, int32_t nsys, const VT *c, const VT *d, VT *x,
                           const double *bslots, const int *flag, const int *bact, const int *pred) {
  pdl_trigger();
  pdl_wait();
  if (pred && *pred == 0) return;
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int32_t s = sys[i];
    if (!bact[s]) continue;
    x[i] = flag[s] ? (VT)BS(S_CC, s) * c[i] + (VT)BS(S_CD, s) * d[i] : (VT)BS(S_S1, s) * c[i];
  }
}

// exact coarsest solve, one dense inverse per system; one warp per row
template <class VT>
__global__ void k_bcoarse(int32_t nL, const int32_t *__restrict__ sys, const int32_t *__restrict__ off,
                          const double *__restrict__ binv, const int64_t *__restrict__ boff, const VT *b, VT *__restrict__ x,
                          const int *bact, const int *pred) {
  pdl_trigger();
  pdl_wait();
  if (pred && *pred == 0) return;
  const int lane = threadIdx.x & 31;
  for (int32_t i = blockIdx.x * kWarps + (threadIdx.x >> 5); i < nL; i += gridDim.x * kWarps) {
    const int32_t s = sys[i];
    if (!bact[s]) continue;
    const int32_t r0 = off[s], m = off[s + 1] - r0;
    const double *Bi = binv + boff[s] + (int64_t)(i - r0) * m;
    double acc = 0.0;
    for (int32_t j = lane; j < m; j += 32) acc += Bi[j] * (double)b[r0 + j];
    acc = warp_sum(acc);
    if (lane == 0) x[i] = (VT)acc;
  }
}

// flexible CG per system: p = z + beta p, p = z right after a restart (brs), whatever an
// earlier solve left in p.  bact[s]: still iterating
template <class VT>
__global__ void k_bfcg_p(int32_t n, const int32_t *__restrict__ sys, int32_t nsys, const VT *z, double *p,
                         const double *bslots, const int *bact, const int *brs) {
  pdl_trigger();
  pdl_wait();
  const int32_t step = gridDim.x * blockDim.x;
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += kRows * step) {
    int32_t sv[kRows];
    VT zv[kRows];
    double pv[kRows];
#pragma unroll
    for (int u = 0; u < kRows; ++u) sv[u] = i + u * step < n ? sys[i + u * step] : -1;
#pragma unroll
    for (int u = 0; u < kRows; ++u)
      if (sv[u] >= 0 && !bact[sv[u]]) sv[u] = -1;
#pragma unroll
    for (int u = 0; u < kRows; ++u)
      if (sv[u] >= 0) {
        zv[u] = z[i + u * step];
        pv[u] = p[i + u * step];
      }
#pragma unroll
    for (int u = 0; u < kRows; ++u)
      if (sv[u] >= 0) p[i + u * step] = brs[sv[u]] ? (double)zv[u] : (double)zv[u] + BS(S_BETA, sv[u]) * pv[u];
  }
}

// x += alpha p, r -= alpha q, the next preconditioner input and its smoothing start,
// ||r||^2; stopped systems keep x and r untouched
template <class VT>
__global__ void __launch_bounds__(kSegThreads) k_bfcg_update(SegArgs g, double *x, double *r, const double *p,
                                                             const double *q, VT *rvt, const VT *__restrict__ wd,
                                                             VT *x0) {
  pdl_trigger();
  pdl_wait();
  for (int32_t t = blockIdx.x; t < g.ntiles; t += gridDim.x) {
    const int32_t s = g.tile_sys[t];
    if (!g.bact[s]) continue;
    const double a = g.bslots[(int64_t)S_ALPHA * g.nsys + s];
    double acc[1] = {0.0};
    const int32_t i1 = g.tile_row[t + 1];
    for (int32_t i = g.tile_row[t] + threadIdx.x; i < i1; i += kRows * kSegThreads) {
      FcgRows<VT> rows;
      rows.load(i, kSegThreads, i1, x, r, p, q, wd);
      rows.apply(i, kSegThreads, i1, a, x, r, rvt, x0, acc[0]);
    }
    seg_finish<1>(acc, g, t, s);
    __syncthreads();
  }
}

// end of an iteration: per-system relative residual, iteration count, status;
// bact[nsys] = number of systems still iterating, also in the mapped pinned word
// host; hist[k] (k < hist_len) gets the largest relative residual of pass k
__global__ void k_bfcg_fin(int32_t nsys, double *__restrict__ bslots, int *__restrict__ bact, int *__restrict__ brs,
                           int *__restrict__ bit, int *__restrict__ bstat, double tol, int max_iter,
                           double *__restrict__ hist, int hist_len, int *__restrict__ it, volatile int *host) {
  pdl_wait_and_trigger();
  __shared__ int nact;
  __shared__ double worst;
  if (threadIdx.x == 0) {
    nact = 0;
    worst = 0.0;
  }
  __syncthreads();
  for (int32_t s = threadIdx.x; s < nsys; s += blockDim.x) {
    brs[s] = 0;
    if (!bact[s]) continue;
    const double rel = sqrt(BS(S_RR, s) / BS(S_NB2, s));
    BS(S_REL, s) = rel;
    const int k = bit[s] + 1;
    bit[s] = k;
    atomicMax(reinterpret_cast<unsigned long long *>(&worst), __double_as_longlong(isfinite(rel) ? rel : 1e300));
    if (!(BS(S_PQ, s) > 0.0)) {
      bstat[s] = AMG_ERR_BREAKDOWN;
      bact[s] = 0;
    } else if (!isfinite(rel)) {
      bstat[s] = AMG_ERR_NAN;
      bact[s] = 0;
    } else if (rel <= tol) {
      bstat[s] = kUpdatedConverged;
      bact[s] = 0;
    } else if (k >= max_iter) {
      bstat[s] = AMG_ERR_NOT_CONVERGED;
      bact[s] = 0;
    } else {
      atomicAdd(&nact, 1);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    bact[nsys] = nact;
    const int k = *it + 1;
    *it = k;
    if (k < hist_len) hist[k] = worst;
    *host = nact;
    __threadfence_system();
  }
}

#undef BS

template <class VT>
__global__ void k_convert_row_data(int32_t n, const double *diag, double omega_host, const double *omega_dev,
                                   const double *__restrict__ pw64,
                                   VT *__restrict__ wd, VT *__restrict__ dinv, VT *__restrict__ pw,
                                   const int32_t *__restrict__ amem, VT *__restrict__ pwm) {
  pdl_wait_and_trigger();
  const double omega = omega_dev ? *omega_dev : omega_host;
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    wd[i] = (VT)(omega / diag[i]);
    dinv[i] = (VT)(1.0 / diag[i]);
    if (pw64) {
      pw[i] = (VT)pw64[i];
      pwm[i] = (VT)pw64[amem[i]];
    }
  }
}

template <class VT>
__global__ void k_copy_cast(int32_t n, const double *in, VT *__restrict__ out) {
  pdl_wait_and_trigger();
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) out[i] = (VT)in[i];
}

// ============================================================== host engine
namespace {

inline int ew_grid(int64_t n) { return grid_for(n, kThreads, kRedBlocks); }
void prepare_batched(Hierarchy &h, cudaStream_t s);
template <class MV, class VT>
void autotune_t(Hierarchy &h, cudaStream_t s);
// Grid of a level's SpMV launches: one wave of resident blocks (6 per SM with
// FP32 vectors, 4 with FP64) unless the autotuner chose another size (at most
// kRedBlocks, the capacity of the partial-sum buffers).  The FP64 products of the
// outer iteration on level 0 use the FP64 kernel's wave whatever the precision.
template <class VT>
inline int default_sell_grid(const Level &L) {
  return grid_for((int64_t)L.nslices, kWarps, sell_min_blocks<VT>() * 152);
}
// launches with fused inner products: one wave of their kernel, which runs
// dot_blocks per SM (a second, short wave and its reductions took the 190k-row
// level of 128^3 from 10 to 17 us), or the autotuner's choice up to it
template <class VT>
constexpr int dot_wave() { return dot_blocks<VT>() * 152; }
inline int dot_grid(const Level &L) { return L.sell_blocks; }
// launches without inner products have no partial-sum buffer to fill, so the
// autotuner may give them up to one warp per slice; by default they take the
// same wave of resident blocks (one warp per slice measured slower on the 128^3
// level 0: 34.4 against 27.4 us under ncu)
inline int full_plain_grid(const Level &L) { return grid_for((int64_t)L.nslices, kWarps, 1 << 30); }
inline int plain_grid(const Level &L) { return L.sell_plain_blocks; }
// Levels of at most kSmallSlices slices (fewer warps than the GPU holds at a
// quarter of its occupancy) run the product with 2^split_log warps a slice: enough
// that a warp takes its entries in one step of eight, or until the level has
// kSplitWarps warps (the GPU's at three quarters of its occupancy), beyond which
// more warps only wait for each other.
constexpr int32_t kSmallSlices = 2048;
constexpr int32_t kSplitWarps = 152 * 48;
inline int split_log_for(const Level &L) {
  if (L.nslices > kSmallSlices || L.nslices == 0) return -1;
  const int64_t width = L.sell_entries / (32 * (int64_t)L.nslices);  // average entries a row
  int wl = 0;
  while (wl < 3 && (width >> wl) > 6 && ((int64_t)L.nslices << (wl + 1)) <= kSplitWarps) ++wl;
  return wl;
}
inline int outer_grid(const Level &L0) { return default_sell_grid<double>(L0); }

template <class MV, class VT>
struct Engine {
  Hierarchy &h;
  cudaStream_t s;
  int64_t launches = 0;
  bool gmres_variant;
  // products skip the slices whose systems have all stopped (a batch's cycle); a
  // product of its own (amg_spmv) computes every row whatever the last solve stopped
  bool gate;

  Engine(Hierarchy &hh, cudaStream_t ss) : h(hh), s(ss) { gmres_variant = h.p.outer == 1, gate = h.batched; }

  VT *V(void *p) { return static_cast<VT *>(p); }
  // batch: the system map of a level and the systems still iterating (null otherwise)
  const int32_t *bsys(const Level &L) const { return h.batched ? L.sys_of : nullptr; }
  const int *bact() const { return h.batched ? h.bactive : nullptr; }

  void check() {
    ++launches;
    AMG_LAUNCH_CHECK();
  }

  SellArgs<VT> sell_args(int k, const VT *x, VT *out, const int *pred) {
    const Level &L = h.lev[k];
    SellArgs<VT> a{};
    a.n = L.n;
    a.nslices = L.nslices;
    a.sptr = L.sptr;
    a.scol = L.scol;
    a.sval = L.sval;
    a.spair = L.spair;
    a.sdiag = L.sdiag;
    if (gate) a.live = L.slive;
    a.x = x;
    a.out = out;
    a.pred = pred;
    return a;
  }

  unsigned *ticket(const Level &L) const { return reinterpret_cast<unsigned *>(L.flag + 1); }

  // ND fused inner products: after the plain product (Alg. 5) and on the last
  // post-smoothing step of level 0 (z^T q of the outer flexible CG)
  // (returns the launch's blocks: the partial sums of each product)
  template <int EPI, int ND = 0>
  int sell(const SellArgs<VT> &a, int k) {
    const Level &L = h.lev[k];
    if (h.batched && ND)  // inner products of a batch are per system (segdot)
      throw Error{AMG_ERR_UNSUPPORTED, "batched SpMV was given fused inner products"};
    if constexpr (EPI == E_Y || EPI == E_RESID)
      if (L.split_log >= 0) {
        const int grid = grid_for(L.nslices, kWarps >> L.split_log, kRedBlocks);
        if (gate)
          klaunch(k_sell_small<MV, VT, EPI, 0, true>, grid, kThreads, s, a, (int)L.split_log);
        else
          klaunch(k_sell_small<MV, VT, EPI, ND, false>, grid, kThreads, s, a, (int)L.split_log);
        check();
        return grid;
      }
    const int grid = ND ? dot_grid(L) : plain_grid(L);
    if (gate)
      klaunch(k_sell<MV, VT, EPI, 0, true>, grid, kThreads, s, a);
    else
      klaunch(k_sell<MV, VT, EPI, ND, false>, grid, kThreads, s, a);
    check();
    return grid;
  }

  // out = approximately A_k^-1 rhs with a zero initial guess (Alg. 4/5).
  // If x0_ready, lev[k].tmp already holds wd_k * rhs.
  void cycle(int k, const VT *rhs, VT *out, bool x0_ready, const int *pred) {
    Level &L = h.lev[k];
    if (k == h.L - 1) {
      if (h.batched)
        klaunch(k_bcoarse<VT>, grid_for(h.nL, kWarps, 152 * 8), kThreads, s, h.nL, (const int32_t *)L.sys_of,
                (const int32_t *)L.sys_off, (const double *)h.binv, (const int64_t *)h.binv_off, rhs, out,
                (const int *)h.bactive, pred);
      else
        klaunch(k_coarse<VT>, grid_for(h.nL, kWarps, 152), kThreads, s, h.nL, h.coarse_inv, rhs, out, pred);
      check();
      return;
    }
    Level &C = h.lev[k + 1];
    VT *tmp = V(L.tmp);
    const bool poly = h.p.smoother == 1 && L.poly != nullptr && !L.poly_off;
    if (poly) {  // x = sum_q diag(c_q) (D^-1 A)^q D^-1 b
      klaunch(k_scale<VT>, ew_grid(L.n), kThreads, s, L.n, V(L.u0), V(L.dinv), rhs, pred, bsys(L), bact());
      check();
      SellArgs<VT> a = sell_args(k, V(L.u0), V(L.u1), pred);
      a.dinv = V(L.dinv);
      sell<E_DSCALE>(a, k);
      a = sell_args(k, V(L.u1), tmp, pred);
      a.dinv = V(L.dinv);
      a.coef = V(L.poly);
      a.p0 = V(L.u0);
      a.p1 = V(L.u1);
      sell<E_POLYPRE>(a, k);
    } else if (!x0_ready) {
      klaunch(k_scale<VT>, ew_grid(L.n), kThreads, s, L.n, tmp, V(L.wd), rhs, pred, bsys(L), bact());  // pre-smoothing
      check();
    }
    {  // r_k = b_k - A_k x_k
      SellArgs<VT> a = sell_args(k, tmp, V(L.r), pred);
      a.rhs = rhs;
      sell<E_RESID>(a, k);
    }
    const bool coarse_is_last = (k + 1 == h.L - 1);
    const bool tail = (k + 1 == h.tail_t);
    // single systems: the restriction to the coarsest level and its solve in one launch
    const bool fuse_coarse = coarse_is_last && !tail && !h.batched && h.nL <= kFusedCoarseMax;
    if (fuse_coarse) {
      klaunch(k_restrict_coarse<VT>, std::min(h.nL, 152), kCoarseThreads, s, h.nL, L.aptr, L.amem,
              (const VT *)V(L.pwm), (const VT *)V(L.r), h.coarse_inv, V(C.xc), pred);
      check();
    } else {
      // r_{k+1} = R_k r_k  (and x0 of level k+1 when it smooths)
      klaunch(k_restrict<VT>, grid_for((int64_t)L.nc * kRestrictLanes, kThreads, 152 * 32), kThreads, s, L.nc, L.aptr,
              L.amem, (const VT *)V(L.pwm), (const VT *)V(L.r), V(C.bc),
              (const VT *)((coarse_is_last || tail) ? nullptr : V(C.wd)), V(C.tmp), pred, bsys(C), bact());
      check();
    }
    if (tail) {  // levels k+1..L-1 in one cluster launch
      TailArgs ta{};
      ta.t = k + 1;
      ta.L = h.L;
      ta.mode = k < h.p.kcycle_levels ? 1 : 0;
      ta.nL = h.nL;
      ta.gmres = gmres_variant ? 1 : 0;
      ta.kt = h.p.kcycle_t;
      ta.Ainv = h.coarse_inv;
      ta.lev = h.tail_dev;
      ta.pred = pred;
      tail_launch<MV, VT>(ta, h.p.tail == 2 ? 1 : 8, s);
      ++launches;
    } else if (coarse_is_last) {
      if (!fuse_coarse) cycle(k + 1, V(C.bc), V(C.xc), true, pred);  // exact coarse solve
    } else if (k < h.p.kcycle_levels) {
      krylov2(k + 1, pred);  // Alg. 5 coarse correction
    } else {
      cycle(k + 1, V(C.bc), V(C.xc), true, pred);  // Alg. 4 recursion
    }
    if (!poly) {  // x_k += P_k x_{k+1}, then the post-smoothing step on the updated residual
      PostArgs<VT> a{};
      a.n = L.n;
      a.nslices = L.nslices;
      a.ptr = L.ap_ptr;
      a.pair = L.ap_pair;
      a.col = L.ap_col;
      a.val = L.ap_val;
      a.own = V(L.ap_own);
      a.pw = V(L.pw);
      a.wd = V(L.wd);
      a.agg = L.agg;
      a.x = tmp;
      a.r = V(L.r);
      a.xc = V(C.xc);
      a.out = out;
      a.pred = pred;
      const int grid = grid_for(L.nslices, kWarps, post_blocks<VT>() * 152);
      if (h.batched) {
        a.live = L.slive;
        klaunch(k_post<VT, 0, true>, grid, kThreads, s, a);
      } else if (k == 0 && zq_fuse) {  // z^T q of the outer flexible CG
        a.q64 = h.q;
        a.partials = L.partials;
        zq_blocks = grid;
        klaunch(k_post<VT, 1, false>, grid, kThreads, s, a);
      } else {
        klaunch(k_post<VT, 0, false>, grid, kThreads, s, a);
      }
      check();
      return;
    }
    // x_k += P_k x_{k+1}
    klaunch(k_prolong<VT>, ew_grid(L.n), kThreads, s, L.n, L.agg, V(L.pw), V(C.xc), tmp, pred, bsys(L), bact());
    check();
    // r_k = b_k - A_k x_k, then the transposed polynomial in Horner form
    SellArgs<VT> b = sell_args(k, tmp, V(L.r), pred);
    b.rhs = rhs;
    b.dinv = V(L.dinv);
    b.coef = V(L.poly);
    b.out2 = V(L.u0);
    sell<E_RESID_POLY>(b, k);
    b = sell_args(k, V(L.u0), V(L.u1), pred);
    b.dinv = V(L.dinv);
    b.coef = V(L.poly);
    b.res = V(L.r);
    sell<E_HORNER>(b, k);
    SellArgs<VT> a = sell_args(k, V(L.u1), out, pred);
    a.xin = tmp;
    a.dinv = V(L.dinv);
    a.coef = V(L.poly);
    a.res = V(L.r);
    if (k == 0 && zq_fuse) {
      a.q64 = h.q;
      a.partials = L.partials;
      zq_blocks = sell<E_HORNER_LAST, 1>(a, k);
    } else {
      sell<E_HORNER_LAST>(a, k);
    }
  }
  bool zq_fuse = false;
  int zq_blocks = 0;  // partial sums of z^T q

  // tiles of level k and the scalar step that ends its per-system inner products;
  // gate: systems still iterating only
  SegArgs seg_args(int k, BFin kind, bool gate, int slot0 = 0) {
    Level &L = h.lev[k];
    SegArgs g{};
    g.ntiles = L.ntiles;
    g.nsys = h.nsys;
    g.tile_row = L.tile_row;
    g.tile_sys = L.tile_sys;
    g.sys_tile = L.sys_tile;
    g.bact = gate ? h.bactive : nullptr;
    g.tpart = L.tpart;
    g.ticket = L.bticket;
    g.bslots = L.bslots;
    g.kind = kind;
    g.slot0 = slot0;
    g.flag = L.bflag;
    g.t = h.p.kcycle_t;
    g.brs = h.bactive + h.nsys + 1;
    return g;
  }
  static int seg_grid(const SegArgs &g) { return grid_for(g.ntiles, 1, 152 * 8); }
  template <int ND, class VS, class VY>
  void segdot(const SegArgs &g, const VS *sv, const VY *y0, const VY *y1, const VY *y2, const int *pred) {
    klaunch(k_segdot<VS, VY, ND>, seg_grid(g), kSegThreads, s, g, sv, y0, y1, y2, pred);
    check();
  }

  // Alg. 5 coarse part at level m for every system of a batch, with per-system
  // scalars; the second inner step runs when any system needs it
  void krylov2_batched(int m, const int *pred) {
    Level &L = h.lev[m];
    const int32_t ns = h.nsys;
    const VT *nil = nullptr;
    cycle(m, V(L.bc), V(L.c), true, pred);
    sell<E_Y>(sell_args(m, V(L.c), V(L.v), pred), m);
    segdot<2>(seg_args(m, BF_K1, true), (const VT *)V(L.c), (const VT *)V(L.v), (const VT *)V(L.bc), nil, pred);
    const SegArgs g = seg_args(m, BF_DECIDE, true);
    klaunch(k_baxpy_rt<VT>, seg_grid(g), kSegThreads, s, g, (const VT *)V(L.bc), (const VT *)V(L.v), V(L.rt),
            (const VT *)V(L.wd), V(L.tmp), pred);
    check();
    const int *any = L.bflag + ns;
    cycle(m, V(L.rt), V(L.d), true, any);
    sell<E_Y>(sell_args(m, V(L.d), V(L.w), any), m);
    segdot<3>(seg_args(m, BF_K3, true), (const VT *)V(L.d), (const VT *)V(L.v), (const VT *)V(L.w),
              (const VT *)V(L.rt), any);
    klaunch(k_bcombine<VT>, ew_grid(L.n), kThreads, s, L.n, (const int32_t *)L.sys_of, ns, (const VT *)V(L.c),
            (const VT *)V(L.d), V(L.xc), (const double *)L.bslots, (const int *)L.bflag, (const int *)h.bactive, pred);
    check();
  }

  // Alg. 5 coarse part at level m: rhs = bc[m], result in xc[m]; lev[m].tmp holds wd*bc.
  void krylov2(int m, const int *pred) {
    if (h.batched) {
      krylov2_batched(m, pred);
      return;
    }
    Level &L = h.lev[m];
    // c = cycle(m, r)
    cycle(m, V(L.bc), V(L.c), true, pred);
    int nb;
    {  // v = A c with the sums that rho_1, alpha_1 and the test need
      SellArgs<VT> a = sell_args(m, V(L.c), V(L.v), pred);
      a.u1 = V(L.bc);
      a.partials = L.partials;
      nb = sell<E_Y, 5>(a, m);
    }
    const int ng = sum_grid(L.n);
    klaunch(k_axpy_rt<VT>, ng, kSumThreads, s, L.n, (const VT *)V(L.bc), (const VT *)V(L.v), V(L.rt),
            (const VT *)V(L.wd), V(L.tmp), h.p.kcycle_t, gmres_variant ? 1 : 0, L.slots, L.flag,
            (const double *)L.partials, nb, pred);
    check();
    if (!(h.p.kcycle_t >= kTestBySums)) {
      klaunch(k_test<VT>, ew_grid(L.n), kThreads, s, L.n, (const VT *)V(L.bc), (const VT *)V(L.rt), h.p.kcycle_t,
              L.slots, L.flag, L.partials, ticket(L), pred);
      check();
    }
    // second inner step, predicated on the decision
    cycle(m, V(L.rt), V(L.d), true, L.flag);
    {
      SellArgs<VT> a = sell_args(m, V(L.d), V(L.w), L.flag);
      a.u1 = V(L.v);
      a.u2 = V(L.rt);
      a.dot_y = gmres_variant;  // GMRES: w^T w, w^T v, w^T r~; CG: d^T w, d^T v, d^T r~
      a.partials = L.partials;
      nb = sell<E_Y, 3>(a, m);
    }
    klaunch(k_combine<VT>, ng, kSumThreads, s, L.n, (const VT *)V(L.c), (const VT *)V(L.d), V(L.xc),
            (const double *)L.slots, (const int *)L.flag, (const double *)L.partials, nb, pred);
    check();
  }

  // flexible CG: out = M r with the smoothing start x0 of level 0 already formed
  // (by k_to_vt or k_fcg_update), with the sums of z^T q.  The result stays in VT.
  const VT *precond_fcg(const int *pred) {
    Level &L0 = h.lev[0];
    constexpr bool f64 = std::is_same<VT, double>::value;
    const VT *in = f64 ? (const VT *)h.r : V(h.pre_in);
    VT *out = f64 ? (VT *)h.z : V(h.pre_out);
    zq_fuse = h.L > 1;
    cycle(0, in, out, true, pred);
    zq_fuse = false;
    if (h.L == 1) {
      zq_blocks = ew_grid(L0.n);
      klaunch(k_dot_zq<VT>, zq_blocks, kThreads, s, L0.n, (const VT *)out, (const double *)h.q, L0.partials, pred);
      check();
    }
    return out;
  }

  // the preconditioner input in VT and x0 from the FP64 residual (before the first
  // iteration and after a restart; otherwise k_fcg_update leaves them)
  void input_from_r(const double *r, const int *pred) {
    Level &L0 = h.lev[0];
    klaunch(k_to_vt<VT>, ew_grid(L0.n), kThreads, s, L0.n, r, V(h.pre_in), V(L0.wd), V(L0.tmp), pred);
    check();
  }

  // z = M r for the FP64 outer iteration
  void precond(const double *r, double *z, const int *pred) {
    Level &L0 = h.lev[0];
    if (std::is_same<VT, double>::value) {
      cycle(0, (const VT *)r, (VT *)z, false, pred);
    } else {
      input_from_r(r, pred);
      cycle(0, V(h.pre_in), V(h.pre_out), true, pred);
      klaunch(k_from_vt<VT>, ew_grid(L0.n), kThreads, s, L0.n, (const VT *)V(h.pre_out), z, pred);
      check();
    }
  }

  // one flexible-CG iteration of every system of a batch (graph-capturable)
  void fcg_iteration_batched(double tol, volatile int *host_active) {
    Level &L0 = h.lev[0];
    const int32_t ns = h.nsys, n = L0.n;
    const int ng = ew_grid(n);
    int *bact = h.bactive, *brs = h.bactive + ns + 1;
    {  // slices of the systems still iterating, on every level
      LiveArgs la{};
      for (int k = 0; k < h.L; ++k) {
        const Level &L = h.lev[k];
        la.n[k] = L.n;
        la.nslices[k] = L.nslices;
        la.sys[k] = L.sys_of;
        la.live[k] = L.slive;
      }
      klaunch(k_slice_live, dim3((unsigned)grid_for(L0.nslices, kThreads, 152 * 4), (unsigned)h.L), kThreads, s, la,
              (const int *)bact);
      check();
    }
    // z = M r from the input and smoothing start left by k_bfcg_update
    constexpr bool f64 = std::is_same<VT, double>::value;
    const VT *in = f64 ? (const VT *)h.r : V(h.pre_in);
    VT *z = f64 ? (VT *)h.z : V(h.pre_out);
    cycle(0, in, z, true, nullptr);
    const double *nil = nullptr;
    segdot<1>(seg_args(0, BF_BETA, true), (const VT *)z, (const double *)h.q, nil, nil, nullptr);
    klaunch(k_bfcg_p<VT>, ng, kThreads, s, n, (const int32_t *)L0.sys_of, ns, (const VT *)z, h.pdir,
            (const double *)L0.bslots, (const int *)bact, (const int *)brs);
    check();
    {  // q = A p in FP64
      SellArgs<double> a{};
      a.n = n;
      a.nslices = L0.nslices;
      a.sptr = L0.sptr64;
      a.scol = L0.scol64;
      a.sval = L0.sval64;
      a.x = h.pdir;
      a.out = h.q;
      a.live = L0.slive;
      klaunch(k_sell<double, double, E_Y, 0, true>, outer_grid(L0), kThreads, s, a);
      check();
    }
    segdot<2>(seg_args(0, BF_ALPHA, true), (const double *)h.pdir, (const double *)h.q, (const double *)h.r, nil,
              nullptr);
    const SegArgs g = seg_args(0, BF_STORE, true, S_RR);
    klaunch(k_bfcg_update<VT>, seg_grid(g), kSegThreads, s, g, h.x, h.r, (const double *)h.pdir, (const double *)h.q,
            f64 ? (VT *)nullptr : V(h.pre_in), (const VT *)V(L0.wd), V(L0.tmp));
    check();
    klaunch(k_bfcg_fin, 1, 1024, s, ns, L0.bslots, bact, brs, h.bit, h.bit + ns, tol, h.p.max_iter, h.hist,
            h.p.max_iter + 8, h.it_dev, host_active);
    check();
  }

  // one flexible-CG iteration, all on the device (graph-capturable)
  void fcg_iteration(int *active, int *restart, volatile int *host_state) {
    Level &L0 = h.lev[0];
    const int ng = sum_grid(L0.n);
    // z = M r, z^T q
    const VT *z = precond_fcg(active);
    // p = z + beta p
    klaunch(k_fcg_p<VT>, ng, kSumThreads, s, L0.n, z, h.pdir, L0.slots, (const int *)restart,
            (const double *)L0.partials, zq_blocks, active);
    check();
    const int nb = std::min(outer_grid(L0), dot_wave<double>());
    {  // q = A p (FP64), p^T q, p^T r
      SellArgs<double> a{};
      a.n = L0.n;
      a.nslices = L0.nslices;
      a.sptr = L0.sptr64;
      a.scol = L0.scol64;
      a.sval = L0.sval64;
      a.x = h.pdir;
      a.out = h.q;
      a.u1 = h.r;
      a.partials = L0.partials;
      a.pred = active;
      klaunch(k_sell<double, double, E_Y, 2, false>, nb, kThreads, s, a);
      check();
    }
    // x, r update, the next preconditioner input, and the end of the iteration
    const FcgState st{h.hist, h.it_dev, active, restart, h.status_dev, host_state};
    klaunch(k_fcg_update<VT>, ng, kSumThreads, s, L0.n, h.x, h.r, (const double *)h.pdir, (const double *)h.q, L0.slots,
            (const double *)L0.partials, nb, L0.partials + 2 * kRedBlocks, ticket(L0), std::is_same<VT, double>::value ? (VT *)nullptr : V(h.pre_in),
            (const VT *)V(L0.wd), V(L0.tmp), st, active);
    check();
  }

  // FGMRES: basis passes take two rows a thread at least (fewer partial sums for the
  // last block) and four blocks an SM at most
  int gs_grid() const { return grid_for(h.lev[0].n, 2 * kThreads, 152 * 4); }
  FgArgs fg_args(volatile int *host_state) {
    Level &L0 = h.lev[0];
    FgArgs a{};
    a.n = L0.n;
    a.m = h.p.restart;
    a.V = h.V;
    a.Z = h.Z;
    a.w = h.q;
    a.z = std::is_same<VT, double>::value ? (const double *)h.pre_out : h.z;
    a.H = h.H;
    a.fg = h.fg;
    a.hc = h.hc;
    a.part = h.gpart;
    a.ticket = ticket(L0);
    a.step = h.it_dev + 3;
    a.slots = L0.slots;
    a.hist = h.hist;
    a.it = h.it_dev;
    a.active = h.it_dev + 1;
    a.status = h.status_dev;
    a.host = host_state;
    return a;
  }

  // one Arnoldi step from the preconditioner input left by k_fg_basis (graph-capturable)
  void fgmres_step(const FgArgs &f) {
    Level &L0 = h.lev[0];
    cycle(0, V(h.pre_in), V(h.pre_out), true, f.active);
    if (!std::is_same<VT, double>::value) {
      klaunch(k_from_vt<VT>, ew_grid(L0.n), kThreads, s, L0.n, (const VT *)V(h.pre_out), h.z, (const int *)f.active);
      check();
    }
    {  // w = A z_j in FP64
      SellArgs<double> a{};
      a.n = L0.n;
      a.nslices = L0.nslices;
      a.sptr = L0.sptr64;
      a.scol = L0.scol64;
      a.sval = L0.sval64;
      a.x = f.z;
      a.out = f.w;
      a.pred = f.active;
      klaunch(k_sell<double, double, E_Y, 0, false>, outer_grid(L0), kThreads, s, a);
      check();
    }
    klaunch(k_fg_gs<GS_DOT>, gs_grid(), kThreads, s, f);
    klaunch(k_fg_gs<GS_AGAIN>, gs_grid(), kThreads, s, f);
    klaunch(k_fg_gs<GS_LAST>, gs_grid(), kThreads, s, f);
    klaunch(k_fg_basis<VT, false>, ew_grid(L0.n), kThreads, s, f, (const double *)f.w, V(h.pre_in),
            (const VT *)V(L0.wd), V(L0.tmp));
    launches += 3;
    check();
  }
};

template <class MV, class VT>
void alloc_level_vectors(Hierarchy &h, Level &L, int k) {
  const size_t n = (size_t)L.n;
  auto vec = [&]() { return (void *)h.arena.get<VT>(n + 1); };
  L.r = vec();
  L.bc = vec();
  L.xc = vec();
  L.tmp = vec();
  L.u0 = vec();
  L.u1 = vec();
  if (k >= 1) {
    L.c = vec();
    L.v = vec();
    L.rt = vec();
    L.d = vec();
    L.w = vec();
  }
  if (L.sell_blocks <= 0) L.sell_blocks = grid_for((int64_t)L.nslices, kWarps, dot_wave<VT>());
  if (L.sell_plain_blocks <= 0) L.sell_plain_blocks = default_sell_grid<VT>(L);
  L.split_log = split_log_for(L);
  L.slots = h.arena.get<double>(kNumSlots);
  L.flag = h.arena.get<int>(4);
  L.partials = h.arena.get<double>((size_t)kRedBlocks * 8);
  AMG_CUDA(cudaMemsetAsync(L.slots, 0, sizeof(double) * kNumSlots, current_stream()));
  AMG_CUDA(cudaMemsetAsync(L.flag, 0, sizeof(int) * 4, current_stream()));
  AMG_CUDA(cudaMemsetAsync(L.partials, 0, sizeof(double) * kRedBlocks * 8, current_stream()));
}

// First level t of the cluster tail: at most kTailMaxRows rows, not the
// coarsest, every level in t..L-3 below the K-cycle levels (the tail runs
// V-cycles only), and no polynomial smoother on those levels.
void configure_tail(Hierarchy &h, cudaStream_t s) {
  h.tail_t = -1;
  if (!h.p.tail || h.batched) return;  // the cluster tail has no per-system scalars
  for (int t = 1; t <= h.L - 2; ++t) {
    if (h.lev[t].n > kTailMaxRows) continue;
    bool ok = true;
    for (int k = t; k <= h.L - 3; ++k) ok = ok && k >= h.p.kcycle_levels;
    for (int k = t; k < h.L - 1; ++k) ok = ok && !(h.p.smoother == 1 && h.lev[k].poly && !h.lev[k].poly_off);
    if (ok) {
      h.tail_t = t;
      break;
    }
  }
  if (h.tail_t < 0) return;
  std::vector<TailLevel> tl(h.L);
  for (int k = 0; k < h.L; ++k) {
    const Level &L = h.lev[k];
    TailLevel &T = tl[k];
    T.n = L.n;
    T.nslices = L.nslices;
    T.nc = L.nc;
    T.sptr = L.sptr;
    T.scol = L.scol;
    T.sval = L.sval;
    T.spair = L.spair;
    T.sdiag = L.sdiag;
    T.wd = L.wd;
    T.pw = L.pw;
    T.agg = L.agg;
    T.aptr = L.aptr;
    T.amem = L.amem;
    T.bc = L.bc;
    T.xc = L.xc;
    T.r = L.r;
    T.c = L.c;
    T.v = L.v;
    T.rt = L.rt;
    T.d = L.d;
    T.w = L.w;
  }
  if (!h.tail_dev) h.tail_dev = h.arena.get<TailLevel>(kMaxLevels);
  AMG_CUDA(cudaMemcpyAsync(h.tail_dev, tl.data(), sizeof(TailLevel) * h.L, cudaMemcpyHostToDevice, s));
  AMG_CUDA(cudaStreamSynchronize(s));
}

template <class MV, class VT>
void prepare_t(Hierarchy &h, cudaStream_t s) {
  for (int k = 0; k < h.L; ++k) alloc_level_vectors<MV, VT>(h, h.lev[k], k);
  const size_t n = (size_t)h.lev[0].n;
  h.x = h.arena.get<double>(n);
  h.b = h.arena.get<double>(n);
  h.r = h.arena.get<double>(n);
  h.z = h.arena.get<double>(n);
  h.pdir = h.arena.get<double>(n);
  h.q = h.arena.get<double>(n);
  h.pre_in = h.arena.get<VT>(n);
  h.pre_out = h.arena.get<VT>(n);
  h.hist = h.arena.get<double>((size_t)h.p.max_iter + 8);
  h.it_dev = h.arena.get<int>(8);
  h.status_dev = h.it_dev + 4;
  AMG_CUDA(cudaMemsetAsync(h.q, 0, sizeof(double) * n, s));
  AMG_CUDA(cudaMemsetAsync(h.pdir, 0, sizeof(double) * n, s));
  if (h.p.outer == 1) {
    const int m = h.p.restart;
    h.V = h.arena.get<double>(n * (size_t)(m + 1));
    h.Z = h.arena.get<double>(n * (size_t)m);
    h.H = h.arena.get<double>((size_t)(m + 1) * m);
    h.fg = h.arena.get<double>(4 * (size_t)m + 2);
    h.hc = h.arena.get<double>(kMaxRestart + 2);
    h.gpart = h.arena.get<double>((size_t)(kMaxRestart + 1) * kRedBlocks);
    AMG_CUDA(cudaMemsetAsync(h.H, 0, sizeof(double) * (m + 1) * m, s));
  }
  if (!h.host_pinned) h.host_pinned = pinned_scratch_get();
  if (h.batched) prepare_batched(h, s);
  configure_tail(h, s);
  if (h.p.autotune) autotune_t<MV, VT>(h, s);
}

template <class VT>
void make_row_data_t(Hierarchy &h, Level &L, const double *diag, cudaStream_t s) {
  if (!L.wd) {  // refilled in place by a values-only re-setup
    L.wd = h.arena.get<VT>((size_t)L.n + 1);
    L.dinv = h.arena.get<VT>((size_t)L.n + 1);
    L.pw = h.arena.get<VT>((size_t)L.n + 1);
    L.pwm = h.arena.get<VT>((size_t)L.n + 1);
  }
  klaunch(k_convert_row_data<VT>, ew_grid(L.n), kThreads, s, L.n, diag, L.omega, (const double *)L.omega_dev,
          L.pw64, (VT *)L.wd, (VT *)L.dinv, (VT *)L.pw, (const int32_t *)L.amem, (VT *)L.pwm);
  AMG_LAUNCH_CHECK();
}

__global__ void k_set_state(int *it, int *active, int *restart, int *status, int it_v, int active_v,
                            int restart_v, int status_v) {
  pdl_wait_and_trigger();
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    if (it_v >= 0) *it = it_v;
    *active = active_v;
    *restart = restart_v;
    *status = status_v;
  }
}

__global__ void k_set_slot(double *slots, int idx, double v) {
  pdl_wait_and_trigger();
  if (threadIdx.x == 0 && blockIdx.x == 0) slots[idx] = v;
}

// Copy n doubles between user memory (host or device) and device memory.
void copy_in(double *dst_dev, const double *src, int32_t n, cudaStream_t s) {
  const cudaMemcpyKind k = pointer_kind(src) == PTR_DEVICE ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
  AMG_CUDA(cudaMemcpyAsync(dst_dev, src, sizeof(double) * (size_t)n, k, s));
}
void copy_out(double *dst, const double *src_dev, int32_t n, cudaStream_t s) {
  const cudaMemcpyKind k = pointer_kind(dst) == PTR_DEVICE ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
  AMG_CUDA(cudaMemcpyAsync(dst, src_dev, sizeof(double) * (size_t)n, k, s));
}

// ||b - A x||^2 into slots[dst] (FP64)
void true_residual(Hierarchy &h, int dst, cudaStream_t s, int64_t &launches) {
  Level &L0 = h.lev[0];
  const int nsg = outer_grid(L0);
  klaunch(k_residual64, nsg, kThreads, s, L0.n, L0.nslices, L0.sptr64, L0.scol64, L0.sval64, h.x, h.b, h.r,
                                        L0.partials + 7 * kRedBlocks);
  klaunch(k_store_sum, 1, kThreads, s, L0.partials + 7 * kRedBlocks, nsg, L0.slots + dst);
  launches += 2;
  AMG_LAUNCH_CHECK();
}

// The cycle trace's counts of second inner steps: cleared before a solve, together
// with the slots that its kernels read (k_begin), and written to mapped pinned words
// before its last synchronisation (k_trace).  One launch each: a launch and a copy per
// level took ~45 us of a call (amg_precond on 77^3: 234 -> 188 us).
struct TraceArgs {
  double *slots[kMaxLevels];
  int L;
};
__global__ void k_begin(TraceArgs a, double tol, double maxit) {
  pdl_wait_and_trigger();
  const int k = threadIdx.x;
  if (k < a.L) a.slots[k][S_TAKEN] = 0.0;
  if (k == 0) {
    a.slots[0][S_TOL] = tol;
    a.slots[0][S_MAXIT] = maxit;
  }
}
__global__ void k_trace(TraceArgs a, volatile int *host) {
  pdl_wait_and_trigger();
  const int k = threadIdx.x;
  if (k < a.L) host[k] = (int)a.slots[k][S_TAKEN];
  __threadfence_system();
}
TraceArgs trace_args(const Hierarchy &h) {
  TraceArgs a{};
  a.L = h.L;
  for (int k = 0; k < h.L; ++k) a.slots[k] = h.lev[k].slots;
  return a;
}
constexpr int kTracePinned = 40;  // of host_pinned: kMaxLevels ints

void trace_reset(Hierarchy &h, double tol, cudaStream_t s) {
  klaunch(k_begin, 1, kMaxLevels, s, trace_args(h), tol, (double)h.p.max_iter);
  AMG_LAUNCH_CHECK();
  h.trace_ok = false;
}

// queue the counts' way to the host; trace_collect reads them after a synchronisation
void trace_queue(Hierarchy &h, cudaStream_t s) {
  int *dev = nullptr;
  AMG_CUDA(cudaHostGetDevicePointer(reinterpret_cast<void **>(&dev), h.host_pinned + kTracePinned, 0));
  klaunch(k_trace, 1, kMaxLevels, s, trace_args(h), (volatile int *)dev);
  AMG_LAUNCH_CHECK();
}

// after a solve with `apps` preconditioner applications: the counts of second
// steps, and from them the visits of every level (Alg. 5 at level m runs the
// cycle of m once, twice when its second step is taken; Alg. 4 recurses once)
void trace_collect(Hierarchy &h, int64_t apps) {
  const volatile int *pin = reinterpret_cast<const volatile int *>(h.host_pinned + kTracePinned);
  for (int k = 0; k < kMaxLevels; ++k) h.visits[k] = h.kcalls[k] = h.second[k] = 0;
  h.visits[0] = apps;
  for (int k = 0; k + 1 < h.L; ++k) {
    const int m = k + 1;
    if (m < h.L - 1 && k < h.p.kcycle_levels && h.tail_t != m) {
      h.kcalls[m] = h.visits[k];
      h.second[m] = pin[m];
      h.visits[m] = h.visits[k] + h.second[m];
    } else {
      h.visits[m] = h.visits[k];
    }
  }
  h.trace_ok = h.tail_t < 0;  // the cluster tail runs its levels without the counters
}

template <class MV, class VT>
int run_solve_t(Hierarchy &h, const double *b, double *x, double tol, int32_t *iters, double *res_hist,
                cudaStream_t s) {
  Level &L0 = h.lev[0];
  const int32_t n = L0.n;
  Engine<MV, VT> eng(h, s);
  int64_t launches = 0;
  int *active = h.it_dev + 1, *restart = h.it_dev + 2;
  copy_in(h.b, b, n, s);
  copy_in(h.x, x, n, s);
  trace_reset(h, tol, s);
  // ||b||^2 and the initial residual
  klaunch(k_dot64, ew_grid(n), kThreads, s, n, h.b, h.b, L0.partials + 6 * kRedBlocks, nullptr);
  klaunch(k_store_sum, 1, kThreads, s, L0.partials + 6 * kRedBlocks, ew_grid(n), L0.slots + S_NB2);
  launches += 2;
  AMG_LAUNCH_CHECK();
  true_residual(h, S_RR, s, launches);
  AMG_CUDA(cudaMemcpyAsync(h.host_pinned, L0.slots, sizeof(double) * kNumSlots, cudaMemcpyDeviceToHost, s));
  AMG_CUDA(cudaStreamSynchronize(s));
  double nb2 = h.host_pinned[S_NB2];
  const double rr0 = h.host_pinned[S_RR];
  const bool zero_b = !(nb2 > 0.0);
  if (zero_b) nb2 = 1.0, klaunch(k_set_slot, 1, 32, s, L0.slots, S_NB2, 1.0);
  double rel = std::sqrt(rr0 / nb2);
  std::vector<double> hist(1, rel);
  int status = AMG_OK;
  int it = 0;
  bool checked = false;  // the slots' true residual is that of the final x
  if (!std::isfinite(rel)) status = AMG_ERR_NAN;
  else if (rel > tol) {
    klaunch(k_set_state, 1, 32, s, h.it_dev, active, restart, h.status_dev, 0, 1, 1, 0);
    AMG_CUDA(cudaMemcpyAsync(h.hist, &hist[0], sizeof(double), cudaMemcpyHostToDevice, s));
    AMG_LAUNCH_CHECK();
    // the state of the iteration in mapped pinned words that its last kernel writes
    // (no copy per iteration): [0] iterations, [4] status
    volatile int *st_host = reinterpret_cast<int *>(h.host_pinned + 32);
    int *st_dev = nullptr;
    AMG_CUDA(cudaHostGetDevicePointer(reinterpret_cast<void **>(&st_dev), h.host_pinned + 32, 0));
    st_host[0] = 0;
    st_host[4] = 0;
    // capture one outer iteration as a graph
    int64_t per_iter = 0;
    if (h.p.use_graph && h.graph_kind != 0) {
      if (h.graph_exec) {
        cudaGraphExecDestroy(h.graph_exec);
        cudaGraphDestroy(h.graph);
        h.graph_exec = nullptr;
      }
      AMG_CUDA(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
      eng.fcg_iteration(active, restart, st_dev);
      AMG_CUDA(cudaStreamEndCapture(s, &h.graph));
      AMG_CUDA(cudaGraphInstantiate(&h.graph_exec, h.graph, 0));
      h.graph_kind = 0;
      h.graph_launches = eng.launches;
      eng.launches = 0;
    }
    per_iter = h.graph_launches;
    eng.input_from_r(h.r, nullptr);
    auto enqueue = [&]() {
      if (h.p.use_graph) {
        AMG_CUDA(cudaGraphLaunch(h.graph_exec, s));
        launches += per_iter;
      } else {
        eng.fcg_iteration(active, restart, st_dev);
      }
    };
    // The next iteration is queued before this one's state is read, so the GPU
    // does not wait for the host between iterations; once an iteration stops
    // (*active = 0) every kernel of the next one returns at once.
    EventPair ep;  // destroyed on every exit, including a throw inside the loop
    cudaEvent_t *evs = ep.e;
    auto launch_iter = [&](int slot) {
      enqueue();
      AMG_CUDA(cudaEventRecord(evs[slot], s));
    };
    int slot = 0;
    launch_iter(slot);
    for (;;) {
      launch_iter(slot ^ 1);
      AMG_CUDA(cudaEventSynchronize(evs[slot]));
      const int dst = st_host[4];
      if (dst == 0) {  // still iterating
        slot ^= 1;
        continue;
      }
      AMG_CUDA(cudaStreamSynchronize(s));  // the queued iteration ran and did nothing
      it = st_host[0];
      if (dst == 1) {  // updated residual meets tol: check the true residual
        true_residual(h, S_TRUE_RR, s, launches);
        AMG_CUDA(cudaMemcpyAsync(h.host_pinned, L0.slots, sizeof(double) * kNumSlots, cudaMemcpyDeviceToHost, s));
        AMG_CUDA(cudaStreamSynchronize(s));
        const double rel_true = std::sqrt(h.host_pinned[S_TRUE_RR] / nb2);
        if (rel_true <= tol || it >= h.p.max_iter) {
          status = rel_true <= tol ? AMG_OK : AMG_ERR_NOT_CONVERGED;
          checked = true;
          break;
        }
        // iterative refinement: restart flexible CG from the true residual
        klaunch(k_set_state, 1, 32, s, h.it_dev, active, restart, h.status_dev, -1, 1, 1, 0);
        eng.input_from_r(h.r, nullptr);
        st_host[4] = 0;  // the stream is idle
        slot = 0;
        launch_iter(slot);
        continue;
      }
      status = dst;
      break;
    }
    AMG_CUDA(cudaStreamSynchronize(s));
    hist.resize((size_t)it + 1);
    if (it > 0)
      AMG_CUDA(cudaMemcpyAsync(&hist[1], h.hist + 1, sizeof(double) * (size_t)it, cudaMemcpyDeviceToHost, s));
  }
  launches += eng.launches;
  if (!checked) true_residual(h, S_TRUE_RR, s, launches);  // final FP64 residual
  AMG_CUDA(cudaMemcpyAsync(h.host_pinned, L0.slots, sizeof(double) * kNumSlots, cudaMemcpyDeviceToHost, s));
  copy_out(x, h.x, n, s);
  trace_queue(h, s);
  AMG_CUDA(cudaStreamSynchronize(s));
  h.info.final_relres = zero_b ? std::sqrt(h.host_pinned[S_TRUE_RR]) : std::sqrt(h.host_pinned[S_TRUE_RR] / nb2);
  trace_collect(h, it);
  h.info.iters = it;
  h.info.status = status;
  h.info.kernel_launches = launches;
  if (iters) *iters = it;
  if (res_hist) std::memcpy(res_hist, hist.data(), sizeof(double) * hist.size());
  return status;
}

// Flexible GMRES(m) (Sec. 2.2, Sec. 4): the Arnoldi basis is orthogonalised by
// classical Gram-Schmidt with one reorthogonalisation (two multi-dot passes), in
// FP64; the K-cycle uses the GMRES variant of Alg. 5.  Every restart starts from
// the true FP64 residual.
template <class MV, class VT>
int run_fgmres_t(Hierarchy &h, const double *b, double *x, double tol, int32_t *iters, double *res_hist,
                 cudaStream_t s) {
  Level &L0 = h.lev[0];
  const int32_t n = L0.n;
  const int m = h.p.restart;
  Engine<MV, VT> eng(h, s);
  int64_t launches = 0;
  int *active = h.it_dev + 1;
  copy_in(h.b, b, n, s);
  copy_in(h.x, x, n, s);
  trace_reset(h, tol, s);
  const int ng = ew_grid(n);
  klaunch(k_dot64, ng, kThreads, s, n, h.b, h.b, L0.partials + 6 * kRedBlocks, nullptr);
  klaunch(k_store_sum, 1, kThreads, s, L0.partials + 6 * kRedBlocks, ng, L0.slots + S_NB2);
  klaunch(k_set_state, 1, 32, s, h.it_dev, active, h.it_dev + 2, h.status_dev, 0, 1, 0, 0);
  launches += 3;
  AMG_LAUNCH_CHECK();
  int it = 0, status = AMG_ERR_NOT_CONVERGED;
  std::vector<double> hist;
  double nb2 = 1.0;
  bool first = true;
  // state of the iteration in mapped pinned words: [0] iterations, [4] status
  volatile int *st_host = reinterpret_cast<int *>(h.host_pinned + 32);
  int *st_dev = nullptr;
  AMG_CUDA(cudaHostGetDevicePointer(reinterpret_cast<void **>(&st_dev), h.host_pinned + 32, 0));
  const FgArgs f = eng.fg_args(st_dev);
  EventPair ep;
  auto launch_step = [&](int slot) {
    if (h.p.use_graph) {
      AMG_CUDA(cudaGraphLaunch(h.graph_exec, s));
      launches += h.graph_launches;
    } else {
      eng.fgmres_step(f);
    }
    AMG_CUDA(cudaEventRecord(ep.e[slot], s));
  };
  for (;;) {
    true_residual(h, S_RR, s, launches);
    AMG_CUDA(cudaMemcpyAsync(h.host_pinned, L0.slots, sizeof(double) * kNumSlots, cudaMemcpyDeviceToHost, s));
    AMG_CUDA(cudaStreamSynchronize(s));
    if (first) {
      nb2 = h.host_pinned[S_NB2];
      if (!(nb2 > 0.0)) {
        nb2 = 1.0;
        klaunch(k_set_slot, 1, 32, s, L0.slots, S_NB2, 1.0);
        ++launches;
      }
      hist.push_back(std::sqrt(h.host_pinned[S_RR] / nb2));
      first = false;
    }
    const double rel = std::sqrt(h.host_pinned[S_RR] / nb2);
    if (!std::isfinite(rel)) { status = AMG_ERR_NAN; break; }
    if (rel <= tol) { status = AMG_OK; break; }
    if (it >= h.p.max_iter) { status = AMG_ERR_NOT_CONVERGED; break; }
    if (h.p.use_graph && h.graph_kind != 1) {  // capture one Arnoldi step
      if (h.graph_exec) {
        cudaGraphExecDestroy(h.graph_exec);
        cudaGraphDestroy(h.graph);
        h.graph_exec = nullptr;
      }
      AMG_CUDA(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
      eng.fgmres_step(f);
      AMG_CUDA(cudaStreamEndCapture(s, &h.graph));
      AMG_CUDA(cudaGraphInstantiate(&h.graph_exec, h.graph, 0));
      h.graph_kind = 1;
      h.graph_launches = eng.launches;
      eng.launches = 0;
    }
    klaunch(k_set_state, 1, 32, s, h.it_dev, active, h.it_dev + 2, h.status_dev, -1, 1, 0, 0);
    klaunch(k_fg_basis<VT, true>, ng, kThreads, s, f, (const double *)h.r, eng.V(h.pre_in), (const VT *)eng.V(L0.wd),
            eng.V(L0.tmp));
    launches += 2;
    AMG_LAUNCH_CHECK();
    // the next step is queued before this one's state is read (within a restart);
    // once a step stops (*active = 0) every kernel of the next one returns at once
    int dst = 0;
    st_host[4] = 0;  // the stream was waited for above
    launch_step(0);
    for (int j = 0; j < m && dst == 0; ++j) {
      if (j + 1 < m) launch_step((j + 1) & 1);
      AMG_CUDA(cudaEventSynchronize(ep.e[j & 1]));
      dst = st_host[4];
    }
    klaunch(k_fg_xupdate, eng.gs_grid(), kThreads, s, f, h.x);
    ++launches;
    AMG_LAUNCH_CHECK();
    AMG_CUDA(cudaStreamSynchronize(s));
    it = st_host[0];
    if (dst == AMG_ERR_NAN) { status = AMG_ERR_NAN; break; }
  }
  hist.resize((size_t)it + 1);
  if (it > 0)
    AMG_CUDA(cudaMemcpyAsync(&hist[1], h.hist + 1, sizeof(double) * (size_t)it, cudaMemcpyDeviceToHost, s));
  launches += eng.launches;
  AMG_CUDA(cudaMemcpyAsync(h.host_pinned, L0.slots, sizeof(double) * kNumSlots, cudaMemcpyDeviceToHost, s));
  copy_out(x, h.x, n, s);
  trace_queue(h, s);
  AMG_CUDA(cudaStreamSynchronize(s));
  h.info.final_relres = std::sqrt(h.host_pinned[S_RR] / nb2);
  trace_collect(h, it);
  h.info.iters = it;
  h.info.status = status;
  h.info.kernel_launches = launches;
  if (iters) *iters = it;
  if (res_hist) std::memcpy(res_hist, hist.data(), sizeof(double) * hist.size());
  return status;
}

__global__ void k_bset(int32_t nsys, const double *bslots, double tol, int *__restrict__ bact, int *__restrict__ bit) {
  pdl_wait_and_trigger();
  // bact[0..nsys) active, bact[nsys] count, bact[nsys+1 ..] restart flags; bit: iters, status
  __shared__ int nact;
  if (threadIdx.x == 0) nact = 0;
  __syncthreads();
  for (int32_t s = threadIdx.x; s < nsys; s += blockDim.x) {
    const double rel = sqrt(bslots[(int64_t)S_RR * nsys + s] / bslots[(int64_t)S_NB2 * nsys + s]);
    const int a = rel > tol ? 1 : 0;
    bact[s] = a;
    bact[nsys + 1 + s] = 1;
    bit[s] = 0;
    bit[nsys + s] = a ? kIterating : AMG_OK;
    if (a) atomicAdd(&nact, 1);
  }
  __syncthreads();
  if (threadIdx.x == 0) bact[nsys] = nact;
}

// restart the systems whose updated residual met tol but whose true residual did not
__global__ void k_brestart(int32_t nsys, const double *bslots, double tol, int max_iter, int *__restrict__ bact,
                           int *__restrict__ bit) {
  pdl_wait_and_trigger();
  __shared__ int nact;
  if (threadIdx.x == 0) nact = 0;
  __syncthreads();
  for (int32_t s = threadIdx.x; s < nsys; s += blockDim.x) {
    const double rel = sqrt(bslots[(int64_t)S_TRUE_RR * nsys + s] / bslots[(int64_t)S_NB2 * nsys + s]);
    int &st = bit[nsys + s];
    if (st == kUpdatedConverged) st = rel <= tol ? AMG_OK : (bit[s] >= max_iter ? AMG_ERR_NOT_CONVERGED : kIterating);
    if (st == kIterating) {
      bact[s] = 1;
      bact[nsys + 1 + s] = 1;
      atomicAdd(&nact, 1);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) bact[nsys] = nact;
}

__global__ void k_fix_zero_norm(int32_t nsys, double *__restrict__ bslots) {
  pdl_wait_and_trigger();
  for (int32_t s = blockIdx.x * blockDim.x + threadIdx.x; s < nsys; s += gridDim.x * blockDim.x)
    if (!(bslots[(int64_t)S_NB2 * nsys + s] > 0.0)) bslots[(int64_t)S_NB2 * nsys + s] = 1.0;
}

template <class MV, class VT>
int run_solve_batch_t(Hierarchy &h, const double *b, double *x, double tol, int32_t *iters, double *relres,
                      cudaStream_t s) {
  Level &L0 = h.lev[0];
  const int32_t n = L0.n, ns = h.nsys;
  Engine<MV, VT> eng(h, s);
  Engine<double, double> e64(h, s);
  int64_t launches = 0;
  copy_in(h.b, b, n, s);
  copy_in(h.x, x, n, s);
  const double *nil = nullptr;
  e64.segdot<1>(e64.seg_args(0, BF_STORE, false, S_NB2), (const double *)h.b, (const double *)h.b, nil, nil, nullptr);
  klaunch(k_fix_zero_norm, grid_for(ns, kThreads, 152), kThreads, s, ns, L0.bslots);
  auto residual = [&](int slot) {  // r = b - A x and ||r||^2 of every system
    klaunch(k_residual64, outer_grid(L0), kThreads, s, n, L0.nslices, (const int64_t *)L0.sptr64,
            (const int32_t *)L0.scol64, (const double *)L0.sval64, (const double *)h.x, (const double *)h.b, h.r,
            L0.partials + 7 * kRedBlocks);
    e64.segdot<1>(e64.seg_args(0, BF_STORE, false, slot), (const double *)h.r, (const double *)h.r, nil, nil, nullptr);
    ++launches;
  };
  residual(S_RR);
  klaunch(k_bset, 1, 1024, s, ns, (const double *)L0.bslots, tol, h.bactive, h.bit);
  AMG_CUDA(cudaMemsetAsync(h.it_dev, 0, sizeof(int), s));
  launches += 2;
  AMG_LAUNCH_CHECK();
  // number of systems still iterating, in a mapped pinned word that a pass's last kernel writes
  volatile int *active = reinterpret_cast<int *>(h.host_pinned + 32);
  int *active_dev = nullptr;
  AMG_CUDA(cudaHostGetDevicePointer(reinterpret_cast<void **>(&active_dev), h.host_pinned + 32, 0));
  // capture one iteration of all systems
  if (h.graph_exec) {
    cudaGraphExecDestroy(h.graph_exec);
    cudaGraphDestroy(h.graph);
    h.graph_exec = nullptr;
  }
  if (h.p.use_graph) {
    AMG_CUDA(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
    eng.fcg_iteration_batched(tol, active_dev);
    AMG_CUDA(cudaStreamEndCapture(s, &h.graph));
    AMG_CUDA(cudaGraphInstantiate(&h.graph_exec, h.graph, 0));
    h.graph_launches = eng.launches;
    eng.launches = 0;
    h.graph_kind = -1;  // not the single-system iteration
  }
  int *pin = reinterpret_cast<int *>(h.host_pinned + 36);
  EventPair ep;
  int rounds = 0;
  auto launch_pass = [&](int slot) {
    if (h.p.use_graph) {
      AMG_CUDA(cudaGraphLaunch(h.graph_exec, s));
      launches += h.graph_launches;
    } else {
      eng.fcg_iteration_batched(tol, active_dev);
    }
    AMG_CUDA(cudaEventRecord(ep.e[slot], s));
    ++rounds;
  };
  for (;;) {
    AMG_CUDA(cudaMemcpyAsync(pin, h.bactive + ns, sizeof(int), cudaMemcpyDeviceToHost, s));
    AMG_CUDA(cudaStreamSynchronize(s));
    if (pin[0] > 0 && rounds < 100 * h.p.max_iter) {
      eng.input_from_r(h.r, nullptr);
      // the next pass is queued before this one's count is read (a pass after the
      // last system stopped changes nothing)
      *active = pin[0];
      int slot = 0;
      launch_pass(slot);
      while (rounds < 100 * h.p.max_iter) {
        launch_pass(slot ^ 1);
        AMG_CUDA(cudaEventSynchronize(ep.e[slot]));
        if (*active == 0) break;
        slot ^= 1;
      }
    }
    // every system stopped: check the true residuals, restart those that miss tol
    residual(S_TRUE_RR);
    klaunch(k_brestart, 1, 1024, s, ns, (const double *)L0.bslots, tol, h.p.max_iter, h.bactive, h.bit);
    ++launches;
    AMG_CUDA(cudaMemcpyAsync(pin, h.bactive + ns, sizeof(int), cudaMemcpyDeviceToHost, s));
    AMG_CUDA(cudaStreamSynchronize(s));
    if (pin[0] == 0 || rounds >= 100 * h.p.max_iter) break;
  }
  launches += eng.launches + e64.launches;
  std::vector<int> bit(2 * ns);
  std::vector<double> sl((size_t)kNumSlots * ns);
  AMG_CUDA(cudaMemcpyAsync(bit.data(), h.bit, sizeof(int) * 2 * ns, cudaMemcpyDeviceToHost, s));
  AMG_CUDA(cudaMemcpyAsync(sl.data(), L0.bslots, sizeof(double) * kNumSlots * ns, cudaMemcpyDeviceToHost, s));
  copy_out(x, h.x, n, s);
  AMG_CUDA(cudaStreamSynchronize(s));
  int status = AMG_OK, maxit = 0;
  double worst = 0.0;
  for (int32_t q = 0; q < ns; ++q) {
    const double rel = std::sqrt(sl[(size_t)S_TRUE_RR * ns + q] / sl[(size_t)S_NB2 * ns + q]);
    if (iters) iters[q] = bit[q];
    if (relres) relres[q] = rel;
    maxit = std::max(maxit, bit[q]);
    worst = std::max(worst, rel);
    const int st = bit[ns + q];
    if (st != AMG_OK && status == AMG_OK) status = st < 0 ? st : AMG_ERR_NOT_CONVERGED;
  }
  h.info.iters = maxit;
  h.info.final_relres = worst;
  h.info.status = status;
  h.info.kernel_launches = launches;
  return status;
}

// Row tiles of level L for the per-system inner products, every tile in one system.
// `seg_tile` rows suit a level that fills the GPU with kSegWave of them; smaller levels
// take smaller tiles (two rows a thread at least) so that their FP64 work meets more
// SMs, larger ones up to four times larger tiles with fewer sums to finish.
constexpr int32_t kSegWave = 152 * 4;
int32_t tile_rows(const Level &L, int32_t seg_tile) {
  const int64_t fit = (int64_t)L.n * seg_tile / ((int64_t)kSegWave * 2048);
  return (int32_t)std::max<int64_t>(2 * kSegThreads, std::min<int64_t>(4 * (int64_t)seg_tile, (fit + 255) / 256 * 256));
}
void build_tiles(Hierarchy &h, Level &L, int32_t seg_tile, cudaStream_t s) {
  const int32_t ns = h.nsys, tile = tile_rows(L, seg_tile);
  std::vector<int32_t> trow, tsys, stile(ns + 1, 0);
  for (int32_t q = 0; q < ns; ++q) {
    stile[q] = (int32_t)trow.size();
    for (int32_t r = L.sys_off_host[q]; r < L.sys_off_host[q + 1]; r += tile) {
      trow.push_back(r);
      tsys.push_back(q);
    }
  }
  stile[ns] = (int32_t)trow.size();
  L.ntiles = (int32_t)trow.size();
  L.seg_tile = seg_tile;
  trow.push_back(L.n);
  L.tile_row = h.arena.get<int32_t>(trow.size());
  L.tile_sys = h.arena.get<int32_t>(tsys.size());
  L.sys_tile = h.arena.get<int32_t>(ns + 1);
  L.tpart = h.arena.get<double>(3 * (size_t)L.ntiles + 1);
  AMG_CUDA(cudaMemcpyAsync(L.tile_row, trow.data(), sizeof(int32_t) * trow.size(), cudaMemcpyHostToDevice, s));
  AMG_CUDA(cudaMemcpyAsync(L.tile_sys, tsys.data(), sizeof(int32_t) * tsys.size(), cudaMemcpyHostToDevice, s));
  AMG_CUDA(cudaMemcpyAsync(L.sys_tile, stile.data(), sizeof(int32_t) * (ns + 1), cudaMemcpyHostToDevice, s));
  AMG_CUDA(cudaStreamSynchronize(s));  // trow, tsys and stile leave scope
}

// per-level system map, row tiles and per-system scalars of a batch
void prepare_batched(Hierarchy &h, cudaStream_t s) {
  const int32_t ns = h.nsys;
  constexpr int32_t kTile = 2048;
  h.bit = h.arena.get<int>(2 * (size_t)ns);
  h.bactive = h.arena.get<int>(2 * (size_t)ns + 2);
  {  // before the first solve (amg_precond, the autotuner) every system counts as iterating
    const std::vector<int> one((size_t)ns + 1, 1);
    AMG_CUDA(cudaMemcpyAsync(h.bactive, one.data(), sizeof(int) * (ns + 1), cudaMemcpyHostToDevice, s));
    AMG_CUDA(cudaStreamSynchronize(s));
  }
  for (int k = 0; k < h.L; ++k) {
    Level &L = h.lev[k];
    L.sys_of = h.arena.get<int32_t>((size_t)L.n + 1);
    klaunch(k_sys_of, ew_grid(L.n), kThreads, s, L.n, ns, (const int32_t *)L.sys_off, L.sys_of);
    L.slive = h.arena.get<unsigned char>((size_t)L.nslices + 1);
    AMG_CUDA(cudaMemsetAsync(L.slive, 1, (size_t)L.nslices + 1, s));
    build_tiles(h, L, kTile, s);
    L.bslots = h.arena.get<double>((size_t)kNumSlots * ns);
    L.bflag = h.arena.get<int>((size_t)ns + 1);
    L.bticket = h.arena.get<int>((size_t)ns);
    AMG_CUDA(cudaMemsetAsync(L.bticket, 0, sizeof(int) * ns, s));
    AMG_CUDA(cudaMemsetAsync(L.bslots, 0, sizeof(double) * kNumSlots * ns, s));
    AMG_CUDA(cudaMemsetAsync(L.bflag, 0, sizeof(int) * (ns + 1), s));
  }
  AMG_LAUNCH_CHECK();
}

// Autotuner of the launch shapes (setup time).  For every level the SpMV is
// timed with CUDA events over candidate grid sizes (multiples of the 152 SMs up
// to one warp per slice) and the smallest grid within 3 % of the fastest is
// kept, for the launches that fuse inner products among the grids within one
// wave of their kernel; for a batch, the row tile of the per-system inner products is chosen
// the same way.  The shapes change the grouping of partial sums only.
template <class MV, class VT>
void autotune_t(Hierarchy &h, cudaStream_t s) {
  Engine<MV, VT> eng(h, s);
  cudaEvent_t e0, e1;
  AMG_CUDA(cudaEventCreate(&e0));
  AMG_CUDA(cudaEventCreate(&e1));
  auto time_it = [&](auto &&launch) {
    for (int r = 0; r < 2; ++r) launch();
    AMG_CUDA(cudaEventRecord(e0, s));
    constexpr int kReps = 5;
    for (int r = 0; r < kReps; ++r) launch();
    AMG_CUDA(cudaEventRecord(e1, s));
    AMG_CUDA(cudaEventSynchronize(e1));
    float ms = 0.f;
    AMG_CUDA(cudaEventElapsedTime(&ms, e0, e1));
    return ms / kReps;
  };
  auto pick = [](const std::vector<std::pair<int, float>> &t) {  // smallest within 3 % of the best
    float best = t[0].second;
    for (auto &c : t) best = std::min(best, c.second);
    for (auto &c : t)
      if (c.second <= 1.03f * best) return c.first;
    return t[0].first;
  };
  try {
    for (int k = 0; k < h.L; ++k) {
      Level &L = h.lev[k];
      DevBuf<VT> x((size_t)L.n + 1), y((size_t)L.n + 1);
      AMG_CUDA(cudaMemsetAsync(x.p, 0, sizeof(VT) * (L.n + 1), s));
      // the plain product at each grid; launches with fused inner products take
      // the best grid within one wave of theirs.  The split-row kernel of
      // the small levels covers its slices in one pass and has no grid to choose.
      const int gfull = full_plain_grid(L);
      std::vector<std::pair<int, float>> t, tr;
      if (L.split_log >= 0) tr = t = {{L.sell_blocks, 0.f}};
      else for (int g : {152, 304, 608, 912, 1216, 2432, 4864, 1 << 30}) {
        const int gg = std::min(g, gfull);
        if (!t.empty() && t.back().first == gg) continue;
        L.sell_plain_blocks = gg;
        const SellArgs<VT> a = eng.sell_args(k, x.p, y.p, nullptr);
        t.push_back({gg, time_it([&] { eng.template sell<E_Y>(a, k); })});
        if (gg <= dot_wave<VT>()) tr.push_back(t.back());
      }
      L.sell_plain_blocks = pick(t);
      L.sell_blocks = pick(tr);
      if (h.batched && k < h.L - 1) {
        std::vector<std::pair<int, float>> tt;
        for (int tile : {1024, 2048, 4096, 8192}) {
          if (!tt.empty() && tile_rows(L, tile) == tile_rows(L, tt.back().first)) continue;  // the same tiles
          build_tiles(h, L, tile, s);
          tt.push_back({tile, time_it([&] {
                          const VT *nil = nullptr;
                          eng.template segdot<2>(eng.seg_args(k, BF_STORE, false, S_RHO1), (const VT *)x.p,
                                                 (const VT *)y.p, (const VT *)y.p, nil, nullptr);
                        })});
        }
        build_tiles(h, L, pick(tt), s);
      }
    }
  } catch (...) {
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    throw;
  }
  AMG_CUDA(cudaEventDestroy(e0));
  AMG_CUDA(cudaEventDestroy(e1));
}

template <class MV, class VT>
void run_precond_t(Hierarchy &h, const double *b, double *x, cudaStream_t s) {
  Engine<MV, VT> eng(h, s);
  const int32_t n = h.lev[0].n;
  if (!h.batched) trace_reset(h, 0.0, s);
  else {  // every system takes part, also after a solve that stopped them
    AMG_CUDA(cudaMemsetAsync(h.bactive, 1, sizeof(int) * h.nsys, s));
    for (int k = 0; k < h.L; ++k) AMG_CUDA(cudaMemsetAsync(h.lev[k].slive, 1, (size_t)h.lev[k].nslices + 1, s));
  }
  copy_in(h.r, b, n, s);
  eng.precond(h.r, h.z, nullptr);
  copy_out(x, h.z, n, s);
  if (!h.batched) trace_queue(h, s);
  AMG_CUDA(cudaStreamSynchronize(s));
  if (!h.batched) trace_collect(h, 1);
  h.info.kernel_launches = eng.launches;
}

template <class MV, class VT>
void run_spmv_t(Hierarchy &h, int k, const void *x, void *y, cudaStream_t s) {
  Engine<MV, VT> eng(h, s);
  eng.gate = false;
  SellArgs<VT> a = eng.sell_args(k, static_cast<const VT *>(x), static_cast<VT *>(y), nullptr);
  eng.template sell<E_Y>(a, k);
}

}  // namespace

#define AMG_DISPATCH(prec, CALL)                                   \
  switch (prec) {                                                  \
    case AMG_PREC_F64: { using MV = double; using VT = double; CALL; break; } \
    case AMG_PREC_F32: { using MV = float; using VT = float; CALL; break; }   \
    default: { using MV = __nv_bfloat16; using VT = float; CALL; break; }     \
  }

void set_poly(Hierarchy &h, int level, const double *coef, cudaStream_t s) {
  Level &L = h.lev[level];
  if (!coef) {  // back to damped Jacobi on this level (the buffer stays for a later set)
    L.poly_off = true;
    configure_tail(h, s);
    h.graph_kind = -1;
    return;
  }
  L.poly_off = false;
  const size_t cnt = (size_t)L.n * 3;
  DevBuf<double> tmp(cnt);
  const cudaMemcpyKind kind = pointer_kind(coef) == PTR_DEVICE ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
  AMG_CUDA(cudaMemcpyAsync(tmp.p, coef, sizeof(double) * cnt, kind, s));
  if (h.p.precision == AMG_PREC_F64) {
    if (!L.poly) L.poly = h.arena.get<double>(cnt);
    AMG_CUDA(cudaMemcpyAsync(L.poly, tmp.p, sizeof(double) * cnt, cudaMemcpyDeviceToDevice, s));
  } else {
    if (!L.poly) L.poly = h.arena.get<float>(cnt);
    klaunch(k_copy_cast<float>, ew_grid((int64_t)cnt), kThreads, s, (int32_t)cnt, tmp.p, (float *)L.poly);
    AMG_LAUNCH_CHECK();
  }
  AMG_CUDA(cudaStreamSynchronize(s));
  configure_tail(h, s);
  h.graph_kind = -1;  // the captured iteration no longer matches: capture again
}

void make_row_data(Hierarchy &h, Level &L, const double *diag, cudaStream_t s) {
  if (h.p.precision == AMG_PREC_F64)
    make_row_data_t<double>(h, L, diag, s);
  else
    make_row_data_t<float>(h, L, diag, s);
}

void prepare_solve(Hierarchy &h, cudaStream_t s) {
  AMG_DISPATCH(h.p.precision, (prepare_t<MV, VT>(h, s)));
}

int run_solve_batch(Hierarchy &h, const double *b, double *x, double tol, int32_t *iters, double *relres,
                    cudaStream_t s) {
  int rc = 0;
  AMG_DISPATCH(h.p.precision, (rc = run_solve_batch_t<MV, VT>(h, b, x, tol, iters, relres, s)));
  return rc;
}

int run_solve(Hierarchy &h, const double *b, double *x, double tol, int32_t *iters, double *res_hist,
              cudaStream_t s) {
  int rc = 0;
  if (h.p.outer == 1) {
    AMG_DISPATCH(h.p.precision, (rc = run_fgmres_t<MV, VT>(h, b, x, tol, iters, res_hist, s)));
  } else {
    AMG_DISPATCH(h.p.precision, (rc = run_solve_t<MV, VT>(h, b, x, tol, iters, res_hist, s)));
  }
  return rc;
}

void run_precond(Hierarchy &h, const double *b, double *x, cudaStream_t s) {
  AMG_DISPATCH(h.p.precision, (run_precond_t<MV, VT>(h, b, x, s)));
}

void run_spmv(Hierarchy &h, int level, const void *x, void *y, cudaStream_t s) {
  AMG_DISPATCH(h.p.precision, (run_spmv_t<MV, VT>(h, level, x, y, s)));
}

}  // namespace amg
