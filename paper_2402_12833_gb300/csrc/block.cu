// Tall-skinny block kernels of the MPCG step (Section 2.2, Algorithm 1):
//   * the Gram blocks W_j = (A P_j)^T Z against the stored window,
//   * the A-orthogonalisation P = Z - sum_j P_j beta_j,
//   * the new Gram matrix sym(P^T A P) and the right-hand side P^T r, once
//     the block SpMM has formed A P,
//   * the update x += P alpha, r -= A P alpha with ||r||^2.
//
// These kernels stream the padded arrays (pads are zero, so they take part
// harmlessly) in 16-byte vectors: 4 floats or 2 doubles per thread and step;
// blockIdx.y selects the problem of a batch (see common.cuh).
// Reductions are deterministic: every block writes its partial sums
// (value-major, fixed block count) and one small kernel adds them in a fixed
// order.  In the FP32 path each thread sums at most 64 points in FP32 and the
// warp adds its 32 lanes in FP32; everything above the warp is FP64.
#include "kernels.cuh"
#include "tune.h"
#include "vec.cuh"

namespace mpcg {

namespace {

// Window Gram W_jj[a][b] = sum_i AP_slot(jj)[a][i] Z[b][i].  The cnt * C rows
// (jj, a) are dealt out in tasks of kGramRows<T, C> rows; a warp keeps the
// task's rows x C partial sums in registers and walks the points in chunks of
// 32 W, so a point's Z values are loaded once per task instead of once per
// window block and the warps of a block, which hold different tasks of the
// same chunk, share them in L1.  The row count is set by the register file:
// with all C rows of a block per thread the C = 9 instance spilled 568 bytes
// at 80 registers and ran at a third of the HBM rate (1025^2, m = 5: 102 us
// for 227 MB, now 51 us); a task holds at most 45 FP32 or 24 FP64 sums
// (5 FP64 rows instead of 4 at C = 5: 13.0 instead of 12.8 ms per 65^2 solve;
// 4 double-word rows instead of 5 at C = 6: 235 instead of 213 us at 129^3).
template <typename T, int C>
constexpr int kGramRows = sizeof(T) == 4 ? (45 / C < 6 ? 45 / C : 6)
                                         : (kIsDw<T> ? (30 / C < 8 ? 30 / C : 8) : (24 / C < 8 ? 24 / C : 8));
// points per lane and step: one 16-byte vector in FP32 (8 bytes from C = 10 on,
// registers), one value in FP64 and double-word (small grids then spread over
// more warps, and their arithmetic, not their loads, is the bound)
template <typename T, int C>
constexpr int kGramW = sizeof(T) == 4 ? (C < 10 ? 4 : 2) : 1;
// steps before the lane's partial sums leave it (at most 64 points)
template <typename T, int C>
constexpr int kGramSteps = sizeof(T) == 4 ? 64 / kGramW<T, C> : 32;

// The walkers of a task: the warps of the launch shared out over the tasks
// present (cnt blocks in the window), at most one per chunk or partial slot.
__device__ __forceinline__ int gram_walkers(int cnt, int C, int rows, int nwarps, int slots) {
  const int ntask = (cnt * C + rows - 1) / rows;
  const int w = nwarps / ntask;
  return w < slots ? w : slots;
}

template <typename T, int C>
__global__ void __launch_bounds__(kBlock, 2) k_gram_window(GridDesc g, Window<T> win, const T* __restrict__ Z,
                                                           double* part, int nwarps, int slots,
                                                           const DevState* state) {
  const int pb = blockIdx.y;
  state += pb;
  if (state->done) return;
  const int cnt = state->count;
  if (cnt == 0) return;
  constexpr int RB = kGramRows<T, C>, W = kGramW<T, C>, NV = RB * C;
  const int m = state->m, newest = state->newest;
  const int lane = threadIdx.x & 31;
  const int wid = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nrows = cnt * C, ntask = (nrows + RB - 1) / RB;
  const int walkers = gram_walkers(cnt, C, RB, nwarps, slots);
  const int task = wid % ntask, walker = wid / ntask;
  if (walker >= walkers) return;
  const long long bo = (long long)pb * g.len + g.G;
  const T* row[RB];
#pragma unroll
  for (int k = 0; k < RB; ++k) {
    int r = task * RB + k;
    if (r >= nrows) r = nrows - 1;   // the last task repeats its last row (not stored)
    const int jj = r / C;
    row[k] = win.AP[(newest - jj + m) % m] + bo + (long long)(r - jj * C) * g.cp;
  }
  const T* Zb = Z + bo;
  const long long steps = (g.npts + 32 * W - 1) / (32 * W);
  double hold[rs_count(NV, 5)];
#pragma unroll
  for (int i = 0; i < rs_count(NV, 5); ++i) hold[i] = 0.0;
  int base = 0, nvalid = NV;
  for (long long q = walker; q < steps;) {
    typename Acc<T>::type acc[NV];
#pragma unroll
    for (int e = 0; e < NV; ++e) acc[e] = Acc<T>::of(T(0));
    for (int n = 0; n < kGramSteps<T, C> && q < steps; ++n, q += walkers) {
      const long long i = (q * 32 + lane) * W;
      if (i >= g.npts) continue;
      T z[C][W];
#pragma unroll
      for (int b = 0; b < C; ++b) VecN<T, W>::load_keep(Zb + (long long)b * g.cp + i, z[b]);
      T ap[RB][W];
#pragma unroll
      for (int k = 0; k < RB; ++k) VecN<T, W>::load(row[k] + i, ap[k]);
#pragma unroll
      for (int k = 0; k < RB; ++k)
#pragma unroll
        for (int b = 0; b < C; ++b)
#pragma unroll
          for (int w = 0; w < W; ++w) mac(acc[k * C + b], ap[k][w], z[b][w]);
    }
    // the warp's sums in T, above the warp in FP64
    T v[NV];
#pragma unroll
    for (int e = 0; e < NV; ++e) v[e] = Acc<T>::value(acc[e]);
    warp_reduce_scatter<T, NV>(v, base, nvalid, lane);
#pragma unroll
    for (int i = 0; i < rs_count(NV, 5); ++i) hold[i] += (double)v[i];
  }
  double* pj = part + (long long)pb * m * C * C * slots;
#pragma unroll
  for (int i = 0; i < rs_count(NV, 5); ++i) {
    const int e = task * NV + base + i;   // = (jj C + a) C + b
    if (i < nvalid && e < nrows * C) pj[(long long)e * slots + walker] = hold[i];
  }
}

// P = Z - sum_j P_j beta_j into the next ring slot.  A P of the new block is
// the block SpMM of P itself (not the recurrence A Z - sum_j A P_j beta_j):
// this kernel then reads the window's P_j only and no A Z exists, (m + 2) C
// words a point at a full window instead of (2 m + 4) C + 1 (129^3, FP32,
// C = 6, four blocks in the window: 102 -> 43 us; 1025^2, C = 9, m = 5: 133 ->
// 49 us).
// Bound by HBM in FP32, by the FP64 and FP32 pipes in FP64 and double-word.
template <typename T, int C>
__global__ void __launch_bounds__(kBlock) k_orth_update(GridDesc g, Window<T> win, const T* __restrict__ Z,
                                                        const DevState* state) {
  const int pb = blockIdx.y;
  state += pb;
  if (state->done) return;
  const int cnt = state->count, m = state->m, newest = state->newest;
  const long long bo = (long long)pb * g.len + g.G;
  constexpr int CP = sizeof(T) == 4 ? (C + 3) / 4 * 4 : (C + 1) / 2 * 2;   // rows start on 16 bytes
  __shared__ __align__(16) T nbeta[kMaxWindow][C][CP];                      // -beta
  __shared__ const T* pp[kMaxWindow];
  for (int e = threadIdx.x; e < cnt * C * C; e += blockDim.x) {
    const int jj = e / (C * C), a = (e / C) % C, b = e % C;
    nbeta[jj][a][b] = -(T)state->beta[jj][a][b];
  }
  for (int jj = threadIdx.x; jj < cnt; jj += blockDim.x) pp[jj] = win.P[(newest - jj + m) % m] + bo;
  __syncthreads();
  T* Pn = win.P[(newest + 1) % m] + bo;
  const T* Zb = Z + bo;
  constexpr int W = sizeof(T) == 4 ? (C < 10 ? 4 : 2) : 1;
  using A = typename Acc<T>::type;
  const long long ngroups = g.npts / W;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < ngroups;
       q += (long long)gridDim.x * blockDim.x) {
    const long long i = q * W;
    A pacc[C][W];
#pragma unroll
    for (int b = 0; b < C; ++b) {
      T zv[W];
      VecN<T, W>::load(Zb + (long long)b * g.cp + i, zv);
#pragma unroll
      for (int w = 0; w < W; ++w) pacc[b][w] = Acc<T>::of(zv[w]);
    }
    for (int jj = 0; jj < cnt; ++jj) {
      const T* pj = pp[jj] + i;
      T pa[C][W];
#pragma unroll
      for (int a = 0; a < C; ++a) VecN<T, W>::load(pj + (long long)a * g.cp, pa[a]);
#pragma unroll
      for (int a = 0; a < C; ++a)
#pragma unroll
        for (int b = 0; b < C; ++b) {
          const T bt = nbeta[jj][a][b];
#pragma unroll
          for (int w = 0; w < W; ++w) mac(pacc[b][w], pa[a][w], bt);
        }
    }
#pragma unroll
    for (int b = 0; b < C; ++b) {
      T p[W];
#pragma unroll
      for (int w = 0; w < W; ++w) p[w] = Acc<T>::value(pacc[b][w]);
      VecN<T, W>::store(Pn + (long long)b * g.cp + i, p);
    }
  }
}

// Gram partials of the new block: the upper triangle of G = P^T A P and
// g = P^T r.  A P is the product of A with the very P read here, so p_a^T A p_b
// and p_b^T A p_a differ by the rounding of one product and one of them serves
// for both (the recurrence A Z - sum_j A P_j beta_j drifts from A P and had to
// be symmetrised): 27 instead of 48 multiply-adds a point at C = 6, which the
// FP64 pipe pays for in full (97^3, FP64: 65.5 -> 38 us).
template <typename T, int C>
__global__ void __launch_bounds__(kBlock, (sizeof(T) == 4 || C <= 7) ? 2 : 1)
    k_block_gram(GridDesc g, Window<T> win, const T* __restrict__ r, double* part, const DevState* state) {
  const int pb = blockIdx.y;
  state += pb;
  if (state->done) return;
  const int ns = (state->newest + 1) % state->m;
  const long long bo = (long long)pb * g.len + g.G;
  const T* Pn = win.P[ns] + bo;
  const T* APn = win.AP[ns] + bo;
  const T* rb = r + bo;
  constexpr int W = sizeof(T) == 4 ? (C <= 7 ? 4 : (C <= 9 ? 2 : 1)) : 1;
  constexpr int NG = C * (C + 1) / 2;
  typename Acc<T>::type acc[NG + C];
#pragma unroll
  for (int i = 0; i < NG + C; ++i) acc[i] = Acc<T>::of(T(0));
  const long long ngroups = g.npts / W;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < ngroups;
       q += (long long)gridDim.x * blockDim.x) {
    const long long i = q * W;
    T p[C][W], ap[C][W], rv[W];
    VecN<T, W>::load_keep(rb + i, rv);
#pragma unroll
    for (int a = 0; a < C; ++a) {
      VecN<T, W>::load_keep(Pn + (long long)a * g.cp + i, p[a]);
      VecN<T, W>::load_keep(APn + (long long)a * g.cp + i, ap[a]);
    }
    int k = 0;
#pragma unroll
    for (int a = 0; a < C; ++a) {
#pragma unroll
      for (int b = a; b < C; ++b) {
#pragma unroll
        for (int w = 0; w < W; ++w) mac(acc[k], p[a][w], ap[b][w]);
        ++k;
      }
#pragma unroll
      for (int w = 0; w < W; ++w) mac(acc[NG + a], p[a][w], rv[w]);
    }
  }
  T fin[NG + C];
#pragma unroll
  for (int i = 0; i < NG + C; ++i) fin[i] = Acc<T>::value(acc[i]);
  block_sum_store<T, NG + C>(fin, part + (long long)pb * (NG + C) * gridDim.x, gridDim.x, blockIdx.x);
}

template <typename T, int C>
__global__ void __launch_bounds__(kBlock) k_update_xr(GridDesc g, Window<T> win, T* __restrict__ x,
                                                      T* __restrict__ r, double* part, const DevState* state) {
  const int pb = blockIdx.y;
  state += pb;
  if (state->done) return;
  const int newest = state->newest;
  const long long bo = (long long)pb * g.len + g.G;
  const T* P = win.P[newest] + bo;
  const T* AP = win.AP[newest] + bo;
  T* xb = x + bo;
  T* rb = r + bo;
  T al[C];
#pragma unroll
  for (int a = 0; a < C; ++a) al[a] = (T)state->alpha[a];
  constexpr int W = Vec<T>::W;
  T acc[1] = {0};
  const long long ngroups = g.npts / W;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < ngroups;
       q += (long long)gridDim.x * blockDim.x) {
    const long long i = q * W;
    T px[W] = {}, apx[W] = {};
#pragma unroll
    for (int a = 0; a < C; ++a) {
      T pv[W], av[W];
      Vec<T>::load(P + (long long)a * g.cp + i, pv);
      Vec<T>::load(AP + (long long)a * g.cp + i, av);
#pragma unroll
      for (int w = 0; w < W; ++w) {
        px[w] = fma(pv[w], al[a], px[w]);
        apx[w] = fma(av[w], al[a], apx[w]);
      }
    }
    T xv[W], rv[W];
    Vec<T>::load_keep(xb + i, xv);
    Vec<T>::load_keep(rb + i, rv);
#pragma unroll
    for (int w = 0; w < W; ++w) {
      xv[w] += px[w];
      rv[w] -= apx[w];
      acc[0] = fma(rv[w], rv[w], acc[0]);
    }
    Vec<T>::store(xb + i, xv);
    Vec<T>::store(rb + i, rv);
  }
  block_sum_store<T, 1>(acc, part + (long long)pb * gridDim.x, gridDim.x, blockIdx.x);
}

// Mixed-precision refinement, start of an inner FP32 solve: with the outer
// residual r64 and |r64|^2 in nrm2[2p], b32 = r64 / |r64| (zero for an
// inactive problem, whose inner solve then stops at once).  The inner iterate
// starts at zero, so the inner residual is b32 itself: it is written to r32
// as well, with the block partials of |r32|^2 and |b32|^2 that the residual
// kernel would have produced (value-major, stride gridDim.x).
__global__ void __launch_bounds__(kBlock) k_start_inner(GridDesc g, const double* __restrict__ r64,
                                                        const double* __restrict__ nrm2,
                                                        const int* __restrict__ active, float* __restrict__ b32,
                                                        float* __restrict__ r32, double* part) {
  const int pb = blockIdx.y;
  const bool on = !active || active[pb];
  const double inv = on && nrm2[2 * pb] > 0.0 ? 1.0 / sqrt(nrm2[2 * pb]) : 0.0;
  const long long o = (long long)pb * g.len + g.G;
  float sums[2] = {0.f, 0.f};
  const long long ngroups = g.npts / 4;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < ngroups;
       q += (long long)gridDim.x * blockDim.x) {
    const long long i = o + q * 4;
    double lo[2], hi[2];
    Vec<double>::load(r64 + i, lo);
    Vec<double>::load(r64 + i + 2, hi);
    const float v[4] = {(float)(lo[0] * inv), (float)(lo[1] * inv), (float)(hi[0] * inv), (float)(hi[1] * inv)};
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      sums[0] = fmaf(v[w], v[w], sums[0]);
      sums[1] = fmaf(v[w], v[w], sums[1]);
    }
    Vec<float>::store(b32 + i, v);
    Vec<float>::store(r32 + i, v);
  }
  block_sum_store<float, 2>(sums, part + (long long)pb * 2 * gridDim.x, gridDim.x, blockIdx.x);
}

// End of an inner solve: x64 += |r64| d32 (nrm2[2p] = |r64|^2).
__global__ void __launch_bounds__(kBlock) k_axpy_mixed(GridDesc g, double* __restrict__ x,
                                                       const float* __restrict__ d, const double* __restrict__ nrm2,
                                                       int* xnz) {
  const int pb = blockIdx.y;
  const double sc = sqrt(nrm2[2 * pb]);
  if (xnz && blockIdx.x == 0 && threadIdx.x == 0) xnz[pb] = 1;   // x may be nonzero from here on
  const long long o = (long long)pb * g.len + g.G;
  const long long ngroups = g.npts / 4;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < ngroups;
       q += (long long)gridDim.x * blockDim.x) {
    const long long i = o + q * 4;
    float dv[4];
    double lo[2], hi[2];
    Vec<float>::load(d + i, dv);
    Vec<double>::load_keep(x + i, lo);
    Vec<double>::load_keep(x + i + 2, hi);
    lo[0] = fma(sc, (double)dv[0], lo[0]);
    lo[1] = fma(sc, (double)dv[1], lo[1]);
    hi[0] = fma(sc, (double)dv[2], hi[0]);
    hi[1] = fma(sc, (double)dv[3], hi[1]);
    Vec<double>::store(x + i, lo);
    Vec<double>::store(x + i + 2, hi);
  }
}

}  // namespace

#define MPCG_C_SWITCH(C, BODY)                                                                   \
  switch (C) {                                                                                   \
    case 1: { constexpr int CC = 1; BODY; } break;                                               \
    case 2: { constexpr int CC = 2; BODY; } break;                                               \
    case 3: { constexpr int CC = 3; BODY; } break;                                               \
    case 4: { constexpr int CC = 4; BODY; } break;                                               \
    case 5: { constexpr int CC = 5; BODY; } break;                                               \
    case 6: { constexpr int CC = 6; BODY; } break;                                               \
    case 7: { constexpr int CC = 7; BODY; } break;                                               \
    case 8: { constexpr int CC = 8; BODY; } break;                                               \
    case 9: { constexpr int CC = 9; BODY; } break;                                               \
    case 10: { constexpr int CC = 10; BODY; } break;                                             \
    case 11: { constexpr int CC = 11; BODY; } break;                                             \
    case 12: { constexpr int CC = 12; BODY; } break;                                             \
    default: break;                                                                              \
  }

// Threads per block for `items` elementwise work items: 256, or as few as a
// warp where 256 would leave SMs without a block.  The FP64 pipe takes a warp
// instruction every 64 cycles, so a small FP64 grid has to be spread over all
// SMs: at 65^2 points, C = 5, 8 blocks of 256 became 65 or more of 32, and the
// window Gram went from 34.8 to 9.7 us, the orthogonalisation from 45 to 12 us,
// the block SpMM from 14.3 to 8.1 us (serialised, event-timed launches).
int spread_threads(long long items) {
  const int sms = sm_count() > 0 ? sm_count() : 152;
  int t = kBlock;
  while (t > 32 && (items + t - 1) / t < sms) t /= 2;
  return t;
}

// of the reducing kernels: the same for a problem alone and in a batch
int stream_threads(const GridDesc& g) { return spread_threads(g.npts / 2); }

// Slots of the window Gram's partial sums, the most warps that share a task's
// points (gram_shape): one per 32 points, at most four per SM.
int gram_chunks_default(const GridDesc& g) {
  const long long c = (g.npts + 31) / 32;
  return (int)(c < 2 * kStreamBlocks ? c : 2 * kStreamBlocks);
}
int gram_chunks_min(const GridDesc& g) { return (gram_chunks_default(g) + 1) / 2; }
int gram_chunks_cap(const GridDesc& g) {
  const long long c = 2LL * gram_chunks_default(g);
  return (int)(c < kGramChunksMax ? c : kGramChunksMax);
}
int gram_chunks(const GridDesc& g) {
  const int v = tune::lookup(tune::kGram, tune::kAny, g.npts, g.nb, 0, gram_chunks_default(g));
  const int lo = gram_chunks_min(g), hi = gram_chunks_cap(g);
  return v < lo ? lo : (v > hi ? hi : v);
}

int stream_blocks_min(const GridDesc& g) {
  const long long groups = g.npts / 2, bd = stream_threads(g);
  long long need = (groups + bd * 16 - 1) / (bd * 16);   // <= 64 points per thread
  if (need < 1) need = 1;
  return (int)(need < kStreamBlocksMax ? need : kStreamBlocksMax);
}
int stream_blocks_default(const GridDesc& g) {
  const long long groups = g.npts / 2, bd = stream_threads(g);
  long long need = stream_blocks_min(g);
  long long fill = (groups + bd - 1) / bd;                // no idle threads
  long long nb = kStreamBlocks < fill ? kStreamBlocks : fill;
  if (need > nb) nb = need;
  if (nb < 1) nb = 1;
  return (int)(nb < kStreamBlocksMax ? nb : kStreamBlocksMax);
}
// the most blocks the tuner may choose (and the reduction buffers reserve):
// eight per SM, without idle threads
int stream_blocks_cap(const GridDesc& g) {
  const long long groups = g.npts / 2, bd = stream_threads(g);
  const long long fill = (groups + bd - 1) / bd;
  long long c = 8LL * (sm_count() > 0 ? sm_count() : 152);
  if (c > fill) c = fill;
  const long long d = stream_blocks_default(g);
  if (c < d) c = d;
  return (int)(c < kStreamBlocksMax ? c : kStreamBlocksMax);
}
int stream_blocks(const GridDesc& g) {
  const int v = tune::lookup(tune::kStream, tune::kAny, g.npts, g.nb, 0, stream_blocks_default(g));
  const int lo = stream_blocks_min(g), hi = stream_blocks_cap(g);
  return v < lo ? lo : (v > hi ? hi : v);
}

// Partial slots per value, the most walkers of a task: a warp's set-up and
// its final reduction cost about two steps, so walkers take two or four steps
// each once the grid has enough of them (a batch of 12 problems of 257^2
// points, C = 7: 70 us with one or two steps, 41 us with four); the slow FP64
// and double-word steps are shared out more finely.  The shape depends on the
// grid alone: a problem sums alike on its own and in a batch.
template <typename T>
int gram_slots(const GridDesc& g) {
  const int w = sizeof(T) == 4 ? 4 : 1;
  const long long steps = (g.npts + 32 * w - 1) / (32 * w);
  const int per = sizeof(T) == 4 ? (steps >= 512 ? 4 : (steps >= 128 ? 2 : 1))
                                 : (steps >= 2048 ? 4 : (steps >= 512 ? 2 : 1));
  const long long n = (steps + per - 1) / per;
  const int v = gram_chunks(g);
  return (int)(n < v ? n : v);
}
template int gram_slots<float>(const GridDesc&);
template int gram_slots<double>(const GridDesc&);
template int gram_slots<dw>(const GridDesc&);

template <typename T, int C>
static GramShape gram_shape_c(const GridDesc& g, int m) {
  constexpr int RB = kGramRows<T, C>;
  GramShape s;
  s.rows = RB;
  s.slots = gram_slots<T>(g);
  const int ntask = (m * C + RB - 1) / RB;
  const long long full = (long long)ntask * s.slots;
  const int cap = 16 * (sm_count() > 0 ? sm_count() : 152);   // two blocks of eight warps per SM
  s.nwarps = (int)(full < cap ? full : (cap > ntask ? cap : ntask));
  return s;
}

template <typename T>
GramShape gram_shape(const GridDesc& g, int C, int m) {
  GramShape s = {};
  MPCG_C_SWITCH(C, (s = gram_shape_c<T, CC>(g, m)));
  return s;
}
template GramShape gram_shape<float>(const GridDesc&, int, int);
template GramShape gram_shape<double>(const GridDesc&, int, int);
template GramShape gram_shape<dw>(const GridDesc&, int, int);

template <typename T>
void launch_gram_window(const GridDesc& g, Window<T> win, const T* Z, int C, int m, double* part,
                        const DevState* state, cudaStream_t s) {
  const GramShape q = gram_shape<T>(g, C, m);
  const int threads = spread_threads(32LL * q.nwarps);
  const int blocks = (32 * q.nwarps + threads - 1) / threads;
  MPCG_C_SWITCH(C, (k_gram_window<T, CC><<<dim3(blocks, g.nb), threads, 0, s>>>(g, win, Z, part, q.nwarps, q.slots,
                                                                                state)));
}

template <typename T>
void launch_orth_update(const GridDesc& g, Window<T> win, const T* Z, int C, const DevState* state,
                        cudaStream_t s) {
  const int w = sizeof(T) == 4 ? (C < 10 ? 4 : 2) : 1;
  const long long groups = g.npts / w;
  const int threads = spread_threads(groups * g.nb);   // elementwise: any shape gives the same values
  const long long need = (groups + threads - 1) / threads;
  const int nb = (int)(need < 2 * kStreamBlocks ? need : 2 * kStreamBlocks);
  MPCG_C_SWITCH(C, (k_orth_update<T, CC><<<dim3(nb, g.nb), threads, 0, s>>>(g, win, Z, state)));
}

template <typename T>
void launch_block_gram(const GridDesc& g, Window<T> win, const T* r, int C, double* part, const DevState* state,
                       cudaStream_t s) {
  const int nb = stream_blocks(g);
  MPCG_C_SWITCH(C, (k_block_gram<T, CC><<<dim3(nb, g.nb), stream_threads(g), 0, s>>>(g, win, r, part, state)));
}

template <typename T>
void launch_update_xr(const GridDesc& g, Window<T> win, T* x, T* r, int C, double* part, const DevState* state,
                      cudaStream_t s) {
  const int nb = stream_blocks(g);
  MPCG_C_SWITCH(C, (k_update_xr<T, CC><<<dim3(nb, g.nb), stream_threads(g), 0, s>>>(g, win, x, r, part, state)));
}

void launch_start_inner(const GridDesc& g, const double* r64, const double* nrm2, const int* active, float* b32,
                        float* r32, double* part, cudaStream_t s) {
  k_start_inner<<<dim3(stream_blocks(g), g.nb), stream_threads(g), 0, s>>>(g, r64, nrm2, active, b32, r32, part);
}
void launch_axpy_mixed(const GridDesc& g, double* x, const float* d, const double* scale, int* xnz,
                       cudaStream_t s) {
  k_axpy_mixed<<<dim3(stream_blocks(g), g.nb), stream_threads(g), 0, s>>>(g, x, d, scale, xnz);
}

template void launch_gram_window<double>(const GridDesc&, Window<double>, const double*, int, int, double*, const DevState*,
                                         cudaStream_t);
template void launch_orth_update<double>(const GridDesc&, Window<double>, const double*, int, const DevState*, cudaStream_t);
template void launch_block_gram<double>(const GridDesc&, Window<double>, const double*, int, double*, const DevState*,
                                        cudaStream_t);
template void launch_update_xr<double>(const GridDesc&, Window<double>, double*, double*, int, double*, const DevState*,
                                       cudaStream_t);
template void launch_gram_window<float>(const GridDesc&, Window<float>, const float*, int, int, double*, const DevState*,
                                         cudaStream_t);
template void launch_orth_update<float>(const GridDesc&, Window<float>, const float*, int, const DevState*, cudaStream_t);
template void launch_block_gram<float>(const GridDesc&, Window<float>, const float*, int, double*, const DevState*,
                                        cudaStream_t);
template void launch_update_xr<float>(const GridDesc&, Window<float>, float*, float*, int, double*, const DevState*,
                                       cudaStream_t);
template void launch_gram_window<dw>(const GridDesc&, Window<dw>, const dw*, int, int, double*, const DevState*,
                                         cudaStream_t);
template void launch_orth_update<dw>(const GridDesc&, Window<dw>, const dw*, int, const DevState*, cudaStream_t);
template void launch_block_gram<dw>(const GridDesc&, Window<dw>, const dw*, int, double*, const DevState*,
                                        cudaStream_t);
template void launch_update_xr<dw>(const GridDesc&, Window<dw>, dw*, dw*, int, double*, const DevState*,
                                       cudaStream_t);

}  // namespace mpcg
