// FP32 stencil products that read every grid row in aligned vectors only.
//
// A thread owns the four points of a group.  Gathering the neighbours
// x[i - 1], x[i + 1] of a row costs, besides the 16-byte vector, two scalars
// whose lanes are 16 bytes apart and touch four L1 lines each, so two thirds of
// the L1 wavefronts of a multi-column product fetch values that the neighbour
// lanes hold (129^3, C = 6: 756 wavefronts a warp and group, L1 86 % busy, DRAM
// 42 %).  Here a thread takes its own four values of a row and adds their
// products to the targets they belong to: its own four points acc[1 .. 4] and,
// over the edges, one point to the left (acc[0]) and one to the right
// (acc[5]).  Only these two sums, over all rows, change lanes at the end, two
// shuffles a column.
//
// Warps are dealt so that no sum has to leave one (RowMap): where whole rows
// fill a warp (pitches dividing 128), what would cross its ends are products
// of the pad between two rows, zero; otherwise consecutive warps overlap by two
// groups and the outer lanes only compute sums for their neighbours.  A point's
// sum has the same products in the same order either way.
#pragma once

#include "kernels.cuh"
#include "vec.cuh"

namespace mpcg {

struct RowMap {
  int stride;            // groups from one warp to the next: 32 (whole rows), or 30 with overlap
  long long nwarps;
};
inline RowMap row_map(const GridDesc& g) {
  RowMap m;
  m.stride = 128 % g.px == 0 ? 32 : 30;
  m.nwarps = (g.npts / 4 + m.stride - 1) / m.stride;
  return m;
}
// This lane's group q in warp w: a lane outside the grid (active = false)
// contributes nothing, an outer lane of an overlap stores nothing.
__device__ __forceinline__ void row_group(const RowMap& m, long long w, int lane, long long ngroups, long long& q,
                                          bool& active, bool& store) {
  q = m.stride == 32 ? w * 32 + lane : w * 30 + lane - 1;
  active = q >= 0 && q < ngroups;
  store = active && (m.stride == 32 || (lane > 0 && lane < 31));
}

// Warps of one problem's launch (the same for a problem alone and in a batch:
// the partial sums below follow them): a warp per segment up to two blocks of
// eight per SM, which then walk the segments (with sixteen blocks per SM the
// block sums cost more than the balance gains: 1025^2, C = 9 32.7 against 28.6
// us, matrix-free 113^3 35.9 against 28.8).
struct RowLaunch {
  int blocks, threads;
};
inline RowLaunch row_launch(const RowMap& m) {
  RowLaunch l;
  l.threads = spread_threads(32 * m.nwarps);
  const long long need = (32 * m.nwarps + l.threads - 1) / l.threads;
  const int cap = 2 * (sm_count() > 0 ? sm_count() : 152) * (kBlock / l.threads);
  l.blocks = (int)(need < cap ? need : cap);
  return l;
}

// Gram sums of the new block beside the product that forms it: with the lane's
// four values of every A p_c in o, the upper triangle of P^T A P and P^T r over
// its points, summed over the warp in FP32 and added to `hold` in FP64 (value
// base + i of the lane's i-th, as warp_reduce_scatter deals them).  p(a, v)
// gives the values of P's column a.  A kernel of its own reads P, A P and r from
// memory again (1025^2, C = 9: 23.5 + 16.3 us against 28.6 together, 257^2 batch,
// C = 7: 20.4 + 18.4 against 28.6, matrix-free 113^3, C = 5: 28.6 + 12.2 against
// 28.7, 33^3 8 + 6 against 8).
template <int C, typename P>
__device__ __forceinline__ void gram_add(P p, const float (&rv)[4], const float (&o)[C][4], bool store,
                                         double (&hold)[rs_count(C * (C + 1) / 2 + C, 5)], int& base, int& nvalid,
                                         int lane) {
  constexpr int NG = C * (C + 1) / 2;
  float v[NG + C];
#pragma unroll
  for (int i = 0; i < NG + C; ++i) v[i] = 0.f;
  if (store) {
    int k = 0;
#pragma unroll
    for (int a = 0; a < C; ++a) {
      float pa[4];
      p(a, pa);
#pragma unroll
      for (int b = a; b < C; ++b) {
#pragma unroll
        for (int w = 0; w < 4; ++w) v[k] = fmaf(pa[w], o[b][w], v[k]);
        ++k;
      }
#pragma unroll
      for (int w = 0; w < 4; ++w) v[NG + a] = fmaf(pa[w], rv[w], v[NG + a]);
    }
  }
  warp_reduce_scatter<float, NG + C>(v, base, nvalid, lane);
#pragma unroll
  for (int i = 0; i < rs_count(NG + C, 5); ++i) hold[i] += (double)v[i];
}
// Columns up to which P's own rows are loaded again as one more row of the
// product's pipeline and kept in registers for gram_add; wider blocks would
// spill and read them one column at a time.
constexpr int kGramRegs = 6;

// the block's sums of the warps' `hold` to part[value * gridDim.x + blockIdx.x];
// every thread of the block calls it
template <int NV>
__device__ __forceinline__ void gram_store(const double (&hold)[rs_count(NV, 5)], int base, int nvalid, double* part) {
  __shared__ double sh[kBlock / 32][NV];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int i = lane; i < NV; i += 32) sh[warp][i] = 0.0;   // a warp without a segment holds nothing
  __syncwarp();
#pragma unroll
  for (int i = 0; i < rs_count(NV, 5); ++i)
    if (i < nvalid) sh[warp][base + i] = hold[i];
  __syncthreads();
  for (int i = threadIdx.x; i < NV; i += blockDim.x) {
    double s = 0.0;
    for (int w = 0; w < nw; ++w) s += sh[w][i];
    part[(long long)i * gridDim.x + blockIdx.x] = s;
  }
}

// acc[1], acc[4] get the sums of the neighbour lanes
__device__ __forceinline__ void edge_shift(float (&acc)[6], int lane) {
  const float l = __shfl_up_sync(0xffffffffu, acc[5], 1);
  const float r = __shfl_down_sync(0xffffffffu, acc[0], 1);
  if (lane > 0) acc[1] += l;
  if (lane < 31) acc[4] += r;
}

// acc += the products of one row: x[w] times the coefficient of its target,
// cl[w] for target w - 1, cc[w] for w, cr[w] for w + 1.
__device__ __forceinline__ void row_products(const float (&cl)[4], const float (&cc)[4], const float (&cr)[4],
                                             const float (&x)[4], float (&acc)[6]) {
#pragma unroll
  for (int w = 0; w < 4; ++w) {
    acc[w] = fmaf(cl[w], x[w], acc[w]);
    acc[w + 1] = fmaf(cc[w], x[w], acc[w + 1]);
    acc[w + 2] = fmaf(cr[w], x[w], acc[w + 2]);
  }
}

// ---- the symmetric half of a stored scalar stencil ------------------------
// (launch_sym_half: plane p holds tap 3^DIM / 2 + p, the couplings to the point
// itself and to the later neighbours.)

// Coefficients of stencil row k (offset ro) for the sources at idx + ro.  Rows
// before the centre are read transposed, A(t, s) = A(s, t), where all three
// planes sit at the source; of the later rows the two side planes sit at the
// target, one point off the source.
template <int DIM>
__device__ __forceinline__ void half_row_coeffs(const float* __restrict__ st, long long pitch, long long idx,
                                                long long ro, int k, float (&cl)[4], float (&cc)[4], float (&cr)[4]) {
  constexpr int R = DIM == 3 ? 9 : 3, kc = R / 2, tc = 3 * kc + 1;
  if (k < kc) {
    const float* p = st + (long long)(3 * (R - 1 - k) - tc) * pitch + idx + ro;
    Vec<float>::load(p, cl);
    Vec<float>::load(p + pitch, cc);
    Vec<float>::load(p + 2 * pitch, cr);
  } else if (k == kc) {
    Vec<float>::load(st + idx, cc);
    Vec<float>::load_keep(st + pitch + idx, cr);
#pragma unroll
    for (int w = 1; w < 4; ++w) cl[w] = cr[w - 1];
    cl[0] = st[pitch + idx - 1];
  } else {
    const float* p = st + (long long)(3 * k - tc) * pitch + idx;
    float a[4], b[4];
    Vec<float>::load_keep(p, a);
    Vec<float>::load_keep(p + pitch, cc);
    Vec<float>::load_keep(p + 2 * pitch, b);
#pragma unroll
    for (int w = 0; w < 3; ++w) {
      cr[w] = a[w + 1];
      cl[w + 1] = b[w];
    }
    cr[3] = p[4];
    cl[0] = p[2 * pitch - 1];
  }
}

}  // namespace mpcg
