// Matrix-free fine-grid operator of the Q1 diffusion problem (Section 1's
// model problem, -div(kappa grad u) with kappa constant on each element),
// the matrix-free direction the paper names as future work (Section 4):
// instead of streaming 27 stored coefficients per unknown, the FP32 kernels
// of the inner solve rebuild each row from the coefficients of the 8
// elements around the node.
//
// 3D Q1 hexahedron of side h: the element stiffness entry between two of its
// nodes depends only on how many coordinates differ: h/3 (same node), 0
// (one), -h/12 (two or three).  Hence, with k_e = -(h/12) kappa_e:
//   centre           -4 * (sum of the 8 k_e around the node)
//   face neighbour    0
//   edge neighbour    sum of the 2 k_e sharing that edge
//   corner neighbour  the 1 k_e sharing that corner.
// 2D Q1 square: 4/6, -1/6, -2/6 for 0, 1, 2 differing coordinates
// (independent of h); with k_e = -kappa_e / 6: centre -4 * (sum of the 4
// k_e), edge neighbour the sum of the 2 k_e sharing the edge, corner twice
// the 1 k_e sharing it (all 9 couplings non-zero).
// k is stored in the padded node layout at the element's lowest node
// (unknown coordinates -1 .. n-1 per axis; the -1 entries sit in pads and
// guards, see common.cuh), zero for elements outside the domain.  Couplings
// to eliminated Dirichlet nodes multiply pad entries of X (zero), and the
// outputs at pad points are set to zero, so the result equals the stored
// operator's.
#include <string.h>

#include "kernels.cuh"
#include "rows.cuh"
#include "vec.cuh"

namespace mpcg {

namespace {

// k_e of element e (lowest node: global node (ex, ey[, ez])) of problem
// blockIdx.y at its padded slot.
__global__ void k_place_kappa(GridDesc g, const double* __restrict__ kappa, int ne, double scale,
                              float* __restrict__ k32, double* __restrict__ k64) {
  const int pb = blockIdx.y;
  const long long n = g.dim == 3 ? (long long)ne * ne * ne : (long long)ne * ne;
  kappa += (long long)pb * n;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    const int ex = (int)(e % ne), ey = (int)((e / ne) % ne), ez = g.dim == 3 ? (int)(e / ((long long)ne * ne)) : 0;
    const long long i = (long long)pb * g.len + g.G + (long long)(ex - g.lox) + (long long)(ey - g.loy) * g.px +
                        (g.dim == 3 ? (long long)(ez - g.loz) * g.pxy : 0);
    const double k = scale * kappa[e];
    k64[i] = k;
    k32[i] = (float)k;
  }
}

// Largest |a_stored - a_kappa| and |a_stored| over the couplings between
// unknowns (FP64) of problem blockIdx.y, as order-preserving bit patterns of
// non-negative doubles.
__global__ void k_check_kappa(GridDesc g, const double* __restrict__ st, const double* __restrict__ k64,
                              unsigned long long* out) {
  const int pb = blockIdx.y;
  const int S = g.dim == 3 ? 27 : 9;
  double dmax = 0.0, amax = 0.0;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < g.npts;
       t += (long long)gridDim.x * blockDim.x) {
    int x, y, z, a;
    decode(g, t, x, y, z, a);
    if (!interior(g, x, y, z)) continue;
    const long long i = (long long)pb * g.len + g.G + t;
    for (int s = 0; s < S; ++s) {
      const int dx = s % 3 - 1, dy = (s / 3) % 3 - 1, dz = g.dim == 3 ? s / 9 - 1 : 0;
      const int qx = x + dx, qy = y + dy, qz = z + dz;
      if (qx < 0 || qy < 0 || qx >= g.nx || qy >= g.ny) continue;
      if (g.dim == 3 && (qz < 0 || qz >= g.nz)) continue;
      const int nd = (dx != 0) + (dy != 0) + (dz != 0);
      double sum = 0.0;   // k_e over the elements holding both nodes
      for (int c = (g.dim == 3 ? 0 : 1); c < 2; ++c) {
        if ((dz < 0 && c == 1) || (dz > 0 && c == 0)) continue;
        for (int b = 0; b < 2; ++b) {
          if ((dy < 0 && b == 1) || (dy > 0 && b == 0)) continue;
          for (int e = 0; e < 2; ++e) {
            if ((dx < 0 && e == 1) || (dx > 0 && e == 0)) continue;
            sum += k64[i + (e - 1) + (long long)(b - 1) * g.px + (g.dim == 3 ? (long long)(c - 1) * g.pxy : 0)];
          }
        }
      }
      double ak;
      if (nd == 0) ak = -4.0 * sum;
      else if (g.dim == 3) ak = nd == 1 ? 0.0 : sum;
      else ak = nd == 1 ? sum : 2.0 * sum;
      const double as = st[(long long)s * g.cp + i];
      dmax = fmax(dmax, fabs(as - ak));
      amax = fmax(amax, fabs(as));
    }
  }
  atomicMax(out, (unsigned long long)__double_as_longlong(dmax));
  atomicMax(out + 1, (unsigned long long)__double_as_longlong(amax));
}

// k_e of the elements around the points x0 .. x0+3 of a group: kq[2b + c][k]
// (2D: kq[b][k]) for the element whose lowest node is (x0 - 1 + k, y - 1 + b,
// z - 1 + c).
template <int DIM>
__device__ __forceinline__ void load_kappa(const float* __restrict__ k32, long long idx, long long px, long long pxy,
                                           float (&kq)[DIM == 3 ? 4 : 2][5]) {
#pragma unroll
  for (int e = 0; e < (DIM == 3 ? 4 : 2); ++e) {
    const int b = DIM == 3 ? e >> 1 : e, c = DIM == 3 ? e & 1 : 1;
    const float* p = k32 + idx + (long long)(b - 1) * px + (long long)(c - 1) * pxy;
    float m[4];
    Vec<float>::load_keep(p, m);
    kq[e][0] = p[-1];
#pragma unroll
    for (int w = 0; w < 4; ++w) kq[e][w + 1] = m[w];
  }
}

// Coefficients of stencil row k (dy = k % 3 - 1, dz = k / 3 - 1; 2D: dy = k - 1)
// for the group's points as sources (rows.cuh): the coupling of a point to its
// left neighbour's column and to its right one's both come from the element
// between them, e[w] and e[w + 1].
template <int DIM>
__device__ __forceinline__ void mf_row_coeffs(const float (&kq)[DIM == 3 ? 4 : 2][5], int k, float (&cl)[4],
                                              float (&cc)[4], float (&cr)[4]) {
  const int dy = k % 3 - 1, dz = DIM == 3 ? k / 3 - 1 : 0;
  float e[5];
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    if constexpr (DIM == 3) {
      const int b = dy > 0, c = dz > 0;
      if (dy == 0 && dz == 0) e[i] = kq[0][i] + kq[1][i] + kq[2][i] + kq[3][i];
      else if (dz == 0) e[i] = kq[2 * b][i] + kq[2 * b + 1][i];   // edges (+-1, dy, 0), face (0, dy, 0)
      else if (dy == 0) e[i] = kq[c][i] + kq[2 + c][i];           // edges (+-1, 0, dz), face (0, 0, dz)
      else e[i] = kq[2 * b + c][i];                               // corners (+-1, dy, dz), edge (0, dy, dz)
    } else {
      e[i] = dy == 0 ? kq[0][i] + kq[1][i] : kq[dy > 0][i];
    }
  }
#pragma unroll
  for (int w = 0; w < 4; ++w) {
    const float s = e[w] + e[w + 1];
    if constexpr (DIM == 3) {
      cl[w] = e[w];
      cr[w] = e[w + 1];
      cc[w] = dy == 0 && dz == 0 ? -4.f * s : s;
    } else {
      cl[w] = dy == 0 ? e[w] : 2.f * e[w];
      cr[w] = dy == 0 ? e[w + 1] : 2.f * e[w + 1];
      cc[w] = dy == 0 ? -4.f * s : s;
    }
  }
}

// the products of row k: in 3D the face couplings are zero, and the row through
// the point has no others
template <int DIM>
__device__ __forceinline__ void mf_row_products(int k, const float (&cl)[4], const float (&cc)[4],
                                                const float (&cr)[4], const float (&x)[4], float (&acc)[6]) {
  const bool centre_row = DIM == 3 && k == 4, edges = DIM == 3 && k != 4 && (k & 1);
  if (centre_row) {
#pragma unroll
    for (int w = 0; w < 4; ++w) acc[w + 1] = fmaf(cc[w], x[w], acc[w + 1]);
  } else if (edges) {
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      acc[w] = fmaf(cl[w], x[w], acc[w]);
      acc[w + 2] = fmaf(cr[w], x[w], acc[w + 2]);
    }
  } else {
    row_products(cl, cc, cr, x, acc);
  }
}

// Y = A X over C columns, A from k, rows read in aligned vectors only
// (rows.cuh; the next row's loads are issued before the present one's
// products): 113^3, C = 5, 36.8 -> 28.6 us, the fused Jacobi 21 -> 15 us against
// gathering the neighbours (event-timed).
// The Gram partial sums of the new block X = P go to part.
template <int DIM, int C>
__global__ void __launch_bounds__(kBlock, C <= 3 ? 3 : 2) k_spmm_mf(GridDesc g, RowMap map,
                                                                    const float* __restrict__ k32, SpmmIO<float> io,
                                                                    const float* __restrict__ r, double* part,
                                                                    const DevState* state) {
  const int pb = blockIdx.y;
  if (state && state[pb].done) return;
  const float* X;
  float* Y;
  spmm_operands(io, state + pb, X, Y);
  constexpr int R = DIM == 3 ? 9 : 3, NV = C * (C + 1) / 2 + C;
  const int lane = threadIdx.x & 31;
  const long long ngroups = g.npts / 4, bo = (long long)pb * g.len + g.G;
  double hold[rs_count(NV, 5)] = {};
  int base = 0, nvalid = 0;
  for (long long wid = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; wid < map.nwarps;
       wid += (long long)gridDim.x * (blockDim.x >> 5)) {
    long long q;
    bool active, store;
    row_group(map, wid, lane, ngroups, q, active, store);
    const long long idx = bo + q * 4;
    float acc[C][6];
#pragma unroll
    for (int c = 0; c < C; ++c)
#pragma unroll
      for (int i = 0; i < 6; ++i) acc[c][i] = 0.f;
    float x[2][C][4], rv[4];
    constexpr bool kP = C <= kGramRegs;
    auto own_rows = [&]() {   // P's own rows and r, for the Gram sums
#pragma unroll
      for (int c = 0; c < C; ++c) Vec<float>::load_keep(X + (long long)c * g.cp + idx, x[R & 1][c]);
      Vec<float>::load_keep(r + idx, rv);
    };
    if (active) {
      float kq[DIM == 3 ? 4 : 2][5];
      auto load = [&](int k) {
        const long long ro = (k % 3 - 1) * (long long)g.px + (DIM == 3 ? (k / 3 - 1) * g.pxy : 0);
#pragma unroll
        for (int c = 0; c < C; ++c) Vec<float>::load_keep(X + (long long)c * g.cp + idx + ro, x[k & 1][c]);
      };
      load_kappa<DIM>(k32, idx, g.px, g.pxy, kq);
      load(0);
#pragma unroll
      for (int k = 0; k < R; ++k) {
        if (k + 1 < R) load(k + 1);
        else if (kP) own_rows();
        float cl[4], cc[4], cr[4];
        mf_row_coeffs<DIM>(kq, k, cl, cc, cr);
#pragma unroll
        for (int c = 0; c < C; ++c) mf_row_products<DIM>(k, cl, cc, cr, x[k & 1][c], acc[c]);
      }
    }
    int x0 = 0, y = 0, z = 0, a;
    if (store) decode(g, q * 4, x0, y, z, a);
    const bool row_in = y < g.ny && (DIM == 2 || z < g.nz);
    float o[C][4];
#pragma unroll
    for (int c = 0; c < C; ++c) {
      edge_shift(acc[c], lane);
#pragma unroll
      for (int w = 0; w < 4; ++w) o[c][w] = row_in && x0 + w < g.nx ? acc[c][w + 1] : 0.f;   // pad points: zero rows
      if (store) Vec<float>::store(Y + (long long)c * g.cp + idx, o[c]);
    }
    if (!kP && store) Vec<float>::load_keep(r + idx, rv);
    gram_add<C>(
        [&](int a, float(&v)[4]) {
          if constexpr (kP) {
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = x[R & 1][a][i];
          } else {
            Vec<float>::load_keep(X + (long long)a * g.cp + idx, v);
          }
        },
        rv, o, store, hold, base, nvalid, lane);
  }
  gram_store<NV>(hold, base, nvalid, part + (long long)pb * NV * gridDim.x);
}

// Two damped-Jacobi sweeps from zero on the fine grid, fused (as k_jacobi
// mode 1): s1 = dinv r, s = s1 + dinv (r - A s1), A from k; dinv (stored) is
// omega / diagonal, zero at pads.
template <int DIM>
__global__ void __launch_bounds__(kBlock, 4) k_jacobi_mf(GridDesc g, RowMap map, const float* __restrict__ k32,
                                                         const float* __restrict__ dinv, const float* __restrict__ r,
                                                         float* __restrict__ out, const DevState* state) {
  const int pb = blockIdx.y;
  if (state && state[pb].done) return;
  constexpr int R = DIM == 3 ? 9 : 3;
  const int lane = threadIdx.x & 31;
  const long long wid = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (wid >= map.nwarps) return;
  long long q;
  bool active, store;
  row_group(map, wid, lane, g.npts / 4, q, active, store);
  const long long idx = (long long)pb * g.len + g.G + q * 4;
  float acc[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, di[4] = {}, ri[4] = {};
  if (active) {
    float kq[DIM == 3 ? 4 : 2][5];
    load_kappa<DIM>(k32, idx, g.px, g.pxy, kq);
#pragma unroll
    for (int k = 0; k < R; ++k) {
      const long long ro = (k % 3 - 1) * (long long)g.px + (DIM == 3 ? (k / 3 - 1) * g.pxy : 0);
      float dv[4], x[4], cl[4], cc[4], cr[4];
      Vec<float>::load_keep(dinv + idx + ro, dv);
      Vec<float>::load_keep(r + idx + ro, x);
      if (k == R / 2) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          di[i] = dv[i];
          ri[i] = x[i];
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) x[i] *= dv[i];
      mf_row_coeffs<DIM>(kq, k, cl, cc, cr);
      mf_row_products<DIM>(k, cl, cc, cr, x, acc);
    }
  }
  edge_shift(acc, lane);
  if (!store) return;
  float o[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) o[i] = di[i] * ri[i] + di[i] * (ri[i] - acc[i + 1]);
  Vec<float>::store(out + idx, o);
}

}  // namespace

mpcg_status place_kappa(const GridDesc& g, const double* kappa, int ne, double h, float* k32, double* k64,
                        unsigned long long* check, const double* st64, double* maxdiff, double* maxabs,
                        cudaStream_t s) {
  if ((g.dim != 2 && g.dim != 3) || g.ncomp != 1) return MPCG_ERR_ARG;
  const long long n = g.dim == 3 ? (long long)ne * ne * ne : (long long)ne * ne;
  const double scale = g.dim == 3 ? -h / 12.0 : -1.0 / 6.0;
  k_place_kappa<<<dim3(grid_for(n, 4096), g.nb), kBlock, 0, s>>>(g, kappa, ne, scale, k32, k64);
  cudaMemsetAsync(check, 0, 2 * sizeof(unsigned long long), s);
  k_check_kappa<<<dim3(grid_for(g.npts, 2048), g.nb), kBlock, 0, s>>>(g, st64, k64, check);
  unsigned long long hv[2] = {0, 0};
  if (cudaMemcpyAsync(hv, check, sizeof(hv), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return MPCG_ERR_CUDA;
  memcpy(maxdiff, &hv[0], sizeof(double));
  memcpy(maxabs, &hv[1], sizeof(double));
  return MPCG_OK;
}

template <int DIM>
static int spmm_mf(const GridDesc& g, const float* k32, const SpmmIO<float>& io, int C, const float* r, double* part,
                   const DevState* state, cudaStream_t s) {
  const RowMap map = row_map(g);
  const RowLaunch l = row_launch(map);
  const dim3 grid(l.blocks, g.nb);
#define MPCG_MF_CASE(CC)                                                                     \
  case CC:                                                                                   \
    k_spmm_mf<DIM, CC><<<grid, l.threads, 0, s>>>(g, map, k32, io, r, part, state);          \
    break;
  switch (C) {
    MPCG_MF_CASE(1) MPCG_MF_CASE(2) MPCG_MF_CASE(3) MPCG_MF_CASE(4) MPCG_MF_CASE(5) MPCG_MF_CASE(6)
    MPCG_MF_CASE(7) MPCG_MF_CASE(8) MPCG_MF_CASE(9) MPCG_MF_CASE(10) MPCG_MF_CASE(11) MPCG_MF_CASE(12)
    default: break;
  }
#undef MPCG_MF_CASE
  return l.blocks;
}

int launch_spmm_mf(const GridDesc& g, const float* k32, const SpmmIO<float>& io, int C, const float* r, double* part,
                   const DevState* state, cudaStream_t s) {
  return g.dim == 3 ? spmm_mf<3>(g, k32, io, C, r, part, state, s) : spmm_mf<2>(g, k32, io, C, r, part, state, s);
}

void launch_jacobi_mf(const GridDesc& g, const float* k32, const float* dinv, const float* r, float* out,
                      const DevState* state, cudaStream_t s) {
  const RowMap map = row_map(g);
  const dim3 grid((unsigned)((32 * map.nwarps + kBlock - 1) / kBlock), g.nb);
  if (g.dim == 3) k_jacobi_mf<3><<<grid, kBlock, 0, s>>>(g, map, k32, dinv, r, out, state);
  else k_jacobi_mf<2><<<grid, kBlock, 0, s>>>(g, map, k32, dinv, r, out, state);
}

}  // namespace mpcg
