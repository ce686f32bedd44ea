// leaf_factor.cuh - cell elimination of the leaf level from the stencil (FP64).
//
// A leaf cell's interior block A_II is the stencil on an m^d grid (m = leaf - 1),
// a band matrix of half bandwidth b = m^(d-1) in lexicographic order, and each
// boundary DOF couples to at most one interior DOF.  So the operators of
// Sec. 2.2, Eq. 2_3, need far less work than on a dense front:
//   A_II = L L^T            banded Cholesky, n b^2 / 2 products
//   G = L^{-1}              column by column, n^2 b / 2 (dense: n^3 / 6)
//   S = A_II^{-1}           L^T S = G by columns, lower triangle, n^2 b / 2
//   V = A_BI A_II^{-1}      row p is -w_p times the row of S at p's interior
//                           neighbour (w_p its stencil coupling), no products
//   X_BB = A_BB - V A_IB    entry (p, q) is -w_p w_q S(p', q')
// For n = 225, b = 15 (leaf 16, 2D) that is 0.8 M products a cell against 9.4 M,
// and no front is stored.  The FP64 pipe (1.89 lanes a clock and SM) bounds both.
// The entries of L outside the band are zero, so L and G take the same operations
// as before; S and V are sums of terms of one sign (A_II is an M-matrix).
//
// One CTA per cell.  L's band sits in shared memory; a warp owns 32 columns of G
// and then of S and walks the rows with the last b values of each column in
// registers (shifted by one a row: moves are free beside the FP64 pipe).
// Measured (the setup's leaf phase with its host planning): 2D 511^2, 1024 cells of
// leaf 16: 41.2 -> 7.6 ms; 3D, 512 cells: leaf 6 13.2 -> 4.8 ms, leaf 8 91 -> 20 ms.
#pragma once

#include "internal.h"

namespace hifcn {
namespace leaf {

constexpr int kMaxBand = 64;
constexpr size_t kMaxSmem = 200 * 1024;

// cells along one axis containing both coordinates a and b; is c the smallest?
__device__ __forceinline__ bool owns(int a, int b, int s, int nc, int c) {
  const int lo_a = (a % s == 0) ? a / s - 1 : a / s, lo_b = (b % s == 0) ? b / s - 1 : b / s;
  return c == max(max(lo_a, lo_b), 0);
}

// shared memory of one cell: band (nI + b rows of b + 1), reciprocal pivots,
// the boundary DOFs' couplings, interior neighbours, box map, window table
__host__ __device__ inline size_t smem_bytes(int nI, int nB, int band, int dim, int s) {
  const size_t box = dim == 3 ? (size_t)(s + 1) * (s + 1) * (s + 1) : (size_t)(s + 1) * (s + 1);
  return ((size_t)(nI + band) * (band + 1) + nI + nB) * sizeof(double) + (nB + box) * sizeof(int) +
         (size_t)band * (band + 1) / 2 * sizeof(unsigned short) + 64;
}

// whether the leaf level of a grid takes this path
inline bool supported(int dim, int leaf, int max_nB, int *band, size_t *smem) {
  const long long m = leaf - 1;
  const long long b = dim == 3 ? m * m : m;
  if (b > kMaxBand) return false;
  *band = (int)b;
  *smem = smem_bytes((int)(m * b), max_nB, (int)b, dim, leaf);
  return *smem <= kMaxSmem;
}

// Cell must provide nI, nB, G_off, V_off, S_off (< 0: S to the scratch),
// Fb_off, dofs_off (I then B); S is stored packed with its diagonal halved.
template <int BW, class Cell>
__global__ void __launch_bounds__(BW > 32 ? 384 : 256)
    k_leaf_factor(const Cell *__restrict__ cells, int cell0, const int *__restrict__ cdofs,
                  const double *__restrict__ diag, const double *__restrict__ wx, const double *__restrict__ wy,
                  const double *__restrict__ wz, int dim, int n, int s, int nc, int band,
                  double *__restrict__ vals, double *__restrict__ scratch, long long scratch_stride,
                  double *__restrict__ Fb, int *__restrict__ err) {
  extern __shared__ __align__(16) unsigned char leaf_smem[];
  const int cid = cell0 + (int)blockIdx.x;
  const Cell c = cells[cid];
  const int nI = c.nI, nB = c.nB, b1 = band + 1, m = s - 1;
  double *Lb = reinterpret_cast<double *>(leaf_smem);      // Lb[i b1 + k] = L[i][i - k]
  double *ri = Lb + (size_t)(nI + band) * b1;              // 1 / L[i][i]
  double *wB = ri + nI;                                    // coupling of a boundary DOF to its interior neighbour
  int *nbr = reinterpret_cast<int *>(wB + nB);             // that neighbour (interior position), -1: none
  int *box = nbr + nB;                                     // boundary position at each point of the cell's box
  const int bs = s + 1, boxn = dim == 3 ? bs * bs * bs : bs * bs;
  unsigned short *tab = reinterpret_cast<unsigned short *>(box + boxn);  // window entries (row << 8 | column)
  const int t = threadIdx.x, nt = blockDim.x, warp = t >> 5, lane = t & 31, nw = nt / 32;
  const int *dofs = cdofs + c.dofs_off;
  const int cc[3] = {cid % nc, (cid / nc) % nc, dim == 3 ? cid / (nc * nc) : 0};
  const long long S1 = n - 1;

  // ---- band of A_II, boundary couplings, tables
  for (int i = t; i < nI + band; i += nt) {
    double *row = Lb + (size_t)i * b1;
    for (int k = 0; k <= band; ++k) row[k] = 0.0;
    if (i < nI) {
      const long long d = dofs[i];
      const int x = i % m, y = (i / m) % m, z = i / (m * m);
      row[0] = diag[d];
      if (x > 0) row[1] = -wx[d - 1];
      if (y > 0) row[m] = -wy[d - S1];
      if (dim == 3 && z > 0) row[m * m] = -wz[d - S1 * S1];
    }
  }
  for (int e = t; e < boxn; e += nt) box[e] = -1;
  for (int r = 1 + t; r <= band; r += nt)
    for (int q = 1; q <= r; ++q) tab[r * (r - 1) / 2 + q - 1] = (unsigned short)(r << 8 | q);
  __syncthreads();
  for (int p = t; p < nB; p += nt) {
    const long long d = dofs[nI + p];
    const int j[3] = {(int)(d % S1) + 1 - cc[0] * s, (int)((d / S1) % S1) + 1 - cc[1] * s,
                      dim == 3 ? (int)(d / (S1 * S1)) + 1 - cc[2] * s : 0};
    box[j[0] + bs * j[1] + bs * bs * j[2]] = p;
    int at = -1;
    double w = 0.0;
    for (int ax = 0; ax < dim; ++ax) {
      if (j[ax] != 0 && j[ax] != s) continue;
      int q[3] = {j[0], j[1], j[2]};
      q[ax] += j[ax] == 0 ? 1 : -1;
      bool in = true;
      for (int e = 0; e < dim; ++e) in = in && q[e] >= 1 && q[e] <= m;
      if (!in) continue;
      at = (q[0] - 1) + m * (q[1] - 1) + (dim == 3 ? m * m * (q[2] - 1) : 0);
      const long long e = j[ax] == 0 ? d : d - (ax == 0 ? 1 : ax == 1 ? S1 : S1 * S1);
      w = (ax == 0 ? wx : ax == 1 ? wy : wz)[e];
    }
    nbr[p] = at;
    wB[p] = w;
  }
  __syncthreads();

  // ---- banded Cholesky: one warp (narrow bands) or the CTA
  const bool wide = band > 24;
  if (wide || warp == 0) {
    const int nth = wide ? nt : 32;
    for (int k = 0; k < nI; ++k) {
      double *col = Lb + (size_t)k * b1;  // L[k + r][k] sits at col[r b1 + r]
      double d = col[0];
      if (!(d > 0.0)) {
        if (t == 0) atomicExch(err, 1);
        d = 1.0;
      }
      const double r1 = rsqrt(d);
      if (wide) __syncthreads();
      else __syncwarp();
      if (t == 0) {
        col[0] = d * r1;
        ri[k] = r1;
      }
      for (int r = 1 + t; r <= band; r += nth) col[r * b1 + r] *= r1;  // rows past nI are zero
      if (wide) __syncthreads();
      else __syncwarp();
      for (int e = t; e < band * b1 / 2; e += nth) {
        const int r = tab[e] >> 8, q = tab[e] & 255;
        col[r * b1 + r - q] -= col[r * b1 + r] * col[q * b1 + q];
      }
      if (wide) __syncthreads();
      else __syncwarp();
    }
  }
  __syncthreads();

  // ---- G = L^{-1} and S = A_II^{-1} by columns, 32 a warp
  double *G = vals + c.G_off;
  double *Sp = c.S_off >= 0 ? vals + c.S_off : scratch + (long long)blockIdx.x * scratch_stride;
  for (int j0 = warp * 32; j0 < nI; j0 += nw * 32) {
    const int j = j0 + lane;
    double h[BW];  // the column's values of the last BW rows, most recent first
#pragma unroll
    for (int k = 0; k < BW; ++k) h[k] = 0.0;
    for (int i = j0; i < nI; ++i) {
      const double *row = Lb + (size_t)i * b1 + 1;
      double a = i == j ? 1.0 : 0.0, a2 = 0.0;
#pragma unroll
      for (int k = BW - 1; k >= 0; --k)
        if (k < band) {
          if (k & 1) a2 -= row[k] * h[k];
          else a -= row[k] * h[k];
        }
      const double g = (a + a2) * ri[i];
#pragma unroll
      for (int k = BW - 1; k > 0; --k) h[k] = h[k - 1];
      h[0] = g;
      if (j <= i) G[tri_off(i) + j] = g;
    }
#pragma unroll
    for (int k = 0; k < BW; ++k) h[k] = 0.0;
    double g = j < nI ? G[tri_off(nI - 1) + j] : 0.0;
    for (int i = nI - 1; i >= j0; --i) {
      const double gn = i > j0 && j <= i - 1 ? G[tri_off(i - 1) + j] : 0.0;
      const double *col = Lb + (size_t)(i + 1) * b1 + 1;  // L[i + 1 + k][i] at col[k b1 + k]
      double a = g, a2 = 0.0;
#pragma unroll
      for (int k = BW - 1; k >= 0; --k)
        if (k < band) {
          if (k & 1) a2 -= col[k * (b1 + 1)] * h[k];
          else a -= col[k * (b1 + 1)] * h[k];
        }
      const double x = (a + a2) * ri[i];
#pragma unroll
      for (int k = BW - 1; k > 0; --k) h[k] = h[k - 1];
      h[0] = x;
      if (j <= i) Sp[tri_off(i) + j] = i == j ? 0.5 * x : x;
      g = gn;
    }
  }
  __syncthreads();

  // ---- V and the Schur complement
  auto S_at = [&](int i, int j) {
    const double v = i >= j ? Sp[tri_off(i) + j] : Sp[tri_off(j) + i];
    return i == j ? 2.0 * v : v;
  };
  double *V = vals + c.V_off;
  const long long vs = pad4(nI);
  for (int p = warp; p < nB; p += nw) {
    const int ip = nbr[p];
    if (ip < 0) {
      for (int j = lane; j < nI; j += 32) V[p * vs + j] = 0.0;
      continue;
    }
    const double w = wB[p];
    for (int j = lane; j < nI; j += 32) V[p * vs + j] = -(w * S_at(ip, j));
  }
  double *X = Fb + c.Fb_off;
  for (int e = t; e < nB * nB; e += nt) {
    const int p = e % nB, q = e / nB;
    X[e] = nbr[p] >= 0 && nbr[q] >= 0 ? -(wB[p] * wB[q] * S_at(nbr[p], nbr[q])) : 0.0;
  }
  __syncthreads();
  // A_BB: the diagonal and the couplings this cell holds (smallest index)
  for (int p = t; p < nB; p += nt) {
    const long long d = dofs[nI + p];
    const int a[3] = {(int)(d % S1) + 1, (int)((d / S1) % S1) + 1, dim == 3 ? (int)(d / (S1 * S1)) + 1 : 0};
    bool own = true;
    for (int ax = 0; ax < dim; ++ax) own = own && owns(a[ax], a[ax], s, nc, cc[ax]);
    if (own) X[p + (long long)p * nB] += diag[d];
    for (int ax = 0; ax < dim; ++ax)
      for (int sg = -1; sg <= 1; sg += 2) {
        int b[3] = {a[0], a[1], a[2]};
        b[ax] += sg;
        if (b[ax] < 1 || b[ax] > n - 1) continue;
        const int lb[3] = {b[0] - cc[0] * s, b[1] - cc[1] * s, dim == 3 ? b[2] - cc[2] * s : 0};
        bool in = true;
        for (int q = 0; q < dim; ++q) in = in && lb[q] >= 0 && lb[q] <= s;
        if (!in) continue;
        const int q = box[lb[0] + bs * lb[1] + bs * bs * lb[2]];
        if (q < 0) continue;
        bool ow = true;
        for (int e = 0; e < dim; ++e) ow = ow && owns(a[e], b[e], s, nc, cc[e]);
        if (!ow) continue;
        const long long e = sg > 0 ? d : d - (ax == 0 ? 1 : ax == 1 ? S1 : S1 * S1);
        X[p + (long long)q * nB] -= (ax == 0 ? wx : ax == 1 ? wy : wz)[e];
      }
  }
}

// Factor ncells leaf cells starting at cell0; scratch (needed when the level
// stores no S) holds tri_off(nI) doubles per cell of the launch.
template <class Cell>
int factor_cells(const Cell *cells_d, int cell0, int ncells, const int *cdofs, const double *diag, const double *wx,
                 const double *wy, const double *wz, int dim, int n, int s, int nc, int band, size_t smem,
                 double *vals, double *scratch, long long scratch_stride, double *Fb, int *err, cudaStream_t st) {
  auto launch = [&](auto kern, int threads) -> int {
    HIF_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    kern<<<ncells, threads, smem, st>>>(cells_d, cell0, cdofs, diag, wx, wy, wz, dim, n, s, nc, band, vals, scratch,
                                        scratch_stride, Fb, err);
    note_launch();
    HIF_CUDA_TRY(cudaGetLastError());
    return HIF_OK;
  };
  if (band <= 8) return launch(k_leaf_factor<8, Cell>, 256);
  if (band <= 16) return launch(k_leaf_factor<16, Cell>, 256);
  if (band <= 32) return launch(k_leaf_factor<32, Cell>, 256);
  return launch(k_leaf_factor<64, Cell>, 384);
}

}  // namespace leaf
}  // namespace hifcn
