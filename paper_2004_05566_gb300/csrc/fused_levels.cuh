// fused_levels.cuh - one launch per level and direction for the small upper levels
// (included by apply.cu inside its anonymous namespace).
//
// Above the levels that stream from HBM, an apply is a chain of dependent launches
// that each move little data: an entity step and a cell step per level and
// direction, about 3.7 us each at 351^2 whatever they do.  The interior DOFs of a
// cell of level l + 1 are exactly the surviving DOFs of the entities of level l
// inside it (in 2D four edges and a corner), so the two steps meet inside a cell:
//   forward   k_level_fwd:  entities of level l, then the cell step of level l + 1:
//     every work item of a cell (rows of [V; G]) forms x_g <- H (x_g - contributions)
//     of the cell's inner entities in shared memory, takes x_I from it and goes on
//     with its rows; the first item of a cell writes the entities' values.
//   backward  k_level_bwd:  the cell step of level l + 1, then the entities of level
//     l inside it: x_I stays in shared memory and enters x_g <- H^T x_g.
//   top       k_level_top:  entities of the last level, the root, the entities back.
// Entities on the faces between cells run as units of their own in the same launch.
// An apply takes 2 L + 1 launches instead of 4 L + 1.
//
// No step may overwrite what another CTA of its launch reads, so the vector
// alternates between two buffers: forward level l reads buffer l and writes buffer
// l + 1 (mod 2); backward it reads what it wrote and writes what it read, so the
// result ends where the input was (a level's redundant DOFs wait in its forward
// output, which no level above touches).  The contributions of consecutive levels
// lie in disjoint parts of the scratch for the same reason.
//
// Rule (build_level_plan): levels whose cells and entities fit one CTA's shared
// memory here, whose cells the bulk-copy kernels do not take and whose entities are
// not split.  Bigger levels are bound by their bytes, not by their launches.
// FP32 only: the FP64 apply is bound by the FP64 pipe in these steps too (63^2: 75.3
// us per CG iteration either way, 511^2 435.8 and 447.1 fused).
// What the chain waits on is latency, not launches (two steps in one launch with the
// same loads took as long as two launches), so everything that does not depend on the
// previous kernel is in registers before the dependency point: positions, slots, the
// first rows of H, G and V.  Per launch at 351^2 about 0.6 us gather, 0.5 us per
// product, 0.8 us from one kernel's end to the next one's data.
// Measured, us per CG iteration (captured solve): 351^2 112.6 -> 102.0, 703^2 200.7
// -> 192.8, 1023^2 356.8 -> 338.5, 2047^2 1083 -> 1065.

// One cell of level l + 1 with its inner entities of level l.  Positions of the
// entities' DOFs are concatenated, each entity padded to a multiple of 4.
struct FusedCell {
  CellDesc c;
  int nsum, ng;        // concatenated positions, entities
  long long cat_off;   // into the position tables
  long long map_off;   // into imap: interior DOF -> position
  int g_off, pad;      // into fgroups
};
struct FusedGroup {
  long long H_off;
  int n, soff;         // DOFs, first position
};
struct FusedItem {
  int cell, a, b, first;  // rows [a, b) of [V; G]; writes the entities' values
};
// a concatenated position: its DOF (-1: padding), its row of H, and where its value
// comes from backward (interior index of the cell, -1: redundant, from memory)
struct __align__(16) FusedPos {
  long long h_off;
  int dof, soff, nq, ipos;
  int n;               // DOFs of its entity
  int c0, nc, pad;     // contribution slots [c0, c0 + nc) of cslot
};

struct FusedLevel {      // of level l
  const FusedCell *cells;
  const FusedItem *items;
  const FusedGroup *fgroups;
  const FusedPos *pos;
  const int *imap;
  const int *small, *large;  // entities on the faces between the cells
  const GroupDesc *groups;
  int nitems, ncells, nsmall, nlarge;
  int max_sum, max_nI, max_nB, max_ng;
  int nt;  // threads of a CTA, forward and backward
};

// CTAs of 512 threads where a level has at most kFuseWideCells cells (twice the rows
// in a batch), else of 256, two an SM; at most about kFuseItems forward items, one
// an SM, so that the next launch's prologue runs beside them.  351^2, us per CG
// iteration: 304 items 103.7 (256 threads) and 101.7, 152 items 102.8 and 102.0;
// 1023^2: 341.9, 340.0, 341.3 and 338.5; 64 wide cells cost 703^2 3 us.
constexpr int kFuseWideCells = 16;
constexpr int kFuseItems = 152;
constexpr int kFuseTopThreads = 512;
constexpr int kFuseMaxSum = 1024;   // concatenated positions of a cell
constexpr int kFuseMaxNI = 1024;

// x_g - contributions at the concatenated positions into gin.  What the thread's
// first position needs besides the vectors is loaded before the dependency point.
constexpr int kFuseSlots = 4;  // cells around a 2D corner
struct FusedPre {
  FusedPos p;
  long long s[kFuseSlots];
};
__device__ __forceinline__ FusedPre fused_pre(const FusedPos *__restrict__ pos, int nsum,
                                              const long long *__restrict__ cslot) {
  FusedPre f;
  f.p = FusedPos{0, -1, 0, 0, -1, 0, 0, 0, 0};
  if ((int)threadIdx.x < nsum) f.p = pos[threadIdx.x];
#pragma unroll
  for (int k = 0; k < kFuseSlots; ++k) f.s[k] = k < f.p.nc ? cslot[f.p.c0 + k] : 0;
  return f;
}
template <int NT>
__device__ __forceinline__ void fused_gather(const FusedPre &pre, const FusedPos *__restrict__ pos, int nsum,
                                             const long long *__restrict__ cslot, const float *__restrict__ contrib,
                                             const float *xin, float *gin) {
  if ((int)threadIdx.x < nsum) {
    float v = 0.f;
    if (pre.p.dof >= 0) {
      v = __ldcg(xin + pre.p.dof);
#pragma unroll
      for (int k = 0; k < kFuseSlots; ++k)
        if (k < pre.p.nc) v -= __ldcg(contrib + pre.s[k]);
      for (int k = kFuseSlots; k < pre.p.nc; ++k) v -= __ldcg(contrib + cslot[pre.p.c0 + k]);
    }
    gin[threadIdx.x] = v;
  }
  for (int t = threadIdx.x + NT; t < nsum; t += NT) {
    const FusedPos p = pos[t];
    float v = 0.f;
    if (p.dof >= 0) {
      v = __ldcg(xin + p.dof);
      for (int k = 0; k < p.nc; ++k) v -= __ldcg(contrib + cslot[p.c0 + k]);
    }
    gin[t] = v;
  }
}

// gout = H gin of the concatenated entities: eight lanes a row, four rows a warp,
// U rows a lane group in flight.  The first batch (its rows of H do not
// depend on the previous kernel) is loaded before the dependency point.
template <int NT>
struct FusedRows {
  static constexpr int U = 4, RS = NT / 8;
  float h[U][2][4];
  int nq[U], so[U];
  const float *row[U];
  __device__ __forceinline__ void load(const FusedPos *__restrict__ pos, int nsum, const float *__restrict__ vals,
                                       int rb) {
    const int sub = threadIdx.x & 7, r0 = threadIdx.x >> 3;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int r = rb + r0 + u * RS;
      nq[u] = 0;
      so[u] = 0;
      row[u] = vals;
      if (r < nsum) {
        const FusedPos p = pos[r];
        nq[u] = p.nq;
        so[u] = p.soff;
        row[u] = vals + p.h_off;
      }
#pragma unroll
      for (int q = 0; q < 2; ++q) ld4_stream(row[u] + 4 * (sub + 8 * q), sub + 8 * q < nq[u], h[u][q]);
    }
  }
  __device__ __forceinline__ void dot(int nsum, int rb, const float *gin, float *gout) const {
    const int sub = threadIdx.x & 7, r0 = threadIdx.x >> 3;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      float acc = 0.f;
#pragma unroll
      for (int q = 0; q < 2; ++q)
        if (sub + 8 * q < nq[u]) {
          float x[4];
          ld4(gin + so[u] + 4 * (sub + 8 * q), x);
          acc += h[u][q][0] * x[0] + h[u][q][1] * x[1] + h[u][q][2] * x[2] + h[u][q][3] * x[3];
        }
      for (int q = sub + 16; q < nq[u]; q += 8) {
        float w[4], x[4];
        ld4(row[u] + 4 * q, w);
        ld4(gin + so[u] + 4 * q, x);
        acc += w[0] * x[0] + w[1] * x[1] + w[2] * x[2] + w[3] * x[3];
      }
      acc += __shfl_xor_sync(0xffffffffu, acc, 4);
      acc += __shfl_xor_sync(0xffffffffu, acc, 2);
      acc += __shfl_xor_sync(0xffffffffu, acc, 1);
      const int r = rb + r0 + u * RS;
      if (sub == 0 && r < nsum) gout[r] = acc;
    }
  }
};

// after the barrier on gin; rows holds the first batch
template <int NT>
__device__ __forceinline__ void fused_rows(FusedRows<NT> &rows, const FusedPos *__restrict__ pos, int nsum,
                                           const float *__restrict__ vals, const float *gin, float *gout) {
  constexpr int B = FusedRows<NT>::U * FusedRows<NT>::RS;
  for (int rb = 0; rb < nsum; rb += B) {
    if (rb > 0) rows.load(pos, nsum, vals, rb);
    rows.dot(nsum, rb, gin, gout);
  }
}

// gout = H^T gin of the concatenated entities: a thread owns a column quad and a
// part of the entity's rows; the parts meet in part (NT quads).  As FusedRows, the
// first U rows of the first block of quads are loaded before the dependency point.
template <int NT>
struct FusedCols {
  static constexpr int U = 8;
  float v[U][4];
  int QW, RG, n, so, np;
  const float *H;  // column quad of the thread in row 0 of its entity
  __device__ __forceinline__ void block(const FusedPos *__restrict__ pos, int nsum, const float *__restrict__ vals,
                                        int q0) {
    const int q = q0 + (int)threadIdx.x % QW;
    n = 0;
    so = np = 0;
    H = vals;
    if (4 * q < nsum) {  // the quad's first position is a DOF; row 4 q - soff of H starts at h_off
      const FusedPos p = pos[4 * q];
      np = 4 * p.nq;
      so = p.soff;
      n = p.n;
      H = vals + p.h_off - (long long)(4 * q - so) * np + (4 * q - so);
    }
    load(threadIdx.x / QW);
  }
  __device__ __forceinline__ void load(int i) {
#pragma unroll
    for (int u = 0; u < U; ++u) ld4_stream(H + (long long)(i + u * RG) * np, i + u * RG < n, v[u]);
  }
  __device__ __forceinline__ void first(const FusedPos *__restrict__ pos, int nsum, const float *__restrict__ vals) {
    pow2_layout(nsum / 4, NT, QW, RG);
    block(pos, nsum, vals, 0);
  }
  // after the barrier on gin; ends with a barrier
  __device__ __forceinline__ void run(const FusedPos *__restrict__ pos, int nsum, const float *__restrict__ vals,
                                      const float *gin, float *gout, float *part) {
    for (int q0 = 0; 4 * q0 < nsum; q0 += QW) {
      if (q0 > 0) block(pos, nsum, vals, q0);
      float acc[4] = {0.f, 0.f, 0.f, 0.f};
      for (int i = threadIdx.x / QW; i < n; i += U * RG) {
        if (i >= RG) load(i);
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const float xv = i + u * RG < n ? gin[so + i + u * RG] : 0.f;
          acc[0] += v[u][0] * xv; acc[1] += v[u][1] * xv; acc[2] += v[u][2] * xv; acc[3] += v[u][3] * xv;
        }
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) part[4 * threadIdx.x + e] = acc[e];
      __syncthreads();
      for (int t = threadIdx.x; t < 4 * QW && 4 * q0 + t < nsum; t += NT) {
        float sum = part[t];
        for (int k = 1; k < RG; ++k) sum += part[4 * k * QW + t];
        gout[4 * q0 + t] = sum;
      }
      __syncthreads();
    }
  }
};

// kRows rows of the stacked [V; G] a warp takes, their first quads in registers
struct FusedItemRows {
  static constexpr int QV = 1;  // quads a lane holds (rows of up to 128 DOFs)
  float v[kRows][QV][4];
  const float *rp[kRows];
  int nq[kRows];
  __device__ __forceinline__ void load(const FusedItem &it, const CellDesc &c, const float *__restrict__ vals, int r0) {
    const int lane = threadIdx.x & 31, nIp = (int)pad4(c.nI);
#pragma unroll
    for (int u = 0; u < kRows; ++u) {
      const int r = r0 + u;
      rp[u] = vals;
      nq[u] = 0;
      if (r < it.b) {
        if (r < c.nB) {
          rp[u] = vals + c.V_off + (long long)r * nIp;
          nq[u] = nIp / 4;
        } else {
          rp[u] = vals + c.G_off + tri_off(r - c.nB);
          nq[u] = (r - c.nB + 4) / 4;
        }
      }
#pragma unroll
      for (int h = 0; h < QV; ++h) ld4_stream(rp[u] + 4 * (lane + 32 * h), lane + 32 * h < nq[u], v[u][h]);
    }
  }
  __device__ __forceinline__ void dot(const float *xs, float (&acc)[kRows]) const {
    const int lane = threadIdx.x & 31;
    int maxq = 0;
#pragma unroll
    for (int u = 0; u < kRows; ++u) {
      acc[u] = 0.f;
      maxq = max(maxq, nq[u]);
    }
#pragma unroll
    for (int h = 0; h < QV; ++h) {
      float x[4] = {0.f, 0.f, 0.f, 0.f};
      if (lane + 32 * h < maxq) ld4(xs + 4 * (lane + 32 * h), x);
#pragma unroll
      for (int u = 0; u < kRows; ++u)
        acc[u] += v[u][h][0] * x[0] + v[u][h][1] * x[1] + v[u][h][2] * x[2] + v[u][h][3] * x[3];
    }
    for (int q = lane + 32 * QV; q < maxq; q += 32) {
      float x[4];
      ld4(xs + 4 * q, x);
#pragma unroll
      for (int u = 0; u < kRows; ++u) {
        float w[4];
        ld4_stream(rp[u] + 4 * q, q < nq[u], w);
        acc[u] += w[0] * x[0] + w[1] * x[1] + w[2] * x[2] + w[3] * x[3];
      }
    }
    // sums of rows 0 to 3 in lanes 0, 8, 16, 24 (a reduce-scatter: six exchanges)
    const bool h16 = (lane & 16) != 0, h8 = (lane & 8) != 0;
    float a = h16 ? acc[2] : acc[0], b = h16 ? acc[3] : acc[1];
    a += __shfl_xor_sync(0xffffffffu, h16 ? acc[0] : acc[2], 16);
    b += __shfl_xor_sync(0xffffffffu, h16 ? acc[1] : acc[3], 16);
    float k = h8 ? b : a;
    k += __shfl_xor_sync(0xffffffffu, h8 ? a : b, 8);
    k += __shfl_xor_sync(0xffffffffu, k, 4);
    k += __shfl_xor_sync(0xffffffffu, k, 2);
    k += __shfl_xor_sync(0xffffffffu, k, 1);
    acc[0] = k;  // row lane / 8
  }
};

// Forward: entities of level l and cells of level l + 1.  smem: gin, gout
// (max_sum each), x_I (pad4(max_nI)); or the entity units' buffers.
template <int NT>
__global__ void __launch_bounds__(NT, 512 / NT) k_level_fwd(FusedLevel L, const int *__restrict__ idx,
                                                               const long long *__restrict__ cptr,
                                                               const long long *__restrict__ cslot,
                                                               const float *__restrict__ vals,
                                                               const float *__restrict__ contrib_in,
                                                               float *__restrict__ contrib_out, float *__restrict__ xI,
                                                               const float *__restrict__ xin, float *__restrict__ xout) {
  constexpr int NW = NT / 32;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float *sm = reinterpret_cast<float *>(smem_raw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if ((int)blockIdx.x >= L.nitems) {
    const int u = blockIdx.x - L.nitems;
    if (u < L.nlarge) {
      group_fwd_unit<float, NT, float, true>(L.groups[L.large[u]], idx, cptr, cslot, vals, contrib_in, xin, xout, sm);
    } else {
      const int t = (u - L.nlarge) * NW + warp;
      if (t < L.nsmall)
        group_fwd_small_warp<float, float, true, true>(L.groups[L.small[t]], idx, cptr, cslot, vals, contrib_in, xin, xout,
                                                sm + 32 * warp);
      else
        pdl_enter();
    }
    return;
  }
  const FusedItem it = L.items[blockIdx.x];
  const FusedCell f = L.cells[it.cell];
  const CellDesc &c = f.c;
  const FusedPos *pos = L.pos + f.cat_off;
  const int nIp = (int)pad4(c.nI);
  float *gin = sm, *gout = gin + L.max_sum, *xs = gout + L.max_sum;
  const FusedPre pre = fused_pre(pos, f.nsum, cslot);
  const int im0 = (int)threadIdx.x < c.nI ? L.imap[f.map_off + threadIdx.x] : 0;
  FusedRows<NT> rows;
  rows.load(pos, f.nsum, vals, 0);
  FusedItemRows ir;
  ir.load(it, c, vals, it.a + warp * kRows);
  unit_dependency_point<true>();
  fused_gather<NT>(pre, pos, f.nsum, cslot, contrib_in, xin, gin);
  __syncthreads();
  fused_rows<NT>(rows, pos, f.nsum, vals, gin, gout);
  __syncthreads();
  for (int i = threadIdx.x; i < nIp; i += NT)
    xs[i] = i < c.nI ? gout[i == (int)threadIdx.x ? im0 : L.imap[f.map_off + i]] : 0.f;
  __syncthreads();
  const int *I = idx + c.I_off;
  for (int r0 = it.a + warp * kRows; r0 < it.b; r0 += NW * kRows) {
    // the lane that will hold a row's sum fetches its index beside the row's values
    const int rl = r0 + (lane >> 3);
    const bool mine = (lane & 7) == 0 && rl < it.b;
    const int il = mine && rl >= c.nB ? I[rl - c.nB] : 0;
    if (r0 != it.a + warp * kRows) ir.load(it, c, vals, r0);
    float acc[kRows];
    ir.dot(xs, acc);
    if (mine) {
      if (rl < c.nB) contrib_out[c.C_off + rl] = acc[0];
      else xI[il] = acc[0];
    }
  }
  if (it.first)
    for (int t = threadIdx.x; t < f.nsum; t += NT) {
      const int d = t == (int)threadIdx.x ? pre.p.dof : pos[t].dof;
      if (d >= 0) xout[d] = gout[t];
    }
}

// Backward: cells of level l + 1 and entities of level l.  smem: x_I forward values
// (pad4(max_nI)), x_B (pad4(max_nB)), x_I (pad4(max_nI)), gin, gout (max_sum each),
// partial sums (4 NT).
template <int NT>
__global__ void __launch_bounds__(NT, 512 / NT) k_level_bwd(FusedLevel L, const int *__restrict__ idx,
                                                               const float *__restrict__ vals,
                                                               const float *__restrict__ xI,
                                                               const float *__restrict__ xin, float *__restrict__ xout) {
  constexpr int NW = NT / 32;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float *sm = reinterpret_cast<float *>(smem_raw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if ((int)blockIdx.x >= L.ncells) {
    const int u = blockIdx.x - L.ncells;
    if (u < L.nlarge) {
      group_bwd_unit<float, NT, float, true>(L.groups[L.large[u]], idx, vals, xin, xout, sm);
    } else {
      const int t = (u - L.nlarge) * NW + warp;
      if (t < L.nsmall)
        group_bwd_small_warp<float, float, true, true>(L.groups[L.small[t]], idx, vals, xin, xout, sm + 32 * warp);
      else
        pdl_enter();
    }
    return;
  }
  const FusedCell f = L.cells[blockIdx.x];
  const CellDesc &c = f.c;
  const FusedPos *pos = L.pos + f.cat_off;
  const int nIp = (int)pad4(c.nI);
  float *xs = sm, *xb = xs + pad4(L.max_nI), *xi = xb + pad4(L.max_nB), *gin = xi + pad4(L.max_nI),
    *gout = gin + L.max_sum, *part = gout + L.max_sum;
  const int *I = idx + c.I_off, *B = idx + c.B_off;
  const float *V = vals + c.V_off, *G = vals + c.G_off;
  // layout of x_I = G^T x_I - V^T x_B by column quads, as cell_bwd_cols_f32; the
  // first rows of G and V, like the first rows of H, are loaded before the
  // dependency point
  const int nqc = nIp / 4, nblk = (nqc + 31) / 32, per = nblk ? (nqc + nblk - 1) / nblk : 0;
  int LW = 1;
  while (LW < per) LW <<= 1;
  const int ql = lane & (LW - 1), rg = (warp * 32 + lane) / LW, RG = NT / LW;
  constexpr int kU = 8;
  float vg[kU][4], vv[kU][4];
  auto load_g = [&](int q0, int i0) {
    const int q = q0 + ql;
    const bool ok = ql < per && q < nqc;
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int i = i0 + u * RG;
      ld4_stream(G + tri_off(i) + 4 * q, ok && i < c.nI && i >= 4 * q, vg[u]);
    }
  };
  auto load_v = [&](int q0, int r0) {
    const int q = q0 + ql;
    const bool ok = ql < per && q < nqc;
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int r = r0 + u * RG;
      ld4_stream(V + (long long)r * nIp + 4 * q, ok && r < c.nB, vv[u]);
    }
  };
  const int t0 = threadIdx.x;
  const int iI = t0 < c.nI ? I[t0] : -1, iB = t0 < c.nB ? B[t0] : -1;
  int d0 = -1, ip0 = -1;
  if (t0 < f.nsum) {
    d0 = pos[t0].dof;
    ip0 = pos[t0].ipos;
  }
  load_g(0, rg);
  load_v(0, rg);
  if (t0 < f.ng) {
    const FusedGroup g = L.fgroups[f.g_off + t0];
    prefetch_block_l2(vals + g.H_off, (long long)g.n * pad4(g.n));
  }
  unit_dependency_point<true>();
  {
    const float a = iI >= 0 ? __ldcg(xI + iI) : 0.f, b = iB >= 0 ? __ldcg(xin + iB) : 0.f;
    const float d = ip0 < 0 && d0 >= 0 ? __ldcg(xin + d0) : 0.f;  // redundant DOFs: their forward values
    if (t0 < c.nI) xs[t0] = a;
    if (t0 < c.nB) xb[t0] = b;
    if (t0 < f.nsum) gin[t0] = d;
  }
  for (int i = t0 + NT; i < c.nI; i += NT) xs[i] = __ldcg(xI + I[i]);
  for (int q = t0 + NT; q < c.nB; q += NT) xb[q] = __ldcg(xin + B[q]);
  for (int t = t0 + NT; t < f.nsum; t += NT) {
    const FusedPos p = pos[t];
    gin[t] = p.ipos < 0 && p.dof >= 0 ? __ldcg(xin + p.dof) : 0.f;
  }
  __syncthreads();
  for (int q0 = 0; q0 < nqc; q0 += per) {
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    for (int i0 = 4 * q0 + rg; i0 < c.nI; i0 += kU * RG) {
      if (q0 > 0 || i0 != rg) load_g(q0, i0);
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const float xv = i0 + u * RG < c.nI ? xs[i0 + u * RG] : 0.f;
        acc[0] += vg[u][0] * xv; acc[1] += vg[u][1] * xv; acc[2] += vg[u][2] * xv; acc[3] += vg[u][3] * xv;
      }
    }
    for (int r0 = rg; r0 < c.nB; r0 += kU * RG) {
      if (q0 > 0 || r0 != rg) load_v(q0, r0);
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const float xv = r0 + u * RG < c.nB ? xb[r0 + u * RG] : 0.f;
        acc[0] -= vv[u][0] * xv; acc[1] -= vv[u][1] * xv; acc[2] -= vv[u][2] * xv; acc[3] -= vv[u][3] * xv;
      }
    }
    for (int o = LW; o < 32; o <<= 1) {
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], o);
    }
    if (lane < LW) {
#pragma unroll
      for (int e = 0; e < 4; ++e) part[warp * 128 + 4 * lane + e] = acc[e];
    }
    __syncthreads();
    for (int t = t0; t < 4 * per && 4 * q0 + t < c.nI; t += NT) {
      float sum = part[t];
#pragma unroll
      for (int w = 1; w < NW; ++w) sum += part[w * 128 + t];
      xi[4 * q0 + t] = sum;
    }
    __syncthreads();
  }
  FusedCols<NT> cols;
  cols.first(pos, f.nsum, vals);
  for (int t = t0; t < f.nsum; t += NT) {
    const int ip = t == t0 ? ip0 : pos[t].ipos;
    if (ip >= 0) gin[t] = xi[ip];
  }
  __syncthreads();
  cols.run(pos, f.nsum, vals, gin, gout, part);
  for (int t = t0; t < f.nsum; t += NT) {
    const int d = t == t0 ? d0 : pos[t].dof;
    if (d >= 0) xout[d] = gout[t];
  }
}

// The entities of the last level around the root, in one CTA.  The "cell" is the
// root: its interior DOFs are the root's, in root order; the root is applied as the
// full symmetric matrix of k_root_dense.  smem: gin, gout (max_sum each), x_r, y_r
// (pad4(nr) each), partial sums (4 NT).
__global__ void __launch_bounds__(kFuseTopThreads) k_level_top(FusedLevel L, int nr, const float *__restrict__ vals,
                                                               const long long *__restrict__ cslot,
                                                               const float *__restrict__ Sr, int lds,
                                                               const float *__restrict__ contrib, const float *xin,
                                                               float *xout) {
  constexpr int NT = kFuseTopThreads, NW = NT / 32;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float *sm = reinterpret_cast<float *>(smem_raw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const FusedCell f = L.cells[0];
  const FusedPos *pos = L.pos + f.cat_off;
  const int nrp = (int)pad4(nr);
  float *gin = sm, *gout = gin + L.max_sum, *xr = gout + L.max_sum, *yr = xr + nrp, *part = yr + nrp;
  if ((int)threadIdx.x < f.ng) {
    const FusedGroup g = L.fgroups[f.g_off + threadIdx.x];
    prefetch_block_l2(vals + g.H_off, (long long)g.n * pad4(g.n));
  }
  if (threadIdx.x == 32) prefetch_block_l2(Sr, (long long)nr * lds);
  const FusedPre pre = fused_pre(pos, f.nsum, cslot);
  const int im0 = (int)threadIdx.x < nr ? L.imap[f.map_off + threadIdx.x] : 0;
  FusedRows<NT> rows;
  rows.load(pos, f.nsum, vals, 0);
  FusedCols<NT> cols;
  cols.first(pos, f.nsum, vals);
  unit_dependency_point<true>();
  fused_gather<NT>(pre, pos, f.nsum, cslot, contrib, xin, gin);
  __syncthreads();
  fused_rows<NT>(rows, pos, f.nsum, vals, gin, gout);
  __syncthreads();
  for (int i = threadIdx.x; i < nrp; i += NT)
    xr[i] = i < nr ? gout[i == (int)threadIdx.x ? im0 : L.imap[f.map_off + i]] : 0.f;
  __syncthreads();
  for (int r0 = warp * kRows; r0 < nr; r0 += NW * kRows) {  // x_r = S_r x_r
    float acc[kRows];
    int nq[kRows];
    const float *rp[kRows];
#pragma unroll
    for (int u = 0; u < kRows; ++u) {
      rp[u] = Sr + (long long)(r0 + u < nr ? r0 + u : 0) * lds;
      nq[u] = r0 + u < nr ? nrp / 4 : 0;
    }
    warp_rows_dot4<float, float>(rp, nq, xr, acc);
    if (lane == 0) {
#pragma unroll
      for (int u = 0; u < kRows; ++u)
        if (r0 + u < nr) yr[r0 + u] = acc[u];
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < f.nsum; t += NT) {
    const int ip = t == (int)threadIdx.x ? pre.p.ipos : pos[t].ipos;
    gin[t] = ip >= 0 ? yr[ip] : gout[t];
  }
  __syncthreads();
  cols.run(pos, f.nsum, vals, gin, gout, part);
  for (int t = threadIdx.x; t < f.nsum; t += NT) {
    const int d = t == (int)threadIdx.x ? pre.p.dof : pos[t].dof;
    if (d >= 0) xout[d] = gout[t];
  }
}
