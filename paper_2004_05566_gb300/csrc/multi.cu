// Inverse apply for k right-hand sides at once (hif_apply_multi): the top
// levels of F^{-1} (Eq. Ainv: R_l for the levels stored in BF16, and the root
// A_L^{-1} of Eq. 3_4) as tensor-core products on GB300.
//
// With k columns stacked, every per-box step of the apply is a small matrix
// product Y (m x k) = A (m x K) X (K x k), A a stored factor block:
//   cells, forward  (E_l^T):  [xI_I ; c_B] = [G ; V] x_I
//   cells, backward (E_l):    x_I = [G^T | -V^T] [xI_I ; x_B]
//   entities, forward / backward (K_l^T C_l^T / C_l K_l): x_g = H x_g, x_g = H^T x_g
//   root (A_L^{-1} = G_r^T G_r): t = G_r x_r, then x_r = G_r^T t
// (G = L^{-1}, V = A_BI A_II^{-1}, H = K^T C^T restricted to the entity).  A is
// read from the BF16 copy of the factor, X is split into a high and a low
// BF16 part (X = X_hi + X_lo to about 16 bits), and both products accumulate in
// FP32 in tensor memory: the result is that of BF16 factor blocks applied to
// the FP32 vectors, the arithmetic of the single-column BF16 levels.
//
// Kernel (one CTA of 256 threads per 128-row tile of one box): the K
// dimension is walked in chunks of 64; each chunk of A and of X_hi / X_lo is
// staged by the threads into shared memory in the canonical K-major layout
// without swizzle (8 x 16-byte core matrices), three chunks deep; one thread
// issues tcgen05.mma (M = 128, N = k rounded up to 16, K = 16 per
// instruction, kind::f16 with BF16 operands and FP32 accumulation) and
// commits each chunk to an mbarrier, so the staging of chunk c + 1 overlaps the
// products of chunk c.  What bounds it is the latency of the staging loads and
// the stores into the layout: the operands of chunk c + 1 are in registers
// before chunk c is stored, and a transposed block goes out as 16-byte rows
// (63^3, 16 columns: level-1 cells backward 283 -> 171 us, forward 154 -> 73 us;
// root 54 + 52 -> 29 + 37 us).  The accumulator lives in tensor memory (128 lanes x N
// columns, allocated per CTA) and is read back with tcgen05.ld, a 32-lane
// quarter and half the columns by each of the eight warps.  Every mbarrier wait is bounded; on expiry
// the CTA records the failure in the handle's error slot and skips its
// results (reported as HIF_ETIMEOUT by the solve).
#include "internal.h"

#include <cuda_bf16.h>

#include <algorithm>
#include <vector>

namespace hifcn {

namespace {

using bf16 = __nv_bfloat16;

constexpr int kTM = 128;      // rows of a tile (M of the MMA)
constexpr int kKC = 64;       // K of a staged chunk (4 MMAs of K = 16)
constexpr int kMThreads = 256;   // 8 warps stage; warp w reads TMEM lanes 32 (w % 4)..
constexpr int kMStages = 3;      // staged chunks in flight
constexpr uint32_t kSbo = 128;               // bytes between core matrices along M / N
constexpr uint32_t kLboA = 16 * 128 + 16;    // bytes between core matrices along K (A), padded
constexpr long long kMmaWaitLimit = 1LL << 24;

enum MPhase { kMCellFwd = 0, kMCellBwd, kMGroupFwd, kMGroupBwd, kMRootRows, kMRootCols };

// One CTA's work: rows [r0, r0 + 128) of a box, K chunks [c0, c1).  When a
// box's K is split over several CTAs (poff >= 0) each writes its partial tile
// (128 rows of npad floats) to the scratch at poff, and k_box_reduce adds the
// splits in order; otherwise (poff < 0) the CTA stores the results itself.
struct MTile {
  int unit, r0, c0, c1;
  long long poff;
};
// floats of one partial tile (any k up to kMultiMaxCols)
constexpr long long kPartTile = (long long)kTM * kMultiMaxCols;
// a tile whose K was split: nks partial tiles at poff, poff + kPartTile, ...
struct RTile {
  int unit, r0, nks, pad;
  long long poff;
};

struct MArgs {
  const MTile *tiles;
  const CellDesc *cells;
  const GroupDesc *groups;
  const int *idx;
  const bf16 *v16;
  const float *v32;         // FP32 values (the levels below the BF16 ones)
  const long long *gs_off;  // per entity of the level: offset of its inputs in gs
  long long root_G_off;
  const int *ridx;
  int nr;
  int ncols, npad;          // right-hand sides, and N of the MMA (ncols rounded up to 16)
  float *x, *xI, *contrib, *gs, *rt;
  long long ldx, ldc, ldg, ldr;  // column strides of x / xI, contrib, gs, rt
  float *part;                   // partial tiles of split boxes
  double *err;
};

__device__ __forceinline__ uint32_t su32(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// shared-memory matrix descriptor of tcgen05 (K-major, no swizzle):
// start address, leading (K) and stride (M/N) byte offsets, version 1
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo & 0x3FFFFu) >> 4) << 16) |
         ((uint64_t)((sbo & 0x3FFFFu) >> 4) << 32) | ((uint64_t)1 << 46);
}

// instruction descriptor of tcgen05.mma kind::f16: FP32 accumulator, BF16 A
// and B, both K-major, N >> 3, M >> 4
__host__ __device__ constexpr uint32_t mma_idesc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t parity) {
  for (long long it = 0; it < kMmaWaitLimit; ++it) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

// rows m and K of a box's operator, by phase
struct Box {
  int m, K;
};

__device__ __forceinline__ Box box_of(const MArgs &a, int ph, int unit) {
  switch (ph) {
    case kMCellFwd: {
      const CellDesc &c = a.cells[unit];
      return {c.nI + c.nB, c.nI};
    }
    case kMCellBwd: {
      const CellDesc &c = a.cells[unit];
      return {c.nI, c.nI + c.nB};
    }
    case kMGroupFwd:
    case kMGroupBwd: {
      const int n = a.groups[unit].n;
      return {n, n};
    }
    default:
      return {a.nr, a.nr};
  }
}

// Stored row `row` of the block a product reads (A's row for the forward
// phases, A's column for the transposed ones): its BF16 pointer and the padded
// length that may be read (zeros beyond the row's own entries).
struct SRow {
  const bf16 *p;
  int len;
};

__device__ __forceinline__ SRow stored_row(const MArgs &a, int ph, const CellDesc &c, const GroupDesc &g, int row) {
  switch (ph) {
    case kMCellFwd:
    case kMCellBwd:
      if (row < c.nI) return {a.v16 + c.G_off + tri_off(row), (int)pad4(row + 1)};
      return {a.v16 + c.V_off + (long long)(row - c.nI) * pad4(c.nI), (int)pad4(c.nI)};
    case kMGroupFwd:
    case kMGroupBwd:
      return {a.v16 + g.H_off + (long long)row * pad4(g.n), (int)pad4(g.n)};
    default:
      return {a.v16 + a.root_G_off + tri_off(row), (int)pad4(row + 1)};
  }
}

__device__ __forceinline__ uint32_t a_off(int i, int kk) {  // i in [0,128), kk in [0,64)
  return (uint32_t)(kk >> 3) * kLboA + (uint32_t)(i >> 3) * kSbo + (uint32_t)(i & 7) * 16 + (uint32_t)(kk & 7) * 2;
}

// The thread's share of a chunk of A (tile rows r0.., K k0..k0+63) in
// registers.  Forward: quads (row t / 16 + 16 j, K 4 (t % 16)).  Transposed:
// rows i = 4 (t % 32).. of the stored rows k0 + 8 (t / 32) + j, i.e. an
// 8 (K) x 4 (M) block.
__device__ __forceinline__ void load_a(const MArgs &a, int ph, bool transposed, const CellDesc &c,
                                       const GroupDesc &g, const Box &bx, int r0, int k0, uint2 (&v)[8]) {
  const int t = threadIdx.x;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    v[j] = make_uint2(0u, 0u);
    if (!transposed) {
      const int row = r0 + (t >> 4) + 16 * j, k = k0 + 4 * (t & 15);
      if (row < bx.m) {
        const SRow sr = stored_row(a, ph, c, g, row);
        if (k < sr.len) v[j] = *reinterpret_cast<const uint2 *>(sr.p + k);
      }
    } else {
      const int row = k0 + 8 * (t >> 5) + j, i = r0 + 4 * (t & 31);
      if (row < bx.K) {
        const SRow sr = stored_row(a, ph, c, g, row);
        if (i < sr.len) v[j] = *reinterpret_cast<const uint2 *>(sr.p + i);
        if (ph == kMCellBwd && row >= c.nI) {  // -V^T
          v[j].x ^= 0x80008000u;
          v[j].y ^= 0x80008000u;
        }
      }
    }
  }
}

// ... and into shared memory.  The transposed block becomes four 16-byte core
// matrix rows (8 K of one M each); the four go out in an order rotated by lane so
// that a quarter warp covers all banks (2-byte stores at a stride of 64 bytes
// were 16-way conflicts, most of the kernel's time).
__device__ __forceinline__ void store_a(bool transposed, const uint2 (&v)[8], unsigned char *sA) {
  const int t = threadIdx.x;
  if (!transposed) {
#pragma unroll
    for (int j = 0; j < 8; ++j) *reinterpret_cast<uint2 *>(sA + a_off((t >> 4) + 16 * j, 4 * (t & 15))) = v[j];
    return;
  }
  uint4 o[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    uint32_t w[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const uint32_t lo = u < 2 ? v[2 * e].x : v[2 * e].y, hi = u < 2 ? v[2 * e + 1].x : v[2 * e + 1].y;
      w[e] = __byte_perm(lo, hi, (u & 1) ? 0x7632 : 0x5410);
    }
    o[u] = make_uint4(w[0], w[1], w[2], w[3]);
  }
  const int q = t & 31, rot = (q >> 1) & 3;
  if (rot & 1) {
    const uint4 x = o[0];
    o[0] = o[1]; o[1] = o[2]; o[2] = o[3]; o[3] = x;
  }
  if (rot & 2) {
    uint4 x = o[0];
    o[0] = o[2]; o[2] = x;
    x = o[1];
    o[1] = o[3]; o[3] = x;
  }
#pragma unroll
  for (int u = 0; u < 4; ++u)
    *reinterpret_cast<uint4 *>(sA + a_off(4 * q + ((u + rot) & 3), 8 * (t >> 5))) = o[u];
}

// The thread's share of a chunk of X: K index k (-1 row index: absent),
// columns t / 64 + 4 j.  x_row gives the row of the source vector, load_b the values.
__device__ __forceinline__ int x_row(const MArgs &a, int ph, const CellDesc &c, const Box &bx, int k) {
  if (k >= bx.K) return -1;
  switch (ph) {
    case kMCellFwd: return a.idx[c.I_off + k];
    case kMCellBwd: return k < c.nI ? a.idx[c.I_off + k] : a.idx[c.B_off + k - c.nI];
    case kMRootRows: return a.ridx[k];
    default: return k;
  }
}

template <int NQ>
__device__ __forceinline__ void load_b(const MArgs &a, int ph, const CellDesc &c, const float *gsrc, int k, int xi,
                                       float (&v)[NQ]) {
  const float *src = a.x;
  long long ld = a.ldx;
  if (ph == kMCellBwd && k < c.nI) src = a.xI;
  if (ph == kMGroupFwd || ph == kMGroupBwd) {
    src = gsrc;
    ld = a.ldg;
  }
  if (ph == kMRootCols) {
    src = a.rt;
    ld = a.ldr;
  }
#pragma unroll
  for (int j = 0; j < NQ; ++j) {
    const int n = ((int)threadIdx.x >> 6) + 4 * j;
    v[j] = xi >= 0 && n < a.ncols ? src[n * ld + xi] : 0.f;
  }
}

// X_hi and X_lo into the canonical layout (K-direction stride padded by 16
// bytes, as A's)
template <int NQ>
__device__ __forceinline__ void store_b(const float (&v)[NQ], unsigned char *sBh, unsigned char *sBl, uint32_t lboB) {
  const int kk = threadIdx.x & (kKC - 1);
#pragma unroll
  for (int j = 0; j < NQ; ++j) {
    const int n = ((int)threadIdx.x >> 6) + 4 * j;
    const bf16 hi = __float2bfloat16_rn(v[j]);
    const bf16 lo = __float2bfloat16_rn(v[j] - __bfloat162float(hi));
    const uint32_t off = (uint32_t)(kk >> 3) * lboB + (uint32_t)(n >> 3) * kSbo + (uint32_t)(n & 7) * 16 +
                         (uint32_t)(kk & 7) * 2;
    *reinterpret_cast<bf16 *>(sBh + off) = hi;
    *reinterpret_cast<bf16 *>(sBl + off) = lo;
  }
}

__device__ __forceinline__ void store_out(const MArgs &a, int ph, int unit, const Box &bx, int row, int n,
                                          float y) {
  if (row >= bx.m || n >= a.ncols) return;
  switch (ph) {
    case kMCellFwd: {
      const CellDesc &c = a.cells[unit];
      if (row < c.nI) a.xI[n * a.ldx + a.idx[c.I_off + row]] = y;
      else a.contrib[n * a.ldc + c.C_off + row - c.nI] = y;
      return;
    }
    case kMCellBwd: {
      const CellDesc &c = a.cells[unit];
      a.x[n * a.ldx + a.idx[c.I_off + row]] = y;
      return;
    }
    case kMGroupFwd:
    case kMGroupBwd: {
      const GroupDesc &g = a.groups[unit];
      a.x[n * a.ldx + a.idx[g.idx_off + row]] = y;
      return;
    }
    case kMRootRows:
      a.rt[n * a.ldr + row] = y;
      return;
    default:
      a.x[n * a.ldx + a.ridx[row]] = y;
  }
}

// Dynamic shared memory: kMStages x (A chunk, X_hi chunk, X_lo chunk).
__host__ __device__ constexpr size_t a_chunk_bytes() { return (size_t)(kKC / 8) * kLboA; }
__host__ __device__ inline uint32_t b_lbo(int npad) { return (uint32_t)(npad / 8) * kSbo + 16; }
__host__ __device__ inline size_t b_chunk_bytes(int npad) { return (size_t)(kKC / 8) * b_lbo(npad); }
inline size_t mma_smem_bytes(int npad) { return kMStages * (a_chunk_bytes() + 2 * b_chunk_bytes(npad)); }

template <int NQ>  // columns padded to 4 NQ
__global__ void __launch_bounds__(kMThreads, NQ <= 8 ? 3 : 2) k_box_mma(MArgs a, int ph) {
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ uint32_t s_tmem;
  __shared__ __align__(8) unsigned long long s_bar[kMStages];
  __shared__ int s_fail;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const MTile tile = a.tiles[blockIdx.x];
  const Box bx = box_of(a, ph, tile.unit);
  const bool transposed = ph == kMCellBwd || ph == kMGroupBwd || ph == kMRootCols;
  const bool group = ph == kMGroupFwd || ph == kMGroupBwd;
  CellDesc cd{};
  GroupDesc gd{};
  if (ph == kMCellFwd || ph == kMCellBwd) cd = a.cells[tile.unit];
  if (group) gd = a.groups[tile.unit];
  const float *gsrc = group ? a.gs + a.gs_off[tile.unit] : nullptr;
  constexpr int npad = 4 * NQ;
  const uint32_t ncol_alloc = npad <= 32 ? 32u : (npad <= 64 ? 64u : 128u);
  const uint32_t lboB = b_lbo(npad);
  const size_t stage_bytes = a_chunk_bytes() + 2 * b_chunk_bytes(npad);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&s_tmem)),
                 "r"(ncol_alloc)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (t == 0) {
    for (int b = 0; b < kMStages; ++b)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(&s_bar[b])) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_fail = 0;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = s_tmem;
  const int nch = tile.c1 - tile.c0;  // chunks of this CTA (K chunks [c0, c1))
  const uint32_t idesc = mma_idesc(kTM, npad);
  bool ok = true;
  // chunk c + 1 is loaded into registers while chunk c is stored and multiplied,
  // and the rows of X it needs are looked up one chunk earlier still: the
  // loads' latency was what bound the kernel
  const int kx = t & (kKC - 1);
  uint2 av[8];
  float bv[NQ];
  int xi = -1;
  if (nch > 0) {
    const int k0 = tile.c0 * kKC;
    load_b<NQ>(a, ph, cd, gsrc, k0 + kx, x_row(a, ph, cd, bx, k0 + kx), bv);
    load_a(a, ph, transposed, cd, gd, bx, tile.r0, k0, av);
    xi = x_row(a, ph, cd, bx, k0 + kKC + kx);
  }
  for (int c = 0; c < nch; ++c) {
    const int b = c % kMStages;
    unsigned char *sA = smem + b * stage_bytes;
    unsigned char *sBh = sA + a_chunk_bytes(), *sBl = sBh + b_chunk_bytes(npad);
    // the products of chunk c - kMStages read this stage: wait for their commit
    if (c >= kMStages &&
        !mbar_wait_bounded(su32(&s_bar[b]), (uint32_t)(((c - kMStages) / kMStages) & 1)))
      ok = false;
    if (!ok) s_fail = 1;  // benign race: every writer stores 1
    if (ok) {
      store_a(transposed, av, sA);
      store_b<NQ>(bv, sBh, sBl, lboB);
      if (c + 1 < nch) {
        const int k1 = (tile.c0 + c + 1) * kKC;
        load_b<NQ>(a, ph, cd, gsrc, k1 + kx, xi, bv);
        load_a(a, ph, transposed, cd, gd, bx, tile.r0, k1, av);
        xi = x_row(a, ph, cd, bx, k1 + kKC + kx);
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (s_fail) {
      ok = false;
      break;
    }
    if (t == 0) {
      const uint32_t a0 = su32(sA), h0 = su32(sBh), l0 = su32(sBl);
#pragma unroll
      for (int ks = 0; ks < kKC / 16; ++ks) {
        const uint64_t ad = smem_desc(a0 + (uint32_t)ks * 2 * kLboA, kLboA, kSbo);
        const uint64_t hd = smem_desc(h0 + (uint32_t)ks * 2 * lboB, lboB, kSbo);
        const uint64_t ld = smem_desc(l0 + (uint32_t)ks * 2 * lboB, lboB, kSbo);
        const uint32_t acc = (c > 0 || ks > 0) ? 1u : 0u;
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
            "l"(ad), "l"(hd), "r"(idesc), "r"(acc)
            : "memory");
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
            "l"(ad), "l"(ld), "r"(idesc), "r"(1u)
            : "memory");
      }
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                       su32(&s_bar[b]))
                   : "memory");
    }
  }
  // the last commit covers every product issued before it
  if (ok && nch > 0 &&
      !mbar_wait_bounded(su32(&s_bar[(nch - 1) % kMStages]), (uint32_t)(((nch - 1) / kMStages) & 1)))
    ok = false;
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  // epilogue: warp w reads lanes 32 (w % 4) + lane, columns of half w / 4
  const int quarter = warp & 3, half = warp >> 2, hcols = npad / 2;
  if (ok && nch > 0) {
    const int row = tile.r0 + quarter * 32 + lane;
    for (int c0 = half * hcols; c0 < (half + 1) * hcols; c0 += 8) {
      uint32_t r[8];
      const uint32_t ta = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)c0;
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
          : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
          : "r"(ta));
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      if (tile.poff >= 0) {  // partial tile of a split box
        float *pt = a.part + tile.poff + (long long)(quarter * 32 + lane) * npad + c0;
#pragma unroll
        for (int j = 0; j < 8; ++j) pt[j] = __uint_as_float(r[j]);
      } else {
#pragma unroll
        for (int j = 0; j < 8; ++j) store_out(a, ph, tile.unit, bx, row, c0 + j, __uint_as_float(r[j]));
      }
    }
  } else if (ok && half == 0) {  // K = 0: the product is zero
    const int row = tile.r0 + quarter * 32 + lane;
    if (tile.poff >= 0) {
      float *pt = a.part + tile.poff + (long long)(quarter * 32 + lane) * npad;
      for (int n = 0; n < npad; ++n) pt[n] = 0.f;
    } else {
      for (int n = 0; n < a.ncols; ++n) store_out(a, ph, tile.unit, bx, row, n, 0.f);
    }
  } else if (t == 0) {
    a.err[0] = 1.0;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncol_alloc) : "memory");
}

// ------------------------------------------- FP32 levels, all columns at once
//
// The levels below the BF16 ones keep FP32 blocks and FP32 arithmetic, so
// their products Y (m x k) = A (m x K) X (K x k) run on the FP32 cores, each
// block read once for up to 32 columns instead of once per column.  One CTA of
// 128 threads takes a 128-row tile of a box; K is walked in chunks of 32,
// A and the gathered X staged by asynchronous copies three chunks deep.  A
// thread owns 4 rows x NC / 4 columns: per four K it reads 4 + 4 quads of
// shared memory for 4 NC multiply-adds.  A value of A enters NC products (four a
// byte at NC = 16), so at k = 16 the chip's 40e12 FMA/s would take 2.5e12 values/s,
// more than HBM delivers (1.7e12); the kernel stays below both (see the figures).
// Each chunk is summed on its own and added to the total, so a sum of K products
// rounds like one of 32 + K / 32.  kComp (the levels whose single-column backward step sums the
// boundary products with compensation): four products at a time enter the
// total by Kahan's summation.  Backward cells: the K index runs over the G
// rows padded to a multiple of 64, then the V rows, whose chunks are
// subtracted.
// Bound by shared-memory latency at 12 warps an SM, so four CTAs fit an SM
// (quads of a staged row swizzled instead of padded), and tiles skip the chunks
// that are zero by the triangle of G.
// Measured at 63^3 with 16 columns (level 0, 353 MB of blocks), per apply:
// forward 1720 us column by column, 206 at three CTAs, 162 now; backward 1568,
// 263, 222 (52 each at the copy rate).  Every tile of a box gathers the box's X
// again, 2.6 times the blocks' bytes in L2 sectors.
constexpr int kFThreads = 128;
constexpr int kFC = 32;          // K of a staged chunk
constexpr int kFStages = 3;

template <int NC>
__host__ __device__ constexpr size_t f32_stage_floats() { return (size_t)kTM * kFC + (size_t)kFC * NC; }

__device__ __forceinline__ void cp_async16(void *dst, const void *src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(su32(dst)), "l"(src), "r"(ok ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_async4(void *dst, const void *src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(su32(dst)), "l"(src), "r"(ok ? 4 : 0)
               : "memory");
}

// stored FP32 row `row` of a box and its padded length
struct FRow {
  const float *p;
  int len;
};
__device__ __forceinline__ FRow f32_row(const float *v, const CellDesc &c, const GroupDesc &g, bool cell, int row) {
  if (!cell) return {v + g.H_off + (long long)row * pad4(g.n), (int)pad4(g.n)};
  if (row < c.nI) return {v + c.G_off + tri_off(row), (int)pad4(row + 1)};
  return {v + c.V_off + (long long)(row - c.nI) * pad4(c.nI), (int)pad4(c.nI)};
}

template <int NC, bool kTrans, bool kComp>
__global__ void __launch_bounds__(kFThreads, NC <= 16 ? 4 : 3) k_box_f32(MArgs a, int ph) {
  extern __shared__ __align__(16) float fsm[];
  constexpr int CP = NC / 4;  // columns per thread
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const MTile tile = a.tiles[blockIdx.x];
  const int n0 = blockIdx.y * NC;
  const bool cell = ph == kMCellFwd || ph == kMCellBwd;
  CellDesc cd{};
  GroupDesc gd{};
  if (cell) cd = a.cells[tile.unit];
  else gd = a.groups[tile.unit];
  // rows of the product, stored rows (transposed: the K range), and the K
  // index of the first V row of a backward cell
  const int m = ph == kMCellFwd ? cd.nI + cd.nB : cell ? cd.nI : gd.n;
  const int K = cell ? cd.nI : gd.n;                       // K of the forward forms and of G
  const int kV = ph == kMCellBwd ? (cd.nI + 63) & ~63 : 1 << 30;
  const int c_begin = tile.c0 * (kKC / kFC), c_end = tile.c1 * (kKC / kFC);
  // staging of A: thread t copies quads t, t + 128, ... of the chunk
  const int sq = kTrans ? (t & 31) : (t & 7);              // quad within a staged row
  const int srow = kTrans ? (t >> 5) : (t >> 3);           // first staged row of the thread
  constexpr int kSRows = 8;                                // staged rows per thread
  constexpr int kSStep = kTrans ? kFThreads / 32 : kFThreads / 8;
  FRow fr[kTrans ? 1 : kSRows];
  if constexpr (!kTrans) {
#pragma unroll
    for (int j = 0; j < kSRows; ++j) {
      const int row = tile.r0 + srow + kSStep * j;
      fr[j] = row < m ? f32_row(a.v32, cd, gd, cell, row) : FRow{a.v32, 0};
    }
  }
  // gathered input row kk of the chunk at K index k: index -1 when absent
  auto x_index = [&](int k) -> int {
    if (!cell) return k < K ? k : -1;
    if (ph == kMCellFwd) return k < K ? a.idx[cd.I_off + k] : -1;
    if (k < kV) return k < cd.nI ? a.idx[cd.I_off + k] : -1;
    return k - kV < cd.nB ? a.idx[cd.B_off + k - kV] : -1;
  };
  const float *gsrc = cell ? nullptr : a.gs + a.gs_off[tile.unit];
  const int xk = t & (kFC - 1), xn = t / kFC;              // X element: row xk, columns xn + 4 j
  int xi = c_begin < c_end ? x_index(c_begin * kFC + xk) : -1;  // of the next chunk to stage
  auto stage = [&](int c) {
    if (c < c_end) {
      float *sA = fsm + (size_t)((c - c_begin) % kFStages) * f32_stage_floats<NC>();
      float *sX = sA + (size_t)kTM * kFC;
      const int k0 = c * kFC;
      if constexpr (kTrans) {
#pragma unroll
        for (int j = 0; j < kSRows; ++j) {
          const int kk = srow + kSStep * j, k = k0 + kk;
          const int row = k < kV ? (k < K ? k : -1) : (k - kV < cd.nB ? cd.nI + k - kV : -1);
          FRow f{a.v32, 0};
          if (row >= 0) f = f32_row(a.v32, cd, gd, cell, row);
          const int i = tile.r0 + 4 * sq;
          const bool ok = i < f.len;
          cp_async16(sA + kk * kTM + 4 * sq, f.p + (ok ? i : 0), ok);
        }
      } else {
#pragma unroll
        for (int j = 0; j < kSRows; ++j) {
          const int k = k0 + 4 * sq;
          const bool ok = k < fr[j].len;
          const int r = srow + kSStep * j;  // quads of a row swizzled against bank conflicts
          cp_async16(sA + r * kFC + 4 * (sq ^ (r & 7)), fr[j].p + (ok ? k : 0), ok);
        }
      }
      const float *src;
      long long ld;
      if (!cell) {
        src = gsrc + (xi >= 0 ? xi : 0);
        ld = a.ldg;
      } else {
        src = (ph == kMCellBwd && k0 < kV ? a.xI : a.x) + (xi >= 0 ? xi : 0);
        ld = a.ldx;
      }
#pragma unroll
      for (int j = 0; j < CP; ++j) {
        const int n = n0 + xn + 4 * j;
        const bool ok = xi >= 0 && n < a.ncols;
        cp_async4(sX + xk * NC + xn + 4 * j, src + (ok ? n * ld : 0), ok);
      }
      if (c + 1 < c_end) xi = x_index(k0 + kFC + xk);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  stage(c_begin);
  stage(c_begin + 1);
  const int cg = lane & 3, rg = warp * 8 + (lane >> 2);
  float tot[4][CP], cmp[4][kComp ? CP : 1];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
#pragma unroll
    for (int j = 0; j < CP; ++j) tot[u][j] = 0.f;
#pragma unroll
    for (int j = 0; j < (kComp ? CP : 1); ++j) cmp[u][j] = 0.f;
  }
  for (int c = c_begin; c < c_end; ++c) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kFStages - 2) : "memory");
    __syncthreads();
    stage(c + kFStages - 1);
    const float *sA = fsm + (size_t)((c - c_begin) % kFStages) * f32_stage_floats<NC>();
    const float *sX = sA + (size_t)kTM * kFC;
    const bool neg = c * kFC >= kV;
    float acc[4][CP];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int j = 0; j < CP; ++j) acc[u][j] = 0.f;
#pragma unroll 2
    for (int kk = 0; kk < kFC; kk += 4) {
      float av[4][4];  // [row][k] or, transposed, [k][row]
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float4 v = *reinterpret_cast<const float4 *>(kTrans ? sA + (kk + u) * kTM + 4 * rg
                                                                  : sA + (rg + 32 * u) * kFC + (kk ^ (4 * (rg & 7))));
        av[u][0] = v.x; av[u][1] = v.y; av[u][2] = v.z; av[u][3] = v.w;
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float xv[CP];
        const float *px = sX + (kk + q) * NC + cg * CP;
        if constexpr (CP == 2) {
          const float2 v = *reinterpret_cast<const float2 *>(px);
          xv[0] = v.x; xv[1] = v.y;
        } else {
#pragma unroll
          for (int j = 0; j < CP; j += 4) {
            const float4 v = *reinterpret_cast<const float4 *>(px + j);
            xv[j] = v.x; xv[j + 1] = v.y; xv[j + 2] = v.z; xv[j + 3] = v.w;
          }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int j = 0; j < CP; ++j) acc[u][j] = fmaf(kTrans ? av[q][u] : av[u][q], xv[j], acc[u][j]);
      }
      if constexpr (kComp) {  // Kahan's summation of the four products' sum
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int j = 0; j < CP; ++j) {
            const float y = __fsub_rn(neg ? -acc[u][j] : acc[u][j], cmp[u][j]);
            const float s = __fadd_rn(tot[u][j], y);
            cmp[u][j] = __fsub_rn(__fsub_rn(s, tot[u][j]), y);
            tot[u][j] = s;
            acc[u][j] = 0.f;
          }
      }
    }
    if constexpr (!kComp) {
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int j = 0; j < CP; ++j) tot[u][j] += neg ? -acc[u][j] : acc[u][j];
    }
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int lr = kTrans ? 4 * rg + u : rg + 32 * u, row = tile.r0 + lr;
    if constexpr (kComp)
#pragma unroll
      for (int j = 0; j < CP; ++j) tot[u][j] -= cmp[u][j];
    if (tile.poff >= 0) {  // partial tile of a split box
#pragma unroll
      for (int j = 0; j < CP; ++j) {
        const int n = n0 + cg * CP + j;
        if (n < a.npad) a.part[tile.poff + (long long)lr * a.npad + n] = tot[u][j];
      }
      continue;
    }
    if (row >= m) continue;
    float *dst;
    long long ld = a.ldx;
    if (!cell) {
      dst = a.x + a.idx[gd.idx_off + row];
    } else if (ph == kMCellBwd) {
      dst = a.x + a.idx[cd.I_off + row];
    } else if (row < cd.nI) {
      dst = a.xI + a.idx[cd.I_off + row];
    } else {
      dst = a.contrib + cd.C_off + row - cd.nI;
      ld = a.ldc;
    }
#pragma unroll
    for (int j = 0; j < CP; ++j) {
      const int n = n0 + cg * CP + j;
      if (n < a.ncols) dst[n * ld] = tot[u][j];
    }
  }
}

// the split boxes: rows of a tile added over its K splits in order, then stored
__global__ void __launch_bounds__(kTM) k_box_reduce(MArgs a, int ph, const RTile *__restrict__ rt) {
  const RTile r = rt[blockIdx.x];
  const Box bx = box_of(a, ph, r.unit);
  const int row = threadIdx.x;
  const long long stride = kPartTile;
  for (int n = 0; n < a.ncols; ++n) {
    float y = 0.f;
    for (int k = 0; k < r.nks; ++k) y += a.part[r.poff + k * stride + (long long)row * a.npad + n];
    store_out(a, ph, r.unit, bx, r.r0 + row, n, y);
  }
}

// entity inputs of a level for all columns: gs_c[goff_g + i] = x_c[g_i]
// (forward: minus the cells' contributions to g_i)
__global__ void __launch_bounds__(256) k_multi_gather(const GroupDesc *__restrict__ groups, int ngroups,
                                                      const int *__restrict__ idx,
                                                      const long long *__restrict__ cptr,
                                                      const long long *__restrict__ cslot,
                                                      const long long *__restrict__ gs_off, bool fwd,
                                                      const float *__restrict__ x, long long ldx,
                                                      const float *__restrict__ contrib, long long ldc,
                                                      float *__restrict__ gs, long long ldg, int ncols) {
  const int gi = blockIdx.x;
  if (gi >= ngroups) return;
  const GroupDesc g = groups[gi];
  const long long o = gs_off[gi];
  for (int e = threadIdx.x; e < g.n * ncols; e += blockDim.x) {
    const int i = e % g.n, n = e / g.n;
    float v = x[n * ldx + idx[g.idx_off + i]];
    if (fwd) {
      const long long p0 = cptr[g.cptr_off + i], p1 = cptr[g.cptr_off + i + 1];
      for (long long q = p0; q < p1; ++q) v -= contrib[n * ldc + cslot[q]];
    }
    gs[n * ldg + o + i] = v;
  }
}

__global__ void k_cols_to_float(const double *__restrict__ X, float *__restrict__ Y, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    Y[i] = (float)X[i];
}
__global__ void k_cols_to_double(const float *__restrict__ X, double *__restrict__ Y, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    Y[i] = (double)X[i];
}

}  // namespace

// The CTAs of one phase (tiles, possibly split along K) and the tiles to
// reduce afterwards (device arrays).
struct PhaseWork {
  MTile *tiles = nullptr;
  int ntiles = 0;
  RTile *rtiles = nullptr;
  int nrtiles = 0;
  long long part_floats = 0;
};

// Per-handle state of the multi-column apply (built on first use).
struct MultiState {
  int cap = 0;  // columns the buffers hold
  float *x = nullptr, *xI = nullptr, *contrib = nullptr, *gs = nullptr, *rt = nullptr;
  // per-column CG state of cn_step_multi (FP64 vectors, scalars, partials, tickets)
  int cg_cap = 0;
  double *g = nullptr, *cx = nullptr, *r = nullptr, *p = nullptr, *q = nullptr, *w = nullptr;
  double *scal = nullptr, *part = nullptr;
  unsigned *tk = nullptr;
  long long ldc = 0, ldg = 0, ldr = 0;
  // per top level: the work of the cell forward, cell backward and entity
  // phases (the entity forward and backward share theirs), per-entity gs
  // offsets; the root's rows and columns
  std::vector<PhaseWork> cf, cb, grp;
  std::vector<long long *> goff;
  PhaseWork root, root_t;
  float *tpart = nullptr;  // partial tiles of split boxes (largest phase)
};

void destroy_multi_state(Handle *h) {
  // all device buffers of the state are handle allocations (freed with it)
  delete static_cast<MultiState *>(h->multi);
  h->multi = nullptr;
}

namespace {

template <typename T>
int upload_vec(Handle *h, const std::vector<T> &v, T **out) {
  *out = nullptr;
  if (v.empty()) return HIF_OK;
  HIF_TRY(dev_alloc(h, (void **)out, v.size() * sizeof(T)));
  HIF_CUDA_TRY(cudaMemcpy(*out, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice));
  return HIF_OK;
}

// A box's operator: m rows, K; tri > 0: its first tri rows are lower
// triangular (row r ends at K index r), tri < 0: its columns start at the
// diagonal (row r begins at K index r).
struct BoxSize {
  int m, K, tri;
};

// CTAs of a phase: every 128-row tile of every box, over the K chunks that are
// not zero by the triangle; a phase with few tiles splits K so that about
// kTargetCtas CTAs run (at least 4 chunks per split), the splits of a tile
// adding up in k_box_reduce.
int build_phase(Handle *h, const std::vector<BoxSize> &sizes, PhaseWork *w) {
  constexpr int kTargetCtas = 3 * 152;
  long long T = 0;
  for (const BoxSize &b : sizes) T += (b.m + kTM - 1) / kTM;
  const int ks = (int)std::max<long long>(1, std::min<long long>(16, (kTargetCtas + T - 1) / std::max<long long>(T, 1)));
  std::vector<MTile> tiles;
  std::vector<RTile> rts;
  long long poff = 0;
  for (int u = 0; u < (int)sizes.size(); ++u) {
    const int m = sizes[u].m, K = sizes[u].K, tri = sizes[u].tri;
    for (int r = 0; r < m; r += kTM) {
      const int lo = tri < 0 ? r / kKC : 0;
      const int hi = tri > 0 && r + kTM <= tri ? (r + kTM + kKC - 1) / kKC : (K + kKC - 1) / kKC;
      const int nch = hi - lo;
      int nks = std::max(1, std::min(ks, nch / 4));
      const int cps = nks > 1 ? (nch + nks - 1) / nks : nch;
      nks = nks > 1 ? (nch + cps - 1) / cps : 1;
      if (nks == 1) {
        tiles.push_back({u, r, lo, hi, -1});
        continue;
      }
      rts.push_back({u, r, nks, 0, poff});
      for (int k = 0; k < nks; ++k) {
        tiles.push_back({u, r, lo + k * cps, lo + std::min(nch, (k + 1) * cps), poff});
        poff += kPartTile;
      }
    }
  }
  HIF_TRY(upload_vec(h, tiles, &w->tiles));
  HIF_TRY(upload_vec(h, rts, &w->rtiles));
  w->ntiles = (int)tiles.size();
  w->nrtiles = (int)rts.size();
  w->part_floats = poff;
  return HIF_OK;
}

int build_multi_state(Handle *h, int k) {
  MultiState *M = static_cast<MultiState *>(h->multi);
  if (M && M->cap >= k) return HIF_OK;
  const int cap = std::max(k, M ? 2 * M->cap : 16);
  if (!M) {
    M = new MultiState();
    h->multi = M;
    const int L = h->L, lb = std::min(h->bf16_lb, L);
    M->cf.assign(L, PhaseWork{});
    M->cb.assign(L, PhaseWork{});
    M->grp.assign(L, PhaseWork{});
    M->goff.assign(L, nullptr);
    long long gsz = 0, part = 0;
    for (int l = 0; l < L; ++l) {
      const LevelHost &H = h->lv_host[l];
      std::vector<BoxSize> cf, cb, gr;
      for (const CellDesc &d : H.cells) {
        cf.push_back({d.nI + d.nB, d.nI, d.nI});
        // the FP32 kernel starts the V rows on a chunk of their own
        cb.push_back({d.nI, (l < lb ? (d.nI + kKC - 1) / kKC * kKC : d.nI) + d.nB, -1});
      }
      std::vector<long long> off(std::max<size_t>(1, H.groups.size()), 0);
      long long o = 0;
      for (int g = 0; g < (int)H.groups.size(); ++g) {
        off[g] = o;
        o += pad4(H.groups[g].n);
        gr.push_back({H.groups[g].n, H.groups[g].n, 0});
      }
      gsz = std::max(gsz, o);
      HIF_TRY(build_phase(h, cf, &M->cf[l]));
      HIF_TRY(build_phase(h, cb, &M->cb[l]));
      HIF_TRY(build_phase(h, gr, &M->grp[l]));
      part = std::max({part, M->cf[l].part_floats, M->cb[l].part_floats, M->grp[l].part_floats});
      HIF_TRY(dev_alloc(h, (void **)&M->goff[l], off.size() * sizeof(long long)));
      HIF_CUDA_TRY(cudaMemcpy(M->goff[l], off.data(), off.size() * sizeof(long long), cudaMemcpyHostToDevice));
    }
    if (h->root_n > 0) {
      HIF_TRY(build_phase(h, {{h->root_n, h->root_n, h->root_n}}, &M->root));
      HIF_TRY(build_phase(h, {{h->root_n, h->root_n, -1}}, &M->root_t));
    }
    part = std::max({part, M->root.part_floats, M->root_t.part_floats});
    HIF_TRY(dev_alloc(h, (void **)&M->tpart, (size_t)std::max<long long>(part, 4) * sizeof(float)));
    M->ldg = std::max<long long>(gsz, 4);
  }
  M->ldc = std::max<long long>(h->max_contrib, 4);
  M->ldr = std::max<long long>(pad4(h->root_n), 4);
  const long long N = h->N;
  HIF_TRY(dev_alloc(h, (void **)&M->x, (size_t)cap * N * sizeof(float)));
  HIF_TRY(dev_alloc(h, (void **)&M->xI, (size_t)cap * N * sizeof(float)));
  HIF_TRY(dev_alloc(h, (void **)&M->contrib, (size_t)cap * M->ldc * sizeof(float)));
  HIF_TRY(dev_alloc(h, (void **)&M->gs, (size_t)cap * M->ldg * sizeof(float)));
  HIF_TRY(dev_alloc(h, (void **)&M->rt, (size_t)cap * M->ldr * sizeof(float)));
  M->cap = cap;  // earlier (smaller) buffers stay allocated until the handle is destroyed
  return HIF_OK;
}

MArgs phase_args(Handle *h, MultiState *M, int level, const PhaseWork &w, int k) {
  const LevelDev *lv = level >= 0 ? &h->lv[level] : nullptr;
  MArgs a{};
  a.tiles = w.tiles;
  a.part = M->tpart;
  a.cells = lv ? lv->cells : nullptr;
  a.groups = lv ? lv->groups : nullptr;
  a.idx = h->idx;
  a.v16 = static_cast<const bf16 *>(h->bf16_vals);
  a.v32 = h->f32.vals;
  a.gs_off = level >= 0 ? M->goff[level] : nullptr;
  a.root_G_off = h->root_G_off;
  a.ridx = h->idx + h->root_idx_off;
  a.nr = h->root_n;
  a.ncols = k;
  a.npad = std::max(16, (k + 15) / 16 * 16);
  a.x = M->x;
  a.xI = M->xI;
  a.contrib = M->contrib;
  a.gs = M->gs;
  a.rt = M->rt;
  a.ldx = h->N;
  a.ldc = M->ldc;
  a.ldg = M->ldg;
  a.ldr = M->ldr;
  a.err = h->scal + kScalErr;
  return a;
}

// the FP32 levels: column tiles of 8, 16 or 32
template <int NC, bool kTrans, bool kComp>
int launch_f32_nc(const MArgs &a, int ph, int ntiles, int k, cudaStream_t s) {
  const size_t sm = kFStages * f32_stage_floats<NC>() * sizeof(float);
  HIF_CUDA_TRY(cudaFuncSetAttribute(k_box_f32<NC, kTrans, kComp>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)sm));
  k_box_f32<NC, kTrans, kComp><<<dim3(ntiles, (k + NC - 1) / NC), kFThreads, sm, s>>>(a, ph);
  return HIF_OK;
}
template <bool kTrans, bool kComp>
int launch_f32_cols(const MArgs &a, int ph, int ntiles, int k, cudaStream_t s) {
  if (k <= 8) return launch_f32_nc<8, kTrans, kComp>(a, ph, ntiles, k, s);
  if (k <= 16) return launch_f32_nc<16, kTrans, kComp>(a, ph, ntiles, k, s);
  return launch_f32_nc<32, kTrans, kComp>(a, ph, ntiles, k, s);
}

int launch_f32(Handle *h, MultiState *M, int ph, int level, const PhaseWork &w, int k, cudaStream_t s) {
  if (w.ntiles <= 0) return HIF_OK;
  const MArgs a = phase_args(h, M, level, w, k);
  StatScope sc(h, ph == kMCellFwd ? "multi_cell_fwd" : ph == kMCellBwd ? "multi_cell_bwd"
                  : ph == kMGroupFwd ? "multi_group_fwd" : "multi_group_bwd", level, 0.0, s);
  if (ph == kMCellBwd && level_uses_sform(h, level)) HIF_TRY((launch_f32_cols<true, true>(a, ph, w.ntiles, k, s)));
  else if (ph == kMCellBwd || ph == kMGroupBwd) HIF_TRY((launch_f32_cols<true, false>(a, ph, w.ntiles, k, s)));
  else HIF_TRY((launch_f32_cols<false, false>(a, ph, w.ntiles, k, s)));
  note_launch();
  if (w.nrtiles > 0) {
    k_box_reduce<<<w.nrtiles, kTM, 0, s>>>(a, ph, w.rtiles);
    note_launch();
  }
  HIF_CUDA_TRY(cudaGetLastError());
  return HIF_OK;
}

int launch_mma(Handle *h, MultiState *M, int ph, int level, const PhaseWork &w, int k, cudaStream_t s) {
  if (w.ntiles <= 0) return HIF_OK;
  const MArgs a = phase_args(h, M, level, w, k);
  const size_t sm = mma_smem_bytes(a.npad);
  auto kern = a.npad == 16 ? k_box_mma<4> : a.npad == 32 ? k_box_mma<8> : a.npad == 48 ? k_box_mma<12> : k_box_mma<16>;
  HIF_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  StatScope sc(h, ph == kMCellFwd ? "mma_cell_fwd" : ph == kMCellBwd ? "mma_cell_bwd"
                  : ph == kMGroupFwd ? "mma_group_fwd" : ph == kMGroupBwd ? "mma_group_bwd"
                  : ph == kMRootRows ? "mma_root_rows" : "mma_root_cols",
               level, 0.0, s);
  kern<<<w.ntiles, kMThreads, sm, s>>>(a, ph);
  note_launch();
  if (w.nrtiles > 0) {
    k_box_reduce<<<w.nrtiles, kTM, 0, s>>>(a, ph, w.rtiles);
    note_launch();
  }
  HIF_CUDA_TRY(cudaGetLastError());
  return HIF_OK;
}

int launch_gather(Handle *h, MultiState *M, int level, bool fwd, int k, cudaStream_t s) {
  const LevelDev &lv = h->lv[level];
  if (!lv.ngroups) return HIF_OK;
  k_multi_gather<<<lv.ngroups, 256, 0, s>>>(lv.groups, lv.ngroups, h->idx, h->cptr, h->cslot, M->goff[level],
                                           fwd, M->x, h->N, M->contrib, M->ldc, M->gs, M->ldg, k);
  note_launch();
  HIF_CUDA_TRY(cudaGetLastError());
  return HIF_OK;
}

}  // namespace

int multi_cg_buffers(Handle *h, int k, MultiCG *out) {
  HIF_TRY(build_multi_state(h, k));
  MultiState *M = static_cast<MultiState *>(h->multi);
  const long long N = h->N;
  const int nb = h->nblocks_vec;
  if (M->cg_cap < k) {
    const int cap = M->cap;
    for (double **v : {&M->g, &M->cx, &M->r, &M->p, &M->q, &M->w})
      HIF_TRY(dev_alloc(h, (void **)v, (size_t)cap * N * sizeof(double)));
    HIF_TRY(dev_alloc(h, (void **)&M->scal, (size_t)cap * 16 * sizeof(double)));
    HIF_TRY(dev_alloc(h, (void **)&M->part, (size_t)cap * 4 * nb * sizeof(double)));
    HIF_TRY(dev_alloc(h, (void **)&M->tk, (size_t)cap * 4 * sizeof(unsigned)));
    HIF_CUDA_TRY(cudaMemset(M->scal, 0, (size_t)cap * 16 * sizeof(double)));
    HIF_CUDA_TRY(cudaMemset(M->tk, 0, (size_t)cap * 4 * sizeof(unsigned)));
    M->cg_cap = cap;
  }
  out->g = M->g;
  out->x = M->cx;
  out->r = M->r;
  out->p = M->p;
  out->q = M->q;
  out->w = M->w;
  out->scal = M->scal;
  out->part = M->part;
  out->tk = M->tk;
  out->z = M->x;
  out->nb = nb;
  return HIF_OK;
}

// X (N x k FP32, column-major) <- F^{-1} X for all columns at once: the FP32
// levels on the FP32 cores, the BF16 levels and the root on the tensor cores.
int apply_multi_f32(Handle *h, int k, cudaStream_t s) {
  MultiState *M = static_cast<MultiState *>(h->multi);
  const int L = h->L, lb = std::min(h->bf16_lb, L);
  auto launch_box = [&](int ph, int l, const PhaseWork &w) {
    return l < lb ? launch_f32(h, M, ph, l, w, k, s) : launch_mma(h, M, ph, l, w, k, s);
  };
  for (int l = 0; l < L; ++l) {
    HIF_TRY(launch_box(kMCellFwd, l, M->cf[l]));
    HIF_TRY(launch_gather(h, M, l, true, k, s));
    HIF_TRY(launch_box(kMGroupFwd, l, M->grp[l]));
  }
  if (h->root_n > 0) {
    HIF_TRY(launch_mma(h, M, kMRootRows, -1, M->root, k, s));
    HIF_TRY(launch_mma(h, M, kMRootCols, -1, M->root_t, k, s));
  }
  for (int l = L - 1; l >= 0; --l) {
    HIF_TRY(launch_gather(h, M, l, false, k, s));
    HIF_TRY(launch_box(kMGroupBwd, l, M->grp[l]));
    HIF_TRY(launch_box(kMCellBwd, l, M->cb[l]));
  }
  return HIF_OK;
}

int multi_check(Handle *h, int k, const char *fn) {
  if (!h->has_bf16 || !h->has_f32) {
    set_last_error(std::string(fn) + ": the handle was not set up with HIF_FP32_BF16TOP");
    return HIF_EINVAL;
  }
  if (k < 1 || k > kMultiMaxCols) {
    set_last_error(std::string(fn) + ": k must lie in [1, HIF_MULTI_MAX_COLS]");
    return HIF_EINVAL;
  }
  return HIF_OK;
}

int apply_multi(Handle *h, const double *X, double *Y, int k, cudaStream_t s) {
  HIF_TRY(multi_check(h, k, "hif_apply_multi"));
  HIF_TRY(build_multi_state(h, k));
  MultiState *M = static_cast<MultiState *>(h->multi);
  const long long n = (long long)k * h->N;
  k_cols_to_float<<<1216, 256, 0, s>>>(X, M->x, n);
  note_launch();
  HIF_TRY(apply_multi_f32(h, k, s));
  k_cols_to_double<<<1216, 256, 0, s>>>(M->x, Y, n);
  note_launch();
  HIF_CUDA_TRY(cudaGetLastError());
  return HIF_OK;
}

}  // namespace hifcn
