// Grid kernels of the PCG extension solve: right-hand side, masked biharmonic apply, CG vector
// update, residual replacement and output.  All are persistent launches over a work list of
// (slot, tile) items so that one launch serves a single solve, a batch or the serving loop.
//
// The operator is eq. (discrete_biharmonic) of Sec. 2.1 with the boundary rules of Algorithm 1
// (Dirichlet padding), half-sample reflection (symmetric) or wrap-around (periodic), evaluated
// matrix-free ("no need to form the 13-banded matrix", Sec. 2.2).
//
// CG vectors are double-float pairs of FP32 planes (hi, lo); see SlotDesc.
#include <algorithm>

#include "async.cuh"
#include "common.cuh"
#include "kernels.h"

namespace bx {

constexpr int kHX = kStTileX + 4;  // 68
constexpr int kHY = kStTileY + 4;  // 36
constexpr int kHalo = kHX * kHY;

__device__ __forceinline__ void tile_origin(const SlotDesc& S, int tile, int& x0, int& y0) {
  const int tx = (S.nx + kStTileX - 1) / kStTileX;
  x0 = (tile % tx) * kStTileX;
  y0 = (tile / tx) * kStTileY;
}

// Map halo position i of the tile to (global index, sign); sign 0 = outside / zero node.
__device__ __forceinline__ int halo_src(const SlotDesc& S, int x0, int y0, int i, float& s) {
  const int ly = i / kHX, lx = i - ly * kHX;
  const int gy = y0 - 2 + ly, gx = x0 - 2 + lx;
  if (gx > S.nx + 1 || gy > S.ny + 1) { s = 0.f; return 0; }
  float sx, sy;
  const int mx = ghost(gx, S.nx, S.bcx, sx);
  const int my = ghost(gy, S.ny, S.bcy, sy);
  s = sx * sy;
  return my * S.nx + mx;
}

// The operator on unequal spacings: the 13-point sum of a smem tile (row stride RS) at local
// (ly+2, lx+2), as a compensated FP32 sum (s, c) that carries the exact sum of the 13 products to about
// 48 bits.
template <int RS>
__device__ __forceinline__ CompSum stencil13_acc(const SlotDesc& S, const float* t, int ly, int lx) {
  const float* c = t + (ly + 2) * RS + (lx + 2);
  const float C = c[0];
  const float E0 = c[-1], E1 = c[1], N0 = c[-RS], N1 = c[RS];
  const float D0 = c[-RS - 1], D1 = c[-RS + 1], D2 = c[RS - 1], D3 = c[RS + 1];
  const float F0 = c[-2], F1 = c[2], G0 = c[-2 * RS], G1 = c[2 * RS];
  CompSum acc;
  acc.add_prod(S.wc, C);
  acc.add_prod(S.wex, E0); acc.add_prod(S.wex, E1);
  acc.add_prod(S.wey, N0); acc.add_prod(S.wey, N1);
  acc.add_prod(S.wd, D0); acc.add_prod(S.wd, D1); acc.add_prod(S.wd, D2); acc.add_prod(S.wd, D3);
  acc.add_prod(S.wfx, F0); acc.add_prod(S.wfx, F1);
  acc.add_prod(S.wfy, G0); acc.add_prod(S.wfy, G1);
  // low parts of the weights: products far below the result's ulp, plain FP32 suffices
  float lo = S.wc_l * C + S.wex_l * (E0 + E1) + S.wey_l * (N0 + N1) +
             S.wd_l * ((D0 + D1) + (D2 + D3)) + S.wfx_l * (F0 + F1) + S.wfy_l * (G0 + G1);
  acc.c = __fadd_rn(acc.c, lo);
  return acc;
}

// The same stencil applied in plain FP32 (for the lo plane of a double-float vector, whose
// contribution is 2^-24 of the hi plane's: its own rounding is far below the result's ulp).
template <int RS>
__device__ __forceinline__ float stencil13_plain(const SlotDesc& S, const float* t, int ly, int lx) {
  const float* c = t + (ly + 2) * RS + (lx + 2);
  const float e = (c[-1] + c[1]), n = (c[-RS] + c[RS]);
  const float d = (c[-RS - 1] + c[-RS + 1]) + (c[RS - 1] + c[RS + 1]);
  const float f = c[-2] + c[2], g = c[-2 * RS] + c[2 * RS];
  return S.wc * c[0] + S.wex * e + S.wey * n + S.wd * d + S.wfx * f + S.wfy * g;
}

// The operator on equal spacings is the five-point g(u) = (sum of the four neighbours) - 4 u taken
// twice (M g(g(p)); the boundary rules make g at a ghost node the reflected, wrapped or zero one).
// One application at two adjacent nodes (x, x+1) of the smem planes h (hi) and l (lo) with an even
// row stride RS, h and l pointing at node x, an even index: error-free TwoSums of the hi plane
// (4 u is exact), the errors and the lo plane's five points in plain FP32.  33 packed operations;
// the 13-point sum of fourteen TwoSums that this replaced took 124 for the two planes, the two
// applications take 66 (and one node of w's ring per tile edge).
__device__ __forceinline__ float2 ld2(const float* p) { return *reinterpret_cast<const float2*>(p); }
template <int RS, bool LO = true>
__device__ __forceinline__ f2x2 lap_pair(const float* h, const float* l) {
  static_assert(RS % 2 == 0, "pairs of nodes start on 8-byte boundaries");
  const float2 C = ld2(h), Cm = ld2(h - 2), Cp = ld2(h + 2);
  float2 a, ea, b, eb, t, et, s, es;
  two_sum2(make_float2(Cm.y, C.x), make_float2(C.y, Cp.x), a, ea);
  two_sum2(ld2(h - RS), ld2(h + RS), b, eb);
  two_sum2(a, b, t, et);
  two_sum2(t, mul2(-4.f, C), s, es);
  float2 e = add2(es, add2(et, add2(ea, eb)));
  if (LO) {
    const float2 c = ld2(l), cm = ld2(l - 2), cp = ld2(l + 2);
    const float2 n = add2(add2(make_float2(cm.y, c.x), make_float2(c.y, cp.x)), add2(ld2(l - RS), ld2(l + RS)));
    e = add2(e, fma2(make_float2(-4.f, -4.f), c, n));
  }
  return {s, e};
}
// The first application over a tile's nodes and their ring of one: rows 1 .. TY + 2 and columns
// 2 .. 69 of the windows h, l into the same places of sh, sl.
template <int TY, int RS, bool LO = true>
__device__ __forceinline__ void lap_tile(const float* h, const float* l, float* sh, float* sl) {
  constexpr int kPairs = kStTileX / 2 + 2;
  for (int k = threadIdx.x; k < kPairs * (TY + 2); k += kStThreads) {
    const int r = k / kPairs, c = (1 + r) * RS + 2 + 2 * (k - r * kPairs);
    const f2x2 w = lap_pair<RS, LO>(h + c, l + c);
    *reinterpret_cast<float2*>(sh + c) = w.hi;
    *reinterpret_cast<float2*>(sl + c) = w.lo;
  }
}

__device__ __forceinline__ double stencil13_f64(const SlotDesc& S, const double* t, int ly, int lx) {
  const double* c = t + (ly + 2) * kHX + (lx + 2);
  return S.dwc * c[0] + S.dwex * (c[-1] + c[1]) + S.dwey * (c[-kHX] + c[kHX]) +
         S.dwd * ((c[-kHX - 1] + c[-kHX + 1]) + (c[kHX - 1] + c[kHX + 1])) +
         S.dwfx * (c[-2] + c[2]) + S.dwfy * (c[-2 * kHX] + c[2 * kHX]);
}

// ---------------------------------------------------------------------------------------------
// Setup: known mask from sign(phi) (Sec. 2.1), b = -M L^2 E_K f in FP64 (Algorithm 1, first
// statement), zero CG state.  Partials: ||b||^2, number of known nodes, number of invalid inputs
// (NaN phi, or a non-finite f at a known node).
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kStThreads)
k_setup(const SlotDesc* __restrict__ slots, const WorkItem* __restrict__ items,
        const int* __restrict__ n_items, const float* const* __restrict__ phis,
        const float* const* __restrict__ fs, const int* __restrict__ dirs) {
  __shared__ double sf[kHalo];
  __shared__ double red[64];
  __shared__ int s_last;
  const int total = *n_items;
  for (int w = blockIdx.x; w < total; w += gridDim.x) {
    const WorkItem it = items[w];
    const SlotDesc& S = slots[it.slot];
    const float* phi = phis[it.slot];
    const float* f = fs[it.slot];
    const bool out_dir = dirs[it.slot] == 0;
    int x0, y0;
    tile_origin(S, it.tile, x0, y0);
    for (int i = threadIdx.x; i < kHalo; i += blockDim.x) {
      float s;
      const int g = halo_src(S, x0, y0, i, s);
      double v = 0.0;
      if (s != 0.f) {
        const float ph = phi[g];
        const bool known = out_dir ? (ph < 0.f) : (ph > 0.f);
        v = known ? (double)s * (double)f[g] : 0.0;
      }
      sf[i] = v;
    }
    __syncthreads();
    double bb = 0.0, cnt = 0.0, bad = 0.0;
    for (int k = threadIdx.x; k < kStTileX * kStTileY; k += blockDim.x) {
      const int ly = k / kStTileX, lx = k - ly * kStTileX;
      const int gx = x0 + lx, gy = y0 + ly;
      if (gx >= S.nx || gy >= S.ny) continue;
      const int g = gy * S.nx + gx;
      const float ph = phi[g];
      const bool known = out_dir ? (ph < 0.f) : (ph > 0.f);
      if (ph != ph || (known && !isfinite(f[g]))) bad += 1.0;
      double bv = 0.0;
      if (!known) bv = -stencil13_f64(S, sf, ly, lx);
      S.mask[g] = known ? 0 : 1;
      S.b[g] = bv;
      S.xhi[g] = 0.f;
      S.xlo[g] = 0.f;
      S.r[g] = 0.f;
      S.r_lo[g] = 0.f;
      S.p[0][g] = 0.f;
      S.p[1][g] = 0.f;
      S.p_lo[0][g] = 0.f;
      S.p_lo[1][g] = 0.f;
      S.q[g] = 0.f;
      S.q_lo[g] = 0.f;
      S.z[g] = 0.f;
      S.z_lo[g] = 0.f;
      bb += bv * bv;
      cnt += known ? 1.0 : 0.0;
    }
    block_sum2<kStThreads>(bb, cnt, red);
    double nn = bad, dummy = 0.0;
    block_sum2<kStThreads>(nn, dummy, red);
    if (threadIdx.x == 0) {
      S.part[it.tile * 4 + 0] = bb;
      S.part[it.tile * 4 + 1] = cnt;
      S.part[it.tile * 4 + 2] = nn;
    }
    if (last_item_block(&S.sc->cnt[0], S.n_st_tiles, &s_last)) {
      double sums[3];
      reduce_partials<kStThreads, 3>(S.part, S.n_st_tiles, sums, red);
      if (threadIdx.x == 0) {
        const double sb = sums[0], sk = sums[1], sn = sums[2];
        SlotScalars* sc = S.sc;
        // The extension is linear in f: the iteration runs on 2^e b with e chosen so that the
        // root mean square of 2^e b over the unknowns is near 1, which keeps the FP32 vectors
        // and their pairwise products inside FP32's range for any magnitude of f.  A power of
        // two changes no rounding; k_output scales the answer back.
        int e = 0;
        const double n_unk = (double)S.nx * (double)S.ny - sk;
        if (sb > 0.0 && isfinite(sb) && n_unk > 0.0) {
          int k;
          frexp(sb / n_unk, &k);
          e = max(-1000, min(1000, -(k / 2)));
        }
        sc->bexp = e;
        const double sbs = ldexp(sb, 2 * e);
        sc->bb = sbs;
        sc->rr = sbs;
        sc->rr_true = sbs;
        sc->rr_ref = sbs;
        sc->rho2[0] = sc->rho2[1] = 0.0;
        sc->beta = 0.0;
        sc->beta_f[0] = sc->beta_f[1] = 0.f;
        sc->alpha = 0.0;
        sc->it = 0;
        sc->fold = 0;
        sc->n_known = (int)sk;
        if (sn > 0.0 || !isfinite(sb)) {
          sc->status = -1;  // EXT_EINVAL: NaN in phi or a non-finite known value
          sc->active = 0;
          sc->need_prec = 0;
        } else if (sb == 0.0) {
          sc->status = ST_OK;  // b = 0: x = 0 is exact
          sc->active = 0;
          sc->need_prec = 0;
        } else {
          sc->status = ST_RUNNING;
          sc->active = 1;
          sc->need_prec = 1;
        }
      }
    }
    __syncthreads();
  }
}

// Set-up, second pass: r = 2^e b as a double-float pair, once the slot's scale exponent e is
// known.
__global__ void __launch_bounds__(kStThreads)
k_rhs_scale(const SlotDesc* __restrict__ slots, const WorkItem* __restrict__ items,
            const int* __restrict__ n_items) {
  const int total = *n_items;
  for (int w = blockIdx.x; w < total; w += gridDim.x) {
    const WorkItem it = items[w];
    const SlotDesc& S = slots[it.slot];
    if (S.sc->status != ST_RUNNING) continue;
    const int e = S.sc->bexp;
    int x0, y0;
    tile_origin(S, it.tile, x0, y0);
    for (int k = threadIdx.x; k < kStTileX * kStTileY; k += blockDim.x) {
      const int ly = k / kStTileX, lx = k - ly * kStTileX;
      const int gx = x0 + lx, gy = y0 + ly;
      if (gx >= S.nx || gy >= S.ny) continue;
      const int g = gy * S.nx + gx;
      const f2 v = df_of(ldexp(S.b[g], e));
      S.r[g] = v.hi;
      S.r_lo[g] = v.lo;
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Set-up of the single-stage entry points: the slot's mask from sign(phi) and the stage's input
// vector v.  OPERATOR: z = v, z_lo = 0 and a zero direction p[0], as at iteration 0 of a solve;
// otherwise the residual r = v, r_lo = 0.  25 (17) bytes a node, bound by HBM; the solve's full
// set-up (FP64 right-hand side, thirteen planes) took 40% of these calls at 2048^2 nodes and more.
// ---------------------------------------------------------------------------------------------
template <bool OPERATOR>
__global__ void __launch_bounds__(kVecThreads)
k_stage_setup(const SlotDesc* __restrict__ slots, const float* __restrict__ phi, const float* __restrict__ v,
              int extend_out) {
  const SlotDesc& S = slots[0];
  const int n = S.nx * S.ny;
  uint8_t* __restrict__ mask = S.mask;
  float* __restrict__ hi = OPERATOR ? S.z : S.r;
  float* __restrict__ lo = OPERATOR ? S.z_lo : S.r_lo;
  float* __restrict__ p = S.p[0];
  float* __restrict__ p_lo = S.p_lo[0];
  constexpr int U = 4;
  for (int e0 = blockIdx.x * U * kVecThreads + threadIdx.x; e0 < n; e0 += gridDim.x * U * kVecThreads) {
    float ph[U], x[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * kVecThreads;
      ph[u] = e < n ? __ldg(phi + e) : 0.f;
      x[u] = e < n ? __ldg(v + e) : 0.f;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * kVecThreads;
      if (e >= n) break;
      const bool known = extend_out ? (ph[u] < 0.f) : (ph[u] > 0.f);
      mask[e] = known ? 0 : 1;
      hi[e] = x[u];
      lo[e] = 0.f;
      if (OPERATOR) {
        p[e] = 0.f;
        p_lo[e] = 0.f;
      }
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Iteration, stage 1: p = z + beta p_old (formed in shared memory including the halo, in
// double-float), q = M L^2 p (Algorithm 1, matvec, with the mask in the epilogue), and p.q as
// partial sums over fixed 64 x 16 node blocks; k_pq_finish then forms alpha = rho / p.q.
//
// q is a double-float pair: on equal spacings the five-point g of p's pair taken twice (lap_pair: the
// first application into the p_old windows, a barrier, the second at the tile's nodes; tiles with
// no unknown node skip both), on unequal ones the exact 13-point sum of p's hi plane (compensated
// FP32) plus the same stencil of its lo plane in plain FP32.
//
// Tiles are 64 nodes wide and TY rows high (TY = 16 or 32, chosen per workspace by the
// autotuner).  Each block walks its share of the (slot, tile) list with two shared-memory window
// sets.  For a slot whose rows span a multiple of 16 bytes in the mask (nx % 16 == 0), the window
// set of the block's next tile arrives by tensor copies while it computes the current one: the hi
// and lo planes of z and p_old over rows y0-2 .. y0+TY+1 and columns x0-4 .. x0+67 (two columns
// wider on the left than the halo, so that each copy starts on a 16-byte boundary) and the tile's
// mask bytes.  Cells outside the grid arrive as zeros; the ghost cells of a boundary tile
// (reflected, wrapped or negated copies of grid nodes under the boundary rule) are gathered by
// plain loads.  Tiles of other slots fill the free window set with plain loads.
//
// The p.q partials do not depend on TY: they are per 64 x 16 block (a tile holds TY / 16 of
// them), each thread adds its nodes of a block in step order (the steps cover the block's rows
// in the same order for either TY), the warp adds its lanes in a fixed butterfly and the producer
// warp the eight warps in FP64 while the next tile is computed (added by a computing warp, the FP64 chain
// held up each tile: 288 us an operator call on 4096^2 nodes, 277 now), but for a block's last tile, whose
// sum the computing warps have sooner (1 us an iteration of 60 at 389 x 251); k_pq_finish adds the
// blocks in index order, so every tile height gives the same bits.
// ---------------------------------------------------------------------------------------------
constexpr int kWX = kStWinX;  // 72: window row, floats
static_assert(kStWinX == kStTileX + 8, "window columns");

template <int TY>
struct StGeom {
  static constexpr int kHYt = TY + 4;                       // halo rows
  static constexpr int kHalo = kHX * kHYt;                   // halo cells
  static constexpr int kWinBytes = kWX * kHYt * 4;           // one FP32 plane window
  static constexpr int kMaskBytes = kStTileX * TY;           // the tile's mask
  static constexpr int kBufBytes = 4 * kWinBytes + kMaskBytes;  // z, z_lo, p, p_lo, mask
  static constexpr int kGhostSlots = 4 * kHYt + 4 * kHX;     // candidate ghost cells of one halo
  static constexpr int kBlocksPerSm = TY == 32 ? 2 : 3;
  static constexpr int kSmemBytes = 2 * kBufBytes + 128;     // two window sets, alignment slack
  static constexpr int kOwn = kStTileX * TY / kStThreads;    // nodes per thread
  static_assert(kWinBytes % 128 == 0 && kBufBytes % 128 == 0, "tensor copy destinations");
  static_assert(kGhostSlots <= 2 * kStThreads, "two ghost candidates per thread");
  static_assert(kOwn * kStThreads == kStTileX * TY && kOwn % 2 == 0, "tile / block size");
  static_assert(kBlocksPerSm * (kSmemBytes + 1280) <= 228 * 1024, "window sets per SM");
};

__device__ __forceinline__ void tile_origin_ty(const SlotDesc& S, int tile, int ty, int& x0, int& y0) {
  const int tx = (S.nx + kStTileX - 1) / kStTileX;
  x0 = (tile % tx) * kStTileX;
  y0 = (tile / tx) * ty;
}

// Candidate k of a tile's ghost cells: the four ghost columns (x = -2, -1, nx, nx+1) over the
// halo's rows, then the four ghost rows over the halo's in-grid columns.  Returns false when the
// candidate lies outside the halo or beyond the second ghost line; (wy, wx) is its window cell.
template <int TY>
__device__ __forceinline__ bool ghost_cell(const SlotDesc& S, int x0, int y0, int k, int& wy,
                                           int& wx) {
  constexpr int kHYt = StGeom<TY>::kHYt;
  if (k < 4 * kHYt) {
    const int j = k / kHYt;
    wy = k - j * kHYt;
    const int gx = j < 2 ? j - 2 : S.nx + (j - 2);
    const int lx = gx - (x0 - 2);
    wx = lx + 2;
    return lx >= 0 && lx < kHX && y0 - 2 + wy <= S.ny + 1;
  }
  const int kk = k - 4 * kHYt;
  const int j = kk / kHX, lx = kk - j * kHX;
  const int gy = j < 2 ? j - 2 : S.ny + (j - 2);
  const int gx = x0 - 2 + lx;
  wy = gy - (y0 - 2);
  wx = lx + 2;
  return wy >= 0 && wy < kHYt && gx >= 0 && gx < S.nx;
}

// Halo cell i of a TY-row tile: (global index, sign); sign 0 = outside / zero node.
template <int TY>
__device__ __forceinline__ int halo_src_ty(const SlotDesc& S, int x0, int y0, int i, float& s) {
  const int ly = i / kHX, lx = i - ly * kHX;
  const int gy = y0 - 2 + ly, gx = x0 - 2 + lx;
  if (gx > S.nx + 1 || gy > S.ny + 1) { s = 0.f; return 0; }
  float sx, sy;
  const int mx = ghost(gx, S.nx, S.bcx, sx);
  const int my = ghost(gy, S.ny, S.bcy, sy);
  s = sx * sy;
  return my * S.nx + mx;
}

// A tile as the block's producer warp hands it to the eight that compute: what they need of the item,
// its slot and the slot's scalars, and whether its windows were copied.
struct StTile {
  const SlotDesc* S;  // null: the end of the list
  int x0, y0, par, copied;
  float beta_hi, beta_lo;
  bool last;          // the block's last item: the computing warps add its p.q themselves
};
constexpr int kStBlock = kStThreads + 32;  // the computing warps and the producer

__device__ __forceinline__ void st_bar() { asm volatile("bar.sync 1, %0;" ::"n"(kStThreads) : "memory"); }
// the same barrier, telling whether v is set in any of the computing threads
__device__ __forceinline__ bool st_bar_or(bool v) {
  uint32_t any;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "bar.red.or.pred q, 1, %2, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(any)
      : "r"(v ? 1u : 0u), "n"(kStThreads)
      : "memory");
  return any != 0;
}

// One warp: p.q of a tile's 16-row blocks (TY / 16 of them, so the partials do not depend on TY), each the FP64
// sum of eight warps' pairs.
template <int TY>
__device__ __forceinline__ void put_pq(const StTile& t, const float2 (&blk)[TY / 16][kStThreads / 32]) {
  const int lane = threadIdx.x & 31;
  const int j = (lane >> 3) & (TY / 16 - 1);  // eight lanes per block, one per warp's pair
  const double v = sum_of_eight(blk[j]);
  const int by = (t.y0 >> 4) + j;
  if ((lane & 7) == 0 && lane < TY / 2 && 16 * by < t.S->ny)
    t.S->pq_part[by * ((t.S->nx + kStTileX - 1) / kStTileX) + t.x0 / kStTileX] = v;
}

// The producer warp: for each of the block's tiles (those whose slot iterates) it waits for a free
// window set, starts the tensor copies (lane 0), forms beta (FUSE: from the preconditioner's partials,
// once per slot), stores p.q of the tile that the set held before and hands the tile over.  Done by a
// computing thread between two tiles, these dependent loads, tensor-map fences and copies took 3.5 K of a
// tile's 11.5 K cycles.
template <int TY, bool FUSE>
__device__ __forceinline__ void stencil_producer(const SlotDesc* __restrict__ slots,
                                                 const WorkItem* __restrict__ items, int total, unsigned char* sbuf,
                                                 uint64_t* full, uint64_t* empty, StTile* info,
                                                 const float2 (*blk_sm)[TY / 16][kStThreads / 32],
                                                 volatile int* abort_flag, long long wait_cycles) {
  using G = StGeom<TY>;
  const int lane = threadIdx.x & 31;
  // p.q of the tile that set b held, once the computing warps have released it
  auto flush = [&](int b) {
    const StTile t = info[b];
    if (!t.last) put_pq<TY>(t, blk_sm[b]);
    __syncwarp();  // the set's entry is written again next
  };
  int n = 0, slot = -1;
  bool last = true;  // of the tile handed over last
  f2 beta = {0.f, 0.f};
  auto acquire = [&](const SlotDesc& S) {
    if (lane < kStMaps && S.st_maps != nullptr)
      tmap_acquire(static_cast<const unsigned char*>(S.st_maps) + 128 * lane);
    __syncwarp();
  };
  if (static_cast<int>(blockIdx.x) < total) {  // what no kernel writes, before the wait
    slot = items[blockIdx.x].slot;
    acquire(slots[slot]);
  }
  int beta_slot = -1;
  pdl_wait();
  bool ok = true;
  for (int w = blockIdx.x; w < total && ok; w += gridDim.x) {
    const WorkItem it = items[w];
    const SlotDesc& S = slots[it.slot];
    SlotScalars* sc = S.sc;
    if (!sc->active) continue;
    if (it.slot != slot) {
      slot = it.slot;
      acquire(S);
    }
    const int b = n & 1, par = sc->it & 1;
    int x0, y0;
    tile_origin_ty(S, it.tile, TY, x0, y0);
    const unsigned char* maps = static_cast<const unsigned char*>(S.st_maps);
    if (lane == 0) {
      ok = mbar_wait(&empty[b], ((n >> 1) & 1) ^ 1, abort_flag, wait_cycles);
      if (ok && maps != nullptr) {
        unsigned char* dst = sbuf + b * G::kBufBytes;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_expect_tx_only(&full[b], G::kBufBytes);
        tma_load_2d(dst, maps, &full[b], x0 - 4, y0 - 2);
        tma_load_2d(dst + G::kWinBytes, maps + 128, &full[b], x0 - 4, y0 - 2);
        tma_load_2d(dst + 2 * G::kWinBytes, maps + 128 * (2 + 2 * par), &full[b], x0 - 4, y0 - 2);
        tma_load_2d(dst + 3 * G::kWinBytes, maps + 128 * (3 + 2 * par), &full[b], x0 - 4, y0 - 2);
        tma_load_2d(dst + 4 * G::kWinBytes, maps + 128 * 6, &full[b], x0, y0);
      }
    }
    ok = __shfl_sync(0xffffffffu, ok, 0);
    if (!ok) break;
    if (it.slot != beta_slot) {
      beta_slot = it.slot;
      if (FUSE) {
        // r.z, z.q -> beta in every block; the tile-0 block records the scalars.  A breakdown (a
        // non-finite r.z or beta) reaches p.q and rho, where the update finds it.
        double rz, zq;
        sum_rz(S, sc->flexible != 0, rz, zq);
        if (lane == 0) {
          const double bd = prec_beta(sc, rz, zq);
          beta = df_of(bd);
          if (it.tile == 0) record_preconditioner(sc, rz, zq, bd);
        }
      } else {
        beta = f2{sc->beta_f[0], sc->beta_f[1]};
      }
    }
    __syncwarp();  // every lane behind the wait for the set
    if (n >= 2) flush(b);
    last = w + static_cast<int>(gridDim.x) >= total;
    if (lane == 0) {
      info[b] = StTile{&S, x0, y0, par, maps != nullptr, beta.hi, beta.lo, last};
      mbar_arrive(&full[b]);
    }
    ++n;
  }
  // the end of the list, and p.q of the last two tiles
  auto released = [&](int k) {  // tile k's set, by the computing warps
    bool r = true;
    if (lane == 0) r = mbar_wait(&empty[k & 1], (k >> 1) & 1, abort_flag, wait_cycles);
    r = __shfl_sync(0xffffffffu, r, 0);
    __syncwarp();
    return r;
  };
  if (ok && n >= 2) {
    ok = released(n - 2);
    if (ok) flush(n & 1);
  }
  if (ok && lane == 0) {
    info[n & 1].S = nullptr;
    mbar_arrive(&full[n & 1]);
  }
  if (ok && !last && released(n - 1)) flush((n - 1) & 1);
  if (lane == 0) {
    // after an abort: the copies already issued (the last into each set) land before the block's
    // memory is released
    if (*abort_flag) {
      const long long t0 = clock64();
      for (int b = 0; b < 2; ++b) {
        const int k = (n - b + 1) / 2;  // tiles handed over in set b
        if (k > 0)
          while (!mbar_try(&full[b], (k - 1) & 1) && clock64() - t0 < kWaitCycles / 4) {
          }
      }
    }
  }
}

// Whether any of the calling thread's share of a tile's mask bytes is set (all threads: the tile).
template <int BYTES>
__device__ __forceinline__ int mask_any(const unsigned char* m) {
  static_assert(BYTES % (4 * kStThreads) == 0, "whole words per thread");
  unsigned v = 0;
#pragma unroll
  for (int i = 0; i < BYTES / (4 * kStThreads); ++i)
    v |= reinterpret_cast<const unsigned*>(m)[threadIdx.x + i * kStThreads];
  return v != 0;
}

template <bool ANISO, int TY, bool FUSE>
__global__ void __launch_bounds__(kStBlock, StGeom<TY>::kBlocksPerSm)
k_stencil(const SlotDesc* __restrict__ slots, const WorkItem* __restrict__ items,
          const int* __restrict__ n_items, int* __restrict__ err, long long wait_cycles) {
  using G = StGeom<TY>;
  extern __shared__ unsigned char st_smem_raw[];
  unsigned char* sbuf = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(st_smem_raw) + 127) & ~static_cast<uintptr_t>(127));
  __shared__ __align__(8) uint64_t full[2], empty[2];
  __shared__ StTile info[2];
  __shared__ int s_abort;
  __shared__ float2 blk_sm[2][TY / 16][kStThreads / 32];  // p.q of each warp in each 16-row block, by window set
  const int total = *n_items;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    for (int b = 0; b < 2; ++b) {
      mbar_init(&full[b], 1);
      mbar_init(&empty[b], 1);
    }
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncthreads();
  volatile int* abort_flag = &s_abort;
  if (warp == kStThreads / 32) {
    stencil_producer<TY, FUSE>(slots, items, total, sbuf, full, empty, info, blk_sm, abort_flag, wait_cycles);
  } else {
  pdl_wait();
  for (int n = 0;; ++n) {
    const int b = n & 1;
    if (st_bar_or(!mbar_wait(&full[b], (n >> 1) & 1, abort_flag, wait_cycles))) break;
    const StTile tile = info[b];
    if (tile.S == nullptr) break;
    const SlotDesc& S = *tile.S;
    const f2 beta = {tile.beta_hi, tile.beta_lo};
    const int par = tile.par, x0 = tile.x0, y0 = tile.y0;
    // plain loads of what the kernels before wrote: their lifetimes overlap this one's, so nothing here
    // may be read as read-only data (__ldg, const __restrict__)
    const float* pold = S.p[par];
    const float* pold_lo = S.p_lo[par];
    float* __restrict__ pnew = S.p[par ^ 1];
    float* __restrict__ pnew_lo = S.p_lo[par ^ 1];
    const float* z = S.z;
    const float* z_lo = S.z_lo;
    // a tile whose halo lies inside the grid has no ghost cell
    const bool interior = x0 >= 2 && y0 >= 2 && x0 + kStTileX + 2 <= S.nx && y0 + TY + 2 <= S.ny;
    unsigned char* buf = sbuf + b * G::kBufBytes;
    bool unknown;  // whether the tile has an unknown node
    if (tile.copied) {
      // ghost cells by plain loads, whose latency passes under the window's p
      int gcell[2] = {-1, -1};
      float gs[2] = {0.f, 0.f};
      f2 gz[2] = {{0.f, 0.f}, {0.f, 0.f}}, gp[2] = {{0.f, 0.f}, {0.f, 0.f}};
      if (!interior) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int k = threadIdx.x + h * kStThreads;
          int wy, wx;
          if (k < G::kGhostSlots && ghost_cell<TY>(S, x0, y0, k, wy, wx)) {
            float s;
            const int g = halo_src_ty<TY>(S, x0, y0, wy * kHX + (wx - 2), s);
            if (s != 0.f) {  // zero-sign ghosts stay the zeros the copy filled in
              gcell[h] = wy * kWX + wx;
              gs[h] = s;
              gz[h] = f2{z[g], z_lo[g]};
              gp[h] = f2{pold[g], pold_lo[g]};
            }
          }
        }
      }
      unknown = mask_any<G::kMaskBytes>(buf + 4 * G::kWinBytes);
      // p = z + beta p_old over the whole window, in place of z
      float4* zh = reinterpret_cast<float4*>(buf);
      float4* zl = reinterpret_cast<float4*>(buf + G::kWinBytes);
      const float4* ph = reinterpret_cast<const float4*>(buf + 2 * G::kWinBytes);
      const float4* pl = reinterpret_cast<const float4*>(buf + 3 * G::kWinBytes);
      for (int v = threadIdx.x; v < kWX * G::kHYt / 4; v += kStThreads) {
        const float4 a = zh[v], al = zl[v], c = ph[v], cl = pl[v];
        const f2x2 u = df_axpy2(beta, {make_float2(c.x, c.y), make_float2(cl.x, cl.y)},
                                {make_float2(a.x, a.y), make_float2(al.x, al.y)});
        const f2x2 t = df_axpy2(beta, {make_float2(c.z, c.w), make_float2(cl.z, cl.w)},
                                {make_float2(a.z, a.w), make_float2(al.z, al.w)});
        zh[v] = make_float4(u.hi.x, u.hi.y, t.hi.x, t.hi.y);
        zl[v] = make_float4(u.lo.x, u.lo.y, t.lo.x, t.lo.y);
      }
      unknown = st_bar_or(unknown);
      if (!interior) {
        float* wh = reinterpret_cast<float*>(buf);
        float* wl = reinterpret_cast<float*>(buf + G::kWinBytes);
#pragma unroll
        for (int h = 0; h < 2; ++h)
          if (gcell[h] >= 0) {
            const f2 v = df_add(gz[h], df_mul(gp[h], beta));
            wh[gcell[h]] = gs[h] * v.hi;
            wl[gcell[h]] = gs[h] * v.lo;
          }
        st_bar();
      }
    } else {
      // plain loads into the window set, kChunk cells per thread in flight at a time (a round is one
      // memory latency)
      float* wh = reinterpret_cast<float*>(buf);
      float* wl = reinterpret_cast<float*>(buf + G::kWinBytes);
      uint8_t* mt = buf + 4 * G::kWinBytes;
      for (int e = threadIdx.x; e < G::kMaskBytes; e += kStThreads) {
        const int ly = e / kStTileX, lx = e - ly * kStTileX;
        const int gx = x0 + lx, gy = y0 + ly;
        mt[e] = (gx < S.nx && gy < S.ny) ? S.mask[gy * S.nx + gx] : 0;
      }
      unknown = true;
      constexpr int kChunk = TY == 16 ? 6 : 5;  // one round of loads or two
#pragma unroll 1
      for (int i0 = 0; i0 < G::kHalo; i0 += kChunk * kStThreads) {
        int gi[kChunk];
        float gsg[kChunk];
        f2 zv[kChunk], pv[kChunk];
#pragma unroll
        for (int j = 0; j < kChunk; ++j) {
          const int i = i0 + threadIdx.x + j * kStThreads;
          gsg[j] = 0.f;
          gi[j] = 0;
          if (i < G::kHalo) gi[j] = halo_src_ty<TY>(S, x0, y0, i, gsg[j]);
        }
#pragma unroll
        for (int j = 0; j < kChunk; ++j) {
          const bool on = gsg[j] != 0.f;
          zv[j] = on ? f2{z[gi[j]], z_lo[gi[j]]} : f2{0.f, 0.f};
          pv[j] = on ? f2{pold[gi[j]], pold_lo[gi[j]]} : f2{0.f, 0.f};
        }
#pragma unroll
        for (int j = 0; j < kChunk; ++j) {
          const int i = i0 + threadIdx.x + j * kStThreads;
          if (i < G::kHalo) {
            const int ly = i / kHX, lx = i - ly * kHX;
            const f2 v = df_add(zv[j], df_mul(pv[j], beta));
            wh[ly * kWX + lx + 2] = gsg[j] * v.hi;
            wl[ly * kWX + lx + 2] = gsg[j] * v.lo;
          }
        }
      }
      st_bar();
    }
    const float* wh = reinterpret_cast<const float*>(buf);
    const float* wl = reinterpret_cast<const float*>(buf + G::kWinBytes);
    const uint8_t* mt = buf + 4 * G::kWinBytes;
    float* __restrict__ qh = S.q;
    float* __restrict__ ql = S.q_lo;
    // p.q of the tile's 64 x 16 blocks: each thread sums its nodes of one block in step order, the
    // warp its lanes in a fixed butterfly, and the producer the eight warps
    CompDotDF dot;
    if (!ANISO) {
      float* sh = reinterpret_cast<float*>(buf + 2 * G::kWinBytes);  // g(p), in place of p_old
      float* sl = reinterpret_cast<float*>(buf + 3 * G::kWinBytes);
      if (unknown) {  // uniform
        lap_tile<TY, kWX>(wh, wl, sh, sl);
        st_bar();
      }
      // node pairs (x, x+1): the window's row stride is even and x - x0 is even.  In a step the warp
      // covers one tile row; two steps (eight rows each) make a 16-row block, unrolled so that their
      // dependent chains overlap.
      const int gx = x0 + 2 * lane;
      const bool in0 = gx < S.nx, in1 = gx + 1 < S.nx;
      const int nx = S.nx, rows = S.ny - y0;
      const int wc0 = (warp + 2) * kWX + 2 * lane + 4;
#pragma unroll 1
      for (int j = 0; j < TY / 16; ++j) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int ly = warp + 8 * (2 * j + h);
          if (ly >= rows || !in0) continue;
          const int g = (y0 + ly) * nx + gx;
          const int wc = wc0 + 8 * (2 * j + h) * kWX;
          const float2 pvh = ld2(wh + wc), pvl = ld2(wl + wc);
          const unsigned m2 = *reinterpret_cast<const uint16_t*>(mt + ly * kStTileX + 2 * lane);
          f2x2 q2 = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
          if (m2) {
            const f2x2 a = lap_pair<kWX>(sh + wc, sl + wc);
            q2 = df_norm2(a.hi, a.lo);
          }
          const bool m0 = (m2 & 0xffu) != 0, m1 = (m2 >> 8) != 0;
          q2.hi = make_float2(m0 ? q2.hi.x : 0.f, m1 ? q2.hi.y : 0.f);
          q2.lo = make_float2(m0 ? q2.lo.x : 0.f, m1 ? q2.lo.y : 0.f);
          if (m0) dot.add(pvh.x, pvl.x, q2.hi.x, q2.lo.x);
          if (in1 && m1) dot.add(pvh.y, pvl.y, q2.hi.y, q2.lo.y);
          if (in1 && (g & 1) == 0) {
            *reinterpret_cast<float2*>(pnew + g) = pvh;
            *reinterpret_cast<float2*>(pnew_lo + g) = pvl;
            *reinterpret_cast<float2*>(qh + g) = q2.hi;
            *reinterpret_cast<float2*>(ql + g) = q2.lo;
          } else {
            pnew[g] = pvh.x;
            pnew_lo[g] = pvl.x;
            qh[g] = q2.hi.x;
            ql[g] = q2.lo.x;
            if (in1) {
              pnew[g + 1] = pvh.y;
              pnew_lo[g + 1] = pvl.y;
              qh[g + 1] = q2.hi.y;
              ql[g + 1] = q2.lo.y;
            }
          }
        }
        // the end of a 16-row block: every lane joins the butterfly
        group_sum_pair<32>(dot.s, dot.c);
        if (lane == 0) blk_sm[b][j][warp] = make_float2(dot.s, dot.c);
        dot = CompDotDF{};
      }
    } else {
      // one node per lane; in step j the warp covers 32 consecutive nodes of one tile row; four
      // steps (four rows each) make a 16-row block
#pragma unroll 1
      for (int j = 0; j < G::kOwn; ++j) {
        const int k = threadIdx.x + j * kStThreads;
        const int ly = k / kStTileX, lx = k - ly * kStTileX;
        const int gx = x0 + lx, gy = y0 + ly;
        if (gx < S.nx && gy < S.ny) {
          const int g = gy * S.nx + gx;
          const float pvh = wh[(ly + 2) * kWX + lx + 4], pvl = wl[(ly + 2) * kWX + lx + 4];
          f2 qv = {0.f, 0.f};
          if (mt[ly * kStTileX + lx]) {
            const CompSum a = stencil13_acc<kWX>(S, wh + 2, ly, lx);
            const float l = stencil13_plain<kWX>(S, wl + 2, ly, lx);
            qv = df_norm(a.s, __fadd_rn(a.c, l));
          }
          pnew[g] = pvh;
          pnew_lo[g] = pvl;
          qh[g] = qv.hi;
          ql[g] = qv.lo;
          dot.add(pvh, pvl, qv.hi, qv.lo);
        }
        if ((j & 3) == 3) {
          group_sum_pair<32>(dot.s, dot.c);
          if (lane == 0) blk_sm[b][j >> 2][warp] = make_float2(dot.s, dot.c);
          dot = CompDotDF{};
        }
      }
    }
    st_bar();
    // the window set, the tile's entry and its sums go back to the producer, which adds up the sums
    if (threadIdx.x == 0) mbar_arrive(&empty[b]);
    if (tile.last && warp == 0) put_pq<TY>(tile, blk_sm[b]);
  }
  }
  __syncthreads();
  if (threadIdx.x == 0 && s_abort) raise_flag(err);
}

// One block per slot (the slot's tile-0 item of the per-slot list): p.q from the stencil's
// block partials (64 x 16 nodes) in a fixed order, alpha = rho / p.q, breakdown detection.
__global__ void __launch_bounds__(32)
k_pq_finish(const SlotDesc* __restrict__ slots, const WorkItem* __restrict__ items,
            const int* __restrict__ n_items) {
  const int total = *n_items;
  pdl_wait();
  for (int w = blockIdx.x; w < total; w += gridDim.x) {
    const SlotDesc& S = slots[items[w].slot];
    if (!S.sc->active) continue;
    const double pq = sum_pq(S);
    __syncwarp();  // every lane has read `active`
    if (threadIdx.x == 0) finish_pq(S.sc, pq);
  }
}

// An update item of a small slot among larger ones: the segments, and so the partial sums, of
// k_update_slice.
__device__ __forceinline__ CompDotDF update_segment(const SlotDesc& S, int tile, int pi, f2 alpha) {
  const Seg g = seg_of(S, tile);
  const f2 nalpha = {-alpha.hi, -alpha.lo};
  CompDotDF dot;
  const float4 ph = g.load(S.p[pi]), pl = g.load(S.p_lo[pi]), qh = g.load(S.q), ql = g.load(S.q_lo);
  float4 rh = g.load(S.r), rl = g.load(S.r_lo), xh = g.load(S.xhi), xl = g.load(S.xlo);
  df_axpy(xh.x, xl.x, alpha, ph.x, pl.x);
  df_axpy(xh.y, xl.y, alpha, ph.y, pl.y);
  df_axpy(xh.z, xl.z, alpha, ph.z, pl.z);
  df_axpy(xh.w, xl.w, alpha, ph.w, pl.w);
  g.store(S.xhi, xh);
  g.store(S.xlo, xl);
  df_axpy(rh.x, rl.x, nalpha, qh.x, ql.x);
  df_axpy(rh.y, rl.y, nalpha, qh.y, ql.y);
  df_axpy(rh.z, rl.z, nalpha, qh.z, ql.z);
  df_axpy(rh.w, rl.w, nalpha, qh.w, ql.w);
  g.store(S.r, rh);
  g.store(S.r_lo, rl);
  dot.add(rh.x, rl.x, rh.x, rl.x);
  dot.add(rh.y, rl.y, rh.y, rl.y);
  dot.add(rh.z, rl.z, rh.z, rl.z);
  dot.add(rh.w, rl.w, rh.w, rl.w);
  return dot;
}

// ---------------------------------------------------------------------------------------------
// Iteration, stage 2: x += alpha p, r -= alpha q (all double-float), partial ||r||^2.  The last
// item advances the iteration count and decides stop / residual replacement.  Bound by HBM on large
// batches (48 B a node) and by the chain of dependent loads and reductions on one grid.  Each thread
// moves one 16-byte vector of every plane per step: 96 KB of loads in flight per SM with three blocks
// (batches), 128 KB with four (few grids, where a slot's items then fit one wave).  alpha arrives as a
// double-float pair: an FP64 division or conversion repeated by every thread costs more than a
// step's loads.  A block takes a contiguous range of items, counts its items of a slot at once, and
// has the next item's first loads in flight under an item's sum: 27.3 M nodes in 222 us (5.9 TB/s, 87% of
// the measured copy rate); with items strided over the blocks, a fence and a counter update for
// each, 295.
// ---------------------------------------------------------------------------------------------
template <bool FUSE>
__global__ void __launch_bounds__(kVecThreads, FUSE ? 4 : 3)
k_update(const SlotDesc* __restrict__ slots, const WorkItem* __restrict__ items,
         const int* __restrict__ n_items) {
  __shared__ float2 red[2][kVecThreads / 32];
  __shared__ float2 s_alpha;  // FUSE: alpha of the slot, and whether it runs
  __shared__ int s_run, s_last;
  const int total = *n_items;
  // the block's items: a contiguous range, so that most share a slot
  const int w0 = static_cast<int>(static_cast<long long>(blockIdx.x) * total / gridDim.x);
  const int w1 = static_cast<int>(static_cast<long long>(blockIdx.x + 1) * total / gridDim.x);
  // the first item and its descriptor ahead of the wait for the previous kernel
  WorkItem it = {0, 0};
  if (w0 < w1) it = items[w0];
  pdl_wait();
  for (int w = w0; w < w1;) {
    // the items w .. we - 1 of one slot (tiles it.tile, it.tile + 1, ...)
    if (w != w0) it = items[w];
    const SlotDesc& S = slots[it.slot];
    SlotScalars* sc = S.sc;
    const int we = min(w1, w + S.n_upd_items - it.tile);
    const int count = we - w;
    w = we;
    if (!FUSE && !sc->active) continue;
    const int pi = (sc->it & 1) ^ 1;
    const float* p = S.p[pi];
    const float* p_lo = S.p_lo[pi];
    const int n = S.nx * S.ny;
    const int chunk = S.vec_chunk;
    const bool flat = !S.upd_seg;
    // nodes of the run that lie in whole chunks: one 16-byte vector of every plane per thread and step
    const int e_run = it.tile * chunk;
    const int e_whole = flat ? min(e_run + count * chunk, n / chunk * chunk) : 0;
    float4 ph, pl, qh, ql, rh, rl, xh, xl;
    auto load = [&](int e) {  // plain loads: the stencil, whose lifetime overlaps this kernel's, writes p and q
      ph = *reinterpret_cast<const float4*>(p + e);
      pl = *reinterpret_cast<const float4*>(p_lo + e);
      qh = *reinterpret_cast<const float4*>(S.q + e);
      ql = *reinterpret_cast<const float4*>(S.q_lo + e);
      rh = *reinterpret_cast<const float4*>(S.r + e);
      rl = *reinterpret_cast<const float4*>(S.r_lo + e);
      xh = *reinterpret_cast<const float4*>(S.xhi + e);
      xl = *reinterpret_cast<const float4*>(S.xlo + e);
    };
    // the first step's loads pass under the sum of the p.q partials
    if (e_run < e_whole) load(e_run + 4 * threadIdx.x);
    f2 alpha;
    if (FUSE) {
      if (threadIdx.x < 32) {
        const bool act = sc->active != 0;  // one reading for the whole block
        const double pq = sum_pq(S);
        if (threadIdx.x == 0) {
          const bool ok = act && pq_ok(sc, pq);
          const f2 af = ok ? df_of(sc->rho2[sc->it & 1] / pq) : f2{0.f, 0.f};
          s_alpha = make_float2(af.hi, af.lo);
          s_run = ok;
          if (act && it.tile == 0) finish_pq(sc, pq);
        }
      }
      __syncthreads();
      alpha = f2{s_alpha.x, s_alpha.y};
      const bool run = s_run != 0;
      __syncthreads();  // s_alpha and s_run are written again for the next slot
      // a breakdown: every block finds the same one, the tile-0 block records it
      if (!run) continue;
    } else {
      alpha = f2{sc->alpha_f[0], sc->alpha_f[1]};
    }
    const f2 nalpha = {-alpha.hi, -alpha.lo};
#pragma unroll 1
    for (int k = 0; k < count; ++k) {
      const int e0 = e_run + k * chunk;
      CompDotDF dot;
      if (e0 < e_whole) {
#pragma unroll 1
        for (int e = e0 + 4 * threadIdx.x; e < e0 + chunk; e += kVecStep) {
          df_axpy(xh.x, xl.x, alpha, ph.x, pl.x);
          df_axpy(xh.y, xl.y, alpha, ph.y, pl.y);
          df_axpy(xh.z, xl.z, alpha, ph.z, pl.z);
          df_axpy(xh.w, xl.w, alpha, ph.w, pl.w);
          df_axpy(rh.x, rl.x, nalpha, qh.x, ql.x);
          df_axpy(rh.y, rl.y, nalpha, qh.y, ql.y);
          df_axpy(rh.z, rl.z, nalpha, qh.z, ql.z);
          df_axpy(rh.w, rl.w, nalpha, qh.w, ql.w);
          *reinterpret_cast<float4*>(S.xhi + e) = xh;
          *reinterpret_cast<float4*>(S.xlo + e) = xl;
          *reinterpret_cast<float4*>(S.r + e) = rh;
          *reinterpret_cast<float4*>(S.r_lo + e) = rl;
          dot.add(rh.x, rl.x, rh.x, rl.x);
          dot.add(rh.y, rl.y, rh.y, rl.y);
          dot.add(rh.z, rl.z, rh.z, rl.z);
          dot.add(rh.w, rl.w, rh.w, rl.w);
          // the next step's loads, the next item's too, pass under the item's sum
          if (e + kVecStep < e_whole) load(e + kVecStep);
        }
      } else if (!flat) {
        dot = update_segment(S, it.tile + k, pi, alpha);
      } else {
        for (int e = e0 + threadIdx.x; e < n; e += blockDim.x) {  // the ragged last chunk
          float xh = S.xhi[e], xl = S.xlo[e];
          df_axpy(xh, xl, alpha, p[e], p_lo[e]);
          S.xhi[e] = xh;
          S.xlo[e] = xl;
          float rh = S.r[e], rl = S.r_lo[e];
          df_axpy(rh, rl, nalpha, S.q[e], S.q_lo[e]);
          S.r[e] = rh;
          S.r_lo[e] = rl;
          dot.add(rh, rl, rh, rl);
        }
      }
      // double-buffered: an item's sum is read before the barrier of the next one's
      const double rr = block_sum_comp<kVecThreads>(dot.as_comp(), red[k & 1]);
      if (threadIdx.x == 0) S.part[(it.tile + k) * 4 + 0] = rr;
    }
    if (last_item_block(&sc->cnt[2], S.n_upd_items, &s_last, count)) {
      double s = 0.0;
      if (threadIdx.x < 32) s = warp_sum_strided(S.part, S.n_upd_items, 4);
      if (threadIdx.x == 0) {
        decide_update(sc, s);
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------------------------
// Tail: true residual r = b - M L^2 xhat in FP64, replace the recursive residual, and decide:
// converged / not converged at maxit / continue (with a fresh preconditioner pass).
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kStThreads)
k_true_residual(const SlotDesc* __restrict__ slots, const WorkItem* __restrict__ items,
                const int* __restrict__ n_items) {
  __shared__ double sx[kHalo];
  __shared__ double red[64];
  __shared__ int s_last;
  const int total = *n_items;
  pdl_wait();
  for (int w = blockIdx.x; w < total; w += gridDim.x) {
    const WorkItem it = items[w];
    const SlotDesc& S = slots[it.slot];
    SlotScalars* sc = S.sc;
    if (!sc->fold) continue;
    const int be = sc->bexp;
    int x0, y0;
    tile_origin(S, it.tile, x0, y0);
    for (int i = threadIdx.x; i < kHalo; i += blockDim.x) {
      float s;
      const int g = halo_src(S, x0, y0, i, s);
      sx[i] = (s != 0.f) ? (double)s * ((double)S.xhi[g] + (double)S.xlo[g]) : 0.0;
    }
    __syncthreads();
    double rr = 0.0;
    for (int k = threadIdx.x; k < kStTileX * kStTileY; k += blockDim.x) {
      const int ly = k / kStTileX, lx = k - ly * kStTileX;
      const int gx = x0 + lx, gy = y0 + ly;
      if (gx >= S.nx || gy >= S.ny) continue;
      const int g = gy * S.nx + gx;
      double rv = 0.0;
      if (S.mask[g]) rv = ldexp(S.b[g], be) - stencil13_f64(S, sx, ly, lx);
      const f2 v = df_of(rv);
      S.r[g] = v.hi;
      S.r_lo[g] = v.lo;
      rr += rv * rv;
    }
    double d2 = 0.0;
    block_sum2<kStThreads>(rr, d2, red);
    if (threadIdx.x == 0) S.part[it.tile * 4 + 0] = rr;
    if (last_item_block(&sc->cnt[3], S.n_st_tiles, &s_last)) {
      double sums[1];
      reduce_partials<kStThreads, 1>(S.part, S.n_st_tiles, sums, red);
      if (threadIdx.x == 0) {
        decide_true(sc, sums[0]);
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------------------------
// After the last preconditioner stage: one block per slot (the slot's tile-0 item of the
// transform work list) reduces the per-tile r.z and z.q partials in a fixed order and forms rho
// and beta (flexible or Fletcher-Reeves), or flags breakdown.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(32)
k_prec_finish(const SlotDesc* __restrict__ slots, const WorkItem* __restrict__ items,
              const int* __restrict__ n_items, int mode) {
  const int total = *n_items;
  pdl_wait();
  for (int w = blockIdx.x; w < total; w += gridDim.x) {
    const SlotDesc& S = slots[items[w].slot];
    SlotScalars* sc = S.sc;
    const int run = mode == 0 ? sc->active : (mode == 1 ? sc->need_prec : 1);
    if (!run) continue;
    double rz, zq;
    sum_rz(S, sc->flexible != 0, rz, zq);
    __syncwarp();  // every lane has read the flags
    if (threadIdx.x == 0) finish_preconditioner(sc, rz, zq, mode);
  }
}

// ---------------------------------------------------------------------------------------------
// Output (Algorithm 1, last statement): out = f at known nodes (bit copy), xhat at unknowns.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kVecThreads)
k_output(const SlotDesc* __restrict__ slots, const WorkItem* __restrict__ items,
         const int* __restrict__ n_items, const float* const* __restrict__ fs,
         float* const* __restrict__ outs) {
  const int total = *n_items;
  for (int w = blockIdx.x; w < total; w += gridDim.x) {
    const WorkItem it = items[w];
    const SlotDesc& S = slots[it.slot];
    const float* f = fs[it.slot];
    float* out = outs[it.slot];
    const int n = S.nx * S.ny;
    const int e0 = it.tile * S.vec_chunk;
    const int e1 = min(n, e0 + S.vec_chunk);
    const int be = S.sc->bexp;  // x = 2^-bexp x'
    for (int e = e0 + threadIdx.x; e < e1; e += blockDim.x)
      out[e] = S.mask[e] ? (float)ldexp((double)S.xhi[e] + (double)S.xlo[e], -be) : f[e];
  }
}

// FP64 variant of the output for one slot (lets the caller recompute the residual exactly).
__global__ void __launch_bounds__(kVecThreads)
k_output64(const SlotDesc* __restrict__ slots, const float* __restrict__ f, double* __restrict__ out) {
  const SlotDesc& S = slots[0];
  const int n = S.nx * S.ny;
  const int be = S.sc->bexp;  // x = 2^-bexp x'
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x)
    out[e] = S.mask[e] ? ldexp((double)S.xhi[e] + (double)S.xlo[e], -be) : (double)f[e];
}

// ---------------------------------------------------------------------------------------------
// q = M L^2 p for a caller-supplied FP32 p (the solver's compensated evaluation; used by the entry
// point that allocates nothing): mask from phi's sign, 64 x 16 tiles, the window of p in shared
// memory.  p.q, of whatever magnitude the caller's p has, is an FP64 sum: a warp whose products are
// within the range that Sum3 is exact in adds them so (an FP64 product per node took longer than the
// rest of the kernel), any other in FP64.  12 bytes a node; a call on 1000 x 700 nodes is bound by its
// launches and the copy of p.q back, so the descriptor travels as a kernel argument.
// ---------------------------------------------------------------------------------------------
template <bool ANISO>
__global__ void __launch_bounds__(kStThreads)
k_apply(const __grid_constant__ SlotDesc S, const float* __restrict__ phi, int extend_out,
        const float* __restrict__ p, float* __restrict__ q, double* __restrict__ part) {
  constexpr int TY = kApplyTileY;
  __shared__ __align__(16) float win[kWX * (TY + 4)];  // rows y0-2 .., columns x0-4 ..
  __shared__ __align__(16) float lap[ANISO ? 1 : 2][ANISO ? 4 : kWX * (TY + 4)];  // g(p), hi and lo
  __shared__ float red[3][kStThreads / 32];  // the warps' sums as Sum3 ...
  __shared__ double red_wide[kStThreads / 32];  // ... or, where `wide`, in FP64
  __shared__ bool wide[kStThreads / 32];
  const int ntx = (S.nx + kStTileX - 1) / kStTileX;
  const int tile = blockIdx.x;
  const int x0 = (tile % ntx) * kStTileX, y0 = (tile / ntx) * TY;
  const bool interior = x0 >= 2 && y0 >= 2 && x0 + kStTileX + 2 <= S.nx && y0 + TY + 2 <= S.ny;
  for (int i = threadIdx.x; i < kHX * (TY + 4); i += kStThreads) {
    const int ly = i / kHX, lx = i - ly * kHX;
    float v;
    if (interior) {
      v = __ldg(p + (size_t)(y0 - 2 + ly) * S.nx + x0 - 2 + lx);
    } else {
      float s;
      const int g = halo_src_ty<TY>(S, x0, y0, i, s);
      v = s != 0.f ? s * __ldg(p + g) : 0.f;
    }
    win[ly * kWX + lx + 2] = v;
  }
  __syncthreads();
  if (!ANISO) {
    lap_tile<TY, kWX, false>(win, nullptr, lap[0], lap[ANISO ? 0 : 1]);
    __syncthreads();
  }
  constexpr int kOwn = kStTileX * TY / (2 * kStThreads);  // node pairs per thread
  float pv[2 * kOwn], qv[2 * kOwn];                       // p and q of the products (zeros elsewhere)
#pragma unroll
  for (int j = 0; j < kOwn; ++j) {
    const int k = threadIdx.x + j * kStThreads;
    pv[2 * j] = pv[2 * j + 1] = qv[2 * j] = qv[2 * j + 1] = 0.f;
    const int ly = k / (kStTileX / 2), lx = 2 * (k - ly * (kStTileX / 2));
    const int gx = x0 + lx, gy = y0 + ly;
    if (gx >= S.nx || gy >= S.ny) continue;
    const size_t g = (size_t)gy * S.nx + gx;
    const bool two = gx + 1 < S.nx;
    const float f0 = __ldg(phi + g), f1 = two ? __ldg(phi + g + 1) : 0.f;
    const bool u0 = !(extend_out ? f0 < 0.f : f0 > 0.f), u1 = two && !(extend_out ? f1 < 0.f : f1 > 0.f);
    const float* c = win + (ly + 2) * kWX + lx + 4;
    float2 r = make_float2(0.f, 0.f);
    if (u0 || u1) {
      if (!ANISO) {
        const int o = (ly + 2) * kWX + lx + 4;
        const f2x2 a = lap_pair<kWX>(lap[0] + o, lap[ANISO ? 0 : 1] + o);
        r = add2(a.hi, a.lo);
      } else {
        r.x = stencil13_acc<kWX>(S, win + 2, ly, lx).result();
        r.y = two ? stencil13_acc<kWX>(S, win + 2, ly, lx + 1).result() : 0.f;
      }
    }
    const float q0 = u0 ? r.x : 0.f, q1 = u1 ? r.y : 0.f;
    q[g] = q0;
    pv[2 * j] = c[0];
    qv[2 * j] = q0;
    if (two) {
      q[g + 1] = q1;
      pv[2 * j + 1] = c[1];
      qv[2 * j + 1] = q1;
    }
  }
  // a product is zero because a factor is, or it and its error term are normal numbers
  bool plain = true;
#pragma unroll
  for (int i = 0; i < 2 * kOwn; ++i) {
    const float m = fabsf(__fmul_rn(pv[i], qv[i]));
    plain = plain && ((m > 0x1p-90f && m < 0x1p100f) || (m == 0.f && (pv[i] == 0.f || qv[i] == 0.f)));
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (__all_sync(0xffffffffu, plain)) {
    Sum3 sum;
#pragma unroll
    for (int i = 0; i < 2 * kOwn; ++i) sum.add_prod(pv[i], qv[i]);
    sum.reduce<32>();
    if (lane == 0) {
      red[0][warp] = sum.s, red[1][warp] = sum.c, red[2][warp] = sum.d;
      wide[warp] = false;
    }
  } else {
    double t = 0.0;
#pragma unroll
    for (int i = 0; i < 2 * kOwn; ++i) t += (double)pv[i] * (double)qv[i];
    t = warp_sum(t);
    if (lane == 0) {
      red_wide[warp] = t;
      wide[warp] = true;
    }
  }
  __syncthreads();
  if (warp == 0) {
    const int w = lane & 7;
    double t = wide[w] ? red_wide[w] : Sum3(red[0][w], red[1][w], red[2][w]).value();
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) part[tile] = t;
  }
}

// ---------------------------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------------------------
void launch_setup(const LaunchCfg& c, const float* const* phis, const float* const* fs,
                  const int* dirs) {
  k_setup<<<c.grid, kStThreads, 0, c.stream>>>(c.slots, c.items, c.n_items, phis, fs, dirs);
}
void launch_stage_setup(const LaunchCfg& c, bool op, const float* phi, const float* v, int n, int dir) {
  const int grid = std::max(1, std::min((n + 4 * kVecThreads - 1) / (4 * kVecThreads), c.grid));
  if (op) k_stage_setup<true><<<grid, kVecThreads, 0, c.stream>>>(c.slots, phi, v, dir == 0);
  else k_stage_setup<false><<<grid, kVecThreads, 0, c.stream>>>(c.slots, phi, v, dir == 0);
}
void launch_rhs_scale(const LaunchCfg& c) {
  k_rhs_scale<<<c.grid, kStThreads, 0, c.stream>>>(c.slots, c.items, c.n_items);
}
template <int TY, bool FUSE>
static void launch_stencil_ty(const LaunchCfg& c, bool aniso, int* err, long long wc) {
  constexpr int smem = StGeom<TY>::kSmemBytes;
  if (aniso)
    launch_cfg(c, k_stencil<true, TY, FUSE>, c.grid, kStBlock, smem, c.slots, c.items, c.n_items, err, wc);
  else
    launch_cfg(c, k_stencil<false, TY, FUSE>, c.grid, kStBlock, smem, c.slots, c.items, c.n_items, err, wc);
}
void launch_stencil(const LaunchCfg& c, bool aniso, int tile_y, int* err, bool fuse_prec) {
  const long long wc = c.wait_cycles > 0 ? c.wait_cycles : kWaitCycles;
  if (fuse_prec) {
    if (tile_y == 16) launch_stencil_ty<16, true>(c, aniso, err, wc);
    else launch_stencil_ty<32, true>(c, aniso, err, wc);
  } else {
    if (tile_y == 16) launch_stencil_ty<16, false>(c, aniso, err, wc);
    else launch_stencil_ty<32, false>(c, aniso, err, wc);
  }
}
int stencil_blocks_per_sm(int tile_y) {
  return tile_y == 16 ? StGeom<16>::kBlocksPerSm : StGeom<32>::kBlocksPerSm;
}
template <bool ANISO, int TY, bool FUSE>
static cudaError_t stencil_attr() {
  // the window sets live in dynamic shared memory; all of the SM's shared memory to the
  // carveout, so that kBlocksPerSm blocks fit
  const cudaError_t e = cudaFuncSetAttribute(k_stencil<ANISO, TY, FUSE>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             StGeom<TY>::kSmemBytes);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_stencil<ANISO, TY, FUSE>, cudaFuncAttributePreferredSharedMemoryCarveout,
                              cudaSharedmemCarveoutMaxShared);
}
cudaError_t stencil_init() {
  const cudaError_t e[8] = {stencil_attr<false, 32, false>(), stencil_attr<true, 32, false>(),
                            stencil_attr<false, 16, false>(), stencil_attr<true, 16, false>(),
                            stencil_attr<false, 32, true>(),  stencil_attr<true, 32, true>(),
                            stencil_attr<false, 16, true>(),  stencil_attr<true, 16, true>()};
  for (cudaError_t x : e)
    if (x != cudaSuccess) return x;
  return cudaSuccess;
}
void launch_pq_finish(const LaunchCfg& c) {
  launch_cfg(c, k_pq_finish, c.grid, 32, 0, c.slots, c.items, c.n_items);
}
void launch_update(const LaunchCfg& c, bool fuse_pq) {
  if (fuse_pq) launch_cfg(c, k_update<true>, c.grid, kVecThreads, 0, c.slots, c.items, c.n_items);
  else launch_cfg(c, k_update<false>, c.grid, kVecThreads, 0, c.slots, c.items, c.n_items);
}
void launch_true_residual(const LaunchCfg& c) {
  launch_cfg(c, k_true_residual, c.grid, kStThreads, 0, c.slots, c.items, c.n_items);
}
void launch_output(const LaunchCfg& c, const float* const* fs, float* const* outs) {
  k_output<<<c.grid, kVecThreads, 0, c.stream>>>(c.slots, c.items, c.n_items, fs, outs);
}
void launch_prec_finish(const LaunchCfg& c, int mode) {
  launch_cfg(c, k_prec_finish, c.grid, 32, 0, c.slots, c.items, c.n_items, mode);
}
void launch_output64(const SlotDesc* slot, int n, const float* f, double* out, cudaStream_t s) {
  int grid = (n + kVecThreads - 1) / kVecThreads;
  grid = grid < 4096 ? grid : 4096;
  k_output64<<<grid, kVecThreads, 0, s>>>(slot, f, out);
}
void launch_apply(const SlotDesc& slot, const float* phi, bool extend_out, const float* p, float* q,
                  double* part, cudaStream_t s) {
  const int grid = apply_tiles(slot.nx, slot.ny);
  if (slot.aniso) k_apply<true><<<grid, kStThreads, 0, s>>>(slot, phi, extend_out, p, q, part);
  else k_apply<false><<<grid, kStThreads, 0, s>>>(slot, phi, extend_out, p, q, part);
}

}  // namespace bx
