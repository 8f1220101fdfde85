// Shared device-side definitions of the biharmonic extension library.
//
// One "slot" is one extension problem being solved; a batch (or the serving loop) is a set of
// slots.  Every CG stage is one launch over a work list of (slot, tile) items drawn from all
// iterating slots; per-slot scalars live in device memory and are reduced deterministically by
// the last work item of the slot to finish (fixed order, no floating-point atomics).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace bx {

constexpr int kPad = 128;           // transform buffers are padded to multiples of this
constexpr int kStTileX = 64;        // stencil tile (x contiguous)
constexpr int kStTileY = 32;
constexpr int kStThreads = 256;
// The stencil's shared-memory window of one tile (also the box of its tensor copies): the halo
// rows y0-2 .. y0+kStTileY+1 and the columns x0-4 .. x0+kStTileX+3, two columns wider on the
// left than the halo so that a copy starts on a 16-byte boundary.
constexpr int kStWinX = kStTileX + 8;
constexpr int kStWinY = kStTileY + 4;
constexpr int kTcMaps = 11;         // transform tensor maps per problem
constexpr int kStMaps = 7;          // stencil tensor maps per slot
constexpr int kLowM = 32;           // low modes per axis computed in high precision
constexpr int kLowAutoSide = 2048;  // low_modes = 2: grids with a side of at least this many nodes
constexpr long long kLowAutoNodes = 2048LL * 2048;  // low_modes = 2: or calls with this many nodes
// Grids of at most kSixNodes nodes in mixed modes with low_modes = 2: six slices per transform operand
// (outside calls large enough for the low-mode correction).  They save about 29% of the
// iterations; the stages' products double, but up to here an iteration is bound by its launches'
// latency: four / six slices 14.9 / 10.5 ms at 128^2, 36.7 / 26.9 at 256^2, 117 / 86 at 512^2, 249 / 216 at
// 768^2, 520 / 604 at 1024^2, 187 / 174 for 16 grids of 128..512 together, 525 / 537 for 48.
constexpr long long kSixNodes = 768LL * 768;
constexpr int kLowNS = 6;           // integer slices per operand of the low-mode products
constexpr int kLowK3 = 32;          // k extent of the inverse low-mode product
constexpr int kVecThreads = 256;
constexpr int kVecStep = 4 * kVecThreads;  // elements a block moves with one vector per thread
// Elements per work item of the vector kernels (a function of the grid alone, so that the partial
// sums do not depend on the call): one step up to 2^17 nodes (the output only: their updates work in
// segments, seg_of) and two up to 2^21 (more blocks at once: the update of a 1024^2 grid went from 14 to
// 12 us), four beyond (less per-item overhead: 43 us a launch on 48 grids of 5.1 M nodes against 61
// with one step everywhere).
constexpr int vec_chunk_of(long long nodes) {
  return kVecStep * (nodes <= 1LL << 17 ? 1 : nodes <= 1LL << 21 ? 2 : 4);
}

// Calls whose grids are all of up to this size have the residuals sliced by the update itself
// (k_update_slice): one launch less in the chain of an iteration (320 x 256, three fields: 69.7 -> 64 us;
// 64^2: 50.5 -> 46).  Above, a pass of its own is as fast: the joint kernel holds a segment's planes
// across a barrier, so that fewer loads are in flight (1024^2: 28 us either way; 48 grids of up to
// 512^2: 76 us against 62).
constexpr long long kSliceNodes = 1LL << 17;

enum Bc : int { BC_SYM = 0, BC_PER = 1, BC_DIR = 2 };

// Status words (match the public EXT_* codes).
enum : int { ST_OK = 0, ST_RUNNING = 1, ST_ENOTCONV = -5, ST_EBREAKDOWN = -6 };

// Per-slot scalars, FP64 where they feed CG.  Written only by the last work item of a slot.
struct __align__(16) SlotScalars {
  double bb;        // ||b||^2
  double rho2[2];   // r.z of the current z at [it & 1], of the previous iteration's at the other
  double pq;        // p.Ap of the current direction
  double zq;        // z_new.q_old (flexible beta)
  double rr;        // ||r||^2, recursive
  double rr_true;   // ||b - A xhat||^2 at the last replacement
  double alpha, beta;
  float alpha_f[2], beta_f[2];  // the same as double-float pairs, for the kernels that apply them
  double rtol2;     // rtol^2
  double rr_ref;    // ||r||^2 at the last residual replacement
  double delta2;    // replace the residual once ||r||^2 < delta2 * rr_ref
  int it;           // completed iterations
  int maxit;
  int fold_every;   // longest stretch of iterations between residual replacements
  int active;       // 1 while the slot iterates
  int fold;         // 1: the tail replaces r by the FP64 true residual b - A xhat
  int need_prec;    // 1: the tail preconditioner runs (after a replacement that continues)
  int status;       // ST_RUNNING until final
  int flexible;
  unsigned cnt[6];  // completion counters of the last-item reductions, one per kernel kind
  int n_known;      // known nodes, counted by the set-up kernel
  int bexp;         // the iteration solves A x' = 2^bexp b; the answer is x = 2^-bexp x'
  // error estimate: in CG, ||x* - x_k||_A^2 = sum_{j >= k} alpha_j rho_j, so the terms of the last
  // kErrDelay iterations over the sum of all terms estimate the relative A-norm error of the
  // iterate kErrDelay steps before the end (an upper estimate for the returned one)
  double aro_total;
  double aro_ring[8];
  int aro_n;
  int it_ref;       // iterations completed at the last residual replacement
  double rr_rec;    // 3-D: the recursive ||r||^2 of the last iteration
};
constexpr int kErrDelay = 8;

// Static description of one slot (device copy).  Padded transform dims are multiples of kPad.
struct SlotDesc {
  int nx, ny, nxp, nyp;
  int bcx, bcy;
  int n_st_tiles;    // grid tiles of the set-up, residual and slicing kernels: ceil(nx/64) * ceil(ny/32)
  int n_sten_tiles;  // tiles of the stencil kernel: ceil(nx/64) * ceil(ny/sten_ty)
  int sten_ty;       // the stencil kernel's tile height (16 or 32)
  int vec_chunk;     // elements per vector work item
  int n_vec_items;   // vector work items: ceil(nx*ny / vec_chunk)
  int n_gm_tiles;    // output tiles of one transform stage
  float wc, wex, wey, wd, wfx, wfy;  // stencil weights (hi), scaled so that max(a, c) = 1
  float wc_l, wex_l, wey_l, wd_l, wfx_l, wfy_l;  // low parts (anisotropic grids only)
  double dwc, dwex, dwey, dwd, dwfx, dwfy;       // FP64 weights for the true residual
  int aniso;
  // grid vectors [ny][nx].  Every CG vector is a double-float pair v = hi + lo of FP32 planes
  // (about 48 bits), updated with error-free FP32 transformations: with FP32 storage alone the
  // rounding of any one of r, p, q, z costs this operator 60-100% more iterations.
  uint8_t* mask;     // 1 = unknown node
  double* b;
  float* xhi;        // the iterate x = xhi + xlo
  float* xlo;
  float* r;          // hi planes ...
  float* p[2];
  float* q;
  float* z;
  float* r_lo;       // ... and their lo planes
  float* p_lo[2];
  float* q_lo;
  float* z_lo;
  const float* lamx; // [nxp] eigenvalues of T_x (scaled), padding entries never read
  const float* lamy;
  float wnorm;       // 1 / w_max, so that the scaled weights are <= 1
  // transforms: block-scaled integer slices (NS = 4 or 6 16-bit planes) and their TMA descriptors
  void* tc_r;        // [tc_nr][nyp][nxp]  residual
  int tc_ns;         // slices per transform operand: 4 or 6
  int tc_nr;         // slices of the residual: tc_ns, or 6 where the low-mode correction reads them
  void* tc_t1;       // [NS][nxp][nyp]
  void* tc_t2;       // [NS][nyp][nxp] (in place of the residual)
  void* tc_t3;       // [NS][nxp][nyp] (in place of T1)
  int8_t* tc_e[4];   // block exponents of the A operand of stage s: [rows][K/128], 0 and 2, 1 and 3 one array
  const int8_t* tc_eb[4];  // block exponents of the B operand of stage s (transform matrices)
  const void* tmaps; // kTcMaps CUtensorMap (64-byte aligned): A operand of stages 0..3, B of 0..3,
                     // the results of stages 0..2 (store boxes)
  const void* st_maps;  // kStMaps CUtensorMap for the stencil's tensor copies (z, z_lo, p[0],
                        // p_lo[0], p[1], p_lo[1], mask); null when a mask row is not a multiple
                        // of 16 bytes
  // Low-mode correction of the tensor-core preconditioner: the modes kx < lowm_x, ky < lowm_y
  // (the smoothest, with the largest weights) are left out of the four 32-bit transform stages and
  // added from thin transforms with six slices per operand (about 48 bits).  0 = off.
  int lowm_x, lowm_y;
  float* low_gp;            // per forward tile t its share of G = Qy_low^T (r Qx_low): [t][2][32][32]
                            // (hi plane, then lo plane)
  void* low_jt;             // J^T slices [kLowNS][nxp][kLowK3] (16-bit codes), J = W o G Qx_low^T
  int8_t* low_jt_e;         // block exponent of each J^T row [nxp]
  float* low_z;             // zl = Qy_low J: [ny][nx] hi plane, lo plane at + nx * ny
  const float* low_qxd;     // Qx[x][kx < 32] double-float: [nxp][32] hi, lo plane at + nxp * 32
  const float* low_qyd;     // Qy[y][ky < 32] double-float: [nyp][32] hi, lo plane at + nyp * 32
  const int8_t* low_qxt_e;  // exponents of the forward product's B operand: [32][nxp / 128]
  const int8_t* low_qy_e;   // exponents of the inverse product's B operand: [nyp]
  const void* low_maps;     // 4 CUtensorMap: r slices, Qx_low^T slices, J^T slices, Qy_low slices
  int n_l1_tiles;           // tiles of the forward product: nyp / 128
  int n_l2_tiles;           // blocks of the middle: nxp / 32
  int n_l3_tiles;           // tiles of the inverse product: (nxp / 128) * (nyp / 32)
  // Mirror fold of the tensor-core transforms (i -> n-1-i on an axis; even and odd classes of
  // ceil(n/2) nodes each): a slot with a folded axis runs its four stages as two or four
  // half-size problems, the slot's classes, held in the tensor-core problem list at
  // kMirClasses * slot + c, c = 2 cls_y + cls_x.
  int mir;           // slot: bit 0 = x folded, bit 1 = y folded (0: the slot is its own problem)
  int mhx, mhy;      // slot: class nodes along x, y (ceil(n/2) on a folded axis, else n)
  int n_fold_items;  // slot: items of the fold kernel (8 class rows x 128 columns)
  int upd_seg;       // slot of at most kSliceNodes nodes: its update items are segments (seg_of), not chunks
  int n_upd_items;   // slot: items of the update kernels
  int n_prep_items;  // slot with no folded axis: items of its residual slicing (32 rows x 128)
  int n_unfold_tiles;// slot: tiles of the unfold kernel (32 x 8 class nodes)
  int n_prec_parts;  // slot: r.z, z.q partials the preconditioner leaves (stage-3 or unfold tiles)
  int mir_out;       // class problem: stage 3 writes the class result g to z, z_lo ([ny][nx])
  SlotScalars* sc;
  double* part;      // per-work-item partial sums (2 doubles per item), slot-local indexing
  double* pq_part;   // p.q partial sums of the stencil, one per 64 x 16 block [ny/16][nx/64]
};

constexpr int kMirClasses = 4;  // tensor-core problem entries per slot

struct WorkItem {
  int slot;
  int tile;   // tile / chunk index within the slot
};

// Programmatic dependent launch.  The kernels of an iteration follow one another at 2-10 us
// each, so the launch gap between them counts: each is launched with programmatic serialization
// and calls pdl_wait before it reads anything an earlier kernel wrote (the descriptors and work
// lists it may read before: no kernel writes them).  griddepcontrol.wait returns once the previous
// grid has completed and its writes are visible; only then does the block release the next grid
// (launch_dependents), so that at most two grids of a stream are in flight and a grid's
// completion implies that of every earlier one.  Every block of every such kernel makes the
// call, whether or not it has work.  Without the launch attribute both instructions do nothing.
__device__ __forceinline__ void pdl_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// ------------------------------------------------------------------------------------------
// Reductions
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Block sum of up to two values; result valid in thread 0.  `sh` holds >= 2*32 doubles.
template <int NT>
__device__ __forceinline__ void block_sum2(double& a, double& b, double* sh) {
  a = warp_sum(a);
  b = warp_sum(b);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) { sh[w] = a; sh[32 + w] = b; }
  __syncthreads();
  if (w == 0) {
    a = (l < NT / 32) ? sh[l] : 0.0;
    b = (l < NT / 32) ? sh[32 + l] : 0.0;
    a = warp_sum(a);
    b = warp_sum(b);
  }
  __syncthreads();
}

// Last-item protocol, called by every thread of the block after thread 0 has written the partials of
// its `items` items.  Returns true in all threads of the block that completes the slot.
__device__ __forceinline__ bool last_item_block(unsigned* counter, unsigned total, int* sflag, unsigned items = 1) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned prev = atomicAdd(counter, items);
    const int last = (prev + items == total) ? 1 : 0;
    if (last) {
      __threadfence();
      *counter = 0u;
    }
    *sflag = last;
  }
  __syncthreads();
  return *sflag != 0;
}

// Sums of partials part[t*4 + k] (k = 0..K-1) over t < n, by the whole block: thread i adds
// t = i, i + NT, ... in order, then a fixed tree.  The order depends only on n, so the result is
// the same whichever block runs the reduction.  Results valid in thread 0.
template <int NT, int K>
__device__ __forceinline__ void reduce_partials(const double* part, int n, double (&out)[K],
                                                double* sh) {
  double acc[3] = {0.0, 0.0, 0.0};
  for (int t = threadIdx.x; t < n; t += NT) {
#pragma unroll
    for (int k = 0; k < K; ++k) acc[k] += __ldcg(&part[t * 4 + k]);
  }
  double a = acc[0], b = K > 1 ? acc[1] : 0.0;
  block_sum2<NT>(a, b, sh);
  out[0] = a;
  if (K > 1) out[1] = b;
  if (K > 2) {
    double c = acc[2], d = 0.0;
    block_sum2<NT>(c, d, sh);
    out[2] = c;
  }
}

// ------------------------------------------------------------------------------------------
// Error-free transformations in FP32 (Knuth TwoSum, FMA-based TwoProd).  The _rn intrinsics
// are never contracted into FMAs, which keeps the transformations exact.
// ------------------------------------------------------------------------------------------
struct f2 { float hi, lo; };

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// Compensated accumulator (Ogita-Rump-Oishi Sum2): s + c carries about twice FP32 precision.
struct CompSum {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float x) {
    float e;
    two_sum(s, x, s, e);
    c = __fadd_rn(c, e);
  }
  // add w*x for an FP32 weight w (exact product split by FMA)
  __device__ __forceinline__ void add_prod(float w, float x) {
    const float p = __fmul_rn(w, x);
    const float pe = __fmaf_rn(w, x, -p);
    add(p);
    c = __fadd_rn(c, pe);
  }
  __device__ __forceinline__ float result() const { return __fadd_rn(s, c); }
};

// Packed FP32x2 arithmetic (two independent lanes, each rounded exactly as its scalar
// counterpart): a - b is fma(b, -1, a), one rounding.
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
  return __ffma2_rn(b, make_float2(-1.f, -1.f), a);
}
__device__ __forceinline__ float2 mul2(float w, float2 a) { return __fmul2_rn(make_float2(w, w), a); }
__device__ __forceinline__ void two_sum2(float2 a, float2 b, float2& s, float2& e) {
  s = add2(a, b);
  const float2 bb = sub2(s, a);
  e = add2(sub2(a, sub2(s, bb)), sub2(b, bb));
}
// Compensated FP32 dot-product accumulator (TwoProd + TwoSum per term).  GB300 runs FP64 at a
// small fraction of its FP32 rate, so per-element FP64 arithmetic would dominate the
// bandwidth-bound kernels; a thread's terms are summed here and only the per-thread totals are
// combined in FP64.
struct CompDot {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float a, float b) {
    const float p = __fmul_rn(a, b);
    const float pe = __fmaf_rn(a, b, -p);
    float e;
    two_sum(s, p, s, e);
    c = __fadd_rn(c, __fadd_rn(e, pe));
  }
  __device__ __forceinline__ double value() const { return (double)s + (double)c; }
};

// Compensated sum of (s, c) pairs over groups of W consecutive lanes in a fixed butterfly; every
// lane of a group gets the group's pair.
template <int W>
__device__ __forceinline__ void group_sum_pair(float& s, float& c) {
#pragma unroll
  for (int o = W / 2; o > 0; o >>= 1) {
    const float s2 = __shfl_xor_sync(0xffffffffu, s, o);
    const float c2 = __shfl_xor_sync(0xffffffffu, c, o);
    float e;
    two_sum(s, s2, s, e);
    c = __fadd_rn(c, __fadd_rn(c2, e));
  }
}

// One warp: the FP64 sum of the pairs sh[0..7] of a block's eight warps, in every lane.
__device__ __forceinline__ double sum_of_eight(const float2* sh) {
  const float2 p = sh[threadIdx.x & 7];
  double v = (double)p.x + (double)p.y;
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Block sum of compensated per-thread accumulators: FP32 TwoSum butterflies inside the warps, FP64 across
// them, by one warp.  The SM adds two FP64 numbers a cycle (a warp instruction takes 16), so FP64
// stays out of every step that each warp would repeat.  Result valid in the first warp.
// `sh` >= NT / 32 float2.
template <int NT>
__device__ __forceinline__ double block_sum_comp(CompDot d, float2* sh) {
  static_assert(NT / 32 == 8, "eight warps");
  group_sum_pair<32>(d.s, d.c);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) sh[w] = make_float2(d.s, d.c);
  __syncthreads();
  return w == 0 ? sum_of_eight(sh) : 0.0;
}

// Sum of exact products in three FP32 numbers (TwoProd, and a TwoSum for every rounding but the last
// number's): about 70 bits while no product's error term leaves FP32's range, so that its FP64 value is
// as good as a sum kept in FP64, at the rate of FP32.
struct Sum3 {
  float s = 0.f, c = 0.f, d = 0.f;
  __device__ __forceinline__ Sum3() {}
  __device__ __forceinline__ Sum3(float s0, float c0, float d0 = 0.f) : s(s0), c(c0), d(d0) {}
  __device__ __forceinline__ void join(float s2, float c2, float d2) {
    float e, t;
    two_sum(s, s2, s, e);
    two_sum(c, c2, c, t);
    d = __fadd_rn(d, __fadd_rn(d2, t));
    two_sum(c, e, c, t);
    d = __fadd_rn(d, t);
  }
  __device__ __forceinline__ void add_prod(float a, float b) {
    const float p = __fmul_rn(a, b);
    join(p, __fmaf_rn(a, b, -p), 0.f);
  }
  // the sum over groups of W consecutive lanes in a fixed butterfly
  template <int W>
  __device__ __forceinline__ void reduce() {
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) {
      const float s2 = __shfl_xor_sync(0xffffffffu, s, o), c2 = __shfl_xor_sync(0xffffffffu, c, o);
      join(s2, c2, __shfl_xor_sync(0xffffffffu, d, o));
    }
  }
  template <bool THIRD = true>
  __device__ __forceinline__ double value() const {
    return (double)s + (THIRD ? (double)c + (double)d : (double)c);
  }
};
// The sum over W warps of one Sum3 each (the same in all its lanes): FP64 for the result only (the SM adds
// two FP64 numbers a cycle).  Result valid in the first warp.
template <int W>
__device__ __forceinline__ double across_warps(Sum3 v, float (&sh)[3][W]) {
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) sh[0][w] = v.s, sh[1][w] = v.c, sh[2][w] = v.d;
  __syncthreads();
  if (w != 0) return 0.0;
  v = Sum3(sh[0][l % W], sh[1][l % W], sh[2][l % W]);
  v.reduce<W>();
  return v.value();
}
// The preconditioner's dot products over W lanes: as good as FP64 sums in FP32 mode (DOTS3), in pairs in the
// mixed modes (as one form for both, 1 us of 60 an iteration slower: more registers in the unfold).
template <int W, bool DOTS3>
__device__ __forceinline__ void reduce_dots(Sum3& v) {
  if (DOTS3) v.reduce<W>();
  else group_sum_pair<W>(v.s, v.c);
}

// ------------------------------------------------------------------------------------------
// Double-float arithmetic (Dekker, Knuth): a value is an unevaluated FP32 pair hi + lo with
// |lo| <= ulp(hi) / 2.  Sums use TwoSum, products the FMA-based TwoProd; cross terms of size
// 2^-24 relative are added in plain FP32, so results carry about 48 bits.
// ------------------------------------------------------------------------------------------
// (s, e) -> normalised pair, valid when |e| is at most about ulp(s) (Fast2Sum)
__device__ __forceinline__ f2 df_norm(float s, float e) {
  const float h = __fadd_rn(s, e);
  return {h, __fsub_rn(e, __fsub_rn(h, s))};
}
__device__ __forceinline__ f2 df_add(f2 a, f2 b) {
  float s, e;
  two_sum(a.hi, b.hi, s, e);
  e = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
  return df_norm(s, e);
}
// a * b for a double-float a and an FP32 b
__device__ __forceinline__ f2 df_mul(f2 a, float b) {
  const float p = __fmul_rn(a.hi, b);
  float e = __fmaf_rn(a.hi, b, -p);
  e = __fmaf_rn(a.lo, b, e);
  return df_norm(p, e);
}
// a * b for double-float a and b
__device__ __forceinline__ f2 df_mul(f2 a, f2 b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  return df_norm(p, e);
}
// c + a * b, all double-float (one TwoProd, one TwoSum)
__device__ __forceinline__ f2 df_fma(f2 a, f2 b, f2 c) {
  const float p = __fmul_rn(a.hi, b.hi);
  float pe = __fmaf_rn(a.hi, b.hi, -p);
  pe = __fmaf_rn(a.hi, b.lo, pe);
  pe = __fmaf_rn(a.lo, b.hi, pe);
  float s, e;
  two_sum(c.hi, p, s, e);
  e = __fadd_rn(e, __fadd_rn(c.lo, pe));
  return df_norm(s, e);
}
__device__ __forceinline__ f2 df_neg(f2 a) { return f2{-a.hi, -a.lo}; }
// an FP64 value as a double-float pair (host and device)
__host__ __device__ __forceinline__ f2 df_of(double v) {
  const float h = (float)v;
  return {h, (float)(v - (double)h)};
}

// Packed FP32x2 forms of the same operations (two independent lanes, each rounded exactly as its
// scalar counterpart).
struct f2x2 { float2 hi, lo; };
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ f2x2 df_norm2(float2 s, float2 e) {
  const float2 h = add2(s, e);
  return {h, sub2(e, sub2(h, s))};
}
// z + beta * p for double-float z, p (two lanes) and a double-float scalar beta
__device__ __forceinline__ f2x2 df_axpy2(f2 beta, f2x2 p, f2x2 z) {
  const float2 bh = make_float2(beta.hi, beta.hi), bl = make_float2(beta.lo, beta.lo);
  const float2 t = __fmul2_rn(bh, p.hi);
  float2 te = fma2(bh, p.hi, neg2(t));
  te = fma2(bh, p.lo, te);
  te = fma2(bl, p.hi, te);
  float2 s, e;
  two_sum2(z.hi, t, s, e);
  e = add2(e, add2(z.lo, te));
  return df_norm2(s, e);
}

// x += a * p with double-float x, p and scalar a (TwoProd + TwoSum)
__device__ __forceinline__ void df_axpy(float& xh, float& xl, f2 a, float ph, float pl) {
  const f2 r = df_fma(a, f2{ph, pl}, f2{xh, xl});
  xh = r.hi;
  xl = r.lo;
}

// Compensated dot product of double-float vectors: hi * hi by TwoProd into a Sum2 accumulator,
// the two cross terms (2^-24 relative) in plain FP32.
struct CompDotDF {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float ah, float al, float bh, float bl) {
    const float p = __fmul_rn(ah, bh);
    const float pe = __fmaf_rn(ah, bh, -p);
    float e;
    two_sum(s, p, s, e);
    c = __fadd_rn(c, __fadd_rn(e, __fmaf_rn(ah, bl, __fmaf_rn(al, bh, pe))));
  }
  __device__ __forceinline__ double value() const { return (double)s + (double)c; }
  __device__ __forceinline__ CompDot as_comp() const {
    CompDot d;
    d.s = s;
    d.c = c;
    return d;
  }
};
// CompDotDF on two lanes at once (the same operations, in the same order, per lane).
struct CompDotDF2 {
  float2 s = make_float2(0.f, 0.f), c = make_float2(0.f, 0.f);
  __device__ __forceinline__ void add(float2 ah, float2 al, float2 bh, float2 bl) {
    const float2 p = __fmul2_rn(ah, bh);
    const float2 pe = __ffma2_rn(ah, bh, make_float2(-p.x, -p.y));
    float2 e;
    two_sum2(s, p, s, e);
    c = add2(c, add2(e, __ffma2_rn(ah, bl, __ffma2_rn(al, bh, pe))));
  }
};

// ------------------------------------------------------------------------------------------
// Ghost-node maps of one axis (Algorithm 1 padding; symmetric = half-sample reflection;
// periodic = wrap).  Input index i in [-2, n+1].  Returns the node index and a sign
// (+1, -1, or 0 for the zero Dirichlet boundary node).
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ int ghost(int i, int n, int bc, float& sgn) {
  sgn = 1.f;
  if (i >= 0 && i < n) return i;
  if (bc == BC_PER) return i < 0 ? i + n : i - n;
  if (bc == BC_SYM) return i < 0 ? -1 - i : 2 * n - 1 - i;
  // Dirichlet: distance 1 is the boundary node (zero), distance 2 the negated first node
  if (i == -1 || i == n) { sgn = 0.f; return 0; }
  sgn = -1.f;
  return i < 0 ? -i - 2 : 2 * n - i;
}

// wnorm / s^2 by the approximate reciprocal (at most 2 ulp in all; s^2 of the grids' eigenvalue
// sums, 1e-18 to 300, stays far inside the normal range).  The preconditioner is only an
// approximation of the inverse, so a 2-ulp change of its weights is immaterial.
__device__ __forceinline__ float spectral_weight_of(float wnorm, float s) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(s * s));
  return wnorm * r;
}

// The per-slot scalar steps.  Each is computed either by one block per slot in a launch of its own
// (k_pq_finish, k_prec_finish) or, for workspaces of few slots, by every block of the kernel that
// needs the result (the update and the next stencil), from the same partial sums in the same
// order, so both give the same bits; then only the block of the slot's tile 0 writes the scalars,
// and none of the fields it writes is read by the other blocks of that kernel.
constexpr int kFuseParts = 2048;  // most partial sums a consumer kernel adds up itself

// Sum of p[i * stride], i < n, by the calling warp: lane l adds i = l, l + 32, ... on four chains, the
// lanes in a fixed butterfly; the order depends on n alone.  Every lane gets the sum.  One warp: the
// FP64 pipe (two lanes a cycle and SM) is the limit, so more warps would only add butterflies.
__device__ __forceinline__ double warp_sum_strided(const double* p, int n, int stride) {
  const int l = threadIdx.x & 31;
  double a[4] = {0.0, 0.0, 0.0, 0.0};
  int i = l;
  for (; i + 224 < n; i += 256) {  // eight loads in flight: the sum of 1024 partials in four trips, not eight
    double v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = __ldcg(p + (size_t)(i + 32 * k) * stride);
#pragma unroll
    for (int k = 0; k < 8; ++k) a[k & 3] += v[k];
  }
  for (; i + 96 < n; i += 128) {
#pragma unroll
    for (int k = 0; k < 4; ++k) a[k] += __ldcg(p + (size_t)(i + 32 * k) * stride);
  }
#pragma unroll
  for (int k = 0; k < 3; ++k)
    if (i + 32 * k < n) a[k] += __ldcg(p + (size_t)(i + 32 * k) * stride);
  return warp_sum((a[0] + a[1]) + (a[2] + a[3]));
}
// One warp: the sum of the slot's p.q partials.
__device__ __forceinline__ double sum_pq(const SlotDesc& S) {
  return warp_sum_strided(S.pq_part, ((S.ny + 15) >> 4) * ((S.nx + kStTileX - 1) / kStTileX), 1);
}
// One warp: the sums of the slot's r.z and (for the flexible beta) z.q partials.
__device__ __forceinline__ void sum_rz(const SlotDesc& S, bool with_zq, double& rz, double& zq) {
  rz = warp_sum_strided(S.part + 2, S.n_prec_parts, 4);
  zq = with_zq ? warp_sum_strided(S.part + 3, S.n_prec_parts, 4) : 0.0;
}

// A warp's part of an update item in segments (slots of up to kSliceNodes): an item is 8, 4 or 2 class rows
// by 128 class columns, and its eight warps hold the rows' segments at the node and its mirrors.  With
// rows of whole 16-byte vectors a lane holds one vector of each plane (reversed class columns on the
// mirrored side), else nodes 32 apart.
struct Seg {
  int lseg, seg;     // log2 of a class row's segments, and the warp's (bits: mirrored in x, in y, folded ones only)
  bool qx, qy, vec;  // mirrored side along x, along y; rows of whole vectors
  bool whole;        // all four nodes exist and form a vector
  int y, xb;         // class row, block of 128 class columns
  int g0, gs;        // node indices g0 + i gs
  unsigned have;     // which nodes exist (a middle row or column belongs to the unmirrored side)
  __device__ __forceinline__ int col(int i) const {
    const int lane = threadIdx.x & 31;
    return vec ? 4 * lane + (qx ? 3 - i : i) : 32 * i + lane;
  }
  __device__ __forceinline__ float4 load(const float* a) const {
    if (whole) return *reinterpret_cast<const float4*>(a + g0);
    float4 v;
    v.x = (have & 1u) ? a[g0] : 0.f;
    v.y = (have & 2u) ? a[g0 + gs] : 0.f;
    v.z = (have & 4u) ? a[g0 + 2 * gs] : 0.f;
    v.w = (have & 8u) ? a[g0 + 3 * gs] : 0.f;
    return v;
  }
  __device__ __forceinline__ void store(float* a, const float4 v) const {
    if (whole) {
      *reinterpret_cast<float4*>(a + g0) = v;
      return;
    }
    if (have & 1u) a[g0] = v.x;
    if (have & 2u) a[g0 + gs] = v.y;
    if (have & 4u) a[g0 + 2 * gs] = v.z;
    if (have & 8u) a[g0 + 3 * gs] = v.w;
  }
};
__device__ __forceinline__ Seg seg_of(const SlotDesc& S, int tile) {
  Seg g;
  const int warp = threadIdx.x >> 5;
  const bool fx = (S.mir & 1) != 0, fy = (S.mir & 2) != 0;
  g.lseg = (fx ? 1 : 0) + (fy ? 1 : 0);
  g.seg = warp & ((1 << g.lseg) - 1);
  g.qx = fx && (g.seg & 1);
  g.qy = fy && (g.seg >> (g.lseg - 1));
  g.vec = (S.nx & 3) == 0;
  const int nxb = (S.mhx + 127) / 128;
  g.y = (tile / nxb) * (8 >> g.lseg) + (warp >> g.lseg);
  g.xb = tile % nxb;
  const int yy = g.qy ? S.ny - 1 - g.y : g.y;
  g.have = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int x = g.xb * 128 + g.col(i);
    if (g.y < S.mhy && !(g.qy && yy == g.y) && x < S.mhx && !(g.qx && S.nx - 1 - x == x)) g.have |= 1u << i;
  }
  const int x = g.xb * 128 + g.col(0);
  g.g0 = yy * S.nx + (g.qx ? S.nx - 1 - x : x);
  g.gs = g.vec ? 1 : g.qx ? -32 : 32;
  g.whole = g.vec && g.have == 15u;
  return g;
}

// alpha = rho / p.q is usable (p.q > 0, everything finite)
__device__ __forceinline__ bool pq_ok(const SlotScalars* sc, double pq) {
  return pq > 0.0 && isfinite(pq) && isfinite(sc->rho2[sc->it & 1]);
}
// One thread: record p.q and alpha, or the breakdown.
__device__ __forceinline__ void finish_pq(SlotScalars* sc, double pq) {
  sc->pq = pq;
  if (!pq_ok(sc, pq)) {
    sc->status = ST_EBREAKDOWN;
    sc->active = 0;
    sc->fold = 1;  // the tail replaces the residual and reports the best iterate
    return;
  }
  const double rho = sc->rho2[sc->it & 1];
  sc->alpha = rho / pq;
  const f2 af = df_of(sc->alpha);
  sc->alpha_f[0] = af.hi;
  sc->alpha_f[1] = af.lo;
  const double aro = sc->alpha * rho;
  sc->aro_total += aro;
  sc->aro_ring[sc->aro_n % kErrDelay] = aro;
  sc->aro_n += 1;
}

// One thread, after an update with ||r||^2 = s: count the iteration and decide stop or residual
// replacement.
__host__ __device__ __forceinline__ void decide_update(SlotScalars* sc, double s) {
  sc->rr = s;
  const int itn = sc->it + 1;
  sc->it = itn;
  if (s <= sc->rtol2 * sc->bb || itn >= sc->maxit || !isfinite(s)) {
    sc->active = 0;
    sc->fold = 1;
  } else if (s < sc->delta2 * sc->rr_ref || itn % sc->fold_every == 0) {
    sc->fold = 1;
  }
}
// The same in three dimensions, where blocks of iterations have a fixed length: a replacement that is due
// (fold_every counts from the last one) stops the iterations, so that it comes at this one and not at the
// block's end; decide_true lets them go on.
__host__ __device__ __forceinline__ void decide_update3(SlotScalars* sc, double s) {
  sc->rr = sc->rr_rec = s;
  const int itn = sc->it + 1;
  sc->it = itn;
  if (s <= sc->rtol2 * sc->bb || itn >= sc->maxit || !isfinite(s) || s < sc->delta2 * sc->rr_ref ||
      itn - sc->it_ref >= sc->fold_every) {
    sc->active = 0;
    sc->fold = 1;
  }
}
// One thread, after the true residual's ||r||^2 = s: converged, stopped, or continue with a fresh
// preconditioner pass.
__host__ __device__ __forceinline__ void decide_true(SlotScalars* sc, double s) {
  sc->rr_true = s;
  sc->rr = s;
  sc->rr_ref = s;
  sc->it_ref = sc->it;
  sc->fold = 0;
  sc->active = 0;
  sc->need_prec = 0;
  if (s <= sc->rtol2 * sc->bb) {
    sc->status = ST_OK;
  } else if (sc->status == ST_EBREAKDOWN) {
  } else if (sc->it >= sc->maxit || !isfinite(s)) {
    sc->status = ST_ENOTCONV;
  } else {
    sc->active = 1;
    sc->need_prec = 1;
  }
}

// beta of the next direction (flexible or Fletcher-Reeves); 0 before the first iteration.
__device__ __forceinline__ double prec_beta(const SlotScalars* sc, double rz, double zq) {
  if (sc->it == 0) return 0.0;
  return sc->flexible ? -zq / sc->pq : rz / sc->rho2[(sc->it & 1) ^ 1];
}
__device__ __forceinline__ void record_preconditioner(SlotScalars* sc, double rz, double zq, double beta) {
  sc->zq = zq;
  sc->rho2[sc->it & 1] = rz;
  sc->beta = beta;
  const f2 bf = df_of(beta);
  sc->beta_f[0] = bf.hi;
  sc->beta_f[1] = bf.lo;
}
// One thread: record rho and beta, or the breakdown.  Mode 1 (the pass after a residual
// replacement) recomputes them for the same iteration.
__device__ __forceinline__ void finish_preconditioner(SlotScalars* sc, double rz, double zq, int mode) {
  if (mode == 2) {
    sc->rho2[0] = rz;
    sc->zq = zq;
    return;
  }
  const double beta = prec_beta(sc, rz, zq);
  record_preconditioner(sc, rz, zq, beta);
  if (!isfinite(rz) || !isfinite(beta)) {
    sc->status = ST_EBREAKDOWN;
    sc->active = 0;
    sc->fold = 1;
  }
  if (mode == 1) sc->need_prec = 0;
}

}  // namespace bx
