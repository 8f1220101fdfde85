// Fast Poisson preconditioner (Sec. 2.2 / Algorithm 1) on the 5th-generation tensor cores.
//
// z = M Q_y W Q_y^T (M r) Q_x W ... written separably on the padded rectangle:
//   stage 0: T1[kx][y]  = sum_x r[y][x]  Qx[x][kx]       (forward transform along x)
//   stage 1: T2[ky][kx] = w(ky,kx) sum_y T1[kx][y] Qy[y][ky]   (along y, times 1/(lam+mu)^2)
//   stage 2: T3[x][ky]  = sum_kx T2[ky][kx] Qx[x][kx]    (inverse along x)
//   stage 3: z[y][x]    = mask(y,x) sum_ky T3[x][ky] Qy[y][ky] (inverse along y), plus partial
//            r.z, z.q per tile (reduced by k_prec_finish or the next stencil)
// Every stage is D[m][n] = sum_k A[m][k] B[n][k] with both operands k-contiguous, written out
// transposed (Out[n][m]) so the next stage again reads a k-contiguous operand.  The products run
// as tcgen05 MMAs with FP16 or BF16 operands and FP32 accumulation.
// This operator is so ill-conditioned that a plain 16-bit operand ruins the preconditioner, and
// even float hi/lo operand splits lose too much in the tensor core's truncating FP32
// accumulation.  The products are therefore made exact:
//
//  * every operand is cut into blocks of KC = 128 consecutive k; a block with largest magnitude
//    below 2^E (and 2^(8-E) times it below 255.5) is stored as four integer slices,
//    v = c0 2^(E-8) + c1 2^(E-16) + c2 2^(E-24) + c3 2^(E-32), |c0| <= 255, |c1..c3| <= 128
//    (exact in FP16 and BF16), plus the exponent E (int8);
//  * for each slice order d = i + j <= 3 (products c_i c'_j; higher orders are below 2^-32 of
//    the block and dropped) a separate TMEM accumulator sums one k-block.  The B slices are
//    stacked along N, so the ten products of a k-step take four MMAs (N = 256, 192, 128, 64).
//    Per k, the products of one order add up to less than 2^16.6, so over 128 k every partial
//    sum is an exact integer below 2^24 and so is the accumulation;
//  * the epilogue warps scale the four exact sums by 2^(E_A + E_B - 16 - 8d) and add them into
//    a compensated (hi, lo) register pair, k-block after k-block, two columns per packed FP32x2
//    operation.
// The operands carry 32 bits relative to each 128-block's largest value and the products add no
// error along K; the stage outputs stay double-float (hi, lo) pairs and are sliced from them
// directly, and the last stage writes z as a double-float pair.  Three slices on
// 64-blocks (24 bits) cost this operator 30-80% more CG iterations than exact transforms; four on
// 128-blocks come within 5-10% of them.
//
// FP32 mode, and the mixed modes' smaller grids, run the same kernels with six slices per operand
// (48 bits of each 128-block, orders 0..5, 21 products), the accuracy of the double-float vectors:
// they take the FP64 iteration's count plus 10-20%.  Its tiles are 128 x 32 (six accumulators twice in TMEM) and its steps 32 deep.
//
// Kernel structure (one CTA per SM, persistent over the (slot, tile) work list):
//   warp 0      : TMA producer: 128B-swizzled K-major tiles of the slices of A and B, two 64-deep
//                 steps of 96 KB
//   warp 1      : TMEM allocation; issues the MMAs and the tcgen05.commit arrivals
//   warps 2..17 : four per TMEM lane quarter (32 rows), each owning a quarter of the tile's columns:
//                 exact k-block sums -> compensated registers -> the stage's epilogue
//                 (eigenvalue weights; masking and per-tile r.z, z.q partials in stage 3).
//
// What bounds it.  A step's ten products take 1,700 SM cycles at the measured BF16 peak; the
// k-loop runs at 1,660 (clock stamps, 1024^2 grid).  Getting there took the issuing warp out of
// the way: run by one lane under a divergent branch it spent 62 cycles an MMA on moving the
// descriptors to uniform registers and 300 a wait, 2,050 a step, so the whole warp now runs the
// loop (uniform descriptors, one elected lane issues) and a wait first tests its barrier without
// reading the clock.  Per-plane barriers for A (earlier refills, but five waits and commits a step)
// measured 3,250 cycles a step; 32-deep steps with a 64-byte swizzle were no faster either.
// Then the epilogue: it reads TMEM in the 16x256b shape, whose register layout is that of an
// 8 x 8 matrix fragment: a thread holds four rows by a few columns, so row and column factors need a
// few shuffles, a column's maximum over the rows three exchanges, and the 16-bit slices leave by
// transposing stmatrix into a swizzled staging tile that tensor stores write out while the next
// tile runs.  (With one row per thread a tile took 64 two-byte stores and about 80 shuffles per
// thread.)  What is left after the last k-block is FP32 issue: about 1,300 cycles for the merge, 2,000
// for slicing and storing, 2,000 for stage 1's weights.
// Every wait on an mbarrier is bounded; on time-out the CTA raises an error flag, drains its
// outstanding copies and MMAs, frees its TMEM and returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "async.cuh"
#include "common.cuh"
#include "kernels.h"

namespace bx {
namespace {

constexpr int BM = 128;
constexpr int KC = 128;                     // k per exponent / exact accumulation block
constexpr int kEpiWarps = 16;
static_assert(KC == BM, "one exponent block per tile column");
constexpr int kThreads = 64 + 32 * kEpiWarps;
// One CTA per SM.  Each of the SM's four schedulers owns a quarter of the register file and
// holds up to ceil(warps / 4) of the CTA's warps.
constexpr int kMaxRegs = (16384 / (32 * ((kThreads / 32 + 3) / 4))) & ~7;
constexpr int kChunks = 2;                       // TMEM ring of k-block accumulator sets
constexpr int kTmemCols = 512;                   // power of two >= kChunks * sets
constexpr int kMaxSteps = 3;                     // pipeline steps in flight

// The products a launch can be: the preconditioner's four stages, and the low-mode correction's
// forward and inverse products (six slices).
constexpr int kLowFwd = 4, kLowInv = 5;

// Tile geometry by the number of slices: shared memory holds two steps of both operands and the
// staging tile of the outgoing slices; six slices of a 64-deep step would not fit twice.
template <int STAGE, int NSL>
struct TcGeom {
  static constexpr bool kLow = STAGE == kLowFwd || STAGE == kLowInv;
  static constexpr int BN = NSL == 4 ? 64 : 32;   // tile columns
  static constexpr int BK = NSL == 4 ? 64 : 32;   // one swizzle atom (128 or 64 bytes) per pipeline step
  static constexpr int KPC = STAGE == kLowInv ? 1 : KC / BK;  // pipeline steps per accumulation block
  static constexpr int A_PLANE = BM * BK * 2;
  static constexpr int kCb = BN / 32;             // 8-column blocks per epilogue warp
  static constexpr int kEpiCols = 8 * kCb;        // tile columns per epilogue warp
  static constexpr int kBPlane = BN * BK * 2;
  static constexpr int kStageBytes = NSL * (A_PLANE + kBPlane);  // one step of both operands
  // staging of the epilogue: a group of the outgoing slices [slice][64-row half][column] as 128-byte
  // rows (six slices leave in two groups, which makes room for a third step in flight: with two, a
  // 32-deep step waited for its copies); the forward low-mode product's H tile and Qy rows; nothing
  // where the results go straight to memory
  static constexpr int kGroup = NSL == 4 ? 4 : 3;
  static constexpr int kStage = STAGE == kLowFwd ? 8 * BM * 33 + 8 * BM * kLowM
                                                 : STAGE <= 2 ? kGroup * 32 * BM * 2 : 0;
  static constexpr int kSteps = NSL == 6 && STAGE != kLowFwd ? 3 : 2;
  static constexpr int kSetCols = NSL * BN;       // one accumulator per slice order
  static constexpr int kSmem = kSteps * kStageBytes + kStage + 1024 + 2048;
  static_assert(!kLow || NSL == kLowNS, "six slices in the low-mode products");
  static_assert(kChunks * kSetCols <= kTmemCols, "TMEM columns");
  static_assert(kSmem <= 232448 && kStage % 8 == 0, "shared memory of an SM's block");
};

struct Ctl {
  uint64_t full[kMaxSteps];
  uint64_t empty[kMaxSteps];
  uint64_t tfull[kChunks];
  uint64_t tempty[kChunks];
  uint64_t drain;
  uint32_t tmem;
  int abort_flag;
  Sum3 red[2][kEpiWarps];                 // stage 3: per-warp r.z and z.q
  float colmax[4][16][4];                 // [column group][column][lane quarter]
};
static_assert(sizeof(Ctl) <= 2048, "control block too large");

// UMMA shared-memory descriptor: K-major operand, rows of K 16-bit values swizzled over 2 K = 128 or
// 64 bytes, 8-row core groups 16 K bytes apart.
template <int K = 64>
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
  static_assert(K == 64 || K == 32, "swizzle atoms");
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
  d |= static_cast<uint64_t>(1) << 16;          // leading-dimension offset (unused here)
  d |= static_cast<uint64_t>(16 * K >> 4) << 32;  // stride between 8-row groups
  d |= static_cast<uint64_t>(1) << 46;          // descriptor version
  d |= static_cast<uint64_t>(K == 64 ? 2 : 4) << 61;  // 128- or 64-byte swizzle
  return d;
}
// Instruction descriptor of kind::f16: FP32 accumulator, both operands K-major, M x N tile.
__host__ __device__ constexpr uint32_t idesc_f16(bool bf16, int M, int N) {
  return (1u << 4) | ((bf16 ? 1u : 0u) << 7) | ((bf16 ? 1u : 0u) << 10) |
         (static_cast<uint32_t>(N >> 3) << 17) | (static_cast<uint32_t>(M >> 4) << 24);
}
__device__ __forceinline__ void umma(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(a), "l"(b), "r"(idesc), "r"(accum)
      : "memory");
}
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
// One lane of the (converged) warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "elect.sync _|q, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(p));
  return p != 0;
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// Sixteen TMEM lanes by eight columns as a matrix fragment: lane l of the warp gets columns
// 2 (l % 4), 2 (l % 4) + 1 of rows l / 4 (v[0], v[1]) and l / 4 + 8 (v[2], v[3]).
__device__ __forceinline__ void tmem_ld_frag(uint32_t taddr, uint32_t (&v)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
               : "r"(taddr));
}
// Four 8 x 8 matrices of 16-bit values (fragments v[0..3]: lane l holds columns 2 (l % 4), + 1 of row
// l / 4) stored transposed: lanes 8 k .. 8 k + 7 give the addresses of matrix k's columns.
__device__ __forceinline__ void stmatrix4_t(uint32_t saddr, const uint32_t (&v)[4]) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(saddr), "r"(v[0]),
               "r"(v[1]), "r"(v[2]), "r"(v[3])
               : "memory");
}
__device__ __forceinline__ void tma_store_2d(const void* tmap, uint32_t saddr, int c0, int c1) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
                   reinterpret_cast<uint64_t>(tmap)),
               "r"(saddr), "r"(c0), "r"(c1)
               : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// A global load that stays where it is written (volatile asm is not moved across the other
// volatile asm of the k-block loop), so its latency overlaps the loop.
__device__ __forceinline__ float ld_early(const float* p) {
  float v;
  asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}

__device__ __forceinline__ unsigned ld_keep(const void* p) {
  unsigned v;
  asm volatile("ld.global.nc.u32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}

// 2^e as a float for e in the normal range, 0 below it.
__device__ __forceinline__ float pow2f(int e) {
  return e < -126 ? 0.f : __int_as_float((min(e, 127) + 127) << 23);
}

// Exponent E of a block whose largest magnitude is amax: amax < 2^E and amax 2^(8-E) < 255.5, so the
// leading slice stays within +-256 (0 for an all-zero block).
__device__ __forceinline__ int block_exp(float amax) {
  if (!(amax > 0.f)) return 0;
  int e;
  frexpf(amax, &e);
  if (amax * pow2f(8 - e) >= 255.5f) ++e;
  // 2^(16-E) stays finite, and the block's sums are scaled by 2^(E-16) >= 2^-126: smaller blocks lose
  // what FP32's own unit of 2^-149 takes from them
  return max(e, -110);
}

// The NSL integer slices of double-float values (hi, lo) for block exponent E, given up = 2^(16-E), on
// two lanes with their own block factors.  The value is brought to the block's scale (exactly: below
// 2^16 in magnitude at any E) and taken sixteen bits at a time: w = the integer nearest to the leading
// plane, removed exactly, the remainder joined with the lo plane and scaled up by 2^16; and each w is cut
// into its two digits w = 256 c0 + c1, |c1| <= 128.  The slices carry the value to 2^-32 (NSL = 4) or
// 2^-48 (6) of the block.  Roundings to the nearest integer add and remove 1.5 * 2^23 on packed FP32x2
// (exact for magnitudes below 2^22; ties to even); a digit is an integer of magnitude at most 256,
// exact in BF16, whose bits are the upper half of the FP32 bits (one byte permutation packs the two
// lanes' codes).  FP16 codes come from the packed two-value conversion.  About 4 packed operations
// a digit; the form before, one digit at a time with a renormalised remainder, took 12.
template <bool BF16, int NSL>
__device__ __forceinline__ void slice_codes2_df(float2 vh, float2 vl, float2 up, uint32_t (&code)[NSL]) {
  static_assert(NSL == 4 || NSL == 6, "slices in pairs");
  const float2 rnd = make_float2(12582912.f, 12582912.f), rnd_n = make_float2(-12582912.f, -12582912.f);
  float2 rh = __fmul2_rn(vh, up), rl = __fmul2_rn(vl, up);
#pragma unroll
  for (int k = 0; k < NSL; k += 2) {
    const float2 w = __fadd2_rn(__fadd2_rn(rh, rnd), rnd_n);
    if (k + 2 < NSL) {
      const float2 h = sub2(rh, w);
      if (k + 4 < NSL) {
        two_sum2(h, rl, rh, rl);
        rl = mul2(65536.f, rl);
      } else {
        rh = __fadd2_rn(h, rl);
      }
      rh = mul2(65536.f, rh);
    }
    float2 c[2];
    c[0] = __fadd2_rn(__ffma2_rn(w, make_float2(0.00390625f, 0.00390625f), rnd), rnd_n);
    c[1] = __ffma2_rn(c[0], make_float2(-256.f, -256.f), w);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      if (BF16) {
        code[k + j] = __byte_perm(__float_as_uint(c[j].x), __float_as_uint(c[j].y), 0x7632);
      } else {
        const __half2 h2 = __floats2half2_rn(c[j].x, c[j].y);
        code[k + j] = static_cast<uint32_t>(__half_as_ushort(__low2half(h2))) |
                      (static_cast<uint32_t>(__half_as_ushort(__high2half(h2))) << 16);
      }
    }
  }
}

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

__device__ __forceinline__ bool slot_runs(const SlotScalars* sc, int mode) {
  return mode == 0 ? sc->active != 0 : (mode == 1 ? sc->need_prec != 0 : true);
}

__device__ __forceinline__ void epi_bar() {
  asm volatile("bar.sync 1, %0;" ::"r"(32 * kEpiWarps) : "memory");
}

// Barrier of the epilogue warps that also tells whether any of them has failed.
__device__ __forceinline__ bool epi_vote(bool fail) {
  uint32_t any;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "bar.red.or.pred q, 1, %2, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(any)
      : "r"(fail ? 1u : 0u), "r"(32 * kEpiWarps)
      : "memory");
  return any != 0;
}

struct TcStage {
  int M, N, K;                   // padded extents (K: the exponents' row length)
  int n, k;                      // real columns of the result and real k: beyond them all is zero
  const unsigned char *ma, *mb;  // tensor maps of A and B
  const int8_t *ea, *eb;         // block exponents: A rows [M][K / KC], B rows [N][K / KC]
  int8_t* eout;                  // next stage's block exponents [N][M/128]
};

template <int STAGE>
__device__ __forceinline__ TcStage tc_stage(const SlotDesc& S) {
  const unsigned char* maps = static_cast<const unsigned char*>(S.tmaps);
  const unsigned char* low = static_cast<const unsigned char*>(S.low_maps);
  if constexpr (STAGE == kLowFwd)  // H = r Qx_low
    return {S.nyp, kLowM, S.nxp, kLowM, S.nx, low, low + 128, S.tc_e[0], S.low_qxt_e, nullptr};
  else if constexpr (STAGE == kLowInv)  // zl^T = J^T Qy_low^T, one block of 32 k
    return {S.nxp, S.nyp, kLowM, S.ny, kLowM, low + 256, low + 384, S.low_jt_e, S.low_qy_e, nullptr};
  else {
    const int8_t *ea = S.tc_e[STAGE], *eb = S.tc_eb[STAGE];
    int8_t* eo = STAGE < 3 ? S.tc_e[(STAGE + 1) & 3] : nullptr;
    if constexpr (STAGE == 0 || STAGE == 2)
      return {S.nyp, S.nxp, S.nxp, S.nx, S.nx, maps + 128 * STAGE, maps + 128 * (4 + STAGE), ea, eb, eo};
    else
      return {S.nxp, S.nyp, S.nyp, S.ny, S.ny, maps + 128 * STAGE, maps + 128 * (4 + STAGE), ea, eb, eo};
  }
}

// Merge of one pair of columns' order sums (exact integers) into the compensated pair (hi, lo);
// scl = 2^(E_A + E_B - 16) of the two columns.  Four slices: orders 1..3 are combined first, their
// roundings are 2^-24 of terms 2^-8 below hi.  Six: orders 0..2 by TwoSum, 3..5 in plain FP32.
template <int NSL>
__device__ __forceinline__ void merge_orders(const float2 (&v)[NSL], float2 scl, float2& hi, float2& lo) {
  const float2 q8 = make_float2(0.00390625f, 0.00390625f);
  float2 er;
  if constexpr (NSL == 4) {
    const float2 w = __ffma2_rn(v[3], q8, v[2]);
    const float2 u = __ffma2_rn(w, q8, v[1]);
    const float2 t0 = __fmul2_rn(v[0], scl);
    const float2 t1 = __fmul2_rn(u, __fmul2_rn(scl, q8));
    two_sum2(hi, t0, hi, er);
    lo = add2(lo, add2(er, t1));
  } else {
    const float2 w = __ffma2_rn(__ffma2_rn(v[5], q8, v[4]), q8, v[3]);
    const float2 s1 = __fmul2_rn(scl, q8), s2 = __fmul2_rn(s1, q8);
    two_sum2(hi, __fmul2_rn(v[0], scl), hi, er);
    lo = add2(lo, er);
    two_sum2(hi, __fmul2_rn(v[1], s1), hi, er);
    lo = add2(lo, er);
    two_sum2(hi, __fmul2_rn(v[2], s2), hi, er);
    lo = add2(lo, add2(er, __fmul2_rn(w, __fmul2_rn(s2, q8))));
  }
}

// DOTS3: FP32 mode's stage 3 (reduce_dots)
template <bool BF16, int STAGE, int NSL, bool DOTS3 = false>
__global__ void __maxnreg__(kMaxRegs)
k_prec_tc(const SlotDesc* __restrict__ slots, const WorkItem* __restrict__ items,
          const int* __restrict__ n_items, int mode, int* __restrict__ err, long long wait_cycles) {
  using G = TcGeom<STAGE, NSL>;
  constexpr int BN = G::BN, kCb = G::kCb, kEpiCols = G::kEpiCols, BK = G::BK, KPC = G::KPC;
  constexpr int A_PLANE = G::A_PLANE, STAGES = G::kSteps;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  unsigned char* sO = smem + STAGES * G::kStageBytes;
  Ctl* ctl = reinterpret_cast<Ctl*>(sO + G::kStage);
  volatile int* abort_flag = &ctl->abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int total = *n_items;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&ctl->full[s], 1);
      mbar_init(&ctl->empty[s], 1);
    }
    for (int a = 0; a < kChunks; ++a) {
      mbar_init(&ctl->tfull[a], 1);
      mbar_init(&ctl->tempty[a], kEpiWarps);
    }
    mbar_init(&ctl->drain, 1);
    ctl->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = ctl->tmem;
  // Each role reads its first tile's item and descriptor, which no kernel writes, before it waits
  // for the previous kernel (pdl_wait): those dependent loads took 1 us after the wait.

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      struct Tile {
        const SlotScalars* sc;
        const unsigned char *ma, *mb;
        int M, N, steps, m0, n0;
      };
      auto tile_of = [&](int w) -> Tile {
        const WorkItem it = items[w];
        if (it.slot < 0) return {};
        const SlotDesc& S = slots[it.slot];
        const TcStage v = tc_stage<STAGE>(S);
        const int mt = v.M / BM;
        Tile t = {S.sc, v.ma, v.mb, v.M, v.N, (v.k + BK - 1) / BK, (it.tile % mt) * BM, (it.tile / mt) * BN};
        if (t.n0 >= v.n) t.steps = 0;  // nothing but padding
        tmap_acquire(t.ma);
        tmap_acquire(t.mb);
        return t;
      };
      Tile t = {};
      if (blockIdx.x < total) t = tile_of(blockIdx.x);
      pdl_wait();
      int n = 0;  // steps issued
      for (int w = blockIdx.x; w < total && !*abort_flag; w += gridDim.x) {
        if (w != blockIdx.x) t = tile_of(w);
        if (t.sc == nullptr || !slot_runs(t.sc, mode)) continue;
        for (int kb = 0; kb < t.steps; ++kb) {
          const int st = n % STAGES;
          unsigned char* sa = smem + st * G::kStageBytes;
          unsigned char* sb = sa + NSL * A_PLANE;
          if (!mbar_wait(&ctl->empty[st], ((n / STAGES) & 1) ^ 1, abort_flag, wait_cycles)) break;
          mbar_expect_tx(&ctl->full[st], G::kStageBytes);
#pragma unroll
          for (int p = 0; p < NSL; ++p)
            tma_load_2d(sa + p * A_PLANE, t.ma, &ctl->full[st], kb * BK, p * t.M + t.m0);
#pragma unroll
          for (int p = 0; p < NSL; ++p)
            tma_load_2d(sb + p * G::kBPlane, t.mb, &ctl->full[st], kb * BK, p * t.N + t.n0);
          ++n;
        }
      }
      if (*abort_flag) {
        // let the copies already issued (the last into each stage) land before the CTA leaves
        const long long t0 = clock64();
        for (int s = 0; s < STAGES; ++s) {
          const int k = (n - s + STAGES - 1) / STAGES;  // steps issued into stage s
          if (k > 0)
            while (!mbar_try(&ctl->full[s], (k - 1) & 1) && clock64() - t0 < kWaitCycles / 4) {
            }
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    // the whole warp runs the loop, so that the descriptors stay in uniform registers; one elected
    // lane issues
    const bool elected = elect_one();
    int n = 0, chunk = 0;
    bool ok = true;
    const SlotScalars* sc = nullptr;
    int k_tile = 0;
    auto tile_of = [&](int w) {
      const int slot = items[w].slot;
      sc = slot < 0 ? nullptr : slots[slot].sc;
      k_tile = 0;
      if (slot >= 0) {
        const TcStage v = tc_stage<STAGE>(slots[slot]);
        if (items[w].tile / (v.M / BM) * BN < v.n) k_tile = v.k;
      }
    };
    if (blockIdx.x < total) tile_of(blockIdx.x);
    pdl_wait();
    for (int w = blockIdx.x; w < total && ok; w += gridDim.x) {
      if (w != blockIdx.x) tile_of(w);
      if (!__any_sync(0xffffffffu, sc != nullptr && slot_runs(sc, mode))) continue;
      const int steps = __reduce_max_sync(0xffffffffu, (k_tile + BK - 1) / BK);
      for (int kb = 0; kb < steps; ++kb) {
        const int half_kb = kb % KPC;  // position inside the accumulation block
        const int cb = chunk % kChunks, st = n % STAGES;
        bool got = half_kb != 0 || mbar_wait(&ctl->tempty[cb], ((chunk / kChunks) & 1) ^ 1, abort_flag, wait_cycles);
        got = got && mbar_wait(&ctl->full[st], (n / STAGES) & 1, abort_flag, wait_cycles);
        ok = __all_sync(0xffffffffu, got);
        if (!ok) break;
        tc_fence_after();
        const uint32_t dset = tmem_base + cb * G::kSetCols;
        const uint64_t ad = sdesc<BK>(smem_u32(smem + st * G::kStageBytes));
        const uint64_t bd = sdesc<BK>(smem_u32(smem + st * G::kStageBytes + NSL * A_PLANE));
        if (elected) {
          // slice pa of A against the B slices 0 .. NSL-1-pa stacked along N (adjacent in shared
          // memory): one MMA adds A_pa B_pb to the accumulator of order pa + pb for every pb,
          // since the order accumulators are adjacent in TMEM the same way; the first MMA of an
          // accumulation block (pa = 0) starts all orders afresh
#pragma unroll
            for (int j = 0; j < BK / 16; ++j)
#pragma unroll
              for (int pa = 0; pa < NSL; ++pa)
                umma(dset + pa * BN, ad + ((pa * A_PLANE) >> 4) + 2 * j, bd + 2 * j, idesc_f16(BF16, BM, (NSL - pa) * BN),
                     (half_kb > 0 || j > 0 || pa > 0) ? 1u : 0u);
          umma_commit(&ctl->empty[st]);
          if (half_kb == KPC - 1 || kb == steps - 1) umma_commit(&ctl->tfull[cb]);
        }
        ++n;
        if (half_kb == KPC - 1 || kb == steps - 1) ++chunk;
      }
    }
    if (elected) {
      // all MMAs issued by this thread complete before TMEM can be released
      umma_commit(&ctl->drain);
      const long long t0 = clock64();
      while (!mbar_try(&ctl->drain, 0) && clock64() - t0 < kWaitCycles) {
      }
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------------ epilogue
    const int quarter = warp & 3;            // TMEM lanes 32*quarter .. +31
    const int ew = warp - 2;
    const int group = ew >> 2;               // columns 32 cb + 8 group .. + 7 of the tile, cb < kCb
    // the thread's rows of the quarter: 8 rb + t4, rb = 0..3; its columns: 2 tc + e, e = 0, 1, of each
    // of the group's column blocks (one packed pair per rb and cb)
    const int t4 = lane >> 2, tc = lane & 3;
    const bool col_lane = lane < kEpiCols;   // lanes that own one of the warp's columns
    int chunk = 0;
    if (blockIdx.x < total && items[blockIdx.x].slot >= 0) {
      // the first tile's descriptor into this SM's L1
      const SlotDesc& S = slots[items[blockIdx.x].slot];
      if (lane < static_cast<int>((sizeof(SlotDesc) + 127) / 128)) {
        const unsigned first = ld_keep(reinterpret_cast<const char*>(&S) + 128 * lane);
        if (first == 0x7fedcba9u) __nanosleep(1);  // the load has a use
      }
    }
    pdl_wait();
    // the epilogue warps leave the list only together, at a vote: after an abort their waits fail
    for (int w = blockIdx.x; w < total; w += gridDim.x) {
      const WorkItem it = items[w];
      if (it.slot < 0) continue;  // an empty place of the balanced list
      const SlotDesc& S = slots[it.slot];
      SlotScalars* sc = S.sc;
      if (!slot_runs(sc, mode)) continue;
      const TcStage v = tc_stage<STAGE>(S);
      const int mt = v.M / BM;
      const int m0 = (it.tile % mt) * BM, n0 = (it.tile / mt) * BN;
      const int mq = m0 + 32 * quarter;          // first row of the quarter
      const int ng = n0 + 8 * group;             // first column of the group (block cb: + 32 cb)
      const int n_mine = ng + 32 * (lane >> 3) + (lane & 7);  // a column lane's column
      if (n0 >= v.n) continue;                   // nothing but padding
      const int kblocks = STAGE == kLowInv ? 1 : (v.k + KC - 1) / KC;
      const int erow = STAGE == kLowInv ? 1 : v.K / KC;  // the exponents' row length
      if (STAGE == 3 && col_lane && !S.mir_out) {
        // the r, q and mask entries read after the last k-block: start them towards L2 now
        const int n = n_mine;
        if (n < S.ny && mq < S.nx) {
          const size_t g = static_cast<size_t>(n) * S.nx + mq;
          const size_t g1 = static_cast<size_t>(n) * S.nx + min(mq + 31, S.nx - 1);
          asm volatile("prefetch.global.L2 [%0];" ::"l"(S.r + g));
          asm volatile("prefetch.global.L2 [%0];" ::"l"(S.r + g1));
          asm volatile("prefetch.global.L2 [%0];" ::"l"(S.q + g));
          asm volatile("prefetch.global.L2 [%0];" ::"l"(S.q + g1));
          asm volatile("prefetch.global.L2 [%0];" ::"l"(S.mask + g));
        }
      }
      // stage 1's eigenvalues, read now (the MMA waits hide their latency) with the grid's edge
      // folded in: a row or column outside it makes the eigenvalue sum negative, and its weight zero
      float lamx[4], lamy[2 * kCb], wnorm = 0.f;
      if (STAGE == 1) {
#pragma unroll
        for (int rb = 0; rb < 4; ++rb) {
          const int m = mq + 8 * rb + t4;
          lamx[rb] = m < S.nx ? ld_early(S.lamx + m) : -INFINITY;
        }
#pragma unroll
        for (int c = 0; c < 2 * kCb; ++c) {
          const int n = ng + 32 * (c >> 1) + 2 * tc + (c & 1);
          lamy[c] = n < S.ny ? ld_early(S.lamy + n) : -INFINITY;
        }
        wnorm = ld_early(&S.wnorm);
      }
      const int8_t* ea_row = v.ea + static_cast<size_t>(mq + lane) * erow;
      const int8_t* eb_col = v.eb + static_cast<size_t>(col_lane ? n_mine : ng) * erow;
      // the thread's share of the tile's Qy_low rows (the G share's operand), loaded now so that
      // their latency hides behind the k-blocks
      constexpr int kYq = STAGE == kLowFwd ? BM * kLowM / (32 * kEpiWarps) : 1;
      float yq[2 * kYq];
      if (STAGE == kLowFwd) {
#pragma unroll
        for (int i = 0; i < kYq; ++i) {
          const size_t a = static_cast<size_t>(m0) * kLowM + 32 * ew + lane + i * 32 * kEpiWarps;
          yq[i] = ld_early(S.low_qyd + a);
          yq[kYq + i] = ld_early(S.low_qyd + static_cast<size_t>(S.nyp) * kLowM + a);
        }
      }
      // compensated (hi, lo) pairs, one packed register pair per (rb, cb)
      float2 hi[kCb][4], lo[kCb][4];
#pragma unroll
      for (int cb = 0; cb < kCb; ++cb)
#pragma unroll
        for (int rb = 0; rb < 4; ++rb) {
          hi[cb][rb] = make_float2(0.f, 0.f);
          lo[cb][rb] = make_float2(0.f, 0.f);
        }
      bool fail = false;
      for (int kb = 0; kb < kblocks; ++kb) {
        const int cs = chunk % kChunks;
        // factors of the block sums, 2^(E_A - 16) of the lane's row and 2^E_B of its column
        const float sa_mine = pow2f(static_cast<int>(ea_row[kb]) - 16);
        const float sb_mine = pow2f(eb_col[kb]);
        // a warp that gives up waiting leaves with the others at the vote after the k-blocks
        if (!fail) fail = !mbar_wait(&ctl->tfull[cs], (chunk / kChunks) & 1, abort_flag, wait_cycles);
        tc_fence_after();
        float sa[4];
#pragma unroll
        for (int rb = 0; rb < 4; ++rb) sa[rb] = __shfl_sync(0xffffffffu, sa_mine, 8 * rb + t4);
        const uint32_t base = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + cs * G::kSetCols + ng - n0;
#pragma unroll
        for (int cb = 0; cb < kCb; ++cb) {
          const float2 sb = make_float2(__shfl_sync(0xffffffffu, sb_mine, 8 * cb + 2 * tc),
                                        __shfl_sync(0xffffffffu, sb_mine, 8 * cb + 2 * tc + 1));
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            uint32_t o[NSL][4];
#pragma unroll
            for (int d = 0; d < NSL; ++d)
              tmem_ld_frag(base + (static_cast<uint32_t>(16 * h) << 16) + d * BN + 32 * cb, o[d]);
            tmem_wait_ld();
            if (cb == kCb - 1 && h == 1) {
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(&ctl->tempty[cs]);
            }
#pragma unroll
            for (int r = 0; r < 2; ++r) {
              const int rb = 2 * h + r;
              float2 x[NSL];
#pragma unroll
              for (int d = 0; d < NSL; ++d)
                x[d] = make_float2(__uint_as_float(o[d][2 * r]), __uint_as_float(o[d][2 * r + 1]));
              merge_orders<NSL>(x, mul2(sa[rb], sb), hi[cb][rb], lo[cb][rb]);
            }
          }
        }
        ++chunk;
      }
      // the sums as normalised double-float pairs
#pragma unroll
      for (int cb = 0; cb < kCb; ++cb)
#pragma unroll
        for (int rb = 0; rb < 4; ++rb) {
          const f2x2 t = df_norm2(hi[cb][rb], lo[cb][rb]);
          hi[cb][rb] = t.hi;
          lo[cb][rb] = t.lo;
        }
      if (STAGE == 1) {
        // weight 1/(lam_y + lam_x)^2 (normalised); the low block (m < lowm_x, n < lowm_y) comes
        // from the six-slice products instead
        const bool low_tile = S.lowm_x != 0 && mq == 0 && ng < kLowM;
        const int lowx = S.lowm_x, lowy = S.lowm_y;
#pragma unroll
        for (int cb = 0; cb < kCb; ++cb)
#pragma unroll
          for (int rb = 0; rb < 4; ++rb) {
            const float s0 = lamy[2 * cb] + lamx[rb], s1 = lamy[2 * cb + 1] + lamx[rb];
            bool ok0 = s0 > 0.f, ok1 = s1 > 0.f;
            if (low_tile && 8 * rb + t4 < lowx) {
              ok0 = ok0 && ng + 32 * cb + 2 * tc >= lowy;
              ok1 = ok1 && ng + 32 * cb + 2 * tc + 1 >= lowy;
            }
            const float2 wt = make_float2(ok0 ? spectral_weight_of(wnorm, s0) : 0.f,
                                          ok1 ? spectral_weight_of(wnorm, s1) : 0.f);
            const float2 p = __fmul2_rn(hi[cb][rb], wt);
            const float2 e = __ffma2_rn(lo[cb][rb], wt, __ffma2_rn(hi[cb][rb], wt, neg2(p)));
            const f2x2 t = df_norm2(p, e);
            hi[cb][rb] = t.hi;
            lo[cb][rb] = t.lo;
          }
        // the tile's rows n beyond the grid lie in the padding of the residual's operand, which only zeros
        // may reach: a residual of NaNs makes NaNs of their zero sums
        if (n0 + BN > v.n) {
#pragma unroll
          for (int cb = 0; cb < kCb; ++cb)
#pragma unroll
            for (int rb = 0; rb < 4; ++rb) {
              const int n = ng + 32 * cb + 2 * tc;
              if (n >= v.n) hi[cb][rb].x = lo[cb][rb].x = 0.f;
              if (n + 1 >= v.n) hi[cb][rb].y = lo[cb][rb].y = 0.f;
            }
        }
      }
      if (STAGE == kLowFwd) {
        // the tile's share of G = Qy_low^T H (its 128 rows of y), by compensated dot products of
        // double-float operands staged in shared memory; H itself is not stored
        if (epi_vote(fail)) break;  // (also: the previous tile's dot products have read the staging)
        float* hs = reinterpret_cast<float*>(sO);  // H tile [128][33]: hi, then lo
        float* ys = hs + 2 * BM * 33;              // Qy_low rows m0 .. m0+127 [128][32]: hi, lo
#pragma unroll
        for (int rb = 0; rb < 4; ++rb) {
          float* h = hs + (32 * quarter + 8 * rb + t4) * 33 + 8 * group + 2 * tc;
          h[0] = hi[0][rb].x;
          h[1] = hi[0][rb].y;
          h[BM * 33] = lo[0][rb].x;
          h[BM * 33 + 1] = lo[0][rb].y;
        }
#pragma unroll
        for (int i = 0; i < kYq; ++i) {
          ys[32 * ew + lane + i * 32 * kEpiWarps] = yq[i];
          ys[BM * kLowM + 32 * ew + lane + i * 32 * kEpiWarps] = yq[kYq + i];
        }
        epi_bar();
        // thread: kx = lane, ky = 2 ew and 2 ew + 1, the two dot products on packed FP32x2 (one
        // 8-byte broadcast load of each plane's Qy_low pair per row)
        CompDotDF2 g;
        const int ky0 = 2 * ew;
#pragma unroll 4
        for (int rr = 0; rr < BM; ++rr) {
          const float bh = hs[rr * 33 + lane], bl = hs[BM * 33 + rr * 33 + lane];
          const float2 ah = *reinterpret_cast<const float2*>(ys + rr * kLowM + ky0);
          const float2 al = *reinterpret_cast<const float2*>(ys + BM * kLowM + rr * kLowM + ky0);
          g.add(ah, al, make_float2(bh, bh), make_float2(bl, bl));
        }
        float* gp = S.low_gp + static_cast<size_t>(it.tile) * 2 * kLowM * kLowM;
        const f2 a0 = df_norm(g.s.x, g.c.x), a1 = df_norm(g.s.y, g.c.y);
        gp[ky0 * kLowM + lane] = a0.hi;
        gp[kLowM * kLowM + ky0 * kLowM + lane] = a0.lo;
        gp[(ky0 + 1) * kLowM + lane] = a1.hi;
        gp[kLowM * kLowM + (ky0 + 1) * kLowM + lane] = a1.lo;
      } else if (STAGE == kLowInv) {
        // zl[y][x] at rows n = y of the tile's columns
        if (epi_vote(fail)) break;
        const int nx = S.nx, ny = S.ny;
        float* zl = S.low_z;
        const size_t nn = static_cast<size_t>(nx) * ny;
#pragma unroll
        for (int rb = 0; rb < 4; ++rb) {
          const int m = mq + 8 * rb + t4, n = ng + 2 * tc;
          if (m < nx && n < ny) {
            const size_t g = static_cast<size_t>(n) * nx + m;
            zl[g] = hi[0][rb].x;
            zl[nn + g] = lo[0][rb].x;
            if (n + 1 < ny) {
              zl[g + nx] = hi[0][rb].y;
              zl[nn + g + nx] = lo[0][rb].y;
            }
          }
        }
      } else if (STAGE <= 2) {
        // block exponents of the next operand: row n, k-block of the tile's 128 m.  The largest
        // magnitude of each column: over the thread's rows, then by halving exchanges over the
        // lanes of equal tc, after which the lane holds one column
        float mx[2 * kCb];
#pragma unroll
        for (int c = 0; c < 2 * kCb; ++c) {
          mx[c] = 0.f;
#pragma unroll
          for (int rb = 0; rb < 4; ++rb)
            mx[c] = fmaxf(mx[c], fabsf((c & 1) ? hi[c >> 1][rb].y : hi[c >> 1][rb].x));
        }
        int col = 2 * tc;
        if (kCb == 2) {
          const bool up = (lane & 16) != 0;
          const float g0 = __shfl_xor_sync(0xffffffffu, up ? mx[0] : mx[2 % (2 * kCb)], 16);
          const float g1 = __shfl_xor_sync(0xffffffffu, up ? mx[1] : mx[3 % (2 * kCb)], 16);
          mx[0] = fmaxf(up ? mx[2 % (2 * kCb)] : mx[0], g0);
          mx[1] = fmaxf(up ? mx[3 % (2 * kCb)] : mx[1], g1);
          col += up ? 8 : 0;
        } else {
#pragma unroll
          for (int c = 0; c < 2; ++c) mx[c] = fmaxf(mx[c], __shfl_xor_sync(0xffffffffu, mx[c], 16));
        }
        {
          const bool up = (lane & 8) != 0;
          const float g = __shfl_xor_sync(0xffffffffu, up ? mx[0] : mx[1], 8);
          mx[0] = fmaxf(up ? mx[1] : mx[0], g);
          col += up ? 1 : 0;
        }
        mx[0] = fmaxf(mx[0], __shfl_xor_sync(0xffffffffu, mx[0], 4));
        if ((lane & 4) == 0 && (kCb == 2 || (lane & 16) == 0)) ctl->colmax[group][col][quarter] = mx[0];
        // the staging tile is free once the previous tile's stores have read it
        if (ew == 0 && lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        if (epi_vote(fail)) break;
        int E_mine = 0;
        if (col_lane) {
          const float4 q = *reinterpret_cast<const float4*>(ctl->colmax[group][lane]);
          E_mine = block_exp(fmaxf(fmaxf(q.x, q.y), fmaxf(q.z, q.w)));
        }
        // slices, transposed into the staging tile, one 32-column block of the tile at a time: row n of
        // 64 m (128 bytes), 16-byte chunks permuted by n % 8 (the tensor stores' 128-byte swizzle;
        // conflict-free here)
        const void* mo = static_cast<const unsigned char*>(S.tmaps) + 128 * (8 + STAGE);
        if (ew == 0 && lane == 0) tmap_acquire(mo);
        const uint32_t so = smem_u32(sO) + (((quarter >> 1) * 32 + 8 * group + (lane & 7)) << 7) +
                            (((((quarter & 1) << 2) + (lane >> 3)) ^ (lane & 7)) << 4);
#pragma unroll
        for (int cb = 0; cb < kCb; ++cb) {
          const int e0 = __shfl_sync(0xffffffffu, E_mine, 8 * cb + 2 * tc);
          const int e1 = __shfl_sync(0xffffffffu, E_mine, 8 * cb + 2 * tc + 1);
          const float2 up = make_float2(pow2f(16 - e0), pow2f(16 - e1));
          uint32_t code[4][NSL];
#pragma unroll
          for (int rb = 0; rb < 4; ++rb) slice_codes2_df<BF16, NSL>(hi[cb][rb], lo[cb][rb], up, code[rb]);
#pragma unroll
          for (int q0 = 0; q0 < NSL; q0 += G::kGroup) {
            if (cb > 0 || q0 > 0) {
              // the previous group's stores have read the staging tile
              if (ew == 0 && lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
              epi_bar();
            }
#pragma unroll
            for (int q = 0; q < G::kGroup; ++q) {
              const uint32_t f[4] = {code[0][q0 + q], code[1][q0 + q], code[2][q0 + q], code[3][q0 + q]};
              stmatrix4_t(so + (q * 2 * 32 << 7), f);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            epi_bar();
            if (ew == 0 && lane == 0) {
#pragma unroll
              for (int q = 0; q < G::kGroup; ++q)
#pragma unroll
                for (int h = 0; h < 2; ++h)
                  tma_store_2d(mo, smem_u32(sO) + ((q * 2 + h) * 32 << 7), m0 + 64 * h, (q0 + q) * v.N + n0 + 32 * cb);
              asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            }
          }
        }
        if (quarter == 0 && col_lane)
          v.eout[static_cast<size_t>(n_mine) * (v.M / KC) + m0 / KC] = static_cast<int8_t>(E_mine);
      } else {
        if (epi_vote(fail)) break;
        CompDotDF c_rz, c_zq;
        const bool mir_out = S.mir_out != 0;
        const bool with_zq = !mir_out && sc->flexible != 0;
        const int nx = S.nx, ny = S.ny;
        const size_t nn = static_cast<size_t>(nx) * ny;
        float* __restrict__ zh = S.z;
        float* __restrict__ zl = S.z_lo;
        const float* lz = S.lowm_x ? S.low_z : nullptr;
#pragma unroll
        for (int cb = 0; cb < kCb; ++cb) {
          // the eight values' nodes: g < 0 outside the grid
          int g[4][2];
#pragma unroll
          for (int rb = 0; rb < 4; ++rb)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const int m = mq + 8 * rb + t4, n = ng + 32 * cb + 2 * tc + e;
              g[rb][e] = (m < nx && n < ny) ? n * nx + m : -1;
            }
          if (lz) {
            // the low-mode part first: the 32-bit stages' result plus zl, one double-float value
            float wh[4][2], wl[4][2];
#pragma unroll
            for (int rb = 0; rb < 4; ++rb)
#pragma unroll
              for (int e = 0; e < 2; ++e) {
                const int gi = max(g[rb][e], 0);
                wh[rb][e] = lz[gi];
                wl[rb][e] = lz[nn + gi];
              }
#pragma unroll
            for (int rb = 0; rb < 4; ++rb) {
              const f2 a = df_add(f2{hi[cb][rb].x, lo[cb][rb].x}, f2{wh[rb][0], wl[rb][0]});
              const f2 b = df_add(f2{hi[cb][rb].y, lo[cb][rb].y}, f2{wh[rb][1], wl[rb][1]});
              hi[cb][rb] = make_float2(a.hi, b.hi);
              lo[cb][rb] = make_float2(a.lo, b.lo);
            }
          }
          if (mir_out) {
            // one mirror class of a folded slot: its result g, unmasked (k_unfold combines the
            // classes, masks and forms the dot products)
#pragma unroll
            for (int rb = 0; rb < 4; ++rb) {
              if (g[rb][0] >= 0) {
                zh[g[rb][0]] = hi[cb][rb].x;
                zl[g[rb][0]] = lo[cb][rb].x;
              }
              if (g[rb][1] >= 0) {
                zh[g[rb][1]] = hi[cb][rb].y;
                zl[g[rb][1]] = lo[cb][rb].y;
              }
            }
            continue;
          }
          float rv[4][2], rl[4][2], qv[4][2], ql[4][2];
          uint8_t mk[4][2];
#pragma unroll
          for (int rb = 0; rb < 4; ++rb)
#pragma unroll
            for (int e = 0; e < 2; ++e) {  // issue the block's loads together
              const int gi = max(g[rb][e], 0);
              rv[rb][e] = S.r[gi];
              rl[rb][e] = S.r_lo[gi];
              // z.q enters only the flexible beta
              qv[rb][e] = with_zq ? S.q[gi] : 0.f;
              ql[rb][e] = with_zq ? S.q_lo[gi] : 0.f;
              mk[rb][e] = g[rb][e] >= 0 ? S.mask[gi] : 0;
            }
#pragma unroll
          for (int rb = 0; rb < 4; ++rb)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              if (g[rb][e] < 0) continue;
              const float a = mk[rb][e] ? (e ? hi[cb][rb].y : hi[cb][rb].x) : 0.f;
              const float b = mk[rb][e] ? (e ? lo[cb][rb].y : lo[cb][rb].x) : 0.f;
              zh[g[rb][e]] = a;
              zl[g[rb][e]] = b;
              c_rz.add(rv[rb][e], rl[rb][e], a, b);
              if (with_zq) c_zq.add(a, b, qv[rb][e], ql[rb][e]);
            }
        }
        if (mir_out) continue;  // a class problem leaves no partial sums
        // tile partials of r.z and z.q: butterflies in the warps, then across them by warp 0; k_prec_finish forms rho and beta from them
        Sum3 rz(c_rz.s, c_rz.c), zq(c_zq.s, c_zq.c);
        reduce_dots<32, DOTS3>(rz);
        if (with_zq) reduce_dots<32, DOTS3>(zq);
        if (lane == 0) {
          ctl->red[0][ew] = rz;
          if (with_zq) ctl->red[1][ew] = zq;
        }
        epi_bar();
        if (ew == 0) {
          rz = ctl->red[0][lane % kEpiWarps];
          reduce_dots<kEpiWarps, DOTS3>(rz);
          if (with_zq) {
            zq = ctl->red[1][lane % kEpiWarps];
            reduce_dots<kEpiWarps, DOTS3>(zq);
          }
          if (lane == 0) {
            S.part[it.tile * 4 + 2] = rz.value<DOTS3>();
            S.part[it.tile * 4 + 3] = with_zq ? zq.value<DOTS3>() : 0.0;
          }
        }
        // ctl->red is rewritten only after the next tile's vote, which this warp joins later
      }
    }
    if (STAGE <= 2 && ew == 0 && lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols)
                 : "memory");
  }
  if (threadIdx.x == 0 && ctl->abort_flag) raise_flag(err);
}

// One row of a transform operand: the warp's 128 columns (lane pairs 64 k + 2 lane) under their common
// exponent, both codes of a slice in one 4-byte store.  `idx`: the lane's first pair in a plane of
// `half` pairs.  With six slices in a mixed mode the first four are stage 0's operand, all six the
// low-mode product's.
template <bool BF16>
__device__ __forceinline__ void slice_row(const float2 (&vh)[2], const float2 (&vl)[2], uint32_t* out32, size_t idx,
                                          size_t half, int nr, int8_t* e, int lane) {
  float amax = 0.f;
#pragma unroll
  for (int k = 0; k < 2; ++k) amax = fmaxf(amax, fmaxf(fabsf(vh[k].x), fabsf(vh[k].y)));
  const int E = block_exp(warp_max(amax));
  const float2 up = make_float2(pow2f(16 - E), pow2f(16 - E));
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    if (nr == kLowNS) {
      uint32_t code[kLowNS];
      slice_codes2_df<BF16, kLowNS>(vh[k], vl[k], up, code);
#pragma unroll
      for (int q = 0; q < kLowNS; ++q) out32[q * half + idx + 32 * k] = code[q];
    } else {
      uint32_t code[4];
      slice_codes2_df<BF16, 4>(vh[k], vl[k], up, code);
#pragma unroll
      for (int q = 0; q < 4; ++q) out32[q * half + idx + 32 * k] = code[q];
    }
  }
  if (lane == 0) *e = static_cast<int8_t>(E);
}

// Residual -> slices of the first stage's A operand (slots with no folded axis).  One item per
// 32 rows and KC columns; one warp per four of the rows, all four loaded before any is sliced.
template <bool BF16>
__global__ void __launch_bounds__(256)
k_tc_prepare(const SlotDesc* __restrict__ slots, const WorkItem* __restrict__ items,
             const int* __restrict__ n_items, int mode) {
  const int total = *n_items;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  pdl_wait();
  for (int w = blockIdx.x; w < total; w += gridDim.x) {
    const WorkItem it = items[w];
    const SlotDesc& S = slots[it.slot];
    SlotScalars* sc = S.sc;
    if (!slot_runs(sc, mode) || S.mir) continue;  // folded slots: k_tc_fold
    const int tx = (S.nx + KC - 1) / KC;
    const int x0 = (it.tile % tx) * KC;
    const int y0 = (it.tile / tx) * kStTileY;
    const int kblocks = S.nxp / KC;
    const size_t plane = static_cast<size_t>(S.nyp) * S.nxp;
    uint16_t* out = static_cast<uint16_t*>(S.tc_r);
    // every row of the warp loaded before any is sliced
    constexpr int kRows = kStTileY / 8;
    static_assert(kRows * 8 == kStTileY && KC == 128, "rows per warp");
    // each lane takes adjacent pairs (x, x+1) and writes both codes of a slice in one 4-byte
    // store (x even, rows of nxp even: aligned)
    constexpr int kPairs = KC / 64;
    float2 v[kRows][kPairs], vl[kRows][kPairs];
#pragma unroll
    for (int j = 0; j < kRows; ++j) {
      const int y = y0 + warp + 8 * j;
#pragma unroll
      for (int k = 0; k < kPairs; ++k) {
        const int x = x0 + 64 * k + 2 * lane;
        const float* row = S.r + static_cast<size_t>(y) * S.nx;
        const float* row_lo = S.r_lo + static_cast<size_t>(y) * S.nx;
        v[j][k].x = (x < S.nx && y < S.ny) ? row[x] : 0.f;
        v[j][k].y = (x + 1 < S.nx && y < S.ny) ? row[x + 1] : 0.f;
        vl[j][k].x = (x < S.nx && y < S.ny) ? row_lo[x] : 0.f;
        vl[j][k].y = (x + 1 < S.nx && y < S.ny) ? row_lo[x + 1] : 0.f;
      }
    }
    uint32_t* out32 = reinterpret_cast<uint32_t*>(out);
#pragma unroll
    for (int j = 0; j < kRows; ++j) {
      const int y = y0 + warp + 8 * j;
      if (y >= S.ny) break;
      slice_row<BF16>(v[j], vl[j], out32, (static_cast<size_t>(y) * S.nxp + x0 + 2 * lane) / 2, plane / 2, S.tc_nr,
                      S.tc_e[0] + static_cast<size_t>(y) * kblocks + x0 / KC, lane);
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Mirror fold (slots with a folded axis).  On a folded axis the basis splits into even and odd
// vectors under i -> n-1-i (plan.cpp), so the four stages of the slot run as two or four
// independent half-size problems, its classes.  k_tc_fold forms each class's residual on its
// ceil(n/2)-node domain, signed sums of r at a node and its mirrors (the even class adds, the
// odd class subtracts; a middle node, its own mirror, counts once in the even class and not in
// the odd one), in double-float, and slices it like k_tc_prepare.  After stage 3 has written
// each class's result g, k_unfold forms z at a node and its mirrors as the sums of the classes
// with the odd ones' signs flipped on the mirrored side, masks it and leaves the r.z and z.q
// partials that stage 3 leaves for an unfolded slot.
// ---------------------------------------------------------------------------------------------

// An item, its slot and its classes' operands.  The first item's are read before the wait for
// the previous kernel (no kernel writes them), the others' ahead of the residual's loads: read where
// the slices are stored, they were four dependent misses in a row.
// The classes of a slot have equal sizes and lie at equal distances in its arena.
struct FoldItem {
  const SlotDesc* S = nullptr;
  int tile = 0;
  char *out = nullptr, *e = nullptr;  // class 0's operand and exponents
  ptrdiff_t step = 0;                 // bytes from one class to the next
  int nxp = 0, nyp = 0, nr = 4;
};
__device__ __forceinline__ FoldItem fold_item(const SlotDesc* __restrict__ slots, const SlotDesc* __restrict__ tcp,
                                              const WorkItem it) {
  FoldItem t;
  t.S = slots + it.slot;
  t.tile = it.tile;
  const SlotDesc &T = tcp[kMirClasses * it.slot], &U = tcp[kMirClasses * it.slot + ((t.S->mir & 1) ? 1 : 2)];
  t.out = static_cast<char*>(T.tc_r);
  t.e = reinterpret_cast<char*>(T.tc_e[0]);
  t.step = static_cast<char*>(U.tc_r) - t.out;
  t.nxp = T.nxp;
  t.nyp = T.nyp;
  t.nr = T.tc_nr;
  return t;
}

// One warp per (class row y, 128 class columns); lane pairs (x, x+1) at x = 64 k + 2 lane.
template <bool BF16>
__global__ void __launch_bounds__(256, 4)
k_tc_fold(const SlotDesc* __restrict__ slots, const SlotDesc* __restrict__ tcp,
          const WorkItem* __restrict__ items, const int* __restrict__ n_items, int mode) {
  const int total = *n_items;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  FoldItem t;
  if (static_cast<int>(blockIdx.x) < total) t = fold_item(slots, tcp, items[blockIdx.x]);
  pdl_wait();
  for (int w = blockIdx.x; w < total; w += gridDim.x) {
    if (w != static_cast<int>(blockIdx.x)) t = fold_item(slots, tcp, items[w]);
    const SlotDesc& S = *t.S;
    if (!slot_runs(S.sc, mode)) continue;
    const bool fx = (S.mir & 1) != 0, fy = (S.mir & 2) != 0;
    const int nxb = (S.mhx + KC - 1) / KC;
    const int y = (t.tile / nxb) * 8 + warp, xb = t.tile % nxb;
    if (y >= S.mhy) continue;
    const int yy = fy ? S.ny - 1 - y : y;  // the mirrored row (y itself on an unfolded axis)
    const bool ymid = yy == y;
    const float* rh = S.r;
    const float* rl = S.r_lo;
    // class values of the lane's four columns: hi and lo planes of pair k's columns (x, x+1)
    float2 ch[4][2], cl[4][2];  // [class][pair]
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      f2 v[4][2];  // [class][column of the pair]
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int x = xb * KC + 64 * k + 2 * lane + e;
        f2 a{0.f, 0.f}, b{0.f, 0.f}, c{0.f, 0.f}, d{0.f, 0.f};
        const int xx = fx ? S.nx - 1 - x : x;
        const bool xmid = xx == x;
        if (x < S.mhx) {
          const size_t gy = static_cast<size_t>(y) * S.nx, gyy = static_cast<size_t>(yy) * S.nx;
          a = f2{rh[gy + x], rl[gy + x]};
          if (!xmid) b = f2{rh[gy + xx], rl[gy + xx]};
          if (!ymid) {
            c = f2{rh[gyy + x], rl[gyy + x]};
            if (!xmid) d = f2{rh[gyy + xx], rl[gyy + xx]};
          }
        }
        // along x: even = a + b, odd = a - b (b = 0 at a middle node or on an unfolded axis)
        const f2 e0 = df_add(a, b), o0 = df_add(a, df_neg(b));
        const f2 e1 = df_add(c, d), o1 = df_add(c, df_neg(d));
        // along y the same with the mirrored row; class c = 2 cls_y + cls_x
        v[0][e] = df_add(e0, e1);
        v[1][e] = df_add(o0, o1);
        v[2][e] = df_add(e0, df_neg(e1));
        v[3][e] = df_add(o0, df_neg(o1));
        if (xmid && fx) {  // the odd x classes vanish at the middle column
          v[1][e] = f2{0.f, 0.f};
          v[3][e] = f2{0.f, 0.f};
        }
        if (ymid && fy) {
          v[2][e] = f2{0.f, 0.f};
          v[3][e] = f2{0.f, 0.f};
        }
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        ch[c][k] = make_float2(v[c][0].hi, v[c][1].hi);
        cl[c][k] = make_float2(v[c][0].lo, v[c][1].lo);
      }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      if ((c & 1) && !fx) continue;
      if ((c & 2) && !fy) continue;
      const size_t plane = static_cast<size_t>(t.nyp) * t.nxp;
      const ptrdiff_t off = t.step * (fx ? c : c >> 1);
      slice_row<BF16>(ch[c], cl[c], reinterpret_cast<uint32_t*>(t.out + off),
                      (static_cast<size_t>(y) * t.nxp + xb * KC + 2 * lane) / 2, plane / 2, t.nr,
                      reinterpret_cast<int8_t*>(t.e + off + static_cast<ptrdiff_t>(y) * (t.nxp / KC) + xb), lane);
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Iteration, stage 2, for slots of up to kSliceNodes: what k_update does (x += alpha p, r -= alpha q,
// partial ||r||^2, the last item's decision), and the new residual's slices, folded by class where an
// axis is folded (what k_tc_prepare and k_tc_fold form from a stored residual).  Bound by the chain
// of dependent loads and reductions: 7 us at 64^2, 10 at 320 x 256, where the two kernels took 8 and 3,
// 9 and 5.  The block's eight warps hold an item's segments (seg_of), leave the new residual in shared
// memory, and then slice one (class row, class) each.
// ---------------------------------------------------------------------------------------------
template <bool BF16, bool FUSE>
__global__ void __launch_bounds__(kVecThreads, 2)
k_update_slice(const SlotDesc* __restrict__ slots, const SlotDesc* __restrict__ tcp,
               const WorkItem* __restrict__ items, const int* __restrict__ n_items) {
  constexpr int kWarps = kVecThreads / 32;
  __shared__ __align__(16) float sh[kWarps][KC], sl[kWarps][KC];  // the new residual by segment
  __shared__ float2 red[kWarps];
  __shared__ float2 s_alpha;  // FUSE: alpha of slot pq_slot, and whether the slot runs
  __shared__ int s_run, s_last;
  int pq_slot = -1;
  f2 alpha = {0.f, 0.f};
  bool run = false;
  const int total = *n_items;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  WorkItem it = {0, 0};
  FoldItem t;
  if (static_cast<int>(blockIdx.x) < total) {
    it = items[blockIdx.x];
    t = fold_item(slots, tcp, it);
  }
  pdl_wait();
  for (int w = blockIdx.x; w < total; w += gridDim.x) {
    if (w != static_cast<int>(blockIdx.x)) {
      it = items[w];
      t = fold_item(slots, tcp, it);
    }
    const SlotDesc& S = *t.S;
    SlotScalars* sc = S.sc;
    if (!FUSE && !sc->active) continue;
    const int pi = (sc->it & 1) ^ 1;
    const Seg g = seg_of(S, t.tile);
    // all loads pass under the sum of the p.q partials
    const float4 ph = g.load(S.p[pi]), pl = g.load(S.p_lo[pi]), qh = g.load(S.q), ql = g.load(S.q_lo);
    float4 rh = g.load(S.r), rl = g.load(S.r_lo), xh = g.load(S.xhi), xl = g.load(S.xlo);
    if (FUSE) {
      if (it.slot != pq_slot) {
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
        run = s_run != 0;
        pq_slot = it.slot;
        __syncthreads();  // s_alpha and s_run are written again for the next slot
      }
      // a breakdown: every block finds the same one, the tile-0 block records it
      if (!run) continue;
    } else {
      alpha = f2{sc->alpha_f[0], sc->alpha_f[1]};
    }
    const f2 nalpha = {-alpha.hi, -alpha.lo};
    df_axpy(rh.x, rl.x, nalpha, qh.x, ql.x);
    df_axpy(rh.y, rl.y, nalpha, qh.y, ql.y);
    df_axpy(rh.z, rl.z, nalpha, qh.z, ql.z);
    df_axpy(rh.w, rl.w, nalpha, qh.w, ql.w);
    auto stage = [&](float* a, const float4 v) {
      if (!g.vec) {
        a[lane] = v.x;
        a[lane + 32] = v.y;
        a[lane + 64] = v.z;
        a[lane + 96] = v.w;
      } else {
        *reinterpret_cast<float4*>(a + 4 * lane) = g.qx ? make_float4(v.w, v.z, v.y, v.x) : v;
      }
    };
    stage(sh[warp], rh);
    stage(sl[warp], rl);
    __syncthreads();
    g.store(S.r, rh);
    g.store(S.r_lo, rl);
    CompDotDF dot;
    dot.add(rh.x, rl.x, rh.x, rl.x);
    dot.add(rh.y, rl.y, rh.y, rl.y);
    dot.add(rh.z, rl.z, rh.z, rl.z);
    dot.add(rh.w, rl.w, rh.w, rl.w);
    df_axpy(xh.x, xl.x, alpha, ph.x, pl.x);
    df_axpy(xh.y, xl.y, alpha, ph.y, pl.y);
    df_axpy(xh.z, xl.z, alpha, ph.z, pl.z);
    df_axpy(xh.w, xl.w, alpha, ph.w, pl.w);
    g.store(S.xhi, xh);
    g.store(S.xlo, xl);
    if (g.y < S.mhy) {
      // the warp's class row again, its class cls_y, cls_x = qy, qx
      const int s0 = warp & ~((1 << g.lseg) - 1);
      const bool fx = (S.mir & 1) != 0, fy = (S.mir & 2) != 0;
      const bool xodd = (S.nx & 1) != 0, ymid = fy && S.ny - 1 - g.y == g.y;
      float2 vh[2], vl[2];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        f2 v[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int c = 64 * k + 2 * lane + e;
          auto at = [&](int s) { return f2{sh[s0 + s][c], sl[s0 + s][c]}; };
          f2 u = at(0);
          if (fx) u = df_add(u, g.qx ? df_neg(at(1)) : at(1));
          if (fy) {
            f2 m = at(fx ? 2 : 1);
            if (fx) m = df_add(m, g.qx ? df_neg(at(3)) : at(3));
            u = df_add(u, g.qy ? df_neg(m) : m);
          }
          // the odd classes vanish at the middle column, row
          const int x = g.xb * KC + c;
          if ((g.qx && xodd && S.nx - 1 - x == x) || (g.qy && ymid)) u = f2{0.f, 0.f};
          v[e] = u;
        }
        vh[k] = make_float2(v[0].hi, v[1].hi);
        vl[k] = make_float2(v[0].lo, v[1].lo);
      }
      const ptrdiff_t off = t.step * g.seg;
      slice_row<BF16>(vh, vl, reinterpret_cast<uint32_t*>(t.out + off),
                      (static_cast<size_t>(g.y) * t.nxp + g.xb * KC + 2 * lane) / 2, static_cast<size_t>(t.nyp) * t.nxp / 2,
                      t.nr, reinterpret_cast<int8_t*>(t.e + off + static_cast<ptrdiff_t>(g.y) * (t.nxp / KC) + g.xb), lane);
    }
    const double rr = block_sum_comp<kVecThreads>(dot.as_comp(), red);
    if (threadIdx.x == 0) S.part[it.tile * 4 + 0] = rr;
    if (last_item_block(&sc->cnt[2], S.n_upd_items, &s_last)) {
      double s = 0.0;
      if (threadIdx.x < 32) s = warp_sum_strided(S.part, S.n_upd_items, 4);
      if (threadIdx.x == 0) {
        decide_update(sc, s);
      }
    }
    __syncthreads();
  }
}

// One thread per class node (tiles of 32 x 8): z at the node and its mirrors, masked, with the
// tile's compensated r.z and z.q partials.
template <bool DOTS3>
__global__ void __launch_bounds__(256)
k_unfold(const SlotDesc* __restrict__ slots, const SlotDesc* __restrict__ tcp,
         const WorkItem* __restrict__ items, const int* __restrict__ n_items, int mode) {
  __shared__ float4 red[8];  // r.z and z.q of each warp
  __shared__ float2 red_d[DOTS3 ? 8 : 1];
  const int total = *n_items;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  pdl_wait();
  for (int w = blockIdx.x; w < total; w += gridDim.x) {
    const WorkItem it = items[w];
    const SlotDesc& S = slots[it.slot];
    if (!slot_runs(S.sc, mode)) continue;
    const bool fx = (S.mir & 1) != 0, fy = (S.mir & 2) != 0;
    const int ntx = (S.mhx + 31) >> 5;
    const int x = (it.tile % ntx) * 32 + lane, y = (it.tile / ntx) * 8 + warp;
    CompDotDF c_rz, c_zq;
    const bool with_zq = S.sc->flexible != 0;  // z.q enters only the flexible beta
    if (x < S.mhx && y < S.mhy) {
      const int xx = fx ? S.nx - 1 - x : x, yy = fy ? S.ny - 1 - y : y;
      // every load first: the classes' g at (y, x), then mask, r (and q) at the mirror nodes
      f2 g[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        g[c] = f2{0.f, 0.f};
        if (((c & 1) && !fx) || ((c & 2) && !fy)) continue;
        const SlotDesc& T = tcp[kMirClasses * it.slot + c];
        const int gi = y * T.nx + x;
        g[c] = f2{T.z[gi], T.z_lo[gi]};
      }
      int gi[4];
      bool live[4];
      uint8_t mk[4];
      float rh[4], rl[4], qh[4], ql[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) {  // t = 2 (mirrored row) + (mirrored column)
        live[t] = !((t & 1) && xx == x) && !((t & 2) && yy == y);
        gi[t] = ((t & 2) ? yy : y) * S.nx + ((t & 1) ? xx : x);
        mk[t] = 0;
        rh[t] = rl[t] = qh[t] = ql[t] = 0.f;
        if (live[t]) {
          mk[t] = S.mask[gi[t]];
          rh[t] = S.r[gi[t]];
          rl[t] = S.r_lo[gi[t]];
          if (with_zq) {
            qh[t] = S.q[gi[t]];
            ql[t] = S.q_lo[gi[t]];
          }
        }
      }
      // even/odd butterflies along x, then y
      const f2 a = df_add(g[0], g[1]), b = df_add(g[0], df_neg(g[1]));
      const f2 c = df_add(g[2], g[3]), d = df_add(g[2], df_neg(g[3]));
      const f2 v[4] = {df_add(a, c), df_add(b, d), df_add(a, df_neg(c)), df_add(b, df_neg(d))};
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        if (!live[t]) continue;
        const float zh = mk[t] ? v[t].hi : 0.f, zl = mk[t] ? v[t].lo : 0.f;
        S.z[gi[t]] = zh;
        S.z_lo[gi[t]] = zl;
        c_rz.add(rh[t], rl[t], zh, zl);
        if (with_zq) c_zq.add(zh, zl, qh[t], ql[t]);
      }
    }
    // the tile's sums: butterflies inside the warps and, by warp 0, across the eight
    Sum3 rz(c_rz.s, c_rz.c), zq(c_zq.s, c_zq.c);
    reduce_dots<32, DOTS3>(rz);
    if (with_zq) reduce_dots<32, DOTS3>(zq);
    if (lane == 0) {
      red[warp] = make_float4(rz.s, rz.c, zq.s, zq.c);
      if (DOTS3) red_d[warp] = make_float2(rz.d, zq.d);
    }
    __syncthreads();
    if (warp == 0) {
      const float4 v = red[lane & 7];
      const float2 d = DOTS3 ? red_d[lane & 7] : make_float2(0.f, 0.f);
      rz = Sum3(v.x, v.y, d.x);
      zq = Sum3(v.z, v.w, d.y);
      reduce_dots<8, DOTS3>(rz);
      if (with_zq) reduce_dots<8, DOTS3>(zq);
      if (lane == 0) {
        S.part[it.tile * 4 + 2] = rz.value<DOTS3>();
        S.part[it.tile * 4 + 3] = with_zq ? zq.value<DOTS3>() : 0.0;
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------------------------
// Low-mode correction (mixed modes).  The weights 1/(lam_y + lam_x)^2 of the smoothest modes are up
// to (64/lam_min)^2 times those of the roughest, so rounding noise of the 32-bit stages, relative
// to |r|, is amplified in exactly these modes and costs CG iterations.  The modes kx < 32,
// ky < 32 (of each transform problem) are therefore left out of stage 1's weights and computed
// here to about 48 bits:
//   forward (kLowFwd):   H[y][kx] = sum_x r[y][x] Qx[x][kx], six slices each side, and each
//                        128-row tile's share of G = Qy_low^T H (double-float dot products)
//   middle (k_low_mid):  G = the shares in tile order, G' = w o G,
//                        J[ky][x] = sum_kx G'[ky][kx] Qx[x][kx] (double-float), J^T in six slices
//   inverse (kLowInv):   zl[y][x] = sum_ky Qy[y][ky] J[ky][x], six slices each side
// and stage 3 adds zl to its result.  With six 8-bit slices per operand the products of orders
// 0..5 (21 of them) are kept, each order in its own TMEM accumulator; per k, the products of one
// order add up to at most 2^17 in magnitude, so over a 128-wide block every partial sum is an
// exact integer of at most 2^24.  Orders 0..2 are merged into the double-float result with TwoSum,
// orders 3..5 (below 2^-24 of it) in plain FP32.
//
// Both products are launches of the stage kernel (forms kLowFwd and kLowInv): 128 x 32 tiles, 32-deep
// steps copied ahead, MMAs of one accumulation block running while the sixteen warps merge the one
// before.  (As kernels of their own, each tile copying, multiplying and merging in turn and the
// inverse one item per 128 rows of x, the two took 45 + 47 us per application on a batch of 48 grids.)
// ---------------------------------------------------------------------------------------------
static_assert(kLowM == 32 && kLowK3 == kLowM, "the inverse product's k is one step");

// The slices of one double-float value on a single lane (the packed routine on lane x).
template <bool BF16>
__device__ __forceinline__ void slice_codes_df(float vh, float vl, float up, uint16_t (&code)[kLowNS]) {
  uint32_t c2[kLowNS];
  slice_codes2_df<BF16, kLowNS>(make_float2(vh, 0.f), make_float2(vl, 0.f), make_float2(up, up), c2);
#pragma unroll
  for (int k = 0; k < kLowNS; ++k) code[k] = static_cast<uint16_t>(c2[k] & 0xffffu);
}

// Middle of the low-mode correction, one block per (problem, 32 rows of x): G = the forward tiles'
// shares summed in tile order, G' = w o G, and the block's rows of J^T,
// J^T[x][ky] = sum_kx G'[ky][kx] Qx[x][kx], by compensated dot products of double-float operands
// (Ogita-Rump-Oishi), each row then cut into six slices with its block exponent (the inverse
// product's A operand).  Lane ky reads its row of G' from shared memory; the block's rows of Qx_low
// are staged there transposed, so that a warp takes the values of two adjacent rows at one kx by one
// 8-byte broadcast load; each warp runs four rows as two packed chains.  Bound by FP32 issue, so the
// blocks are small (128 rows a block left some SMs two blocks and others one).
constexpr int kMidRows = 32;
constexpr int kQsStride = kMidRows + 2;  // [kx][row] stride: even (8-byte pairs), 2-way staging conflicts
template <bool BF16>
__global__ void __launch_bounds__(256)
k_low_mid(const SlotDesc* __restrict__ slots, const WorkItem* __restrict__ items,
          const int* __restrict__ n_items, int mode) {
  __shared__ float gh[kLowM][kLowM + 1], gl[kLowM][kLowM + 1];
  __shared__ __align__(16) float qs[2][kLowM][kQsStride];  // Qx_low rows of the block: hi, lo
  const int total = *n_items;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  pdl_wait();
  for (int w = blockIdx.x; w < total; w += gridDim.x) {
    const WorkItem it = items[w];
    const SlotDesc& S = slots[it.slot];
    if (!slot_runs(S.sc, mode) || S.lowm_x == 0) continue;
    const float* qx_h = S.low_qxd;
    const float* qx_l = S.low_qxd + static_cast<size_t>(S.nxp) * kLowM;
    const int xb = it.tile * kMidRows;
    for (int e = t; e < kMidRows * kLowM; e += 256) {
      const int r = e / kLowM, kx = e - r * kLowM;
      const size_t a = static_cast<size_t>(xb + r) * kLowM + kx;
      qs[0][kx][r] = __ldg(qx_h + a);
      qs[1][kx][r] = __ldg(qx_l + a);
    }
    for (int e = t; e < kLowM * kLowM; e += 256) {
      f2 g{0.f, 0.f};
      for (int tt = 0; tt < S.n_l1_tiles; ++tt) {
        const float* gp = S.low_gp + static_cast<size_t>(tt) * 2 * kLowM * kLowM;
        g = df_add(g, f2{gp[e], gp[kLowM * kLowM + e]});
      }
      const int ky = e / kLowM, kx = e - ky * kLowM;
      const float sw = S.lamy[min(ky, S.nyp - 1)] + S.lamx[min(kx, S.nxp - 1)];
      const bool ok = ky < S.lowm_y && kx < S.lowm_x && sw > 0.f;
      g = ok ? df_mul(g, spectral_weight_of(S.wnorm, sw)) : f2{0.f, 0.f};
      gh[ky][kx] = g.hi;
      gl[ky][kx] = g.lo;
    }
    __syncthreads();
    uint16_t* jt = static_cast<uint16_t*>(S.low_jt);
    const size_t plane = static_cast<size_t>(S.nxp) * kLowK3;
    constexpr int kRows = kMidRows / 8;  // per warp
    const int rb = warp * kRows;
    CompDotDF2 acc[kRows / 2];
#pragma unroll 4
    for (int kx = 0; kx < kLowM; ++kx) {
      const float ah = gh[lane][kx], al = gl[lane][kx];
#pragma unroll
      for (int q = 0; q < kRows / 2; ++q) {
        const float2 bh = *reinterpret_cast<const float2*>(&qs[0][kx][rb + 2 * q]);
        const float2 bl = *reinterpret_cast<const float2*>(&qs[1][kx][rb + 2 * q]);
        acc[q].add(make_float2(ah, ah), make_float2(al, al), bh, bl);
      }
    }
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      const int x = xb + rb + r;
      const CompDotDF2& d = acc[r / 2];
      const f2 j = (r & 1) ? df_norm(d.s.y, d.c.y) : df_norm(d.s.x, d.c.x);
      const int E = block_exp(warp_max(fabsf(j.hi)));
      uint16_t code[kLowNS];
      slice_codes_df<BF16>(j.hi, j.lo, pow2f(16 - E), code);
#pragma unroll
      for (int p = 0; p < kLowNS; ++p) jt[p * plane + static_cast<size_t>(x) * kLowK3 + lane] = code[p];
      if (lane == 0) S.low_jt_e[x] = static_cast<int8_t>(E);
    }
    __syncthreads();  // gh, gl and qs are rewritten by the next item
  }
}

template <bool BF16, int STAGE, int NSL, bool DOTS3 = false>
cudaError_t set_attr() {
  return cudaFuncSetAttribute(k_prec_tc<BF16, STAGE, NSL, DOTS3>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              TcGeom<STAGE, NSL>::kSmem);
}

template <bool BF16, int STAGE, int NSL, bool DOTS3 = false>
void launch_one(const LaunchCfg& c, int mode, int* err) {
  const long long wc = c.wait_cycles > 0 ? c.wait_cycles : kWaitCycles;
  launch_cfg(c, k_prec_tc<BF16, STAGE, NSL, DOTS3>, c.grid, kThreads, TcGeom<STAGE, NSL>::kSmem, c.slots, c.items,
             c.n_items, mode, err, wc);
}

template <bool BF16, int NSL>
void launch_all(const LaunchCfg& c, int stage, int mode, int* err) {
  switch (stage) {
    case 0: launch_one<BF16, 0, NSL>(c, mode, err); break;
    case 1: launch_one<BF16, 1, NSL>(c, mode, err); break;
    case 2: launch_one<BF16, 2, NSL>(c, mode, err); break;
    default:
      if (NSL == 6 && c.dots3) launch_one<BF16, 3, NSL, NSL == 6>(c, mode, err);
      else launch_one<BF16, 3, NSL>(c, mode, err);
  }
}

}  // namespace

bool tc_supported() {
  int dev = 0;
  cudaDeviceProp p;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaGetDeviceProperties(&p, dev) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  if (p.major != 10 || p.sharedMemPerBlockOptin < static_cast<size_t>(TcGeom<0, 4>::kSmem)) return false;
  // one CTA of kThreads threads at kMaxRegs registers each must fit an SM
  int blocks = 0;
  if (set_attr<true, 0, 4>() != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, k_prec_tc<true, 0, 4>, kThreads, TcGeom<0, 4>::kSmem) !=
          cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return blocks >= 1;
}

int tc_step_k(int ns) { return ns == 4 ? TcGeom<0, 4>::BK : TcGeom<0, 6>::BK; }
int tc_tile_cols(int ns) { return ns == 4 ? TcGeom<0, 4>::BN : TcGeom<0, 6>::BN; }

int tc_block() { return KC; }

cudaError_t tc_init() {
  cudaError_t e = cudaSuccess;
  const cudaError_t r[22] = {set_attr<false, 0, 4>(), set_attr<false, 1, 4>(), set_attr<false, 2, 4>(),
                             set_attr<false, 3, 4>(), set_attr<true, 0, 4>(),  set_attr<true, 1, 4>(),
                             set_attr<true, 2, 4>(),  set_attr<true, 3, 4>(),  set_attr<true, 0, 6>(),
                             set_attr<true, 1, 6>(),  set_attr<true, 2, 6>(),  set_attr<true, 3, 6>(),
                             set_attr<false, 0, 6>(), set_attr<false, 1, 6>(), set_attr<false, 2, 6>(),
                             set_attr<false, 3, 6>(),
                             set_attr<false, kLowFwd, 6>(), set_attr<false, kLowInv, 6>(),
                             set_attr<true, kLowFwd, 6>(), set_attr<true, kLowInv, 6>(),
                             set_attr<false, 3, 6, true>(), set_attr<true, 3, 6, true>()};
  for (cudaError_t x : r)
    if (x != cudaSuccess) e = x;
  return e;
}

void launch_low_tc(const LaunchCfg& c, int kind, int mode, int split_kind, int* err) {
  if (kind == 0) split_kind == 0 ? launch_one<false, kLowFwd, 6>(c, mode, err) : launch_one<true, kLowFwd, 6>(c, mode, err);
  else split_kind == 0 ? launch_one<false, kLowInv, 6>(c, mode, err) : launch_one<true, kLowInv, 6>(c, mode, err);
}

void launch_low_mid(const LaunchCfg& c, int mode, int split_kind) {
  if (split_kind == 0) launch_cfg(c, k_low_mid<false>, c.grid, 256, 0, c.slots, c.items, c.n_items, mode);
  else launch_cfg(c, k_low_mid<true>, c.grid, 256, 0, c.slots, c.items, c.n_items, mode);
}

void launch_tc_fold(const LaunchCfg& c, int mode, int split_kind) {
  if (split_kind == 0) launch_cfg(c, k_tc_fold<false>, c.grid, 256, 0, c.slots, c.tcp, c.items, c.n_items, mode);
  else launch_cfg(c, k_tc_fold<true>, c.grid, 256, 0, c.slots, c.tcp, c.items, c.n_items, mode);
}

template <bool BF16>
static void launch_update_slice_t(const LaunchCfg& c, bool fuse_pq) {
  if (fuse_pq) launch_cfg(c, k_update_slice<BF16, true>, c.grid, kVecThreads, 0, c.slots, c.tcp, c.items, c.n_items);
  else launch_cfg(c, k_update_slice<BF16, false>, c.grid, kVecThreads, 0, c.slots, c.tcp, c.items, c.n_items);
}
void launch_update_slice(const LaunchCfg& c, int split_kind, bool fuse_pq) {
  if (split_kind == 0) launch_update_slice_t<false>(c, fuse_pq);
  else launch_update_slice_t<true>(c, fuse_pq);
}

void launch_unfold(const LaunchCfg& c, int mode) {
  if (c.dots3) launch_cfg(c, k_unfold<true>, c.grid, 256, 0, c.slots, c.tcp, c.items, c.n_items, mode);
  else launch_cfg(c, k_unfold<false>, c.grid, 256, 0, c.slots, c.tcp, c.items, c.n_items, mode);
}

void launch_prec_tc(const LaunchCfg& c, int stage, int mode, int split_kind, int ns, int* err) {
  if (ns == 6) split_kind == 0 ? launch_all<false, 6>(c, stage, mode, err) : launch_all<true, 6>(c, stage, mode, err);
  else split_kind == 0 ? launch_all<false, 4>(c, stage, mode, err) : launch_all<true, 4>(c, stage, mode, err);
}

void launch_prec_tc_prepare(const LaunchCfg& c, int mode, int split_kind) {
  if (split_kind == 0) launch_cfg(c, k_tc_prepare<false>, c.grid, 256, 0, c.slots, c.items, c.n_items, mode);
  else launch_cfg(c, k_tc_prepare<true>, c.grid, 256, 0, c.slots, c.items, c.n_items, mode);
}

}  // namespace bx
