// Three-dimensional extension (Sec. 3 Example 2: the equations of Sec. 2 on an nz x ny x nx box).
//
// The operator is A = R (L_z (+) L_y (+) L_x)^2 R^T, L_a the 1-D second difference of axis a under
// its boundary rule; at an interior node with equal spacings it is the 25-point squared 7-point
// Laplacian.  It is applied as Algorithm 1 does in two dimensions, the Laplacian twice with the
// ghost rule of each axis (both passes need only the ghosts at distance one, and the boundary
// rules make the once-padded Laplacian at a ghost node the reflected, wrapped or zero one).  The
// CG vectors are double-float pairs (hi, lo) of FP32 planes as in the two-dimensional path; each
// Laplacian pass adds the seven products of the hi plane by an error-free TwoProd/TwoSum chain and
// the lo plane's in plain FP32.  The right-hand side and the residual replacements are FP64.
//
// The preconditioner is the fast Poisson solve on the box, (L^2)^+ by separable transforms along
// the three axes (Example 2: Fourier transforms on every axis; the cosine and sine transforms of
// the other rules likewise): six dense transform products with double-float operands accumulated
// by compensated dot products, each contracting the contiguous axis and writing its result with
// that axis moved to the front, so that three products rotate the box through all three axes;
// the eigenvalue weights come between the forward and the inverse three.
//
// The iteration is preconditioned CG from x = 0 with the Fletcher-Reeves beta.  Its scalars live on
// the device (the two-dimensional path's SlotScalars and its decisions: stop, residual
// replacement, breakdown) and its kernels follow one another as dependent launches, in blocks of
// kBlockIters iterations with the replacement work at the block's end (an iteration that calls for a
// replacement is the block's last: those behind it pass by); the host stays one block
// ahead, reading the scalars that the block before left, so the device never waits for it.  (Read
// after every reduction, three times an iteration, the scalars cost a 72 x 60 x 50 solve 80 of
// its 330 us an iteration.)  Kernels whose flag is down return at once.  Every reduction sums
// per-block partials in a fixed order, so results are reproducible bit for bit.
#include <cmath>
#include <algorithm>
#include <string>
#include <type_traits>
#include <vector>

#include "common.cuh"
#include "kernels.h"

namespace bx {
namespace {

struct Grid3 {
  int nx, ny, nz;
  int bcx, bcy, bcz;
  float cx, cy, cz;     // 1/h^2 of each axis over the largest of the three (<= 1)
  double dcx, dcy, dcz;
};

constexpr int kT = 256;  // threads of the grid kernels (32 x 8)

__device__ __forceinline__ size_t node3(const Grid3& G, int x, int y, int z) {
  return (static_cast<size_t>(z) * G.ny + y) * G.nx + x;
}

// Block sum of a double per thread in a fixed order; the result is valid in thread 0.
__device__ __forceinline__ double block_sum_d(double v, double* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int k = 0; k < kT / 32; ++k) s += sh[k];
  return s;
}

// Every kernel of the iteration first waits for the one before it (pdl_wait), then returns if the
// flag that its pass runs under is down (no flag: always on).
__device__ __forceinline__ bool gate_shut(const int* gate) {
  pdl_wait();
  return gate != nullptr && *static_cast<const volatile int*>(gate) == 0;
}

__device__ __forceinline__ int block_linear() {
  return (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
}

// The seven taps of the Laplacian at (x, y, z): node indices and ghost signs (0 = the Dirichlet
// boundary node, whose value is zero).
struct Taps7 {
  size_t g[7];
  float s[7];
  float w[7];
};
__device__ __forceinline__ Taps7 taps7(const Grid3& G, int x, int y, int z) {
  Taps7 t;
  float sg;
  int i;
  t.g[0] = node3(G, x, y, z);
  t.s[0] = 1.f;
  t.w[0] = 2.f * (G.cx + G.cy + G.cz);
  i = ghost(x - 1, G.nx, G.bcx, sg); t.g[1] = node3(G, i, y, z); t.s[1] = sg; t.w[1] = -G.cx;
  i = ghost(x + 1, G.nx, G.bcx, sg); t.g[2] = node3(G, i, y, z); t.s[2] = sg; t.w[2] = -G.cx;
  i = ghost(y - 1, G.ny, G.bcy, sg); t.g[3] = node3(G, x, i, z); t.s[3] = sg; t.w[3] = -G.cy;
  i = ghost(y + 1, G.ny, G.bcy, sg); t.g[4] = node3(G, x, i, z); t.s[4] = sg; t.w[4] = -G.cy;
  i = ghost(z - 1, G.nz, G.bcz, sg); t.g[5] = node3(G, x, y, i); t.s[5] = sg; t.w[5] = -G.cz;
  i = ghost(z + 1, G.nz, G.bcz, sg); t.g[6] = node3(G, x, y, i); t.s[6] = sg; t.w[6] = -G.cz;
  return t;
}

// Double-float Laplacian pass, marching along z.  A block of 32 x 8 threads owns 32 x kBy nodes of
// (x, y) (two rows per thread, ty and ty + 8) and a chunk of zc planes (16, or fewer on boxes too small
// to fill the device with such chunks).  Each thread keeps its
// own two columns in registers (planes z - 1, z, z + 1 and the two in flight); the x and y
// neighbours come from a shared-memory tile of the plane with its one-node halo, written once per
// plane and double-buffered, so one barrier per plane suffices.  Global loads run two planes ahead
// of their use.  Every cell's ghost map in x and y is taken once per thread, the z map once per
// plane; ghost signs are folded into the loaded values.  FINAL = false: out = L in at every node.
// FINAL = true: out = M L in (zero at known nodes), and the block's partial p.out (compensated).
// The terms are added in the order centre, x-1, x+1, y-1, y+1, z-1, z+1, as the single-node form
// would.
constexpr int kBy = 16;                       // rows per block
constexpr int kTw = 34, kTh = kBy + 2;        // tile with halo
constexpr int kHalo = 2 * kTw + 2 * kBy;      // halo cells of a tile
static_assert(kHalo <= kT && kBy == 2 * (kT / 32), "one halo cell per thread, two rows per thread");

// One cell that a thread loads on every plane: its offset within a plane and the product of its
// x and y ghost signs; ok = false for cells that are no node's neighbour (nothing is loaded).
struct Cell3 {
  size_t off = 0;
  float sxy = 0.f;
  bool ok = false;
};
__device__ __forceinline__ Cell3 cell3(const Grid3& G, int gx, int gy) {
  Cell3 c;
  if (gx > G.nx || gy > G.ny) return c;  // farther cells neighbour no node of the grid
  float sx, sy;
  const int mx = ghost(gx, G.nx, G.bcx, sx), my = ghost(gy, G.ny, G.bcy, sy);
  c.sxy = sx * sy;
  c.ok = c.sxy != 0.f;
  c.off = static_cast<size_t>(my) * G.nx + mx;
  return c;
}

// Tile coordinates of halo cell k: the row above, the row below, the left and the right column.
__device__ __forceinline__ int halo_pos(int k) {
  if (k < kTw) return k;
  if (k < 2 * kTw) return (kTh - 1) * kTw + (k - kTw);
  if (k < 2 * kTw + kBy) return (1 + k - 2 * kTw) * kTw;
  return (1 + k - 2 * kTw - kBy) * kTw + kTw - 1;
}

// A thread's values of one plane: its two own cells and its halo cell (hi, lo).
struct Plane3 {
  float h[3] = {0.f, 0.f, 0.f}, l[3] = {0.f, 0.f, 0.f};
};
__device__ __forceinline__ Plane3 k3_fetch(const Grid3& G, const float* ih, const float* il,
                                           const Cell3 (&cl)[3], int zz) {
  Plane3 p;
  float sz;
  const int mz = ghost(zz, G.nz, G.bcz, sz);
  if (sz == 0.f) return p;
  const size_t base = static_cast<size_t>(mz) * G.ny * G.nx;
#pragma unroll
  for (int k = 0; k < 3; ++k)
    if (cl[k].ok) {
      const float s = cl[k].sxy * sz;
      p.h[k] = s * ih[base + cl[k].off];
      p.l[k] = s * il[base + cl[k].off];
    }
  return p;
}

__device__ __forceinline__ void k3_put(const Plane3& p, float* th, float* tl, int ca, int hp) {
  th[ca] = p.h[0];
  tl[ca] = p.l[0];
  th[ca + 8 * kTw] = p.h[1];
  tl[ca + 8 * kTw] = p.l[1];
  if (hp >= 0) {
    th[hp] = p.h[2];
    tl[hp] = p.l[2];
  }
}

// The seven-term double-float Laplacian of one node: x and y neighbours from the tile at c, the
// centre and the z neighbours (below, up) from the thread's registers.
__device__ __forceinline__ f2 k3_node(const Grid3& G, const float* th, const float* tl, int c, float ch,
                                      float cl, float bh, float bl, float uh, float ul) {
  const float w0 = 2.f * (G.cx + G.cy + G.cz);
  const float hv[7] = {ch, th[c - 1], th[c + 1], th[c - kTw], th[c + kTw], bh, uh};
  const float lv[7] = {cl, tl[c - 1], tl[c + 1], tl[c - kTw], tl[c + kTw], bl, ul};
  const float w[7] = {w0, -G.cx, -G.cx, -G.cy, -G.cy, -G.cz, -G.cz};
  CompSum a;
  float lo = 0.f;
#pragma unroll
  for (int k = 0; k < 7; ++k) {
    a.add_prod(w[k], hv[k]);
    lo = __fmaf_rn(w[k], lv[k], lo);
  }
  return df_norm(a.s, __fadd_rn(a.c, lo));
}

template <bool FINAL>
__global__ void __launch_bounds__(kT)
k3_lap(Grid3 G, int zc, const int* __restrict__ gate, const float* ih, const float* il,
       float* __restrict__ oh, float* __restrict__ ol, const uint8_t* __restrict__ mask, const float* ph,
       const float* pl, double* __restrict__ part) {
  if (gate_shut(gate)) return;
  __shared__ double sh[kT / 32];
  __shared__ float tile[2][2][kTh * kTw];  // [buffer][hi, lo]
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int x0 = blockIdx.x * 32, y0 = blockIdx.y * kBy, z0 = blockIdx.z * zc;
  const int z1 = min(z0 + zc, G.nz);
  const int x = x0 + tx;
  const int yr[2] = {y0 + ty, y0 + ty + 8};
  const bool in[2] = {x < G.nx && yr[0] < G.ny, x < G.nx && yr[1] < G.ny};
  const int ca = (ty + 1) * kTw + tx + 1;  // tile position of the first own node
  Cell3 cl[3];
  cl[0] = cell3(G, x, yr[0]);
  cl[1] = cell3(G, x, yr[1]);
  int hp = -1;
  if (threadIdx.x < kHalo) {
    hp = halo_pos(threadIdx.x);
    const int ly = hp / kTw, lx = hp - ly * kTw;
    cl[2] = cell3(G, x0 - 1 + lx, y0 - 1 + ly);
  }
  const size_t plane = static_cast<size_t>(G.ny) * G.nx;
  // p and the mask at the own nodes, loaded one plane ahead (FINAL only)
  uint8_t mk[2] = {0, 0};
  float pph[2] = {0.f, 0.f}, ppl[2] = {0.f, 0.f};
  auto load_p = [&](int z, uint8_t (&m)[2], float (&h)[2], float (&l)[2]) {
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (in[i]) {
        const size_t g = z * plane + cl[i].off;
        m[i] = mask[g];
        h[i] = ph[g];
        l[i] = pl[g];
      }
  };
  Plane3 below = k3_fetch(G, ih, il, cl, z0 - 1);
  Plane3 cur = k3_fetch(G, ih, il, cl, z0);
  Plane3 up = k3_fetch(G, ih, il, cl, z0 + 1);
  Plane3 n1;
  if (z0 + 1 < z1) n1 = k3_fetch(G, ih, il, cl, z0 + 2);
  if (FINAL) load_p(z0, mk, pph, ppl);
  k3_put(cur, tile[0][0], tile[0][1], ca, hp);
  __syncthreads();
  CompDotDF dot;
  for (int z = z0; z < z1; ++z) {
    const int b = (z - z0) & 1;
    Plane3 n2;  // plane z + 3, needed from the step of plane z + 2 on
    if (z + 2 < z1) n2 = k3_fetch(G, ih, il, cl, z + 3);
    uint8_t nmk[2] = {0, 0};
    float nph[2] = {0.f, 0.f}, npl[2] = {0.f, 0.f};
    if (FINAL && z + 1 < z1) load_p(z + 1, nmk, nph, npl);
    const float* th = tile[b][0];
    const float* tl = tile[b][1];
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (in[i]) {
        const size_t g = z * plane + cl[i].off;
        f2 v{0.f, 0.f};
        if (!FINAL || mk[i])
          v = k3_node(G, th, tl, ca + i * 8 * kTw, cur.h[i], cur.l[i], below.h[i], below.l[i], up.h[i], up.l[i]);
        oh[g] = v.hi;
        ol[g] = v.lo;
        if (FINAL) dot.add(pph[i], ppl[i], v.hi, v.lo);
      }
    if (z + 1 < z1) k3_put(up, tile[b ^ 1][0], tile[b ^ 1][1], ca, hp);
    __syncthreads();
    below = cur;
    cur = up;
    up = n1;
    n1 = n2;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      mk[i] = nmk[i];
      pph[i] = nph[i];
      ppl[i] = npl[i];
    }
  }
  if (FINAL) {
    const double s = block_sum_d(dot.value(), sh);
    if (threadIdx.x == 0) part[block_linear()] = s;
  }
}

// FP64 Laplacian pass.  MODE 0: out = L in.  MODE 1: out = -M L in (the right-hand side) and the
// partial ||out||^2.  MODE 2: out = b - M L in (the true residual), its partial ||out||^2, and the
// double-float copy (rh, rl) of out when rh is given.
template <int MODE>
__global__ void __launch_bounds__(kT)
k3_lap64(Grid3 G, const int* __restrict__ gate, const double* in, double* __restrict__ out,
         const uint8_t* __restrict__ mask, const double* __restrict__ b, double* __restrict__ part,
         float* __restrict__ rh, float* __restrict__ rl) {
  if (gate_shut(gate)) return;
  __shared__ double sh[kT / 32];
  const int x = blockIdx.x * 32 + (threadIdx.x & 31);
  const int y = blockIdx.y * 8 + (threadIdx.x >> 5);
  const int z = blockIdx.z;
  double sq = 0.0;
  if (x < G.nx && y < G.ny) {
    const Taps7 t = taps7(G, x, y, z);
    const size_t g = t.g[0];
    const double w[7] = {2.0 * (G.dcx + G.dcy + G.dcz), -G.dcx, -G.dcx, -G.dcy, -G.dcy, -G.dcz, -G.dcz};
    double v = 0.0;
#pragma unroll
    for (int k = 0; k < 7; ++k) v += w[k] * static_cast<double>(t.s[k]) * in[t.g[k]];
    if (MODE == 0) {
      out[g] = v;
    } else {
      const bool unk = mask[g] != 0;
      const double o = MODE == 1 ? (unk ? -v : 0.0) : (unk ? b[g] - v : 0.0);
      out[g] = o;
      sq = o * o;
      if (MODE == 2 && rh != nullptr) {
        const f2 d = df_of(o);
        rh[g] = d.hi;
        rl[g] = d.lo;
      }
    }
  }
  if (MODE != 0) {
    const double s = block_sum_d(sq, sh);
    if (threadIdx.x == 0) part[block_linear()] = s;
  }
}

// mask (1 = unknown), the known field as FP64 with zeros elsewhere, and counts: [0] unknown,
// [1] known, [2] NaN phi, [3] non-finite f at a known node.
__global__ void __launch_bounds__(kT)
k3_setup(size_t n, const float* __restrict__ phi, const float* __restrict__ f, int dir,
         uint8_t* __restrict__ mask, double* __restrict__ fk, unsigned long long* __restrict__ counts) {
  unsigned long long c[4] = {0, 0, 0, 0};
  for (size_t i = blockIdx.x * static_cast<size_t>(kT) + threadIdx.x; i < n; i += static_cast<size_t>(gridDim.x) * kT) {
    const float p = phi[i];
    const bool known = dir == 0 ? (p < 0.f) : (p > 0.f);
    if (p != p) ++c[2];
    const float fv = f[i];
    mask[i] = known ? 0 : 1;
    fk[i] = known ? static_cast<double>(fv) : 0.0;
    if (known) {
      ++c[1];
      if (!isfinite(fv)) ++c[3];
    } else {
      ++c[0];
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    unsigned long long v = c[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0 && v) atomicAdd(&counts[k], v);
  }
}

// r = 2^-e b as a double-float pair, x = 0
__global__ void __launch_bounds__(kT)
k3_init(size_t n, const double* __restrict__ b, double s, float* __restrict__ rh, float* __restrict__ rl,
        float* __restrict__ xh, float* __restrict__ xl) {
  for (size_t i = blockIdx.x * static_cast<size_t>(kT) + threadIdx.x; i < n; i += static_cast<size_t>(gridDim.x) * kT) {
    const f2 d = df_of(b[i] * s);
    rh[i] = d.hi;
    rl[i] = d.lo;
    xh[i] = 0.f;
    xl[i] = 0.f;
  }
}

// x += alpha p, r -= alpha q (double-float), partial ||r||^2 per block
__global__ void __launch_bounds__(kT, 4)
k3_update(size_t n, const SlotScalars* sc, const float* ph, const float* pl, const float* qh,
          const float* ql, float* xh, float* xl, float* rh, float* rl, double* __restrict__ part) {
  __shared__ float sh[3][kT / 32];
  if (gate_shut(&sc->active)) return;
  const f2 alpha{sc->alpha_f[0], sc->alpha_f[1]}, na{-alpha.hi, -alpha.lo};
  CompDotDF rr;
  const size_t n4 = n / 4;
  for (size_t i = blockIdx.x * static_cast<size_t>(kT) + threadIdx.x; i < n4; i += static_cast<size_t>(gridDim.x) * kT) {
    const float4 p = reinterpret_cast<const float4*>(ph)[i], po = reinterpret_cast<const float4*>(pl)[i];
    const float4 q = reinterpret_cast<const float4*>(qh)[i], qo = reinterpret_cast<const float4*>(ql)[i];
    float4 x = reinterpret_cast<float4*>(xh)[i], xo = reinterpret_cast<float4*>(xl)[i];
    float4 r = reinterpret_cast<float4*>(rh)[i], ro = reinterpret_cast<float4*>(rl)[i];
    df_axpy(x.x, xo.x, alpha, p.x, po.x);
    df_axpy(x.y, xo.y, alpha, p.y, po.y);
    df_axpy(x.z, xo.z, alpha, p.z, po.z);
    df_axpy(x.w, xo.w, alpha, p.w, po.w);
    df_axpy(r.x, ro.x, na, q.x, qo.x);
    df_axpy(r.y, ro.y, na, q.y, qo.y);
    df_axpy(r.z, ro.z, na, q.z, qo.z);
    df_axpy(r.w, ro.w, na, q.w, qo.w);
    reinterpret_cast<float4*>(xh)[i] = x;
    reinterpret_cast<float4*>(xl)[i] = xo;
    reinterpret_cast<float4*>(rh)[i] = r;
    reinterpret_cast<float4*>(rl)[i] = ro;
    rr.add(r.x, ro.x, r.x, ro.x);
    rr.add(r.y, ro.y, r.y, ro.y);
    rr.add(r.z, ro.z, r.z, ro.z);
    rr.add(r.w, ro.w, r.w, ro.w);
  }
  if (blockIdx.x == 0)
    for (size_t i = 4 * n4 + threadIdx.x; i < n; i += kT) {
      df_axpy(xh[i], xl[i], alpha, ph[i], pl[i]);
      df_axpy(rh[i], rl[i], na, qh[i], ql[i]);
      rr.add(rh[i], rl[i], rh[i], rl[i]);
    }
  Sum3 v(rr.s, rr.c);
  v.reduce<32>();
  const double s = across_warps<kT / 32>(v, sh);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// p = z + beta p (double-float)
__global__ void __launch_bounds__(kT)
k3_direction(size_t n, const SlotScalars* sc, const float* zh, const float* zl, float* ph, float* pl) {
  if (gate_shut(&sc->active)) return;
  const f2 beta{sc->beta_f[0], sc->beta_f[1]};
  const size_t n4 = n / 4;
  for (size_t i = blockIdx.x * static_cast<size_t>(kT) + threadIdx.x; i < n4; i += static_cast<size_t>(gridDim.x) * kT) {
    const float4 z = reinterpret_cast<const float4*>(zh)[i], zo = reinterpret_cast<const float4*>(zl)[i];
    const float4 p = reinterpret_cast<const float4*>(ph)[i], po = reinterpret_cast<const float4*>(pl)[i];
    const f2 a = df_fma(beta, f2{p.x, po.x}, f2{z.x, zo.x}), b = df_fma(beta, f2{p.y, po.y}, f2{z.y, zo.y});
    const f2 c = df_fma(beta, f2{p.z, po.z}, f2{z.z, zo.z}), d = df_fma(beta, f2{p.w, po.w}, f2{z.w, zo.w});
    reinterpret_cast<float4*>(ph)[i] = make_float4(a.hi, b.hi, c.hi, d.hi);
    reinterpret_cast<float4*>(pl)[i] = make_float4(a.lo, b.lo, c.lo, d.lo);
  }
  if (blockIdx.x == 0)
    for (size_t i = 4 * n4 + threadIdx.x; i < n; i += kT) {
      const f2 v = df_fma(beta, f2{ph[i], pl[i]}, f2{zh[i], zl[i]});
      ph[i] = v.hi;
      pl[i] = v.lo;
    }
}

// One warp: a scalar step from n partials (entry i at part[i * stride]).  KIND 0: p.q -> alpha;
// 1: ||r||^2 after an update; 2: r.z -> rho, beta (mode 0 or 1); 3: ||b - A x||^2 of a replacement.
template <int KIND>
__global__ void __launch_bounds__(32)
k3_finish(SlotScalars* sc, const double* part, int n, int stride, int mode) {
  pdl_wait();
  const int on = KIND == 3 ? sc->fold : (KIND == 2 && mode == 1) ? sc->need_prec : sc->active;
  if (!on) return;
  const double v = warp_sum_strided(part, n, stride);
  __syncwarp();  // every lane has read its flag
  if (threadIdx.x != 0) return;
  if (KIND == 0) finish_pq(sc, v);
  if (KIND == 1) decide_update3(sc, v);
  if (KIND == 2) finish_preconditioner(sc, v, 0.0, mode);
  if (KIND == 3) decide_true(sc, v);
}

// the iterate as FP64 (for the true residual)
__global__ void __launch_bounds__(kT)
k3_to_double(size_t n, const int* __restrict__ gate, const float* h, const float* l, double* __restrict__ d) {
  if (gate_shut(gate)) return;
  for (size_t i = blockIdx.x * static_cast<size_t>(kT) + threadIdx.x; i < n; i += static_cast<size_t>(gridDim.x) * kT)
    d[i] = static_cast<double>(h[i]) + static_cast<double>(l[i]);
}

// masked copy of a float field into double-float planes (zero lo plane)
__global__ void __launch_bounds__(kT)
k3_load_masked(size_t n, const float* __restrict__ v, const uint8_t* __restrict__ mask, float* __restrict__ h,
               float* __restrict__ l) {
  for (size_t i = blockIdx.x * static_cast<size_t>(kT) + threadIdx.x; i < n; i += static_cast<size_t>(gridDim.x) * kT) {
    h[i] = mask[i] ? v[i] : 0.f;
    l[i] = 0.f;
  }
}

// out = f at known nodes (bit copy), 2^e x elsewhere
__global__ void __launch_bounds__(kT)
k3_output(size_t n, const float* __restrict__ xh, const float* __restrict__ xl, int e,
          const uint8_t* __restrict__ mask, const float* __restrict__ f, float* __restrict__ out) {
  for (size_t i = blockIdx.x * static_cast<size_t>(kT) + threadIdx.x; i < n; i += static_cast<size_t>(gridDim.x) * kT)
    out[i] = mask[i] ? static_cast<float>(ldexp(static_cast<double>(xh[i]) + static_cast<double>(xl[i]), e)) : f[i];
}

// Sum of partials in index order by one block (thread t adds t, t + 256, ...; then the block);
// entry i is part[i * stride].
__global__ void __launch_bounds__(kT)
k3_sum(const double* __restrict__ part, int n, double* __restrict__ out, int stride = 1) {
  __shared__ double sh[kT / 32];
  double v = 0.0;
  for (int i = threadIdx.x; i < n; i += kT) v += part[static_cast<size_t>(i) * stride];
  const double s = block_sum_d(v, sh);
  if (threadIdx.x == 0) *out = s;
}

// ---------------------------------------------------------------------------------------------
// Transform products on the CUDA cores (boxes with a side that is no multiple of 128).
// D[m][n] = sum_k A[m][k] B[n][k] for double-float A ([M][K], row-major, lo plane separate) and B
// (rows of length ldb, lo plane at + ldb * ldb), written with n first: out[n * M + m].  Each thread
// keeps 2 x 4 compensated dot products (Ogita-Rump-Oishi Dot2 of double-float operands, pairs of n on
// packed FP32x2).
//
// FORM 0: a plain product.  FORM 1 (the third): times the weights wnorm / (lam_z + lam_y + lam_x)^2
// of the modes [kz][ky][kx], zero for a zero sum (the constant mode when no axis is Dirichlet).
// FORM 2 (the last): z = M Z, zero at known nodes, with the block's partial r.z.
//
// Bound by FP32 issue: twelve operations a multiply-add.  Tiles of 32 x 32 by 128 threads: a
// 72 x 60 x 50 box then has about 280 blocks a product, two an SM, where 64 x 64 tiles left half the
// SMs idle and the rest with eight warps (28-36 us a product); the next 16-deep slab is loaded into
// registers while the current one multiplies.
// ---------------------------------------------------------------------------------------------
constexpr int GM = 32, GN = 32, GK = 16, kGt = 128;

struct Gemm3 {
  const float *A, *Al, *B;
  float *out, *outl;
  int M, K, ldb, N;
  const float *lx, *ly, *lz;  // FORM 1
  int nx;
  float wnorm;
  const uint8_t* mask;        // FORM 2
  const float *rh, *rl;
  double* part;
};

template <int FORM>
__global__ void __launch_bounds__(kGt)
k3_gemm(Gemm3 g, const int* __restrict__ gate) {
  __shared__ __align__(16) float As[2][2][GK][GM + 1];  // [buffer][hi, lo][k][m]
  __shared__ __align__(16) float Bs[2][2][GK][GN + 4];
  __shared__ float sh[3][kGt / 32];
  if (gate_shut(gate)) return;
  const float* Bl = g.B + static_cast<size_t>(g.ldb) * g.ldb;
  const int m0 = blockIdx.x * GM, n0 = blockIdx.y * GN;
  const int t = threadIdx.x, tm = t & 15, tn = t >> 4;
  const int lk = t & 15, lr = t >> 4;  // loads: k and first row of the slab (rows lr + 8 i)
  constexpr int kRows = GM * GK / kGt;
  float ra[2][kRows], rb[2][kRows];
  auto fetch = [&](int k0) {
    const int k = k0 + lk;
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
      const int m = m0 + lr + 8 * i, n = n0 + lr + 8 * i;
      const size_t a = static_cast<size_t>(m) * g.K + k, b = static_cast<size_t>(n) * g.ldb + k;
      const bool oa = m < g.M && k < g.K, ob = n < g.N && k < g.K;
      ra[0][i] = oa ? g.A[a] : 0.f;
      ra[1][i] = oa ? g.Al[a] : 0.f;
      rb[0][i] = ob ? __ldg(g.B + b) : 0.f;
      rb[1][i] = ob ? __ldg(Bl + b) : 0.f;
    }
  };
  auto put = [&](int b) {
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
      As[b][0][lk][lr + 8 * i] = ra[0][i];
      As[b][1][lk][lr + 8 * i] = ra[1][i];
      Bs[b][0][lk][lr + 8 * i] = rb[0][i];
      Bs[b][1][lk][lr + 8 * i] = rb[1][i];
    }
  };
  CompDotDF2 acc[2][2];  // [row tm + 16 i][pair of columns 4 tn + 2 j]
  fetch(0);
  put(0);
  __syncthreads();
  int buf = 0;
  for (int k0 = 0; k0 < g.K; k0 += GK) {
    const bool more = k0 + GK < g.K;
    if (more) fetch(k0 + GK);
#pragma unroll 4
    for (int kk = 0; kk < GK; ++kk) {
      const float4 bh = *reinterpret_cast<const float4*>(&Bs[buf][0][kk][4 * tn]);
      const float4 bl = *reinterpret_cast<const float4*>(&Bs[buf][1][kk][4 * tn]);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const float ah = As[buf][0][kk][tm + 16 * i], al = As[buf][1][kk][tm + 16 * i];
        const float2 a2 = make_float2(ah, ah), l2 = make_float2(al, al);
        acc[i][0].add(a2, l2, make_float2(bh.x, bh.y), make_float2(bl.x, bl.y));
        acc[i][1].add(a2, l2, make_float2(bh.z, bh.w), make_float2(bl.z, bl.w));
      }
    }
    if (more) put(buf ^ 1);
    __syncthreads();
    buf ^= 1;
  }
  CompDotDF dot;
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int m = m0 + tm + 16 * i, n = n0 + 4 * tn + j;
      if (m >= g.M || n >= g.N) continue;
      const CompDotDF2& c = acc[i][j >> 1];
      f2 v = (j & 1) ? df_norm(c.s.y, c.c.y) : df_norm(c.s.x, c.c.x);
      const size_t o = static_cast<size_t>(n) * g.M + m;
      if (FORM == 1) {
        const float s = g.lz[n] + g.ly[m / g.nx] + g.lx[m % g.nx];
        v = s > 0.f ? df_mul(v, spectral_weight_of(g.wnorm, s)) : f2{0.f, 0.f};
      }
      if (FORM == 2) {
        if (!g.mask[o]) v = f2{0.f, 0.f};
        dot.add(g.rh[o], g.rl[o], v.hi, v.lo);
      }
      g.out[o] = v.hi;
      g.outl[o] = v.lo;
    }
  if (FORM == 2) {
    Sum3 v(dot.s, dot.c);
    v.reduce<32>();
    const double s = across_warps<kGt / 32>(v, sh);
    if (t == 0) g.part[blockIdx.y * gridDim.x + blockIdx.x] = s;
  }
}

// ---------------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------------
#define BX3(call)                                                     \
  do {                                                                \
    cudaError_t e_ = (call);                                          \
    if (e_ != cudaSuccess) {                                          \
      *err = std::string(#call) + ": " + cudaGetErrorString(e_);      \
      return EXT_ECUDA;                                               \
    }                                                                 \
  } while (0)

// Device state of one 3-D call: one allocation, freed on every return path.
struct State3 {
  size_t n = 0;
  int vec_blocks = 0, zc = 16;
  dim3 grid3, gridz, block3;  // gridz: the z-marching double-float passes
  int n_parts = 0, n_parts_z = 0, n_parts_g = 0;
  uint8_t* mask = nullptr;
  double *b = nullptr, *d0 = nullptr, *d1 = nullptr, *part = nullptr, *scal = nullptr;
  float *xh = nullptr, *xl = nullptr, *rh = nullptr, *rl = nullptr, *ph = nullptr, *pl = nullptr;
  float *qh = nullptr, *ql = nullptr, *zh = nullptr, *zl = nullptr, *uh = nullptr, *ul = nullptr;
  float *th = nullptr, *tl = nullptr, *lam = nullptr;
  unsigned long long* counts = nullptr;
  SlotScalars* sc = nullptr;
  char* arena = nullptr;
  cudaEvent_t ev[2] = {nullptr, nullptr};
  Tc3 tc;  // the tensor-core preconditioner, when built
  ~State3() {
    cudaFree(arena);
    for (void* p : tc.owned) cudaFree(p);
    for (cudaEvent_t e : ev)
      if (e) cudaEventDestroy(e);
  }
};

Grid3 grid_of(const Solve3Args& a) {
  Grid3 G;
  G.nx = a.nx;
  G.ny = a.ny;
  G.nz = a.nz;
  G.bcx = a.bc[0];
  G.bcy = a.bc[1];
  G.bcz = a.bc[2];
  const double c[3] = {1.0 / (a.h[0] * a.h[0]), 1.0 / (a.h[1] * a.h[1]), 1.0 / (a.h[2] * a.h[2])};
  const double m = std::max(c[0], std::max(c[1], c[2]));
  G.dcx = c[0] / m;
  G.dcy = c[1] / m;
  G.dcz = c[2] / m;
  G.cx = (float)G.dcx;
  G.cy = (float)G.dcy;
  G.cz = (float)G.dcz;
  return G;
}

dim3 gemm_grid(int M, int N) { return dim3((M + GM - 1) / GM, (N + GN - 1) / GN); }

int alloc_state(const Solve3Args& a, State3& s, bool solve, std::string* err) {
  s.n = (size_t)a.nx * a.ny * a.nz;
  s.block3 = dim3(kT);
  s.grid3 = dim3((a.nx + 31) / 32, (a.ny + 7) / 8, a.nz);
  s.n_parts = (int)(s.grid3.x * s.grid3.y * s.grid3.z);
  // chunks of 16 planes, or of 8 or 4 while the blocks would not fill the device twice (the two
  // planes a chunk reads beyond its own then cost less than the idle SMs)
  const int xy = s.grid3.x * ((a.ny + kBy - 1) / kBy);
  s.zc = 16;
  while (s.zc > 4 && xy * ((a.nz + s.zc - 1) / s.zc) < 2 * a.sm_count) s.zc /= 2;
  s.gridz = dim3(s.grid3.x, (a.ny + kBy - 1) / kBy, (a.nz + s.zc - 1) / s.zc);
  s.n_parts_z = (int)(s.gridz.x * s.gridz.y * s.gridz.z);
  const dim3 gl = gemm_grid(a.ny * a.nx, a.nz);
  s.n_parts_g = (int)(gl.x * gl.y);
  s.vec_blocks = (int)std::max<size_t>(1, std::min<size_t>((s.n / 4 + kT - 1) / kT, (size_t)a.sm_count * 8));
  const size_t n = s.n;
  const bool simt = !a.tc_build;
  size_t total = 0;
  auto layout = [&](char* base) {
    size_t off = 0;
    auto take = [&](auto** p, size_t count) {
      *p = reinterpret_cast<std::remove_reference_t<decltype(*p)>>(base + off);
      off = (off + sizeof(**p) * count + 255) / 256 * 256;
    };
    take(&s.mask, n);
    take(&s.part, std::max(std::max(s.n_parts, s.n_parts_g), std::max(s.vec_blocks, s.n_parts_z)));
    take(&s.scal, 8);
    take(&s.counts, 4);
    take(&s.sc, 1);
    take(&s.d0, n);
    for (float** v : {&s.zh, &s.zl, &s.uh, &s.ul}) take(v, n);
    if (simt || !solve)
      for (float** v : {&s.th, &s.tl}) take(v, n);
    take(&s.lam, (size_t)a.nx + a.ny + a.nz);
    if (solve) {
      take(&s.b, n);
      take(&s.d1, n);
      for (float** v : {&s.xh, &s.xl, &s.rh, &s.rl, &s.ph, &s.pl, &s.qh, &s.ql}) take(v, n);
    }
    total = off;
  };
  layout(nullptr);
  if (cudaMalloc(&s.arena, total) != cudaSuccess) {
    cudaGetLastError();
    s.arena = nullptr;
    *err = "cudaMalloc of the 3-D workspace failed";
    return EXT_ENOMEM;
  }
  layout(s.arena);
  return EXT_OK;
}

// Eigenvalues of each axis scaled like the stencil weights, and the weight normaliser wnorm =
// (smallest nonzero eigenvalue sum)^2.
int upload_eigen(const Solve3Args& a, const Grid3& G, State3& s, float* wnorm, std::string* err) {
  const double sc[3] = {G.dcx, G.dcy, G.dcz};
  const int n[3] = {a.nx, a.ny, a.nz};
  std::vector<float> all;
  double lo0[3], lo1[3];  // smallest and smallest nonzero of each axis
  for (int ax = 0; ax < 3; ++ax) {
    lo0[ax] = lo1[ax] = 1e300;
    for (int k = 0; k < n[ax]; ++k) {
      const double v = (float)(a.lam[ax][k] * sc[ax]);
      all.push_back((float)v);
      lo0[ax] = std::min(lo0[ax], v);
      if (v > 0) lo1[ax] = std::min(lo1[ax], v);
    }
  }
  double smin = lo0[0] + lo0[1] + lo0[2];
  if (!(smin > 0))
    smin = std::min(lo1[0] + lo0[1] + lo0[2], std::min(lo0[0] + lo1[1] + lo0[2], lo0[0] + lo0[1] + lo1[2]));
  *wnorm = (float)(smin * smin);
  BX3(cudaMemcpyAsync(s.lam, all.data(), 4 * all.size(), cudaMemcpyHostToDevice, a.stream));
  BX3(cudaStreamSynchronize(a.stream));  // `all` is a pageable source
  return EXT_OK;
}

LaunchCfg dependent(const Solve3Args& a) {
  LaunchCfg c{};
  c.stream = a.stream;
  c.pdl = true;
  return c;
}

// z = M (L^2)^+ M r: six transform products with the weights in the third and the mask and the r.z
// partials in the last (r, z double-float; the products alternate between (th, tl) and (uh, ul)).
// r must be zero at known nodes.  mode as in launch_prec_tc; the CUDA-core kernels take its flag.
void precondition(const Solve3Args& a, const State3& s, float wnorm, const float* rh, const float* rl,
                  float* zh, float* zl, int mode) {
  const int nx = a.nx, ny = a.ny, nz = a.nz;
  LaunchCfg c = dependent(a);
  if (s.tc.on) {
    // the tensor-core path: its descriptors hold r, q, z and the mask of this solve
    const Tc3& t = s.tc;
    c.slots = t.d_descs;
    c.wait_cycles = t.wait_cycles;
    c.dots3 = t.dots3;
    c.items = t.d_items[0];
    c.n_items = t.d_counts;
    c.grid = std::max(1, std::min(t.n_items[0], t.sm_count * 8));
    launch_prec_tc_prepare(c, mode, t.split);
    static const int kForm[7] = {-1, 0, 0, 1, 2, 2, 3};
    for (int k = 1; k < 7; ++k) {
      c.items = t.d_items[k];
      c.n_items = t.d_counts + k;
      c.grid = std::max(1, std::min(t.n_items[k], t.sm_count));
      launch_prec_tc(c, kForm[k], mode, t.split, t.ns, t.err);
    }
    *a.launches += 7;
  } else {
    const int* gate = mode == 0 ? &s.sc->active : mode == 1 ? &s.sc->need_prec : nullptr;
    auto gemm = [&](auto kernel, const float* A, const float* Al, int M, int K, const float* B, int ldb, int N,
                    float* o, float* ol) {
      const Gemm3 g{A, Al, B, o, ol, M, K, ldb, N, s.lam, s.lam + nx, s.lam + nx + ny, nx, wnorm, s.mask, rh, rl,
                    s.part};
      launch_cfg(c, kernel, gemm_grid(M, N), kGt, 0, g, gate);
    };
    // forward: x, y, z (each contracts the contiguous axis and moves it to the front)
    gemm(k3_gemm<0>, rh, rl, nz * ny, nx, a.qt[0], a.np[0], nx, s.th, s.tl);      // [kx][z][y]
    gemm(k3_gemm<0>, s.th, s.tl, nx * nz, ny, a.qt[1], a.np[1], ny, s.uh, s.ul);  // [ky][kx][z]
    gemm(k3_gemm<1>, s.uh, s.ul, ny * nx, nz, a.qt[2], a.np[2], nz, s.th, s.tl);  // [kz][ky][kx]
    // inverse: x, y, z
    gemm(k3_gemm<0>, s.th, s.tl, nz * ny, nx, a.q[0], a.np[0], nx, s.uh, s.ul);   // [x][kz][ky]
    gemm(k3_gemm<0>, s.uh, s.ul, nx * nz, ny, a.q[1], a.np[1], ny, s.th, s.tl);   // [y][x][kz]
    gemm(k3_gemm<2>, s.th, s.tl, ny * nx, nz, a.q[2], a.np[2], nz, zh, zl);       // [z][y][x]
    *a.launches += 6;
  }
  if (mode == 2) return;
  if (s.tc.on) launch_cfg(c, k3_finish<2>, 1, 32, 0, s.sc, s.tc.part + 2, s.tc.n_tiles3, 4, mode);
  else launch_cfg(c, k3_finish<2>, 1, 32, 0, s.sc, s.part, s.n_parts_g, 1, mode);
  ++*a.launches;
}

// q = M L^2 p (p double-float, zero at known nodes), p.q partials in part
void apply_operator(const Solve3Args& a, const Grid3& G, const State3& s, const int* gate, const float* ph,
                    const float* pl, float* qh, float* ql) {
  const LaunchCfg c = dependent(a);
  launch_cfg(c, k3_lap<false>, s.gridz, kT, 0, G, s.zc, gate, ph, pl, s.uh, s.ul, s.mask, nullptr, nullptr, nullptr);
  launch_cfg(c, k3_lap<true>, s.gridz, kT, 0, G, s.zc, gate, s.uh, s.ul, qh, ql, s.mask, ph, pl, s.part);
  *a.launches += 2;
}

// One CG iteration: p = z + beta p, q = A p, alpha, x, r, ||r||^2, z, rho and beta.
void enqueue_iteration(const Solve3Args& a, const Grid3& G, const State3& s, float wnorm) {
  const LaunchCfg c = dependent(a);
  launch_cfg(c, k3_direction, s.vec_blocks, kT, 0, s.n, s.sc, s.zh, s.zl, s.ph, s.pl);
  apply_operator(a, G, s, &s.sc->active, s.ph, s.pl, s.qh, s.ql);
  launch_cfg(c, k3_finish<0>, 1, 32, 0, s.sc, s.part, s.n_parts_z, 1, 0);
  launch_cfg(c, k3_update, s.vec_blocks, kT, 0, s.n, s.sc, s.ph, s.pl, s.qh, s.ql, s.xh, s.xl, s.rh, s.rl, s.part);
  launch_cfg(c, k3_finish<1>, 1, 32, 0, s.sc, s.part, s.vec_blocks, 1, 0);
  *a.launches += 4;
  precondition(a, s, wnorm, s.rh, s.rl, s.zh, s.zl, 0);
}

// The end of a block: the FP64 true residual where one is due, the decision, and the fresh
// preconditioner pass of a solve that continues.
void enqueue_tail(const Solve3Args& a, const Grid3& G, const State3& s, float wnorm) {
  const LaunchCfg c = dependent(a);
  const int* gate = &s.sc->fold;
  launch_cfg(c, k3_to_double, s.vec_blocks, kT, 0, s.n, gate, s.xh, s.xl, s.d0);
  launch_cfg(c, k3_lap64<0>, s.grid3, kT, 0, G, gate, s.d0, s.d1, s.mask, nullptr, nullptr, nullptr, nullptr);
  launch_cfg(c, k3_lap64<2>, s.grid3, kT, 0, G, gate, s.d1, s.d0, s.mask, s.b, s.part, s.rh, s.rl);
  launch_cfg(c, k3_finish<3>, 1, 32, 0, s.sc, s.part, s.n_parts, 1, 0);
  *a.launches += 4;
  precondition(a, s, wnorm, s.rh, s.rl, s.zh, s.zl, 1);
}

// mask and known field; validation of the data
int setup_mask(const Solve3Args& a, State3& s, const float* phi, const float* f, unsigned long long* cnt,
               std::string* err) {
  BX3(cudaMemsetAsync(s.counts, 0, 4 * sizeof(unsigned long long), a.stream));
  k3_setup<<<s.vec_blocks, kT, 0, a.stream>>>(s.n, phi, f, a.dir, s.mask, s.d0, s.counts);
  ++*a.launches;
  BX3(cudaGetLastError());
  BX3(cudaMemcpyAsync(cnt, s.counts, 4 * sizeof(unsigned long long), cudaMemcpyDeviceToHost, a.stream));
  BX3(cudaStreamSynchronize(a.stream));
  if (cnt[2] || cnt[3]) {
    *err = cnt[2] ? "phi holds NaN" : "f is not finite at a known node";
    return EXT_EINVAL;
  }
  return EXT_OK;
}

constexpr int kBlockIters = 8;  // iterations between two readings of the scalars

// Whether a wait of the tensor-core kernels ran out (the CUDA-core kernels have none).
bool wait_ran_out(const State3& s) { return s.tc.on && *static_cast<volatile const int*>(s.tc.err) != 0; }
// Then the flag goes down once the stream has finished, so the next call starts afresh.
int timed_out(const Solve3Args& a, const State3& s, std::string* err) {
  BX3(cudaStreamSynchronize(a.stream));
  *s.tc.err = 0;
  *err = "a bounded device wait (tensor-core pipeline) ran out";
  return EXT_ETIMEOUT;
}

}  // namespace

int solve3d_run(const Solve3Args& a, const float* phi, const float* f, float* out, ext_result* res,
                std::string* err) {
  State3 s;
  int rc = alloc_state(a, s, true, err);
  if (rc) return rc;
  if (a.tc_build) {
    rc = a.tc_build(Tc3Io{s.rh, s.rl, s.qh, s.ql, s.zh, s.zl, s.mask, s.sc}, s.tc);
    if (rc) return rc;
  }
  const Grid3 G = grid_of(a);
  float wnorm = 1.f;
  rc = upload_eigen(a, G, s, &wnorm, err);
  if (rc) return rc;
  unsigned long long cnt[4];
  rc = setup_mask(a, s, phi, f, cnt, err);
  if (rc) return rc;
  res->n_unknown = (int32_t)cnt[0];
  res->n_known = (int32_t)cnt[1];
  const bool has_dirichlet = a.bc[0] == 2 || a.bc[1] == 2 || a.bc[2] == 2;
  if (cnt[1] == 0 && !has_dirichlet) {
    *err = "no known node: the extension is not unique without a Dirichlet axis";
    return EXT_ENOKNOWN;
  }
  cudaStream_t st = a.stream;
  // b = -M L^2 E_K f (FP64) and ||b||^2
  k3_lap64<0><<<s.grid3, s.block3, 0, st>>>(G, nullptr, s.d0, s.d1, s.mask, nullptr, nullptr, nullptr, nullptr);
  ++*a.launches;
  k3_lap64<1><<<s.grid3, s.block3, 0, st>>>(G, nullptr, s.d1, s.b, s.mask, nullptr, s.part, nullptr, nullptr);
  ++*a.launches;
  k3_sum<<<1, kT, 0, st>>>(s.part, s.n_parts, s.scal);
  ++*a.launches;
  double bb = 0.0;
  BX3(cudaMemcpyAsync(&bb, s.scal, sizeof(double), cudaMemcpyDeviceToHost, st));
  BX3(cudaStreamSynchronize(st));
  const double bnorm = std::sqrt(bb);
  res->iters = 0;
  res->relres_true = res->relres_rec = 0.0;
  res->err_est = 0.0;
  if (!(bnorm > 0.0) || cnt[0] == 0) {
    k3_init<<<s.vec_blocks, kT, 0, st>>>(s.n, s.b, 0.0, s.rh, s.rl, s.xh, s.xl);
    ++*a.launches;
    k3_output<<<s.vec_blocks, kT, 0, st>>>(s.n, s.xh, s.xl, 0, s.mask, f, out);
    ++*a.launches;
    BX3(cudaGetLastError());
    BX3(cudaStreamSynchronize(st));
    res->status = EXT_OK;
    return EXT_OK;
  }
  // the iteration runs on 2^-e b with ||2^-e b|| near 1
  int e = 0;
  std::frexp(bnorm, &e);
  const double scale = std::ldexp(1.0, -e);
  k3_init<<<s.vec_blocks, kT, 0, st>>>(s.n, s.b, scale, s.rh, s.rl, s.xh, s.xl);
  ++*a.launches;
  // the scaled right-hand side for the true residual: b <- 2^-e b (exact)
  k3_to_double<<<s.vec_blocks, kT, 0, st>>>(s.n, nullptr, s.rh, s.rl, s.b);
  ++*a.launches;
  const double bn = bnorm * scale;
  SlotScalars& h0 = a.h_sc[0];
  h0 = SlotScalars{};
  h0.bb = h0.rr = h0.rr_rec = h0.rr_true = h0.rr_ref = bn * bn;
  h0.rtol2 = a.rtol * a.rtol;
  h0.delta2 = a.replace_factor * a.replace_factor;
  h0.fold_every = a.true_res_every;
  h0.maxit = a.maxit > 0 ? a.maxit : 10 * std::max(a.nx, std::max(a.ny, a.nz));
  h0.status = ST_RUNNING;
  h0.active = h0.need_prec = 1;
  const int maxit = h0.maxit;
  BX3(cudaMemcpyAsync(s.sc, &h0, sizeof(SlotScalars), cudaMemcpyHostToDevice, st));
  // the first direction is z (beta = 0)
  BX3(cudaMemsetAsync(s.ph, 0, 4 * s.n, st));
  BX3(cudaMemsetAsync(s.pl, 0, 4 * s.n, st));
  for (cudaEvent_t& v : s.ev) BX3(cudaEventCreateWithFlags(&v, cudaEventDisableTiming));
  precondition(a, s, wnorm, s.rh, s.rl, s.zh, s.zl, 1);
  SlotScalars last{};
  // a block of a solve that runs completes an iteration at least (one whose recursive residual converges
  // in each, the true one not, no more than that), so maxit ends the solve before the blocks do
  const long long max_blocks = maxit + 1LL;
  // one block stays ahead of the reading; with nothing left to do it passes by its flags
  for (long long blk = 0; blk <= max_blocks; ++blk) {
    if (blk < max_blocks) {
      const int set = blk & 1;
      for (int i = 0; i < kBlockIters; ++i) enqueue_iteration(a, G, s, wnorm);
      enqueue_tail(a, G, s, wnorm);
      BX3(cudaGetLastError());
      BX3(cudaMemcpyAsync(&a.h_sc[set], s.sc, sizeof(SlotScalars), cudaMemcpyDeviceToHost, st));
      BX3(cudaEventRecord(s.ev[set], st));
    }
    if (blk == 0) continue;
    const int seen = (blk - 1) & 1;
    BX3(cudaEventSynchronize(s.ev[seen]));
    if (wait_ran_out(s)) return timed_out(a, s, err);
    last = a.h_sc[seen];
    if (last.status != ST_RUNNING) break;
  }
  BX3(cudaStreamSynchronize(st));
  int status = last.status == ST_RUNNING ? EXT_ETIMEOUT : last.status;
  res->iters = last.it;
  res->relres_true = std::sqrt(last.rr_true) / bn;
  res->relres_rec = std::sqrt(last.rr_rec) / bn;
  double tail = 0.0;
  for (int k = 0; k < std::min(last.aro_n, kErrDelay); ++k) tail += last.aro_ring[k];
  res->err_est = last.aro_total > 0.0 ? std::sqrt(std::max(0.0, tail) / last.aro_total) : 0.0;
  k3_output<<<s.vec_blocks, kT, 0, st>>>(s.n, s.xh, s.xl, e, s.mask, f, out);
  ++*a.launches;
  BX3(cudaGetLastError());
  BX3(cudaStreamSynchronize(st));
  res->status = status;
  return status;
}

int apply3d_operator(const Solve3Args& a, const float* phi, const float* p, float* q, std::string* err) {
  State3 s;
  int rc = alloc_state(a, s, false, err);
  if (rc) return rc;
  const Grid3 G = grid_of(a);
  unsigned long long cnt[4];
  rc = setup_mask(a, s, phi, phi, cnt, err);  // f is not used: phi stands in (finite at known nodes)
  if (rc) return rc;
  // p masked into (th, tl); q into (zh, zl); the hi plane is the result
  k3_load_masked<<<s.vec_blocks, kT, 0, a.stream>>>(s.n, p, s.mask, s.th, s.tl);
  ++*a.launches;
  apply_operator(a, G, s, nullptr, s.th, s.tl, s.zh, s.zl);
  BX3(cudaMemcpyAsync(q, s.zh, 4 * s.n, cudaMemcpyDeviceToDevice, a.stream));
  BX3(cudaGetLastError());
  BX3(cudaStreamSynchronize(a.stream));
  return EXT_OK;
}

int apply3d_preconditioner(const Solve3Args& a, const float* phi, const float* r, float* z, double* scale,
                           std::string* err) {
  State3 s;
  int rc = alloc_state(a, s, false, err);
  if (rc) return rc;
  const Grid3 G = grid_of(a);
  float wnorm = 1.f;
  rc = upload_eigen(a, G, s, &wnorm, err);
  if (rc) return rc;
  unsigned long long cnt[4];
  rc = setup_mask(a, s, phi, phi, cnt, err);
  if (rc) return rc;
  // the masked copy of r: d0 reinterpreted as two float planes
  float* rh = reinterpret_cast<float*>(s.d0);
  float* rl = rh + s.n;
  if (a.tc_build) {
    SlotScalars h{};  // no flexible beta: the last product leaves z.q out
    BX3(cudaMemcpyAsync(s.sc, &h, sizeof(h), cudaMemcpyHostToDevice, a.stream));
    rc = a.tc_build(Tc3Io{rh, rl, s.uh, s.ul, s.zh, s.zl, s.mask, s.sc}, s.tc);
    if (rc) return rc;
  }
  k3_load_masked<<<s.vec_blocks, kT, 0, a.stream>>>(s.n, r, s.mask, rh, rl);
  ++*a.launches;
  precondition(a, s, wnorm, rh, rl, s.zh, s.zl, 2);
  BX3(cudaMemcpyAsync(z, s.zh, 4 * s.n, cudaMemcpyDeviceToDevice, a.stream));
  BX3(cudaGetLastError());
  BX3(cudaStreamSynchronize(a.stream));
  if (wait_ran_out(s)) return timed_out(a, s, err);
  // weights are (L^2)^+ scaled by wnorm, times the square of the stencil scaling (max 1/h^2)^-2
  const double m = std::max(1.0 / (a.h[0] * a.h[0]), std::max(1.0 / (a.h[1] * a.h[1]), 1.0 / (a.h[2] * a.h[2])));
  if (scale) *scale = (double)wnorm * m * m;
  return EXT_OK;
}

}  // namespace bx
