// Geometric multigrid on the Schur-reduced electrode blocks (paper section 4:
// one V-cycle approximates each electrode-level block inverse; the paper uses
// BoomerAMG, here the structured hex grid gives the hierarchy directly).
//
// Hierarchies h: 0 phi_s anode, 1 phi_s cathode, 2 phi_e, 3 c_e.  The two
// electrodes' phi_s never couple, and the thin separator leaves no coarse
// grid that could represent both electrodes' near-constant modes, so phi_s
// gets one masked hierarchy per electrode (they share the level-0 arrays).
//
// Per level: trilinear prolongation P (rows of masked-out fine nodes zero),
// Galerkin operators A_{l+1} = P^T A_l P split into a fixed part (built once
// at setup from the fixed stencils) and a linearization-dependent part
// (Schur/reaction row sums, rebuilt per Newton step), Chebyshev smoothing on
// D^-1 A over [lam/ratio, lam] (lam: Gershgorin bound), and an explicit FP64
// inverse on the coarsest level.  Stencils are in difference form (slot 13
// = row sum), see p4d_common.cuh.
#include <algorithm>
#include <type_traits>
#include <vector>
#include <cmath>
#include "p4d_common.cuh"

namespace p4d {
namespace {

template <typename T> __device__ __forceinline__ T fromd(double v);
template <> __device__ __forceinline__ double fromd<double>(double v) { return v; }
template <> __device__ __forceinline__ float fromd<float>(double v) { return (float)v; }
template <> __device__ __forceinline__ __nv_bfloat16 fromd<__nv_bfloat16>(double v) {
  return __float2bfloat16((float)v);
}
// stencil entry -> compute precision (identity for float/double, widen bf16)
template <typename T> __device__ __forceinline__ T tof(T v) { return v; }
__device__ __forceinline__ float tof(__nv_bfloat16 v) { return __bfloat162float(v); }


struct LevelDims {
  int nnx, nny, nnz;
  int64_t n;
};

struct HList {
  int h[kNH];
};

__device__ __forceinline__ void node_ijk(const LevelDims& d, int64_t n, int& i, int& j, int& k) {
  i = (int)(n % d.nnx);
  j = (int)((n / d.nnx) % d.nny);
  k = (int)(n / ((int64_t)d.nnx * d.nny));
}

// One-dimensional linear interpolation between a fine node line (ne
// elements) and its coarsening: coarse nodes sit on the even fine nodes and,
// when ne is odd, also on the last fine node (that coarse element spans one
// fine element), so every element count >= 2 can be coarsened.  Per fine
// node: up to two parents; per coarse node: up to three support nodes.
// (struct Axis / Xfer: p4d_common.cuh)

// ---------------------------------------------------------------- masks
__global__ void k_mask0(int64_t nn, const uint8_t* __restrict__ label, uint8_t* m0, uint8_t* m1, uint8_t* m2,
                        uint8_t* m3) {
  const int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (n >= nn) return;
  const uint8_t l = label[n];
  const bool act = l & kLabActive;
  m0[n] = act && (l & kLabAnode);
  m1[n] = act && (l & kLabCathode);
  m2[n] = 1;
  m3[n] = 1;
}

// First and last node of each hierarchy's mask: ext[2 h] = min, ext[2 h + 1]
// = max (initialised to n and -1).
__global__ void k_mask_extent(int64_t n, Ptr4<const uint8_t> m, int* __restrict__ ext) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int h = blockIdx.y;
  if (i >= n || !pk(m.p, h)[i]) return;
  atomicMin(ext + 2 * h, (int)i);
  atomicMax(ext + 2 * h + 1, (int)i);
}

__global__ void k_mask_coarse(LevelDims fd, LevelDims cd, Xfer X, Ptr4<const uint8_t> fm, Ptr4<uint8_t> cm) {
  const int64_t C = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int h = blockIdx.y;
  if (C >= cd.n) return;
  int I, J, K;
  node_ijk(cd, C, I, J, K);
  uint8_t any = 0;
  for (int tz = 0; tz < 3; ++tz) {
    const int fk = X.a[2].sup[K * 3 + tz];
    if (fk < 0) continue;
    for (int ty = 0; ty < 3; ++ty) {
      const int fj = X.a[1].sup[J * 3 + ty];
      if (fj < 0) continue;
      for (int tx = 0; tx < 3; ++tx) {
        const int fi = X.a[0].sup[I * 3 + tx];
        if (fi < 0) continue;
        any |= pk(fm.p, h)[fi + (int64_t)fd.nnx * (fj + (int64_t)fd.nny * fk)];
      }
    }
  }
  pk(cm.p, h)[C] = any ? 1 : 0;
}

// 32-bit (i, j, k) of node n of a level (every level has < 2^31 nodes).
__device__ __forceinline__ void node_ijk_i32(const LevelDims& d, int n, int& i, int& j, int& k) {
  const int sxy = d.nnx * d.nny;
  k = n / sxy;
  const int r = n - k * sxy;
  j = r / d.nnx;
  i = r - j * d.nnx;
}

// Interpolation between a level and its coarsening, computed instead of read
// from the tables of struct Axis (same rule and weights; the weights 1/2 and
// 1 are exact, so the sums round identically): a table entry is a dependent
// load in front of every transferred value, and the transfers are bound by
// that latency.  Coarse node I of a coarsened axis sits on fine node 2 I;
// with an odd element count the last fine node keeps its own coarse node.
struct Axis1 {
  int nf, nc, c;   // fine nodes, coarse nodes, coarsened
};
struct Xfer1 {
  Axis1 a[3];
};

// Entry t of the support of coarse node I: fine node (-1: none) and weight.
template <typename T>
__device__ __forceinline__ int sup_of(const Axis1& a, int I, int t, T& w) {
  w = (T)1;
  if (!a.c) return t == 0 ? I : -1;
  const int f = 2 * I - 1 + t;
  if (f < 0 || f >= a.nf) return -1;
  if (f == a.nf - 1 && !(a.nf & 1)) return I == a.nc - 1 ? f : -1;   // the last fine node of an odd element count
  if (t != 1) w = (T)0.5;
  return f;
}

// Parent q (0, 1) of fine node i: coarse node (-1: none) and weight.
template <typename T>
__device__ __forceinline__ int par_of(const Axis1& a, int i, int q, T& w) {
  w = (T)1;
  if (!a.c) return q == 0 ? i : -1;
  if (i == a.nf - 1 && !(a.nf & 1)) return q == 0 ? a.nc - 1 : -1;
  if (!(i & 1)) return q == 0 ? i >> 1 : -1;
  w = (T)0.5;
  return (i >> 1) + q;
}

// ---------------------------------------------------------------- Galerkin
// Source operator in difference form: off-diagonals O[o][n] (o != 13) and
// row sums s[n] (slot 13, or a separate array at level 0).
struct SrcOp {
  const double* st;      // [27][n] (slot 13 ignored when rs != nullptr)
  const double* rs;      // optional separate row sums [n]
};

// A_c = P^T diag(m) A diag(m) P for one hierarchy; writes difference form.
// identity_out: coarse nodes without support get an identity row (fixed part)
// or a zero row (variable part).  TV: the precision of input, accumulation
// and output (FP64 for the fixed part and the FP64 preconditioner).
//
// One warp per coarse node, lane t < 27 owning fine support node t: each
// lane scatters its row's products into its own column of 27 accumulators
// in shared memory, then lane o sums slot o over the 27 columns in a fixed
// order (deterministic, no atomics).
constexpr int kRapWarps = 4;     // coarse nodes per block
constexpr int kRapLd = 28;       // accumulator column stride (27 lanes, padded)

// acc[stride * oo] += a * w(g -> D) over the (up to 8) coarse parents D of
// fine node (gi, gj, gk), oo the slot of D in the coarse row of (I, J, K).
template <typename TV>
__device__ __forceinline__ void rap_scatter(const Xfer& X, int gi, int gj, int gk, int I, int J, int K, TV a,
                                            TV* acc, int stride) {
  const TV* pwx = parw_t<TV>(X.a[0]);
  const TV* pwy = parw_t<TV>(X.a[1]);
  const TV* pwz = parw_t<TV>(X.a[2]);
  int oyz[4];
  TV wyz[4];
  int nyz = 0;
  for (int c3 = 0; c3 < 2; ++c3) {
    const int pz = X.a[2].par[gk * 2 + c3];
    if (pz < 0) continue;
    for (int c2 = 0; c2 < 2; ++c2) {
      const int py = X.a[1].par[gj * 2 + c2];
      if (py < 0) continue;
      oyz[nyz] = 3 * (py - J + 1) + 9 * (pz - K + 1);
      wyz[nyz] = pwy[gj * 2 + c2] * pwz[gk * 2 + c3];
      ++nyz;
    }
  }
  for (int c1 = 0; c1 < 2; ++c1) {
    const int px = X.a[0].par[gi * 2 + c1];
    if (px < 0) continue;
    const TV t = a * pwx[gi * 2 + c1];
    for (int q = 0; q < nyz; ++q) acc[(oyz[q] + px - I + 1) * stride] += t * wyz[q];
  }
}

// Fine support node of lane t (t < 27) of coarse node (I, J, K): index f and
// weight, or false when absent or masked out.
template <typename TV>
__device__ __forceinline__ bool rap_support(const LevelDims& fd, const Xfer& X, const uint8_t* m, int I, int J, int K,
                                            int t, int& fi, int& fj, int& fk, int64_t& f, TV& wf) {
  const int tx = t % 3, ty = (t / 3) % 3, tz = t / 9;
  fi = X.a[0].sup[I * 3 + tx];
  fj = X.a[1].sup[J * 3 + ty];
  fk = X.a[2].sup[K * 3 + tz];
  if (fi < 0 || fj < 0 || fk < 0) return false;
  f = fi + (int64_t)fd.nnx * (fj + (int64_t)fd.nny * fk);
  if (!m[f]) return false;
  wf = supw_t<TV>(X.a[0])[I * 3 + tx] * (supw_t<TV>(X.a[1])[J * 3 + ty] * supw_t<TV>(X.a[2])[K * 3 + tz]);
  return true;
}

// Slot totals of one warp's accumulator block and the row sum: lane o < 27
// writes slot o of coarse node C.
template <typename TV>
__device__ __forceinline__ void rap_finish(const TV* my, TV rs_lane, bool cin, int identity_out, int lane,
                                           TV* o_, int64_t cn, int64_t C) {
  TV rsum = rs_lane;
  for (int o = 16; o > 0; o >>= 1) rsum += __shfl_xor_sync(0xffffffffu, rsum, o);
  if (lane >= 27) return;
  TV v;
  if (!cin) {
    v = (lane == 13 && identity_out) ? (TV)1 : (TV)0;
  } else if (lane == 13) {
    v = rsum;
  } else {
    v = 0;
    for (int l = 0; l < 27; ++l) v += my[lane * kRapLd + l];
  }
  o_[lane * cn + C] = v;
}

template <typename TV>
__global__ void __launch_bounds__(32 * kRapWarps) k_rap(LevelDims fd, LevelDims cd, Xfer X, Ptr4<const TV> fst,
                                                        Ptr4<const TV> frs, Ptr4<const uint8_t> fm,
                                                        Ptr4<const uint8_t> cm, Ptr4<TV> out, int identity_out) {
  __shared__ TV part[kRapWarps][27 * kRapLd];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t C = (int64_t)blockIdx.x * kRapWarps + warp;
  const int h = blockIdx.y;
  if (C >= cd.n) return;   // per warp
  TV* my = part[warp];
  if (lane < 27)
    for (int o = 0; o < 27; ++o) my[o * kRapLd + lane] = (TV)0;
  int I, J, K;
  node_ijk(cd, C, I, J, K);
  const bool cin = pk(cm.p, h)[C];
  const TV* st = pk(fst.p, h);
  const TV* rs = pk(frs.p, h);
  const int64_t fn = fd.n;
  TV rs_l = 0;
  int fi, fj, fk;
  int64_t f;
  TV wf;
  if (cin && lane < 27 && rap_support<TV>(fd, X, pk(fm.p, h), I, J, K, lane, fi, fj, fk, f, wf)) {
    const uint8_t* m = pk(fm.p, h);
    const TV sf = rs ? rs[f] : st[13 * fn + f];
    rs_l = wf * sf;
    // full-form diagonal of row f
    TV diag = sf;
    for (int o = 0; o < 27; ++o)
      if (o != 13) diag -= st[o * fn + f];
    for (int o = 0; o < 27; ++o) {
      const int dx = o % 3 - 1, dy = (o / 3) % 3 - 1, dz = o / 9 - 1;
      const int gi = fi + dx, gj = fj + dy, gk = fk + dz;
      if (gi < 0 || gj < 0 || gk < 0 || gi >= fd.nnx || gj >= fd.nny || gk >= fd.nnz) continue;
      const int64_t gidx = gi + (int64_t)fd.nnx * (gj + (int64_t)fd.nny * gk);
      if (!m[gidx]) continue;
      const TV a = (o == 13 ? diag : st[o * fn + f]) * wf;
      if (a == (TV)0) continue;
      rap_scatter<TV>(X, gi, gj, gk, I, J, K, a, my + lane, kRapLd);
    }
  }
  __syncwarp();
  rap_finish<TV>(my, rs_l, cin, identity_out, lane, pk(out.p, h), cd.n, C);
}

// The same product in FP32, without scattering: per axis the parents of the
// neighbours f + o of a support node lie on the coarse offsets d in {-1, 0,
// 1} of I, so the lane multiplies its row with 3 x 3 weight maps per axis
// held in registers (absent parents: weight 0, acc + 0 = acc) and adds to 27
// register accumulators, offset by offset as the scatter does; only the 27
// slots then pass through shared memory, summed over the lanes in the same
// order.  The scatter updates shared memory up to 216 times per lane (109 us
// at level 2 of a 65 x 65 x 49 cell, 751 + 188 us at levels 2 and 3 of 129 x
// 129 x 97); with this kernel and the coarsest solve below the linearization
// of the two cells takes 0.51 and 2.27 ms instead of 0.70 and 2.88.  In FP64
// the extra products cost more than the scatter.
struct RapAxis {
  float m[3][3];   // [o][d]: weight from fine node f + o - 1 to coarse node I + d - 1
};
__device__ __forceinline__ RapAxis rap_axis(const Axis1& a, int I, int t, int& f, float& w) {
  RapAxis r;
  f = sup_of<float>(a, I, t, w);
#pragma unroll
  for (int o = 0; o < 3; ++o) {
    const int g = f + o - 1;
    const bool in = f >= 0 && g >= 0 && g < a.nf;
    float w0 = 0.f, w1 = 0.f;
    const int p0 = in ? par_of<float>(a, g, 0, w0) : -9, p1 = in ? par_of<float>(a, g, 1, w1) : -9;
#pragma unroll
    for (int d = 0; d < 3; ++d) r.m[o][d] = p0 == I + d - 1 && p0 >= 0 ? w0 : (p1 == I + d - 1 && p1 >= 0 ? w1 : 0.f);
  }
  return r;
}

__global__ void __launch_bounds__(32 * kRapWarps) k_rap32(LevelDims fd, LevelDims cd, Xfer1 X, Ptr4<const float> fst,
                                                          Ptr4<const uint8_t> fm, Ptr4<const uint8_t> cm,
                                                          Ptr4<float> out) {
  __shared__ float part[kRapWarps][27 * kRapLd];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int C = blockIdx.x * kRapWarps + warp;
  const int h = blockIdx.y;
  if (C >= (int)cd.n) return;   // per warp
  float* my = part[warp];
  int I, J, K;
  node_ijk_i32(cd, C, I, J, K);
  const bool cin = pk(cm.p, h)[C];
  const float* __restrict__ st = pk(fst.p, h);
  const uint8_t* __restrict__ m = pk(fm.p, h);
  const int fn = (int)fd.n;
  float acc[27];
#pragma unroll
  for (int q = 0; q < 27; ++q) acc[q] = 0.f;
  float rs_l = 0.f;
  if (cin && lane < 27) {
    int fi, fj, fk;
    float wx, wy, wz;
    const RapAxis ax = rap_axis(X.a[0], I, lane % 3, fi, wx);
    const RapAxis ay = rap_axis(X.a[1], J, lane / 3 % 3, fj, wy);
    const RapAxis az = rap_axis(X.a[2], K, lane / 9, fk, wz);
    const int f = fi + fd.nnx * (fj + fd.nny * fk);
    if (fi >= 0 && fj >= 0 && fk >= 0 && m[f]) {
      const float wf = wx * (wy * wz);
      float a[27];
#pragma unroll
      for (int o = 0; o < 27; ++o) a[o] = st[o * fn + f];
      unsigned in = 0;   // neighbours inside the grid and the mask
#pragma unroll
      for (int o = 0; o < 27; ++o) {
        const int gi = fi + o % 3 - 1, gj = fj + (o / 3) % 3 - 1, gk = fk + o / 9 - 1;
        const bool g = gi >= 0 && gj >= 0 && gk >= 0 && gi < fd.nnx && gj < fd.nny && gk < fd.nnz;
        if (g && m[gi + fd.nnx * (gj + fd.nny * gk)]) in |= 1u << o;
      }
      const float sf = a[13];
      rs_l = wf * sf;
      float diag = sf;   // full-form diagonal of row f
#pragma unroll
      for (int o = 0; o < 27; ++o)
        if (o != 13) diag -= a[o];
      a[13] = diag;
#pragma unroll
      for (int oz = 0; oz < 3; ++oz)
#pragma unroll
        for (int oy = 0; oy < 3; ++oy) {
          float wzy[9];
#pragma unroll
          for (int q = 0; q < 9; ++q) wzy[q] = az.m[oz][q / 3] * ay.m[oy][q % 3];
#pragma unroll
          for (int ox = 0; ox < 3; ++ox) {
            const int o = ox + 3 * oy + 9 * oz;
            const float v = (in >> o) & 1 ? a[o] * wf : 0.f;
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) {
              const float t = v * ax.m[ox][dx];
#pragma unroll
              for (int q = 0; q < 9; ++q) acc[3 * q + dx] += t * wzy[q];
            }
          }
        }
    }
  }
  if (lane < 27) {
#pragma unroll
    for (int o = 0; o < 27; ++o) my[o * kRapLd + lane] = acc[o];
  }
  __syncwarp();
  rap_finish<float>(my, rs_l, cin, 0, lane, pk(out.p, h), cd.n, C);
}

// V_1 = P^T diag(m s) P by gathering: with a diagonal operator and a
// tensor-product P, entry (C, C + o) is sum_f w_C(f) m_f s_f w_{C+o}(f) over
// the fine nodes f in both supports, and it factors by axis.  One thread per
// coarse node: the m s values of its (at most 3 x 3 x 3) support nodes, the
// per-axis weight products q_a[d][t] = w_C(t) w_{C+d-1}(t) of support entry t,
// then three passes (x, y, z) give all 27 slots.  Slot 13 holds the row sum
// sum_f w_C(f) m_f s_f (a fine node's interpolation weights sum to one).
template <typename TV>
__global__ void __launch_bounds__(128) k_rap_diag_g(LevelDims fd, LevelDims cd, Xfer X, Ptr4<const double> s,
                                                    Ptr4<const uint8_t> fm, Ptr4<const uint8_t> cm,
                                                    Ptr4<TV> out) {
  const int C = blockIdx.x * blockDim.x + threadIdx.x;
  const int h = blockIdx.y;
  if (C >= (int)cd.n) return;
  TV* o_ = pk(out.p, h);
  const int64_t cn = cd.n;
  if (!pk(cm.p, h)[C]) {
#pragma unroll
    for (int o = 0; o < 27; ++o) o_[o * cn + C] = (TV)0;
    return;
  }
  int I, J, K;
  node_ijk(cd, (int64_t)C, I, J, K);
  const int Ic[3] = {I, J, K};
  const int ncd[3] = {cd.nnx, cd.nny, cd.nnz};
  int f[3][3];      // support fine index per axis and entry (-1: none)
  TV w[3][3];       // its weight w_C
  TV q[3][3][3];    // [axis][offset d][entry t]: w_C(t) w_{C+d-1}(t)
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int* sup = X.a[a].sup;
    const TV* sw = supw_t<TV>(X.a[a]);
#pragma unroll
    for (int t = 0; t < 3; ++t) {
      f[a][t] = sup[Ic[a] * 3 + t];
      w[a][t] = f[a][t] >= 0 ? sw[Ic[a] * 3 + t] : (TV)0;
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int I2 = Ic[a] + d - 1;
      const bool in = I2 >= 0 && I2 < ncd[a];
#pragma unroll
      for (int t = 0; t < 3; ++t) {
        TV wv = (TV)0;
#pragma unroll
        for (int u = 0; u < 3; ++u) {
          const int g = in ? sup[I2 * 3 + u] : -1;
          if (f[a][t] >= 0 && g == f[a][t]) wv = sw[I2 * 3 + u];
        }
        q[a][d][t] = w[a][t] * wv;
      }
    }
  }
  // m s of the support nodes
  const double* sv = pk(s.p, h);
  const uint8_t* m = pk(fm.p, h);
  TV S[3][3][3];   // [tz][ty][tx]
#pragma unroll
  for (int tz = 0; tz < 3; ++tz)
#pragma unroll
    for (int ty = 0; ty < 3; ++ty)
#pragma unroll
      for (int tx = 0; tx < 3; ++tx) {
        TV v = (TV)0;
        if (f[0][tx] >= 0 && f[1][ty] >= 0 && f[2][tz] >= 0) {
          const int64_t fi = f[0][tx] + (int64_t)fd.nnx * (f[1][ty] + (int64_t)fd.nny * f[2][tz]);
          if (m[fi]) v = (TV)sv[fi];
        }
        S[tz][ty][tx] = v;
      }
  // row sum
  TV rs = (TV)0;
#pragma unroll
  for (int tz = 0; tz < 3; ++tz)
#pragma unroll
    for (int ty = 0; ty < 3; ++ty)
#pragma unroll
      for (int tx = 0; tx < 3; ++tx) rs += w[2][tz] * (w[1][ty] * (w[0][tx] * S[tz][ty][tx]));
  // x pass: T1[dx][tz][ty]; y pass: T2[dx][dy][tz]; z pass: the slots
  TV T1[3][3][3];
#pragma unroll
  for (int dx = 0; dx < 3; ++dx)
#pragma unroll
    for (int tz = 0; tz < 3; ++tz)
#pragma unroll
      for (int ty = 0; ty < 3; ++ty) {
        TV acc = (TV)0;
#pragma unroll
        for (int tx = 0; tx < 3; ++tx) acc += q[0][dx][tx] * S[tz][ty][tx];
        T1[dx][tz][ty] = acc;
      }
  TV T2[3][3][3];
#pragma unroll
  for (int dx = 0; dx < 3; ++dx)
#pragma unroll
    for (int dy = 0; dy < 3; ++dy)
#pragma unroll
      for (int tz = 0; tz < 3; ++tz) {
        TV acc = (TV)0;
#pragma unroll
        for (int ty = 0; ty < 3; ++ty) acc += q[1][dy][ty] * T1[dx][tz][ty];
        T2[dx][dy][tz] = acc;
      }
#pragma unroll
  for (int dz = 0; dz < 3; ++dz)
#pragma unroll
    for (int dy = 0; dy < 3; ++dy)
#pragma unroll
      for (int dx = 0; dx < 3; ++dx) {
        const int o = dx + 3 * dy + 9 * dz;
        TV v;
        if (o == 13) {
          v = rs;
        } else {
          TV acc = (TV)0;
#pragma unroll
          for (int tz = 0; tz < 3; ++tz) acc += q[2][dz][tz] * T2[dx][dy][tz];
          v = acc;
        }
        o_[o * cn + C] = v;
      }
}

__device__ __forceinline__ void atomic_max_pos(double* addr, double v) {
  atomicMax(reinterpret_cast<unsigned long long*>(addr), (unsigned long long)__double_as_longlong(v));
}

// Block-wide maximum of a non-negative value, one atomic per block (all
// threads of the block must call it).
__device__ __forceinline__ void block_max_to(double* addr, double v) {
  __shared__ double red[32];
  for (int off = 16; off > 0; off >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, off));
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  if (warp == 0) {
    v = lane < (blockDim.x + 31) / 32 ? red[lane] : 0.0;
    for (int off = 16; off > 0; off >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, off));
    if (lane == 0 && v > 0.0) atomic_max_pos(addr, v);
  }
}

// Level 0: variable row sums, storage stencil slot 13, inverse diagonal, lam.
// The fixed off-diagonal sums come from setup; only node-local arithmetic
// remains (the reciprocal and the Gershgorin ratio in the compute precision).
template <typename TS, typename T>
__global__ void k_level0_update(Grid g, double tau, const double* __restrict__ sfix,
                                const double* __restrict__ offsum, const double* __restrict__ absoff,
                                const uint8_t* __restrict__ label, const int32_t* __restrict__ eidx,
                                const double* __restrict__ Aj, const double* __restrict__ ge,
                                const double* __restrict__ gc, const double* __restrict__ zeta, double s0,
                                double s1, double s2, TS* st0, TS* st1, TS* st2, T* di0, T* di1, T* di2,
                                double* __restrict__ svar, double* lam, float2* __restrict__ sd) {
  const int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t nn = g.nn;
  double gl[kNH] = {0.0, 0.0, 0.0, 0.0};
  if (n < nn) {
    const int32_t e = eidx[n];
    const uint8_t l = label[n];
    const bool act = l & kLabActive;
    double sv[3] = {0.0, 0.0, 0.0};
    if (e >= 0) {
      const double zA = zeta[e] * Aj[e];
      if (act) sv[0] = zA * ge[e];
      sv[1] = zA * ge[e];
      sv[2] = -tau * zA * gc[e];
    }
    TS* sts[3] = {st0, st1, st2};
    T* dis[3] = {di0, di1, di2};
    const double sc[3] = {s0, s1, s2};
    for (int f = 0; f < 3; ++f) {
      const double s = sfix[f * nn + n] + sv[f];
      double diag = (f == 0 && !act) ? 1.0 : s - offsum[f * nn + n];
      const double ab = absoff[f * nn + n];
      if (!(diag > 0.0)) diag = fmax(ab, 1e-300);   // keep the smoother finite on a degenerate row
      svar[f * nn + n] = sv[f];
      sts[f][13 * nn + n] = fromd<TS>(sc[f] * s);
      const T dsc = (T)(sc[f] * diag);
      dis[f][n] = (T)1 / dsc;
      // the matrix-free level 0 adds the variable diagonal to the element part;
      // it reads it with 1/diag as one pair
      if (sd) sd[f * nn + n] = make_float2((float)(T)(sc[f] * sv[f]), (float)((T)1 / dsc));
      int h = f + 1;
      if (f == 0) {
        if (!act) continue;
        h = (l & kLabAnode) ? 0 : 1;
      }
      // Gershgorin ratio in FP64: the Chebyshev interval must not depend on
      // the preconditioner precision
      gl[h] = (ab + diag) / diag;
    }
  }
  for (int h = 0; h < kNH; ++h) block_max_to(lam + h, gl[h]);
}

// Level >= 1: A = F + V into storage precision, inverse diagonal and lam.
template <typename TS, typename T, typename TV>
__global__ void k_level_combine(LevelDims d, Ptr4<const double> F, Ptr4<const TV> V, Ptr4<TS> st,
                                Ptr4<T> dinv, Ptr4<const uint8_t> mask, double sc0, double sc1, double sc2,
                                double sc3, double* lam) {
  const int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int h = blockIdx.y;
  double gl = 0.0;
  if (n < d.n) {
    const double sc = h == 0 ? sc0 : (h == 1 ? sc1 : (h == 2 ? sc2 : sc3));
    const double* __restrict__ f = pk(F.p, h);
    const TV* __restrict__ v = pk(V.p, h);
    if (std::is_same<T, float>::value) {
      // FP32 cycle: the sum of the fixed and variable parts, the scaling, the
      // diagonal and the Gershgorin sums in FP32 (the results are stored in
      // FP32 or BF16; the row sum in slot 13 adds its two parts directly)
      const float scf = (float)sc;
      float diag = 0.f, absoff = 0.f, s = 0.f;
      float as[27];   // all loads before the first store
#pragma unroll
      for (int o = 0; o < 27; ++o) as[o] = (float)f[o * d.n + n] + (float)v[o * d.n + n];
#pragma unroll
      for (int o = 0; o < 27; ++o) {
        const float a = as[o];
        pk(st.p, h)[o * d.n + n] = (TS)(scf * a);
        if (o == 13) s = a;
        else { diag -= a; absoff += fabsf(a); }
      }
      diag += s;
      if (!(diag > 0.f)) diag = fmaxf(absoff, 1e-30f);
      pk(dinv.p, h)[n] = (T)(1.0f / (scf * diag));
      if (pk(mask.p, h)[n]) gl = (double)((absoff + fabsf(diag)) / diag);
    } else {
      double diag = 0.0, absoff = 0.0, s = 0.0;
      double as[27];
#pragma unroll
      for (int o = 0; o < 27; ++o) as[o] = f[o * d.n + n] + (double)v[o * d.n + n];
#pragma unroll
      for (int o = 0; o < 27; ++o) {
        const double a = as[o];
        pk(st.p, h)[o * d.n + n] = fromd<TS>(sc * a);
        if (o == 13) s = a;
        else { diag -= a; absoff += fabs(a); }
      }
      diag += s;
      if (!(diag > 0.0)) diag = fmax(absoff, 1e-300);
      pk(dinv.p, h)[n] = fromd<T>(1.0 / (sc * diag));
      if (pk(mask.p, h)[n]) gl = (absoff + fabs(diag)) / diag;
    }
  }
  block_max_to(lam + h, gl);
}

// Dense scaled coarsest operator [n][n] (row major) from difference form.
template <typename TV>
__global__ void k_dense(LevelDims d, Ptr4<const double> F, Ptr4<const TV> V, double sc0, double sc1,
                        double sc2, double sc3, double* out) {
  const int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int h = blockIdx.y;
  if (n >= d.n) return;
  const double sc = h == 0 ? sc0 : (h == 1 ? sc1 : (h == 2 ? sc2 : sc3));
  double* A = out + (size_t)h * d.n * d.n;
  int i, j, k;
  node_ijk(d, n, i, j, k);
  for (int64_t m = 0; m < d.n; ++m) A[n * d.n + m] = 0.0;
  double diag = 0.0;
  for (int o = 0; o < 27; ++o) {
    const double a = pk(F.p, h)[o * d.n + n] + (double)pk(V.p, h)[o * d.n + n];
    if (o == 13) { diag += a; continue; }
    diag -= a;
    const int dx = o % 3 - 1, dy = (o / 3) % 3 - 1, dz = o / 9 - 1;
    const int ii = i + dx, jj = j + dy, kk = k + dz;
    if (ii < 0 || jj < 0 || kk < 0 || ii >= d.nnx || jj >= d.nny || kk >= d.nnz) continue;
    A[n * d.n + (ii + (int64_t)d.nnx * (jj + (int64_t)d.nny * kk))] = sc * a;
  }
  A[n * d.n + n] = sc * diag;
}

// Single-level hierarchy: dense scaled level-0 operator of hierarchy h from
// the fixed stencil (off-diagonals), fixed + variable row sums and the mask
// (masked-out rows/columns become identity).
__global__ void k_dense0(Grid g, const double* __restrict__ Jst, const double* __restrict__ sfix,
                         const double* __restrict__ svar, Ptr4<const uint8_t> mask, double sc0, double sc1,
                         double sc2, double* out) {
  const int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int h = blockIdx.y;
  const int64_t nn = g.nn;
  if (n >= nn) return;
  const int f = h == 0 || h == 1 ? 0 : h - 1;
  const double sc = f == 0 ? sc0 : (f == 1 ? sc1 : sc2);
  double* A = out + (size_t)h * nn * nn;
  for (int64_t m = 0; m < nn; ++m) A[n * nn + m] = 0.0;
  if (!pk(mask.p, h)[n]) {
    A[n * nn + n] = 1.0;
    return;
  }
  const int i = (int)(n % g.nnx), j = (int)((n / g.nnx) % g.nny), k = (int)(n / ((int64_t)g.nnx * g.nny));
  const double* st = Jst + (size_t)f * 27 * nn;
  double diag = sfix[f * nn + n] + svar[f * nn + n];
  for (int o = 0; o < 27; ++o) {
    if (o == 13) continue;
    const double a = st[o * nn + n];
    diag -= a;
    const int dx = o % 3 - 1, dy = (o / 3) % 3 - 1, dz = o / 9 - 1;
    const int ii = i + dx, jj = j + dy, kk = k + dz;
    if (ii < 0 || jj < 0 || kk < 0 || ii >= g.nnx || jj >= g.nny || kk >= g.nnz) continue;
    const int64_t m = ii + (int64_t)g.nnx * (jj + (int64_t)g.nny * kk);
    if (pk(mask.p, h)[m]) A[n * nn + m] = sc * a;
  }
  A[n * nn + n] = sc * diag;
}

// Coarsest-level inverse, n <= kLuMax: LU with partial pivoting of each
// hierarchy's matrix by a cluster of kLuBlocks blocks (perm[i] = the original
// row now at row i; the factors leave column by column), then the columns of
// the inverse, one warp each, by forward and backward substitution.  FP64
// throughout.
//
// Factorization: panels of kLuPanel columns, panel b in the shared memory of
// block b mod kLuBlocks, a row per thread.  Rows stay where they are; their
// positions move.  The owner factors a panel in registers (a step: pivot
// search over the warps, one division, the updates left in the panel) and
// sends the multipliers and pivots to all blocks, one cluster barrier per
// panel.  The owner of the next panel updates that one first and factors it
// while the others update the rest, so that the chain is the n pivot steps.
// An FP64 instruction of a warp occupies its scheduler's FP64 unit for 64
// clocks whatever its lanes: the rows are spread over the warps, and each
// warp forms the reciprocal itself (352 clocks).  Every entry sees the same
// operations in the same order as in the plain row-by-row elimination (a zero
// multiplier is skipped).  One block per hierarchy, all of the trailing block
// by it, took 111 us at 63 rows and 353 us at 120.  Columns per panel x blocks
// (63 / 120 rows, us): 1 x 4 93 / 219, 1 x 8 84 / 182, 2 x 4 82 / 198, 2 x 8
// 80 / 168, 4 x 4 90 / 210, 4 x 8 87 / 180, 8 x 4 109 / 241; 4 x 4 with the
// panel in one warp 104 / 267.
constexpr int kLuMax = 256;
constexpr int kLuBlocks = 8;
constexpr int kLuPanel = 2;
inline int lu_panels(int n) { return (n + kLuPanel - 1) / kLuPanel; }
inline int lu_threads(int n) { return (n + 31) / 32 * 32; }
inline size_t lu_smem(int n) {   // own columns, and three panels of multipliers
  return sizeof(double) * n * (size_t)kLuPanel * ((lu_panels(n) + kLuBlocks - 1) / kLuBlocks + 3);
}

// Row n of the dense scaled coarsest operator, from difference form.
struct DenseRows {
  LevelDims d;
  double sc[kNH];
};

// Tests of doubles on their bits: a floating-point comparison is an FP64
// instruction (20 clocks of an SM's FP64 unit per warp).
__device__ __forceinline__ bool nonzero(double v) { return (__double_as_longlong(v) << 1) != 0; }

__device__ __forceinline__ unsigned cluster_addr(const void* p, int rank) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(p);
  unsigned ra;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(rank));
  return ra;
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;\n" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;\n" ::: "memory"); }

template <typename TV>
__global__ void __cluster_dims__(kLuBlocks, 1, 1) __launch_bounds__(kLuMax)
    k_lu_factor(int n, DenseRows dr, Ptr4<const double> F, Ptr4<const TV> V, const double* __restrict__ mats,
                double* __restrict__ lu, int* __restrict__ perm) {
  constexpr int NB = kLuPanel, C = kLuBlocks;
  extern __shared__ double lu_s[];
  __shared__ int2 pivs[3][NB];               // (row, its position before) of a panel's pivots
  __shared__ double U[kLuMax / C][NB];       // the pivot rows' entries in the own columns
  // candidates of the warps for a pivot, two steps in turn: key, (row,
  // position), the row's entries in the panel
  __shared__ long long ckey[2][kLuMax / 32];
  __shared__ int2 crow[2][kLuMax / 32];
  __shared__ double cval[2][kLuMax / 32][NB];
  const int h = blockIdx.x / C, rank = blockIdx.x % C;
  const int r = threadIdx.x, lane = r & 31, warp = r >> 5, nw = blockDim.x >> 5;
  const bool row = r < n;
  const int np = (n + NB - 1) / NB;
  const int nloc = rank < np ? (np - 1 - rank) / C + 1 : 0;   // own panels
  double* A = lu_s;                                           // [own column][row]
  double* L = lu_s + (size_t)n * NB * ((np + C - 1) / C);     // [3][NB][row]
  if (row) {
    for (int l = 0; l < nloc * NB; ++l) {
      const int c = (l / NB * C + rank) * NB + l % NB;
      A[l * n + r] = mats && c < n ? mats[((size_t)h * n + r) * n + c] : 0.0;
    }
    if (!mats) {
      const double sc = pk(dr.sc, h);
      int i, j, k;
      node_ijk(dr.d, r, i, j, k);
      double a[27];
#pragma unroll
      for (int o = 0; o < 27; ++o) a[o] = pk(F.p, h)[o * dr.d.n + r] + (double)pk(V.p, h)[o * dr.d.n + r];
      auto put = [&](int c, double v) {
        const int b = c / NB;
        if (b % C == rank) A[(b / C * NB + c % NB) * n + r] = v;
      };
      double diag = 0.0;
#pragma unroll
      for (int o = 0; o < 27; ++o) {
        if (o == 13) { diag += a[o]; continue; }
        diag -= a[o];
        const int ii = i + o % 3 - 1, jj = j + (o / 3) % 3 - 1, kk = k + o / 9 - 1;
        if (ii < 0 || jj < 0 || kk < 0 || ii >= dr.d.nnx || jj >= dr.d.nny || kk >= dr.d.nnz) continue;
        put(ii + dr.d.nnx * (jj + dr.d.nny * kk), sc * a[o]);
      }
      put(r, sc * diag);
    }
  }
  int pos = r;

  // Factors panel b (this block's, up to date) and sends it to all blocks.
  auto factor = [&](int b) {
    double* P = A + (size_t)(b / C * NB) * n;
    int at = row ? pos : -1;
    double v[NB];
#pragma unroll
    for (int m = 0; m < NB; ++m) v[m] = row ? P[m * n + r] : 0.0;
#pragma unroll
    for (int m = 0; m < NB; ++m) {
      const int k = b * NB + m;
      if (k >= n) continue;   // uniform
      // magnitudes compared as integers (the bits of non-negative doubles are
      // ordered; a NaN is never chosen), the row that comes first of equal ones
      long long key = __double_as_longlong(v[m]) & 0x7fffffffffffffffll;
      if (key > 0x7ff0000000000000ll) key = -1;
      const bool cand = at >= k;
      const int hi = cand ? (int)(key >> 32) : -2;
      const int mh = __reduce_max_sync(0xffffffffu, hi);
      const unsigned lo = cand && hi == mh ? (unsigned)key : 0u;
      const unsigned ml = __reduce_max_sync(0xffffffffu, lo);
      const bool top = cand && hi == mh && lo == ml;
      const int mp = (int)__reduce_min_sync(0xffffffffu, top ? (unsigned)at : 0xffffu);
      if (mh == -2 ? lane == 0 : top && at == mp) {
        ckey[m & 1][warp] = mh == -2 ? -2 : key;
        crow[m & 1][warp] = make_int2(r, mp);
#pragma unroll
        for (int q = m; q < NB; ++q) cval[m & 1][warp][q] = v[q];
      }
      __syncthreads();
      long long best = ckey[m & 1][0];
      int2 bw = crow[m & 1][0];
      int wb = 0;
#pragma unroll 1
      for (int w = 1; w < nw; ++w) {
        const long long kw = ckey[m & 1][w];
        const int2 cw = crow[m & 1][w];
        if (kw > best || (kw == best && cw.y < bw.y)) { best = kw; bw = cw; wb = w; }
      }
      const double* u = cval[m & 1][wb];
      const double d = u[m];
      const double id = nonzero(d) ? 1.0 / d : 0.0;
      if (r < C)
        asm volatile("st.shared::cluster.v2.s32 [%0], {%1, %2};" ::"r"(cluster_addr(&pivs[b % 3][m], r)), "r"(bw.x),
                     "r"(bw.y) : "memory");
      if (at == bw.y) at = k;
      else if (at == k) at = bw.y;
      if (at > k) {
        v[m] *= id;
        if (nonzero(v[m])) {
#pragma unroll
          for (int q = m + 1; q < NB; ++q) v[q] = fma(-v[m], u[q], v[q]);
        }
      }
      __syncwarp();
    }
    if (row) {
#pragma unroll
      for (int m = 0; m < NB; ++m) {
        P[m * n + r] = v[m];
        // a multiplier where the row's position is below the column's pivot
        const double l = at > b * NB + m ? v[m] : 0.0;
        double* dst = L + ((size_t)(b % 3) * NB + m) * n + r;
#pragma unroll
        for (int q = 0; q < C; ++q)
          asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(cluster_addr(dst, q)), "d"(l) : "memory");
      }
    }
  };

  cluster_arrive();   // every block has started and written its columns
  cluster_wait();
  if (rank == 0) factor(0);
  cluster_arrive();
#pragma unroll 1
  for (int b = 0; b < np; ++b) {
    cluster_wait();
    const double* Lb = L + (size_t)(b % 3) * NB * n;
    double l[NB];
    bool piv = false;
#pragma unroll
    for (int t = 0; t < NB; ++t) {
      l[t] = row ? Lb[t * n + r] : 0.0;
      if (b * NB + t >= n) continue;
      const int2 p = pivs[b % 3][t];
      if (r == p.x) {
        pos = b * NB + t;
        piv = true;
      } else if (pos == b * NB + t) {
        pos = p.y;
      }
    }
    if (b + 1 == np) break;
    // own columns after panel b; the first panel of them may be the next one
    const int c0 = NB * (b < rank ? 0 : (b - rank) / C + 1), c1 = nloc * NB;
    // the pivot rows' entries, a column per lane of the first warp
    if (r < 32) {
      for (int c = c0 + lane; c < c1; c += 32) {
        double u[NB];
#pragma unroll
        for (int t = 0; t < NB; ++t) u[t] = A[c * n + pivs[b % 3][t].x];
#pragma unroll
        for (int t = 0; t < NB; ++t) {
          const int p = pivs[b % 3][t].x;
#pragma unroll
          for (int q = 0; q < t; ++q) {
            const double m = Lb[q * n + p];
            if (nonzero(m)) u[t] = fma(-m, u[q], u[t]);
          }
          A[c * n + p] = u[t];
          U[c][t] = u[t];
        }
      }
    }
    __syncthreads();
    // every other row by its thread
    bool on[NB], any[NB];
#pragma unroll
    for (int t = 0; t < NB; ++t) {
      on[t] = !piv && nonzero(l[t]);
      any[t] = __any_sync(0xffffffffu, on[t]);
    }
    auto update = [&](int e0, int e1) {
#pragma unroll 4
      for (int c = e0; c < e1; ++c) {
        if (!row) break;
        double w = A[c * n + r];
#pragma unroll
        for (int t = 0; t < NB; ++t)
          if (any[t]) {
            const double x = fma(-l[t], U[c][t], w);
            w = on[t] ? x : w;
          }
        if (!piv) A[c * n + r] = w;
      }
    };
    const bool mine = (b + 1) % C == rank;
    if (mine) {
      update(c0, c0 + NB);
      factor(b + 1);
      // (buffers of three panels: this block's work on panel b below is done
      // when it arrives for panel b + 2)
      cluster_arrive();
      update(c0 + NB, c1);
      // the pivot rows' entries of the next step are read and U is written
      // by the first warp
      __syncthreads();
    } else {
      update(c0, c1);
      cluster_arrive();
    }
  }
  double* G = lu + (size_t)h * n * n;
  if (row) {
    for (int l = 0; l < nloc * NB; ++l) {
      const int c = (l / NB * C + rank) * NB + l % NB;
      if (c < n) G[(size_t)c * n + pos] = A[l * n + r];
    }
    if (rank == 0) perm[(size_t)h * n + pos] = r;
  }
}

// x / d from r = 1 / d (correctly rounded): one Newton correction of the
// quotient by its exact remainder gives the correctly rounded quotient
// (Markstein 1990) in three FP64 operations.
__device__ __forceinline__ double div_by(double x, double d, double r) {
  const double q = x * r;
  return finite_bits(q) && finite_bits(r) ? fma(fma(-q, d, x), r, q) : x / d;
}

// Columns of the inverse, a column per warp, its entries in registers (entry
// lane + 32 t in x[t]).  A substitution step is a chain of a shuffle, (going
// back) a quotient and an update; the factors' columns are loaded a batch
// ahead, from the caches.  With the column in shared memory and the factors
// staged there 50 us at 63 rows and 105 us at 120; now 32 and 68.
constexpr int kLuCols = 4;
template <int NT>
__global__ void __launch_bounds__(32 * kLuCols) k_lu_inverse(int n, const double* __restrict__ lu,
                                                             const int* __restrict__ perm, double* __restrict__ inv) {
  constexpr int B = NT > 4 ? 2 : 4;           // factor columns of a batch
  __shared__ double dg[32 * NT], rd[32 * NT];   // the diagonal and its reciprocals
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int j = blockIdx.x * kLuCols + warp;
  const double* G = lu + (size_t)blockIdx.y * n * n;   // [column][row]
  for (int r = threadIdx.x; r < n; r += blockDim.x) {
    const double d = G[(size_t)r * n + r];
    dg[r] = d;
    rd[r] = d != 0.0 ? 1.0 / d : 0.0;
  }
  __syncthreads();
  if (j >= n) return;   // per warp
  const int* P = perm + (size_t)blockIdx.y * n;
  // x = P e_j, then L y = x (unit lower), then U x = y
  double x[NT];
  int k0 = n;
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    const int i = lane + 32 * t;
    const bool one = i < n && P[i] == j;
    x[t] = one ? 1.0 : 0.0;
    if (one) k0 = i;
  }
  k0 = (int)__reduce_min_sync(0xffffffffu, (unsigned)k0);
  double c[B][NT], cn[B][NT];
  auto load = [&](int k, double (&d)[B][NT]) {   // factor columns k .. k + B - 1
#pragma unroll
    for (int q = 0; q < B; ++q)
#pragma unroll
      for (int t = 0; t < NT; ++t) {
        const int i = lane + 32 * t;
        d[q][t] = k + q >= 0 && k + q < n && i < n ? __ldg(G + (size_t)(k + q) * n + i) : 0.0;
      }
  };
  auto next = [&] {
#pragma unroll
    for (int q = 0; q < B; ++q)
#pragma unroll
      for (int t = 0; t < NT; ++t) c[q][t] = cn[q][t];
  };
  const int kb = k0 / B * B;   // x is zero above its unit entry
  load(kb, cn);
#pragma unroll
  for (int tb = 0; tb < NT; ++tb) {
#pragma unroll 1
    for (int k = max(kb, 32 * tb); k < min(n, 32 * tb + 32); k += B) {
      next();
      load(k + B, cn);
#pragma unroll
      for (int q = 0; q < B; ++q) {
        const double xk = __shfl_sync(0xffffffffu, x[tb], (k + q) & 31);
        if (nonzero(xk)) {   // uniform
          const double v = fma(-c[q][tb], xk, x[tb]);
          if (lane > ((k + q) & 31)) x[tb] = v;
#pragma unroll
          for (int t = tb + 1; t < NT; ++t) x[t] = fma(-c[q][t], xk, x[t]);
        }
      }
    }
  }
  load((n - 1) / B * B, cn);
#pragma unroll
  for (int tb = NT - 1; tb >= 0; --tb) {
#pragma unroll 1
    for (int k = (min(n, 32 * tb + 32) - 1) / B * B; k >= 32 * tb; k -= B) {
      next();
      load(k - B, cn);
#pragma unroll
      for (int q = B - 1; q >= 0; --q) {
        if (k + q >= n) continue;
        const double d = dg[k + q];
        double xk = __shfl_sync(0xffffffffu, x[tb], (k + q) & 31);
        xk = nonzero(d) ? div_by(xk, d, rd[k + q]) : 0.0;
        if (lane == ((k + q) & 31)) x[tb] = xk;
        if (nonzero(xk)) {   // uniform
          const double v = fma(-c[q][tb], xk, x[tb]);
          if (lane < ((k + q) & 31)) x[tb] = v;
#pragma unroll
          for (int t = 0; t < tb; ++t) x[t] = fma(-c[q][t], xk, x[t]);
        }
      }
    }
  }
  double* Inv = inv + (size_t)blockIdx.y * n * n;
#pragma unroll
  for (int t = 0; t < NT; ++t)
    if (lane + 32 * t < n) Inv[(size_t)(lane + 32 * t) * n + j] = x[t];
}

__global__ void k_gauss_jordan(int n, double* mats, double* work) {
  double* A = mats + (size_t)blockIdx.x * n * n;
  double* Inv = work + (size_t)blockIdx.x * n * n;
  __shared__ int piv;
  __shared__ double pval;
  for (int r = threadIdx.x >> 5; r < n; r += blockDim.x >> 5)
    for (int cc = threadIdx.x & 31; cc < n; cc += 32) Inv[(size_t)r * n + cc] = r == cc ? 1.0 : 0.0;
  __syncthreads();
  for (int col = 0; col < n; ++col) {
    if (threadIdx.x == 0) {
      int p = col;
      double best = fabs(A[(size_t)col * n + col]);
      for (int r = col + 1; r < n; ++r) {
        const double v = fabs(A[(size_t)r * n + col]);
        if (v > best) { best = v; p = r; }
      }
      piv = p;
      pval = A[(size_t)p * n + col];
    }
    __syncthreads();
    const int p = piv;
    if (p != col)
      for (int t = threadIdx.x; t < n; t += blockDim.x) {
        double a = A[(size_t)col * n + t]; A[(size_t)col * n + t] = A[(size_t)p * n + t]; A[(size_t)p * n + t] = a;
        double b = Inv[(size_t)col * n + t]; Inv[(size_t)col * n + t] = Inv[(size_t)p * n + t]; Inv[(size_t)p * n + t] = b;
      }
    __syncthreads();
    const double inv_p = pval != 0.0 ? 1.0 / pval : 0.0;
    for (int t = threadIdx.x; t < n; t += blockDim.x) {
      A[(size_t)col * n + t] *= inv_p;
      Inv[(size_t)col * n + t] *= inv_p;
    }
    __syncthreads();
    // rows over warps, columns over lanes (no 64-bit index division)
    for (int r = threadIdx.x >> 5; r < n; r += blockDim.x >> 5) {
      if (r == col) continue;
      const double f = A[(size_t)r * n + col];
      if (f == 0.0) continue;
      for (int cc = threadIdx.x & 31; cc < n; cc += 32) {
        if (cc != col) A[(size_t)r * n + cc] -= f * A[(size_t)col * n + cc];
        Inv[(size_t)r * n + cc] -= f * Inv[(size_t)col * n + cc];
      }
    }
    __syncthreads();
    for (int r = threadIdx.x; r < n; r += blockDim.x)
      if (r != col) A[(size_t)r * n + col] = 0.0;
    __syncthreads();
  }
  for (int64_t t = threadIdx.x; t < (int64_t)n * n; t += blockDim.x) A[t] = Inv[t];
}

// ---------------------------------------------------------------- cycle kernels
template <typename TS, typename T>
struct LvlPtrs {
  const TS* st[kNH];
  const T* dinv[kNH];
  const uint8_t* mask[kNH];
  const T* x[kNH];
  T* xo[kNH];
  const T* b[kNH];
  T* r[kNH];
  T* d[kNH];
};

// Stencil kernels: kNpt rows per thread, blockDim apart (each load
// instruction stays coalesced), and the loads of one z-plane of the stencil
// (9 coefficients and 9 neighbour values per row) issued before their
// updates.  The kernels are bound by memory latency unless enough loads are
// in flight; on cube128 level 0 one row per thread with plane-batched loads
// was fastest (two rows per thread with per-offset loads came close, four or
// more were slower from register pressure).
constexpr int kNpt = 1;

// ax[q] = (A x)_{n[q]} in difference form, for the rows with on[q]:
// ax = s_13 x_n + sum_{o != 13} s_o (x_{n+off(o)} - x_n).  Every row takes
// the same unchecked path: the stencils hold exact zeros in the slots of
// neighbours outside the grid, and the x vectors carry zeroed guard zones
// (see alloc_x), so the loads of boundary rows stay in bounds and such a
// slot adds fma(0, finite, acc) = acc.  Indices are 32-bit (every level has
// fewer than 2^31/27 nodes).
template <typename TS, typename T>
__device__ __forceinline__ void stencil_rows(const TS* __restrict__ st, const T* __restrict__ x, const LevelDims& dd,
                                             const int (&n)[kNpt], const bool (&on)[kNpt], T (&ax)[kNpt]) {
  const int N = (int)dd.n;
  const int sy = dd.nnx, sz = dd.nnx * dd.nny;
  T xn[kNpt];
#pragma unroll
  for (int q = 0; q < kNpt; ++q) {
    xn[q] = on[q] ? x[n[q]] : (T)0;
    ax[q] = on[q] ? (T)tof(st[13 * N + n[q]]) * xn[q] : (T)0;
  }
  // one z-plane of the stencil at a time: all of its loads first, then the
  // updates, summed in offset order
#pragma unroll
  for (int pz = 0; pz < 3; ++pz) {
    TS sv[9][kNpt];
    T xv[9][kNpt];
#pragma unroll
    for (int t = 0; t < 9; ++t) {
      const int o = 9 * pz + t;
      if (o == 13) continue;
      const int off = (o % 3 - 1) + ((o / 3) % 3 - 1) * sy + (o / 9 - 1) * sz;
#pragma unroll
      for (int q = 0; q < kNpt; ++q)
        if (on[q]) {
          sv[t][q] = st[o * N + n[q]];
          xv[t][q] = x[n[q] + off];
        }
    }
#pragma unroll
    for (int t = 0; t < 9; ++t) {
      if (9 * pz + t == 13) continue;
#pragma unroll
      for (int q = 0; q < kNpt; ++q)
        if (on[q]) ax[q] = fma((T)tof(sv[t][q]), xv[t][q] - xn[q], ax[q]);
    }
  }
}

// Chebyshev coefficients, on the device (so that captured graphs stay valid
// across linearizations): for level l, step s and hierarchy h,
// tab[((l kMaxDeg + s) 3 + j) kNH + h], j = 0: c0, 1: ca, 2: cb.  Step 0:
// d = c0 z; later steps: d = ca d + cb z, with z = D^-1 (b - A x).
template <typename T>
__device__ __forceinline__ T cheb_at(const T* tab, int level, int step, int j, int h) {
  return tab[((level * kMaxDeg + step) * 3 + j) * kNH + h];
}

// Rows of this thread: n[q] = base + q blockDim + tid with base the first
// row of block blo[h] + blockIdx.x (the launch covers only the blocks that
// hold rows of the hierarchy's mask).  ld[q]: the row is in range, so its
// loads are issued at once -- every array of a level is finite at every
// node, and a row outside the mask computes a value that is never stored;
// on[q]: the row is also inside the mask and its results are written.
// all_on: the hierarchy's mask is all ones (phi_e, c_e at every level), no
// mask load.
__device__ __forceinline__ void stencil_nodes(int N, const uint8_t* __restrict__ mask, bool all_on, int blo,
                                              int (&n)[kNpt], bool (&ld)[kNpt], bool (&on)[kNpt]) {
  const int base = (blo + (int)blockIdx.x) * (blockDim.x * kNpt) + threadIdx.x;
#pragma unroll
  for (int q = 0; q < kNpt; ++q) {
    n[q] = base + q * blockDim.x;
    ld[q] = n[q] < N;
    on[q] = ld[q] && (all_on || mask[n[q]]);
  }
}

// Block ranges of the listed hierarchies for one launch.
struct BRange {
  int lo[kNH];
  int cnt[kNH];
};

// One Chebyshev step, x_out = x + d.
template <typename TS, typename T>
__global__ void __launch_bounds__(256) k_cheb(LevelDims dd, LvlPtrs<TS, T> P, HList hl, BRange br,
                                              const T* __restrict__ ctab, int level, int step, int first) {
  const int hi = blockIdx.y;
  const int h = pk(hl.h, hi);
  if ((int)blockIdx.x >= pk(br.cnt, h)) return;
  int n[kNpt];
  bool ld[kNpt], on[kNpt];
  stencil_nodes((int)dd.n, pk(P.mask, h), h >= 2, pk(br.lo, h), n, ld, on);
  const T* __restrict__ b = pk(P.b, h);
  const T* __restrict__ dinv = pk(P.dinv, h);
  const T* __restrict__ x = pk(P.x, h);
  T* __restrict__ d = pk(P.d, h);
  T* __restrict__ xo = pk(P.xo, h);
  // the row's own values, loaded before the stencil so that their latency
  // overlaps with the stencil loads
  T bq[kNpt], dq[kNpt], iq[kNpt];
#pragma unroll
  for (int q = 0; q < kNpt; ++q) {
    bq[q] = ld[q] ? b[n[q]] : (T)0;
    iq[q] = ld[q] ? dinv[n[q]] : (T)0;
    dq[q] = (ld[q] && step != 0) ? d[n[q]] : (T)0;
  }
  T ax[kNpt];
  if (!first) stencil_rows<TS, T>(pk(P.st, h), x, dd, n, ld, ax);
  const T c0 = cheb_at(ctab, level, step, 0, h), ca = cheb_at(ctab, level, step, 1, h),
          cb = cheb_at(ctab, level, step, 2, h);
#pragma unroll
  for (int q = 0; q < kNpt; ++q) {
    if (!on[q]) continue;
    const int m = n[q];
    T res = bq[q];
    if (!first) res -= ax[q];
    const T z = iq[q] * res;
    const T dn = step == 0 ? c0 * z : fma(cb, z, ca * dq[q]);   // contraction as in k_tail
    d[m] = dn;
    xo[m] = (first ? (T)0 : x[m]) + dn;
  }
}

template <typename TS, typename T>
__global__ void __launch_bounds__(256) k_resid(LevelDims dd, LvlPtrs<TS, T> P, HList hl, BRange br) {
  const int h = pk(hl.h, blockIdx.y);
  if ((int)blockIdx.x >= pk(br.cnt, h)) return;
  int n[kNpt];
  bool ld[kNpt], on[kNpt];   // level-0 phi_s hierarchies share r: never write masked-out nodes
  stencil_nodes((int)dd.n, pk(P.mask, h), h >= 2, pk(br.lo, h), n, ld, on);
  T ax[kNpt];
  stencil_rows<TS, T>(pk(P.st, h), pk(P.x, h), dd, n, ld, ax);
  const T* __restrict__ b = pk(P.b, h);
  T* __restrict__ r = pk(P.r, h);
#pragma unroll
  for (int q = 0; q < kNpt; ++q)
    if (on[q]) r[n[q]] = b[n[q]] - ax[q];
}


// Node planes of the listed hierarchies that hold rows of their masks.
struct PRange {
  int lo[kNH];
  int cnt[kNH];
};

// Full-weighting restriction (P^T r)_C over the fine nodes of the mask.
// The phi_e / c_e masks are all ones (no mask load); elsewhere a masked-out
// residual is selected away (never multiplied: it may hold stale values).
// By planes: a block's coarse plane K (and with it the z support) is uniform,
// one integer division per node is left; absent support nodes of an axis get
// weight 0 on a node of the plane (acc + 0 r = acc; the support is summed in
// increasing node order).  Many planes of fewer than 128 nodes share a block,
// one per threadIdx.y (see for_planes).
template <typename T>
__global__ void __launch_bounds__(256) k_restrict(LevelDims fd, LevelDims cd, Xfer1 X, Ptr4<const T> fr,
                                                  Ptr4<const uint8_t> fm, Ptr4<T> cb, HList hl, PRange pr) {
  const int h = pk(hl.h, blockIdx.z);
  const int p = (int)(blockIdx.y * blockDim.y + threadIdx.y);
  if (p >= pk(pr.cnt, h)) return;
  const int K = pk(pr.lo, h) + p;
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= cd.nnx * cd.nny) return;
  const int J = q / cd.nnx, I = q - J * cd.nnx;
  const T* __restrict__ r = pk(fr.p, h);
  const uint8_t* __restrict__ m = pk(fm.p, h);
  const bool all_on = h >= 2;
  int fx[3], fy[3];
  T wx[3], wy[3];
#pragma unroll
  for (int t = 0; t < 3; ++t) {
    fx[t] = sup_of<T>(X.a[0], I, t, wx[t]);
    if (fx[t] < 0) { fx[t] = 0; wx[t] = (T)0; }
    fy[t] = sup_of<T>(X.a[1], J, t, wy[t]);
    if (fy[t] < 0) { fy[t] = 0; wy[t] = (T)0; }
    fy[t] *= fd.nnx;
  }
  T acc = 0;
#pragma unroll
  for (int tz = 0; tz < 3; ++tz) {
    T wz;
    const int fk = sup_of<T>(X.a[2], K, tz, wz);
    if (fk < 0) continue;   // uniform
    const int o = fd.nnx * fd.nny * fk;
    T v[9];
    bool on[9];
#pragma unroll
    for (int t = 0; t < 9; ++t) {
      const int f = o + fy[t / 3] + fx[t % 3];
      v[t] = r[f];
      on[t] = all_on || m[f];
    }
#pragma unroll
    for (int t = 0; t < 9; ++t) acc += on[t] && wx[t % 3] * wy[t / 3] != (T)0 ? wx[t % 3] * wy[t / 3] * wz * v[t] : (T)0;
  }
  pk(cb.p, h)[K * (cd.nnx * cd.nny) + q] = acc;
}

// Prolongation by planes, as k_restrict.
template <typename T>
__global__ void __launch_bounds__(256) k_prolong(LevelDims fd, LevelDims cd, Xfer1 X, Ptr4<const T> cx_,
                                                 Ptr4<const uint8_t> fm, Ptr4<T> fx, HList hl, PRange pr) {
  const int h = pk(hl.h, blockIdx.z);
  const int y = (int)(blockIdx.y * blockDim.y + threadIdx.y);
  if (y >= pk(pr.cnt, h)) return;
  const int k = pk(pr.lo, h) + y;
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= fd.nnx * fd.nny) return;
  const int j = q / fd.nnx, i = q - j * fd.nnx;
  const int f = k * (fd.nnx * fd.nny) + q;
  // the mask gates only the write: the interpolation's loads do not wait on it
  // (phi_e / c_e masks are all ones)
  const bool on = h >= 2 || pk(fm.p, h)[f];
  const T xf = pk(fx.p, h)[f];
  const T* __restrict__ cx = pk(cx_.p, h);
  int px[2], py[2];
  T wx[2], wy[2];
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    px[t] = par_of<T>(X.a[0], i, t, wx[t]);
    if (px[t] < 0) { px[t] = 0; wx[t] = (T)0; }
    py[t] = par_of<T>(X.a[1], j, t, wy[t]);
    if (py[t] < 0) { py[t] = 0; wy[t] = (T)0; }
    py[t] *= cd.nnx;
  }
  T acc = 0;
#pragma unroll
  for (int c3 = 0; c3 < 2; ++c3) {
    T wz;
    const int pz = par_of<T>(X.a[2], k, c3, wz);
    if (pz < 0) continue;   // uniform
    const T* __restrict__ p = cx + pz * (cd.nnx * cd.nny);
    T v[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) v[t] = p[py[t >> 1] + px[t & 1]];
#pragma unroll
    for (int t = 0; t < 4; ++t) acc += wx[t & 1] * wy[t >> 1] * wz * v[t];
  }
  if (on) pk(fx.p, h)[f] = xf + acc;
}

// x = A^-1 b at the coarsest level (dense FP64 inverse): one warp per row,
// lanes over the columns, a fixed-order warp reduction.
constexpr int kCoarseWarps = 8;
template <typename T>
__device__ __forceinline__ double coarse_row(int n, const double* __restrict__ A, const T* b, int lane) {
  double acc = 0.0;
  for (int cidx = lane; cidx < n; cidx += 32) acc += A[cidx] * (double)b[cidx];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  return acc;
}
template <typename T>
__global__ void __launch_bounds__(32 * kCoarseWarps) k_coarse_solve(int n, const double* __restrict__ inv,
                                                                    Ptr4<const T> b, Ptr4<const uint8_t> mask,
                                                                    Ptr4<T> x, HList hl) {
  const int h = pk(hl.h, blockIdx.y);
  const int lane = threadIdx.x & 31;
  const int r = blockIdx.x * kCoarseWarps + (threadIdx.x >> 5);
  if (r >= n) return;   // per warp
  const double acc = coarse_row<T>(n, inv + (size_t)h * n * n + (size_t)r * n, pk(b.p, h), lane);
  if (lane == 0 && pk(mask.p, h)[r]) pk(x.p, h)[r] = (T)acc;   // masked-out rows are never read (and may be shared)
}

// ---------------------------------------------------------------- coarse tail
// The V-cycle from level l0 down to the coarsest level and back up to l0 in
// one launch, one thread-block cluster per hierarchy.  Launched level by
// level, the small levels are bound by latency: 7 dependent launches per
// level, each waiting on several rounds of L2 loads.  Here every vector of
// the tail lives in shared memory: rows are owned by thread (at most one per
// thread and level; contiguous chunks of rows per block), a thread keeps its
// row's 27 coefficients, b, 1/diag, d and x in registers over the level's
// steps and stores x into the shared memory of every block that owns a
// neighbour row (the residual: of the blocks that own a parent row; the
// final x: a child row), with one cluster barrier per step.  A level of at
// most kTailThreads rows runs on the first block alone (block barriers),
// unless a coarser one takes more blocks (tail_blocks); the coarsest dense
// solve, FP64 and bound by the FP64 rate of an SM, is spread over the
// cluster.  Only the x of level l0 goes back to global memory.  Per row the
// arithmetic, its order and its contractions are those of k_cheb, k_resid,
// k_restrict, k_prolong and k_coarse_solve: the results are bit-identical to
// the level-by-level cycle's.
constexpr int kTailThreads = 512;
constexpr int kTailMaxCluster = 16;
// Rows per block before a level takes another block of the cluster: one per
// thread in FP32; in FP64 the stencil is bound by the FP64 rate of the SM
// (27 clocks per row and step).
template <typename T>
constexpr int kTailRows = kTailThreads;
template <>
constexpr int kTailRows<double> = 128;
constexpr size_t kTailMaxSmem = 216 * 1024;   // dynamic; the static part is under 8 KB

struct TailLevel {
  LevelDims d;
  Xfer1 X;                     // towards the next level
  int oA, oB, ob;              // shared offsets (elements): x buffers (at node 0, inside their guards), own b
  int lo[kNH], hi[kNH];        // row range of each hierarchy's mask
  int nr[kNH];                 // blocks that own rows, not fewer than on a coarser level (tail_blocks)
  const void* st[kNH];
  const void* dinv[kNH];
  const uint8_t* mask[kNH];
};

struct TailArgs {
  int nl;                      // levels of the tail
  int l0;                      // multigrid level of lev[0] (Chebyshev table row)
  int deg, cs;                 // Chebyshev degree, blocks per cluster
  int len;                     // shared elements
  int h[kNH];                  // hierarchy of each cluster
  const void* ctab;
  const double* inv;           // coarsest inverses [kNH][n][n]
  void* b[kNH];                // right-hand side and result of lev[0]
  void* x[kNH];
  TailIO io;                   // whole preconditioner application (see TailIO)
  TailLevel lev[kMaxLevels];
};

// A level as its cluster uses it (copied to shared memory once: the kernel
// parameters of a level are cold in the constant cache at its first use).
struct TailLv {
  const void* st;
  const void* dinv;
  const uint8_t* mask;
  LevelDims d;
  Xfer1 X;
  int lo, rows, chunk, nr;     // first row, rows, rows per block, blocks that own rows
  int oA, oB, ob;
  float rch, rsx, rsxy;        // 1 / chunk, 1 / nnx, 1 / (nnx nny)
};

__device__ __forceinline__ void cluster_barrier() {
  // not .aligned: the rows' branches may leave a warp's lanes unconverged
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;\n" ::: "memory");
}

// a / b for 0 <= a < 2^14 and 1 <= b < 2^14, rb = 1.0f / b: a + 1/2 is at
// least 1/(2 b) of the quotient away from an integer, far above the rounding
// of the FP32 product (an integer division is a chain of ~100 clocks).
__device__ __forceinline__ int small_div(int a, float rb) { return (int)(((float)a + 0.5f) * rb); }

// Block that owns row n of level L (n clamped to the level's rows).
__device__ __forceinline__ int tail_owner(const TailLv& L, int n) {
  if (L.nr == 1) return 0;
  const int i = n - L.lo;
  return small_div(i < 0 ? 0 : (i >= L.rows ? L.rows - 1 : i), L.rch);
}

__device__ __forceinline__ void tail_ijk(const TailLv& L, int n, int (&id)[3]) {
  id[2] = small_div(n, L.rsxy);
  const int r = n - id[2] * (L.d.nnx * L.d.nny);
  id[1] = small_div(r, L.rsx);
  id[0] = r - id[1] * L.d.nnx;
}

// The transfers of k_restrict and k_prolong for one row, the axes' entries
// formed once, absent entries as weight 0 on an index inside the level.
template <typename T>
__device__ __forceinline__ T tail_restrict(const TailLv& F, const TailLv& C, const T* r, int c) {
  int id[3];
  tail_ijk(C, c, id);
  int f[3][3];
  T w[3][3];
  const int str[3] = {1, F.d.nnx, F.d.nnx * F.d.nny};
#pragma unroll
  for (int ax = 0; ax < 3; ++ax) {
    const Axis1 A = F.X.a[ax];
#pragma unroll
    for (int t = 0; t < 3; ++t) {
      const int s = sup_of<T>(A, id[ax], t, w[ax][t]);
      if (s < 0) w[ax][t] = (T)0;
      f[ax][t] = (s < 0 ? 0 : s) * str[ax];
    }
  }
  T acc = 0;
#pragma unroll
  for (int tz = 0; tz < 3; ++tz)
#pragma unroll
    for (int ty = 0; ty < 3; ++ty) {
      const T wyz = w[1][ty] * w[2][tz];
      const int o = f[1][ty] + f[2][tz];
#pragma unroll
      for (int tx = 0; tx < 3; ++tx) acc += w[0][tx] * wyz * r[o + f[0][tx]];
    }
  return acc;
}

template <typename T>
__device__ __forceinline__ T tail_prolong(const TailLv& F, const TailLv& C, const T* x, const int (&id)[3]) {
  int p[3][2];
  T w[3][2];
  const int str[3] = {1, C.d.nnx, C.d.nnx * C.d.nny};
#pragma unroll
  for (int ax = 0; ax < 3; ++ax) {
    const Axis1 A = F.X.a[ax];
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const int s = par_of<T>(A, id[ax], t, w[ax][t]);
      if (s < 0) w[ax][t] = (T)0;
      p[ax][t] = (s < 0 ? 0 : s) * str[ax];
    }
  }
  T acc = 0;
#pragma unroll
  for (int c3 = 0; c3 < 2; ++c3)
#pragma unroll
    for (int c2 = 0; c2 < 2; ++c2) {
      const T wyz = w[1][c2] * w[2][c3];
      const int o = p[1][c2] + p[2][c3];
#pragma unroll
      for (int c1 = 0; c1 < 2; ++c1) acc += w[0][c1] * wyz * x[o + p[0][c1]];
    }
  return acc;
}

// v into entry `off` of the shared memory of blocks r0 .. r1 of the cluster.
template <typename T>
__device__ __forceinline__ void tail_put(T* sm, int off, int r0, int r1, T v) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(sm + off);
  for (int r = r0; r <= r1; ++r) {
    unsigned ra;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(r));
    if constexpr (sizeof(T) == 4)
      asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(ra), "f"(v) : "memory");
    else
      asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(ra), "d"(v) : "memory");
  }
}

// The 27 coefficients of row n, and (A x)_n in difference form summed in
// offset order (as stencil_rows), x in shared memory.
template <typename TS, typename T>
__device__ __forceinline__ void row_coef(const void* st, int N, int n, T (&c)[27]) {
  const TS* p = static_cast<const TS*>(st);
#pragma unroll
  for (int o = 0; o < 27; ++o) c[o] = (T)tof(__ldg(p + o * N + n));
}
template <typename T>
__device__ __forceinline__ T row_apply(const T (&c)[27], const T* x, int sy, int sz, int n, T xn) {
  T ax = fma(c[0], x[n - 1 - sy - sz] - xn, c[13] * xn);
#pragma unroll
  for (int o = 1; o < 27; ++o)
    if (o != 13) ax += c[o] * (x[n + (o % 3 - 1) + ((o / 3) % 3 - 1) * sy + (o / 9 - 1) * sz] - xn);
  return ax;
}

// TS0: storage of lev[0] (multigrid level 0 keeps FP32 stencils under the
// BF16 option), TS: of the levels below.  One loop visits the levels down
// and up, so that every piece of code appears once: instruction fetch of
// code that a launch executes once costs more than its arithmetic.  Measured
// (clocks of one launch at 2,025 rows, 3 levels, 4 blocks per cluster): 40 k
// = 20 us, of which a step (27 shared loads, 8 k clocks in all) plus its
// barrier (0.2 k in one block, 0.9-1.9 k in a cluster of 4-16) take half,
// the first loads of each level most of the rest; with the vectors in global
// memory and global loads of the transfer tables 33 us, launched level by
// level (17 launches) 70 us.  FP64 is bound by the FP64 rate of the SMs.
template <typename TS0, typename TS, typename T>
__global__ void __launch_bounds__(kTailThreads, 1) k_tail(const __grid_constant__ TailArgs a) {
  extern __shared__ __align__(16) unsigned char tail_smem[];
  __shared__ TailLv lv[kMaxLevels];
  __shared__ T ch[kMaxLevels * kMaxDeg * 3];
  T* sm = reinterpret_cast<T*>(tail_smem);
  const int h = a.h[blockIdx.x / a.cs];
  const int rank = blockIdx.x % a.cs;
  const int tid = threadIdx.x;
  const bool all_on = h >= 2;
  for (int i = tid; i < a.len; i += kTailThreads) sm[i] = (T)0;
  if (tid < a.nl) {
    const TailLevel& L = a.lev[tid];
    TailLv v;
    v.st = L.st[h];
    v.dinv = L.dinv[h];
    v.mask = L.mask[h];
    v.d = L.d;
    v.X = L.X;
    v.lo = L.lo[h];
    v.rows = L.hi[h] - L.lo[h];
    v.nr = L.nr[h];
    v.chunk = (v.rows + v.nr - 1) / v.nr;
    v.oA = L.oA;
    v.oB = L.oB;
    v.ob = L.ob;
    v.rch = 1.0f / (float)max(1, v.chunk);
    v.rsx = 1.0f / (float)v.d.nnx;
    v.rsxy = 1.0f / (float)(v.d.nnx * v.d.nny);
    lv[tid] = v;
  }
  const T* __restrict__ ctab = static_cast<const T*>(a.ctab);
  for (int i = tid; i < a.nl * a.deg * 3; i += kTailThreads)
    ch[i] = cheb_at(ctab, a.l0 + i / (3 * a.deg), i / 3 % a.deg, i % 3, h);
  __syncthreads();
  T io_w = (T)0;
  if (a.io.on) {
    const int f = h < 2 ? 0 : h - 1;
    if constexpr (sizeof(T) == sizeof(float)) {
      __shared__ float w;
      if (tid == 0) w = (float)(a.io.iwf[f] * a.io.sc[f]);
      __syncthreads();
      io_w = w;
    }
    if (h == 2) {   // phi_s rows without an unknown are identity rows
      const double* __restrict__ r = a.io.r.get();
      double* z = a.io.z.get();
      for (int n = rank * kTailThreads + tid; n < (int)lv[0].d.n; n += a.cs * kTailThreads)
        if (!(a.io.label[n] & kLabActive)) z[n] = (r[n] * a.io.sqd[n]) * a.io.iwf[0];
    }
  }
  if (a.cs > 1) cluster_barrier();   // no store into a block that has not started and cleared its vectors
  const int nd = a.nl - 1;           // smoothed levels
#pragma unroll 1
  for (int v = 0; v < 2 * nd; ++v) {
    const bool up = v >= nd;
    const int q = up ? 2 * nd - 1 - v : v;
    const TailLv& L = lv[q];
    const TailLv& B = lv[q + 1];
    if (v == nd) {
      // the coarsest level's dense solve, rows over the warps of the cluster
      const int n = (int)B.d.n, lane = tid & 31;
      const double* inv = a.inv + (size_t)h * n * n;
      if (a.cs > 1) cluster_barrier();
      else __syncthreads();
#pragma unroll 1
      for (int r = rank * (kTailThreads / 32) + (tid >> 5); r < n; r += a.cs * (kTailThreads / 32)) {
        const bool on = all_on || __ldg(B.mask + r);
        const double acc = coarse_row<T>(n, inv + (size_t)r * n, sm + B.ob, lane);
        if (lane < L.nr && on) tail_put(sm, B.oA + r, lane, lane, (T)acc);
      }
      if (a.cs > 1) cluster_barrier();
      else __syncthreads();
    }
    const bool multi = L.nr > 1;
    if (!multi && rank > 0) continue;
    const int sy = L.d.nnx, sz = L.d.nnx * L.d.nny;
    const int n = L.lo + rank * L.chunk + tid;
    const bool in = tid < L.chunk && n < L.lo + L.rows;
    const bool on = in && (all_on || __ldg(L.mask + n));
    // x is in the first buffer after an even number of steps
    int x = (up && (a.deg & 1)) ? L.oB : L.oA, xo = (up && (a.deg & 1)) ? L.oA : L.oB;
    T c[27];
    T bq = (T)0, iq = (T)0, dq = (T)0, xq = (T)0;
    int id[3] = {0, 0, 0};
    int r0 = 0, r1 = 0, g0 = 0, g1 = 0;   // blocks of the neighbour rows; of the parent (down) or child (up) rows
    if (in) {   // on the way up these loads are in flight over the barrier
      if (!std::is_same<TS0, TS>::value && q == 0) row_coef<TS0, T>(L.st, (int)L.d.n, n, c);
      else row_coef<TS, T>(L.st, (int)L.d.n, n, c);
      if (q > 0) {
        bq = sm[L.ob + tid];
      } else if (a.io.on && !up) {
        // the load of the preconditioner's input (k_load, macro layout, scaled)
        const int f = h < 2 ? 0 : h - 1;
        const int64_t row = (int64_t)f * L.d.n + n;
        const double* __restrict__ r = a.io.r.get();
        const double rv = r[row];
        if constexpr (sizeof(T) == sizeof(float)) bq = ((float)rv * a.io.sqd32[row]) * io_w;
        else bq = a.io.sc[f] * ((rv * a.io.sqd[row]) * a.io.iwf[f]);
        if (on) static_cast<T*>(a.b[h])[n] = bq;
      } else {
        bq = static_cast<const T*>(a.b[h])[n];
      }
      iq = __ldg(static_cast<const T*>(L.dinv) + n);
      if (up) xq = sm[x + n];
      r0 = tail_owner(L, n - sz - sy - 1);
      r1 = tail_owner(L, n + sz + sy + 1);
      tail_ijk(L, n, id);
      const TailLv& U = lv[up && q > 0 ? q - 1 : q];   // the finer level of the transfer
      const TailLv& G = up ? U : B;                    // the level whose owners get the last vector
      if (G.nr > 1) {
        int c0 = 0, c1 = 0, st = 1;
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
          const Axis1 A = U.X.a[ax];
          T w;
          int e0, e1;
          if (up) {
            const int s0 = sup_of<T>(A, id[ax], 0, w), s1 = sup_of<T>(A, id[ax], 1, w), s2 = sup_of<T>(A, id[ax], 2, w);
            e0 = s0 >= 0 ? s0 : s1;
            e1 = s2 >= 0 ? s2 : (s1 >= 0 ? s1 : s0);
          } else {
            e0 = par_of<T>(A, id[ax], 0, w);
            e1 = par_of<T>(A, id[ax], 1, w);
            if (e1 < 0) e1 = e0;
          }
          c0 += st * e0;
          c1 += st * e1;
          st *= up ? A.nf : A.nc;
        }
        g0 = tail_owner(G, c0);
        g1 = tail_owner(G, c1);
      }
    }
    if (up) {
      if (v > nd) {   // (the coarsest solve ended with a barrier)
        if (multi) cluster_barrier();
        else __syncthreads();
      }
      if (in) {
        xq += tail_prolong<T>(L, B, sm + B.oA, id);
        if (on) tail_put(sm, x + n, r0, r1, xq);
      }
      if (multi) cluster_barrier();
      else __syncthreads();
    }
    // down: deg steps from x = 0, then the residual (s == deg); up: deg steps
    const int ns = up ? a.deg : a.deg + 1;
#pragma unroll 1
    for (int s = 0; s < ns; ++s) {
      if (in) {
        T res = bq;
        if (up || s > 0) res -= row_apply<T>(c, sm + x, sy, sz, n, xq);
        T val = res;
        if (s < a.deg) {
          const T z = iq * res;
          const T* cf = ch + (q * a.deg + s) * 3;
          dq = s == 0 ? cf[0] * z : fma(cf[2], z, cf[1] * dq);
          xq += dq;
          val = xq;
        }
        if (on) {
          const bool last = s == ns - 1;   // the residual, to the parents' blocks; the final x, to the children's
          if (last && up && q == 0) {
            if (a.io.on) a.io.z.get()[(int64_t)(h < 2 ? 0 : h - 1) * L.d.n + n] = (double)val;
            else static_cast<T*>(a.x[h])[n] = val;
          }
          else tail_put(sm, xo + n, last ? g0 : r0, last ? g1 : r1, val);
        }
      }
      if (s < a.deg) {
        const int t = x;
        x = xo;
        xo = t;
      }
      if (up && s == ns - 1) break;   // the level above starts with the barrier
      if (multi) cluster_barrier();
      else __syncthreads();
    }
    if (!up && rank < B.nr) {
      const int C = B.lo + rank * B.chunk + tid;
      if (tid < B.chunk && C < B.lo + B.rows) {
        // rows outside the mask hold exact zeros in the shared vectors
        const T val = tail_restrict<T>(L, B, sm + xo, C);
        if (q + 1 < nd) sm[B.ob + tid] = val;
        else tail_put(sm, B.ob + C, 0, a.cs - 1, val);   // every block solves rows of the coarsest level
      }
    }
  }
}

size_t tsize(int precision, int level) {
  if (precision == 0) return sizeof(double);
  if (precision == 2 && level > 0) return sizeof(__nv_bfloat16);
  return sizeof(float);
}

template <typename T>
HList make_hl(const int* hs, int nhs) {
  HList l{};
  for (int i = 0; i < kNH; ++i) l.h[i] = i < nhs ? hs[i] : hs[0];
  return l;
}

Xfer1 xfer1(const MGLevel& A, const MGLevel& B) {
  return Xfer1{{{A.nnx, B.nnx, A.cx}, {A.nny, B.nny, A.cy}, {A.nnz, B.nnz, A.cz}}};
}

LevelDims dims(const MGLevel& L) { return LevelDims{L.nnx, L.nny, L.nnz, L.n}; }

template <typename TS, typename T>
LvlPtrs<TS, T> ptrs(const MGLevel& L) {
  LvlPtrs<TS, T> P;
  for (int h = 0; h < kNH; ++h) {
    P.st[h] = (const TS*)L.st[h];
    P.dinv[h] = (const T*)L.dinv[h];
    P.mask[h] = L.mask[h];
    P.x[h] = (const T*)L.x[h];
    P.xo[h] = (T*)L.x2[h];
    P.b[h] = (const T*)L.b[h];
    P.r[h] = (T*)L.r[h];
    P.d[h] = (T*)L.d[h];
  }
  return P;
}

void swap_x(MGLevel& L, const int* hs, int nhs) {
  bool done[kNH] = {false, false, false, false};
  for (int t = 0; t < nhs; ++t) {
    int h = hs[t];
    // level-0 hierarchies 0/1 alias one buffer pair: swap it once
    if (L.x[h] == L.x[h ^ 1] && h < 2) {
      if (done[0]) continue;
      done[0] = done[1] = true;
      std::swap(L.x[0], L.x2[0]);
      L.x[1] = L.x[0];
      L.x2[1] = L.x2[0];
      continue;
    }
    if (done[h]) continue;
    done[h] = true;
    std::swap(L.x[h], L.x2[h]);
  }
}


// The Chebyshev coefficient table in the smoother's precision.
template <typename T> const T* cheb_tab(const p4d_ctx* c);
template <> const double* cheb_tab<double>(const p4d_ctx* c) { return c->cheb_dev; }
template <> const float* cheb_tab<float>(const p4d_ctx* c) { return c->cheb_dev32; }

// Node planes that hold a level's block ranges for the listed hierarchies (the
// transfers go by planes), and the widest range.
static_assert(kNpt == 1, "a block of the ranges is kBlock rows");
PRange prange(const MGLevel& A, const int* hs, int nhs, unsigned* gy) {
  PRange r{};
  int w = 1;
  const int sxy = A.nnx * A.nny;
  for (int h = 0; h < kNH; ++h) {
    const int lo = A.blo[h] * kBlock, hi = (int)std::min<int64_t>(A.n, (int64_t)(A.blo[h] + A.bcnt[h]) * kBlock);
    r.lo[h] = lo / sxy;
    r.cnt[h] = A.bcnt[h] ? (hi - 1) / sxy - r.lo[h] + 1 : 0;
  }
  for (int t = 0; t < nhs; ++t) w = std::max(w, r.cnt[hs[t]]);
  *gy = (unsigned)w;
  return r;
}

// Launches of the transfers over the planes of L: f(grid, block, planes).
// Blocks of a multiple of 64 threads that wastes little of the plane's last
// block; planes of fewer than 128 nodes share a block while every SM keeps
// four of them; planes beyond a grid's y extent go in further launches.  One
// application with a block of at least 128 threads per plane / now: 44,001
// planes of 4 nodes FP64 2.13 / 1.04 ms, FP32 1.29 / 0.99; 9,001 of 25 nodes
// 0.92 / 0.76, 0.42 / 0.37; 1,101 of 64 the same.  (Ten planes of 110 nodes in
// five blocks cost an FP64 application 2.5 us.)
template <typename F>
void for_planes(const MGLevel& L, const int* hs, int nhs, F&& f) {
  unsigned planes = 1;
  PRange pr = prange(L, hs, nhs, &planes);
  const int sxy = L.nnx * L.nny;
  dim3 block(256);
  const int share = std::min((int)(planes * nhs / (4 * 152)), 256 / sxy);
  if (sxy < 128 && share > 1) {
    block = dim3(sxy, share);
  } else {
    int waste = 1 << 30;
    for (int t = 256; t >= 128; t -= 64) {
      const int w = (int)nblocks(sxy, t) * t - sxy;
      if (w < waste) { waste = w; block.x = t; }
    }
  }
  const unsigned gy = (planes + block.y - 1) / block.y, most = 65535;
  for (unsigned y = 0; y < gy; y += most) {
    f(dim3(nblocks(sxy, block.x), std::min(gy - y, most), nhs), block, pr);
    for (int h = 0; h < kNH; ++h) {
      pr.lo[h] += most * block.y;
      pr.cnt[h] -= most * block.y;
    }
  }
}

// Block ranges of a level for the listed hierarchies, and the launch's grid
// width (the widest range).
BRange brange(const MGLevel& A, const int* hs, int nhs, unsigned* gx) {
  BRange r{};
  int w = 1;
  for (int h = 0; h < kNH; ++h) {
    r.lo[h] = A.blo[h];
    r.cnt[h] = A.bcnt[h];
  }
  for (int t = 0; t < nhs; ++t) w = std::max(w, A.bcnt[hs[t]]);
  *gx = (unsigned)w;
  return r;
}

// A level-0 step that applies the operator to a nonzero x (mode 0: a
// Chebyshev step, mode 1: the residual) for the hierarchies hs: the fields
// with a matrix-free operator in one mf launch, the others (phi_s with
// collector shells) with the stored stencils.
template <typename TS0, typename T>
p4d_status level0_stencil_step(p4d_ctx* c, MGLevel& A, const int* hs, int nhs, const HList& hl, const BRange& br,
                               dim3 grid, int mode, int step) {
  int fmask = 0, shs[kNH], ns = 0;
  for (int t = 0; t < nhs; ++t) {
    const int f = hs[t] < 2 ? 0 : hs[t] - 1;
    if (mf_field_on(c, f)) fmask |= 1 << f;
    else shs[ns++] = hs[t];
  }
  if (fmask) P4D_TRYS(mf_level0(c, fmask, mode, step));
  if (ns) {
    const HList hl2 = make_hl<T>(shs, ns);
    const dim3 g2(grid.x, ns);
    if (mode == 0)
      ::p4d::count_launch(), k_cheb<TS0, T><<<g2, kBlock, 0, c->stream>>>(dims(A), ptrs<TS0, T>(A), hl2, br, cheb_tab<T>(c), 0, step, 0);
    else
      ::p4d::count_launch(), k_resid<TS0, T><<<g2, kBlock, 0, c->stream>>>(dims(A), ptrs<TS0, T>(A), hl2, br);
  }
  (void)hl;
  return P4D_OK;
}

// Shared-memory layout of the tail from level l0 (elements; offsets into
// `lev` when given): per level two x buffers with guards and the block's own
// b, at the coarsest b and x.
int tail_layout(const p4d_ctx* c, int l0, TailLevel* lev) {
  int o = 0;
  for (int l = l0; l < c->nlev; ++l) {
    const MGLevel& A = c->lev[l];
    const int n = (int)A.n, G = A.nnx * A.nny + A.nnx + 1;
    const bool last = l == c->nlev - 1;
    int oA, oB, ob;
    if (last) {
      oA = o;
      oB = o;
      ob = o + n;
      o += 2 * n;
    } else {
      oA = o + G;
      oB = o + n + 3 * G;
      ob = o + 2 * n + 4 * G;
      o += 2 * n + 4 * G + kTailThreads;
    }
    if (lev) {
      lev[l - l0].oA = oA;
      lev[l - l0].oB = oB;
      lev[l - l0].ob = ob;
    }
  }
  return o;
}

cudaLaunchConfig_t tail_config(int cs, int nhs, size_t smem, cudaStream_t stream, cudaLaunchAttribute* at) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(cs * nhs));
  cfg.blockDim = dim3(kTailThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)cs;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cfg;
}

// Blocks of the cluster that own rows, per level and hierarchy: as many as
// the level's rows need, and at least as many as the next coarser level has.
// A mask's row range is rounded to 256 rows and coarsening along z alone
// halves no plane, so a coarser level can need more (a cathode at 9 x 7 nodes
// per plane: rows 512 to 1007, on the next level 0 to 566).  A level that one
// block owns runs without cluster barriers and without the other blocks: with
// a shared level below it they would neither restrict into their rows nor
// order their stores before the first block reads them.
template <typename T>
void tail_blocks(TailArgs& a) {
  for (int h = 0; h < kNH; ++h) {
    int least = 1;
    for (int q = a.nl - 1; q >= 0; --q) {
      TailLevel& L = a.lev[q];
      const int need = (L.hi[h] - L.lo[h] + kTailRows<T> - 1) / kTailRows<T>;
      least = L.nr[h] = std::max(least, std::min(a.cs, need));
    }
  }
}

// The levels l0 .. L - 1 in one launch (see k_tail).
template <typename TS0, typename TS, typename T>
p4d_status tail_launch(p4d_ctx* c, const int* hs, int nhs, int l0, const TailIO& io) {
  const int L = c->nlev;
  TailArgs a;
  a.nl = L - l0;
  a.l0 = l0;
  a.deg = c->prm.cheb_degree;
  a.cs = c->tail_cs;
  a.ctab = cheb_tab<T>(c);
  a.inv = c->lev[L - 1].inv;
  a.len = tail_layout(c, l0, a.lev);
  a.io = io;
  for (int t = 0; t < kNH; ++t) a.h[t] = t < nhs ? hs[t] : hs[0];
  for (int h = 0; h < kNH; ++h) {
    a.b[h] = c->lev[l0].b[h];
    a.x[h] = c->lev[l0].x[h];
  }
  for (int q = 0; q < a.nl; ++q) {
    const MGLevel& A = c->lev[l0 + q];
    TailLevel& B = a.lev[q];
    B.d = dims(A);
    if (q + 1 < a.nl) B.X = xfer1(A, c->lev[l0 + q + 1]);
    for (int h = 0; h < kNH; ++h) {
      B.lo[h] = A.blo[h] * kBlock;
      B.hi[h] = (int)std::min<int64_t>(A.n, (int64_t)(A.blo[h] + A.bcnt[h]) * kBlock);
      B.st[h] = A.st[h];
      B.dinv[h] = A.dinv[h];
      B.mask[h] = A.mask[h];
    }
  }
  tail_blocks<T>(a);
  cudaLaunchAttribute at[1];
  const cudaLaunchConfig_t cfg = tail_config(a.cs, nhs, sizeof(T) * a.len, c->stream, at);
  ::p4d::count_launch();
  P4D_TRY(cudaLaunchKernelEx(&cfg, l0 == 0 ? k_tail<TS0, TS, T> : k_tail<TS, TS, T>, a));
  return P4D_OK;
}

template <typename TS0, typename TS, typename T>
p4d_status vcycle_t(p4d_ctx* c, const int* hs, int nhs, const TailIO& io = TailIO{}) {
  const int LT = c->tail_l0 >= 0 ? c->tail_l0 : c->nlev - 1;   // levels above: one launch per operation
  const int deg = c->prm.cheb_degree;
  HList hl = make_hl<T>(hs, nhs);
  for (int l = 0; l < LT; ++l) {
    MGLevel& A = c->lev[l];
    MGLevel& B = c->lev[l + 1];
    unsigned gx = 1;
    const BRange br = brange(A, hs, nhs, &gx);
    const dim3 grid(gx, nhs);
    for (int s = 0; s < deg; ++s) {
      if (l == 0 && s > 0) prof_mark(c, 3);
      // (level 0, step 0: with the right-hand side, see mg_first_by_load)
      if (l == 0 && s > 0) P4D_TRYS((level0_stencil_step<TS0, T>(c, A, hs, nhs, hl, br, grid, 0, s)));
      else if (l > 0) ::p4d::count_launch(), k_cheb<TS, T><<<grid, kBlock, 0, c->stream>>>(dims(A), ptrs<TS, T>(A), hl, br, cheb_tab<T>(c), l, s, s == 0);
      if (l == 0 && s > 0) prof_mark(c, 3);
      swap_x(A, hs, nhs);
    }
    if (l == 0) P4D_TRYS((level0_stencil_step<TS0, T>(c, A, hs, nhs, hl, br, grid, 1, 0)));
    else ::p4d::count_launch(), k_resid<TS, T><<<grid, kBlock, 0, c->stream>>>(dims(A), ptrs<TS, T>(A), hl, br);
    Ptr4<const T> fr;
    Ptr4<const uint8_t> fm;
    Ptr4<T> cb;
    for (int h = 0; h < kNH; ++h) { fr.p[h] = (const T*)A.r[h]; fm.p[h] = A.mask[h]; cb.p[h] = (T*)B.b[h]; }
    for_planes(B, hs, nhs, [&](dim3 g, dim3 b, const PRange& pr) {
      ::p4d::count_launch(), k_restrict<T><<<g, b, 0, c->stream>>>(dims(A), dims(B), xfer1(A, B), fr, fm, cb, hl, pr);
    });
  }
  if (c->tail_l0 >= 0) {
    P4D_TRYS((tail_launch<TS0, TS, T>(c, hs, nhs, LT, io)));
  } else {
    MGLevel& C = c->lev[LT];
    Ptr4<const T> b;
    Ptr4<const uint8_t> m;
    Ptr4<T> x;
    for (int h = 0; h < kNH; ++h) { b.p[h] = (const T*)C.b[h]; m.p[h] = C.mask[h]; x.p[h] = (T*)C.x[h]; }
    ::p4d::count_launch(), k_coarse_solve<T><<<dim3((unsigned)((C.n + kCoarseWarps - 1) / kCoarseWarps), nhs), 32 * kCoarseWarps, 0, c->stream>>>((int)C.n, C.inv, b, m, x, hl);
  }
  for (int l = LT - 1; l >= 0; --l) {
    MGLevel& A = c->lev[l];
    MGLevel& B = c->lev[l + 1];
    Ptr4<const T> cxp;
    Ptr4<const uint8_t> fm;
    Ptr4<T> fx;
    for (int h = 0; h < kNH; ++h) { cxp.p[h] = (const T*)B.x[h]; fm.p[h] = A.mask[h]; fx.p[h] = (T*)A.x[h]; }
    unsigned gx = 1;
    const BRange br = brange(A, hs, nhs, &gx);
    const dim3 grid(gx, nhs);
    for_planes(A, hs, nhs, [&](dim3 g, dim3 b, const PRange& pr) {
      ::p4d::count_launch(), k_prolong<T><<<g, b, 0, c->stream>>>(dims(A), dims(B), xfer1(A, B), cxp, fm, fx, hl, pr);
    });
    for (int s = 0; s < deg; ++s) {
      if (l == 0) prof_mark(c, 3);
      if (l == 0) P4D_TRYS((level0_stencil_step<TS0, T>(c, A, hs, nhs, hl, br, grid, 0, s)));
      else ::p4d::count_launch(), k_cheb<TS, T><<<grid, kBlock, 0, c->stream>>>(dims(A), ptrs<TS, T>(A), hl, br, cheb_tab<T>(c), l, s, 0);
      if (l == 0) prof_mark(c, 3);
      swap_x(A, hs, nhs);
    }
  }
  P4D_TRY(cudaGetLastError());
  return P4D_OK;
}

}  // namespace

// ---------------------------------------------------------------- planning
// An x vector of a level (the input of the unchecked stencil loads) with a
// zeroed guard of at least nnx nny + nnx + 1 entries on both sides, rounded
// to 64 entries so that the vector keeps the allocation's alignment.
p4d_status alloc_x(p4d_ctx* c, void** p, size_t ts, const MGLevel& lv) {
  const int64_t G = ((int64_t)lv.nnx * lv.nny + lv.nnx + 1 + 63) / 64 * 64;
  const size_t bytes = ts * (size_t)(lv.n + 2 * G);
  void* base = nullptr;
  P4D_TRYS(dalloc(c, &base, bytes));
  P4D_TRY(cudaMemset(base, 0, bytes));
  *p = static_cast<char*>(base) + ts * G;
  return P4D_OK;
}

// First level of the single-launch tail and its cluster size (-1: no tail).
// The finest level is taken that has at most one row per thread of the
// largest cluster (FP64: two blocks' worth of rows per block, see kTailRows)
// and whose shared vectors fit: one more level in the tail replaces seven
// launches.  Measured per FGMRES solve (level by level / tail from 2,000
// rows / from this rule's level): 9 x 9 x 25 nodes 2.35 / - / 1.74 ms,
// 65 x 65 x 49 5.46 / 5.00 / 4.80 ms, FP64 41 x 37 x 37 8.28 / 7.97 / 7.57
// ms, 129 x 129 x 97 18.5 / 18.0 / 17.7 ms.
p4d_status tail_plan(p4d_ctx* c) {
  c->tail_l0 = -1;
  const int L = c->nlev;
  const bool fp64 = c->prm.precision == 0;
  const size_t tv = fp64 ? sizeof(double) : sizeof(float);
  const int rpb = fp64 ? kTailRows<double> : kTailRows<float>;
  const int64_t most = (int64_t)kTailMaxCluster * (fp64 ? 2 * rpb : rpb);
  if (c->lev[L - 1].n > kTailThreads) return P4D_OK;
  for (int l = 0; l < L - 1 && c->tail_l0 < 0; ++l)
    if (c->lev[l].n <= most && tv * tail_layout(c, l, nullptr) <= kTailMaxSmem) c->tail_l0 = l;
  if (c->tail_l0 < 0) return P4D_OK;
  int cs = 1;
  while (cs < kTailMaxCluster && (int64_t)cs * rpb < c->lev[c->tail_l0].n) cs *= 2;
  c->tail_cs = cs;
  const bool z = c->tail_l0 == 0;
  const void* k = fp64 ? (const void*)k_tail<double, double, double>
                  : c->prm.precision == 1 ? (const void*)k_tail<float, float, float>
                  : z ? (const void*)k_tail<float, __nv_bfloat16, float>
                      : (const void*)k_tail<__nv_bfloat16, __nv_bfloat16, float>;
  // process-wide attributes shared by every handle: always the largest values
  P4D_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  P4D_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTailMaxSmem));
  // a device (partition) that cannot hold such a cluster keeps the launches per level
  cudaLaunchAttribute at[1];
  cudaLaunchConfig_t cfg = tail_config(cs, 1, tv * tail_layout(c, c->tail_l0, nullptr), nullptr, at);
  int fit = 0;
  if (cudaOccupancyMaxActiveClusters(&fit, k, &cfg) != cudaSuccess || fit < 1) {
    cudaGetLastError();
    c->tail_l0 = -1;
  }
  return P4D_OK;
}

p4d_status mg_plan(p4d_ctx* c) {
  const int prec = c->prm.precision;
  const size_t tv = prec == 0 ? sizeof(double) : sizeof(float);
  int nnx = c->g.nnx, nny = c->g.nny, nnz = c->g.nnz;
  int L = 0;
  while (true) {
    MGLevel& lv = c->lev[L];
    lv.nnx = nnx; lv.nny = nny; lv.nnz = nnz;
    lv.n = (int64_t)nnx * nny * nnz;
    // coarsened axes: those with >= 2 elements (odd counts included) whose
    // mean element size is at most twice the smallest among them -- the
    // stiffness couples most strongly across short element edges, and the
    // point smoother reduces only errors smooth along the weak directions,
    // so weakly coupled axes stay fine until the elements are near isotropic
    const int nd[3] = {nnx, nny, nnz};
    int can[3];
    double hm[3], hmin = 0.0;
    bool any = false;
    for (int a = 0; a < 3; ++a) {
      can[a] = (nd[a] - 1) >= 2;
      hm[a] = nd[a] >= 2 ? c->len[a] / (nd[a] - 1) : 0.0;
      if (can[a] && (!any || hm[a] < hmin)) hmin = hm[a];
      any = any || can[a];
    }
    const int cx = can[0] && hm[0] <= 2.0 * hmin, cy = can[1] && hm[1] <= 2.0 * hmin,
              cz = can[2] && hm[2] <= 2.0 * hmin;
    ++L;
    if (lv.n <= c->prm.coarse_max || !(cx || cy || cz) || L >= kMaxLevels) break;
    lv.cx = cx; lv.cy = cy; lv.cz = cz;
    const int dn[3] = {nnx, nny, nnz}, fl[3] = {cx, cy, cz};
    int cn[3];
    for (int a = 0; a < 3; ++a) {
      const int nf = dn[a], ne = nf - 1;
      const int nc = fl[a] ? (ne + 1) / 2 + 1 : nf;
      cn[a] = nc;
      std::vector<int> par(2 * nf, -1), sup(3 * nc, -1);
      std::vector<double> parw(2 * nf, 0.0), supw(3 * nc, 0.0);
      for (int i = 0; i < nf; ++i) {
        if (!fl[a]) { par[2 * i] = i; parw[2 * i] = 1.0; continue; }
        if ((ne & 1) && i == ne) { par[2 * i] = (ne + 1) / 2; parw[2 * i] = 1.0; }
        else if ((i & 1) == 0) { par[2 * i] = i / 2; parw[2 * i] = 1.0; }
        else { par[2 * i] = (i - 1) / 2; par[2 * i + 1] = (i + 1) / 2; parw[2 * i] = parw[2 * i + 1] = 0.5; }
      }
      std::vector<int> cnt(nc, 0);
      for (int i = 0; i < nf; ++i)
        for (int q = 0; q < 2; ++q) {
          const int C = par[2 * i + q];
          if (C < 0) continue;
          if (cnt[C] >= 3) return P4D_ERR_INVALID_ARG;
          sup[3 * C + cnt[C]] = i;
          supw[3 * C + cnt[C]] = parw[2 * i + q];
          ++cnt[C];
        }
      int* dp = nullptr;
      double* dw = nullptr;
      P4D_TRYS(dalloc_t(c, &dp, par.size() + sup.size()));
      P4D_TRYS(dalloc_t(c, &dw, parw.size() + supw.size()));
      P4D_TRY(cudaMemcpy(dp, par.data(), par.size() * sizeof(int), cudaMemcpyHostToDevice));
      P4D_TRY(cudaMemcpy(dp + par.size(), sup.data(), sup.size() * sizeof(int), cudaMemcpyHostToDevice));
      P4D_TRY(cudaMemcpy(dw, parw.data(), parw.size() * sizeof(double), cudaMemcpyHostToDevice));
      P4D_TRY(cudaMemcpy(dw + parw.size(), supw.data(), supw.size() * sizeof(double), cudaMemcpyHostToDevice));
      std::vector<float> wf(parw.size() + supw.size());
      for (size_t q = 0; q < parw.size(); ++q) wf[q] = (float)parw[q];
      for (size_t q = 0; q < supw.size(); ++q) wf[parw.size() + q] = (float)supw[q];
      float* dwf = nullptr;
      P4D_TRYS(dalloc_t(c, &dwf, wf.size()));
      P4D_TRY(cudaMemcpy(dwf, wf.data(), wf.size() * sizeof(float), cudaMemcpyHostToDevice));
      lv.X.a[a] = Axis{dp, dw, dp + par.size(), dw + parw.size(), dwf, dwf + parw.size()};
    }
    nnx = cn[0];
    nny = cn[1];
    nnz = cn[2];
  }
  c->nlev = L;
  // process-wide attributes: the largest sizes the kernels use
  P4D_TRY(cudaFuncSetAttribute(k_lu_factor<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)lu_smem(kLuMax)));
  P4D_TRY(cudaFuncSetAttribute(k_lu_factor<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)lu_smem(kLuMax)));
  if (c->lev[L - 1].n > 4096) return P4D_ERR_INVALID_ARG;   // coarsest level too large for a dense inverse
  P4D_TRYS(tail_plan(c));
  double* lam = nullptr;
  P4D_TRYS(dalloc_t(c, &lam, (size_t)kNH * L));
  for (int l = 0; l < L; ++l) {
    MGLevel& lv = c->lev[l];
    const int64_t n = lv.n;
    const size_t ts = tsize(prec, l);
    lv.lam = lam + (size_t)l * kNH;
    for (int h = 0; h < kNH; ++h) P4D_TRYS(dalloc_t(c, &lv.mask[h], n));
    if (l == 0) {
      // fields: phi_s (hierarchies 0,1 share), phi_e (2), c_e (3)
      void *st[3], *di[3], *x[3], *x2[3], *b[3], *r[3], *d[3];
      for (int f = 0; f < 3; ++f) {
        P4D_TRYS(dalloc(c, &st[f], ts * 27 * n));
        P4D_TRYS(dalloc(c, &di[f], tv * n));
        P4D_TRYS(alloc_x(c, &x[f], tv, lv));
        P4D_TRYS(alloc_x(c, &x2[f], tv, lv));
        P4D_TRYS(dalloc(c, &b[f], tv * n));
        P4D_TRYS(dalloc(c, &r[f], tv * n));
        P4D_TRYS(dalloc(c, &d[f], tv * n));
        P4D_TRY(cudaMemset(x[f], 0, tv * n));
        P4D_TRY(cudaMemset(x2[f], 0, tv * n));
        P4D_TRY(cudaMemset(b[f], 0, tv * n));
        P4D_TRY(cudaMemset(d[f], 0, tv * n));
      }
      const int fh[kNH] = {0, 0, 1, 2};
      for (int h = 0; h < kNH; ++h) {
        lv.st[h] = st[fh[h]]; lv.dinv[h] = di[fh[h]]; lv.x[h] = x[fh[h]]; lv.x2[h] = x2[fh[h]];
        lv.b[h] = b[fh[h]]; lv.r[h] = r[fh[h]]; lv.d[h] = d[fh[h]];
      }
      if (c->tail_l0 == 0) {
        // the tail's clusters run the two phi_s hierarchies unsynchronized,
        // and a row next to the other electrode loads its neighbour there
        // (times an exact zero): iterates of their own
        P4D_TRYS(alloc_x(c, &lv.x[1], tv, lv));
        P4D_TRYS(alloc_x(c, &lv.x2[1], tv, lv));
      }
      ::p4d::count_launch(), k_mask0<<<nblocks(n), kBlock, 0, c->stream>>>(n, c->label, lv.mask[0], lv.mask[1], lv.mask[2], lv.mask[3]);
    } else {
      P4D_TRYS(dalloc_t(c, &lv.Ffix, (size_t)kNH * 27 * n));
      P4D_TRYS(dalloc(c, &lv.Vvar, (prec == 0 ? sizeof(double) : sizeof(float)) * (size_t)kNH * 27 * n));
      for (int h = 0; h < kNH; ++h) {
        P4D_TRYS(dalloc(c, &lv.st[h], ts * 27 * n));
        P4D_TRYS(dalloc(c, &lv.dinv[h], tv * n));
        P4D_TRYS(alloc_x(c, &lv.x[h], tv, lv));
        P4D_TRYS(alloc_x(c, &lv.x2[h], tv, lv));
        P4D_TRYS(dalloc(c, &lv.b[h], tv * n));
        P4D_TRYS(dalloc(c, &lv.r[h], tv * n));
        P4D_TRYS(dalloc(c, &lv.d[h], tv * n));
        P4D_TRY(cudaMemset(lv.x[h], 0, tv * n));
        P4D_TRY(cudaMemset(lv.x2[h], 0, tv * n));
        P4D_TRY(cudaMemset(lv.d[h], 0, tv * n));
      }
      MGLevel& fl = c->lev[l - 1];
      Ptr4<const uint8_t> fm;
      Ptr4<uint8_t> cm;
      for (int h = 0; h < kNH; ++h) { fm.p[h] = fl.mask[h]; cm.p[h] = lv.mask[h]; }
      ::p4d::count_launch(), k_mask_coarse<<<dim3(nblocks(n), kNH), kBlock, 0, c->stream>>>(dims(fl), dims(lv), fl.X, fm, cm);
    }
    if (l == L - 1) {
      P4D_TRYS(dalloc_t(c, &lv.inv, (size_t)2 * kNH * n * n));
      P4D_TRYS(dalloc_t(c, &lv.perm, (size_t)kNH * n));
    }
  }
  // per level and hierarchy, the stencil-kernel blocks that hold mask rows
  {
    int* ext = nullptr;
    P4D_TRYS(dalloc_t(c, &ext, (size_t)2 * kNH * L));
    std::vector<int> init(2 * kNH * L);
    for (int l = 0; l < L; ++l)
      for (int h = 0; h < kNH; ++h) {
        init[2 * (l * kNH + h)] = (int)c->lev[l].n;
        init[2 * (l * kNH + h) + 1] = -1;
      }
    P4D_TRY(cudaMemcpyAsync(ext, init.data(), init.size() * sizeof(int), cudaMemcpyHostToDevice, c->stream));
    for (int l = 0; l < L; ++l) {
      Ptr4<const uint8_t> m;
      for (int h = 0; h < kNH; ++h) m.p[h] = c->lev[l].mask[h];
      ::p4d::count_launch(), k_mask_extent<<<dim3(nblocks(c->lev[l].n), kNH), kBlock, 0, c->stream>>>(
          c->lev[l].n, m, ext + 2 * kNH * l);
    }
    P4D_TRY(cudaMemcpyAsync(init.data(), ext, init.size() * sizeof(int), cudaMemcpyDeviceToHost, c->stream));
    P4D_TRY(cudaStreamSynchronize(c->stream));
    const int rows = kBlock * kNpt;
    for (int l = 0; l < L; ++l)
      for (int h = 0; h < kNH; ++h) {
        const int lo = init[2 * (l * kNH + h)], hi = init[2 * (l * kNH + h) + 1];
        c->lev[l].blo[h] = hi < 0 ? 0 : lo / rows;
        c->lev[l].bcnt[h] = hi < 0 ? 0 : hi / rows - lo / rows + 1;
      }
  }
  // level-0 particle work and variable row sums
  P4D_TRYS(dalloc(c, &c->yc, (prec == 0 ? sizeof(double) : sizeof(float)) * (size_t)std::max<int64_t>(1, c->NE) * c->nc));
  P4D_TRY(cudaGetLastError());
  return P4D_OK;
}

namespace {
template <typename TS>
__global__ void k_level0_offdiag(Grid g, const double* __restrict__ Jst, double s0, double s1, double s2, TS* st0,
                                 TS* st1, TS* st2) {
  const int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (n >= g.nn) return;
  const int64_t nn = g.nn;
  TS* sts[3] = {st0, st1, st2};
  const double sc[3] = {s0, s1, s2};
  for (int f = 0; f < 3; ++f)
    for (int o = 0; o < 27; ++o)
      if (o != 13) sts[f][o * nn + n] = fromd<TS>(sc[f] * Jst[((size_t)f * 27 + o) * nn + n]);
}
}  // namespace

p4d_status mg_setup_fixed(p4d_ctx* c) {
  const int prec = c->prm.precision;
  MGLevel& l0 = c->lev[0];
  if (prec == 0)
    ::p4d::count_launch(), k_level0_offdiag<double><<<nblocks(l0.n), kBlock, 0, c->stream>>>(c->g, c->Jst, c->scale_f[0], c->scale_f[1], c->scale_f[2],
                                                                  (double*)l0.st[0], (double*)l0.st[2], (double*)l0.st[3]);
  else
    ::p4d::count_launch(), k_level0_offdiag<float><<<nblocks(l0.n), kBlock, 0, c->stream>>>(c->g, c->Jst, c->scale_f[0], c->scale_f[1], c->scale_f[2],
                                                                 (float*)l0.st[0], (float*)l0.st[2], (float*)l0.st[3]);
  const int64_t nn = c->g.nn;
  for (int l = 0; l + 1 < c->nlev; ++l) {
    MGLevel& A = c->lev[l];
    MGLevel& B = c->lev[l + 1];
    Ptr4<const double> fst, frs;
    Ptr4<const uint8_t> fm, cm;
    Ptr4<double> out;
    const int fh[kNH] = {0, 0, 1, 2};
    for (int h = 0; h < kNH; ++h) {
      if (l == 0) {
        fst.p[h] = c->Jst + (size_t)fh[h] * 27 * nn;
        frs.p[h] = c->sfix + (size_t)fh[h] * nn;
      } else {
        fst.p[h] = A.Ffix + (size_t)h * 27 * A.n;
        frs.p[h] = nullptr;
      }
      fm.p[h] = A.mask[h];
      cm.p[h] = B.mask[h];
      out.p[h] = B.Ffix + (size_t)h * 27 * B.n;
    }
    ::p4d::count_launch(), k_rap<double><<<dim3(nblocks(B.n, kRapWarps), kNH), 32 * kRapWarps, 0, c->stream>>>(dims(A), dims(B), A.X, fst, frs, fm, cm, out, 1);
  }
  P4D_TRY(cudaGetLastError());
  return P4D_OK;
}

// Variable part of levels >= 1 (Galerkin products in precision TV), the
// stored level operators, and the coarsest dense inverse (FP64).
template <typename TV>
p4d_status mg_update_levels(p4d_ctx* c, const double* svar, const double* sch) {
  const int prec = c->prm.precision;
  const int64_t nn = c->g.nn;
  const double* sf = c->scale_f;
  const int fh[kNH] = {0, 0, 1, 2};
  for (int l = 1; l < c->nlev; ++l) {
    MGLevel& A = c->lev[l - 1];
    MGLevel& B = c->lev[l];
    Ptr4<const uint8_t> fm, cm;
    Ptr4<TV> out;
    for (int h = 0; h < kNH; ++h) { fm.p[h] = A.mask[h]; cm.p[h] = B.mask[h]; out.p[h] = (TV*)B.Vvar + (size_t)h * 27 * B.n; }
    if (l == 1) {
      Ptr4<const double> s;
      for (int h = 0; h < kNH; ++h) s.p[h] = svar + (size_t)fh[h] * nn;
      ::p4d::count_launch(), k_rap_diag_g<TV><<<dim3(nblocks(B.n, 128), kNH), 128, 0, c->stream>>>(dims(A), dims(B), A.X, s, fm, cm, out);
    } else {
      Ptr4<const TV> fst, frs;
      if constexpr (std::is_same<TV, float>::value) {
        for (int h = 0; h < kNH; ++h) fst.p[h] = (const float*)A.Vvar + (size_t)h * 27 * A.n;
        ::p4d::count_launch(), k_rap32<<<dim3(nblocks(B.n, kRapWarps), kNH), 32 * kRapWarps, 0, c->stream>>>(dims(A), dims(B), xfer1(A, B), fst, fm, cm, out);
      } else {
      for (int h = 0; h < kNH; ++h) { fst.p[h] = (const TV*)A.Vvar + (size_t)h * 27 * A.n; frs.p[h] = nullptr; }
      ::p4d::count_launch(), k_rap<TV><<<dim3(nblocks(B.n, kRapWarps), kNH), 32 * kRapWarps, 0, c->stream>>>(dims(A), dims(B), A.X, fst, frs, fm, cm, out, 0);
      }
    }
    Ptr4<const double> F;
    Ptr4<const TV> V;
    Ptr4<const uint8_t> m;
    for (int h = 0; h < kNH; ++h) {
      F.p[h] = B.Ffix + (size_t)h * 27 * B.n;
      V.p[h] = (const TV*)B.Vvar + (size_t)h * 27 * B.n;
      m.p[h] = B.mask[h];
    }
    const dim3 grid(nblocks(B.n), kNH);
    if (prec == 0) {
      Ptr4<double> st, di;
      for (int h = 0; h < kNH; ++h) { st.p[h] = (double*)B.st[h]; di.p[h] = (double*)B.dinv[h]; }
      ::p4d::count_launch(), k_level_combine<double, double, TV><<<grid, kBlock, 0, c->stream>>>(dims(B), F, V, st, di, m, sch[0], sch[1], sch[2], sch[3], B.lam);
    } else if (prec == 1) {
      Ptr4<float> st, di;
      for (int h = 0; h < kNH; ++h) { st.p[h] = (float*)B.st[h]; di.p[h] = (float*)B.dinv[h]; }
      ::p4d::count_launch(), k_level_combine<float, float, TV><<<grid, kBlock, 0, c->stream>>>(dims(B), F, V, st, di, m, sch[0], sch[1], sch[2], sch[3], B.lam);
    } else {
      Ptr4<__nv_bfloat16> st;
      Ptr4<float> di;
      for (int h = 0; h < kNH; ++h) { st.p[h] = (__nv_bfloat16*)B.st[h]; di.p[h] = (float*)B.dinv[h]; }
      ::p4d::count_launch(), k_level_combine<__nv_bfloat16, float, TV><<<grid, kBlock, 0, c->stream>>>(dims(B), F, V, st, di, m, sch[0], sch[1], sch[2], sch[3], B.lam);
    }
  }
  // coarsest: dense scaled operator and its inverse
  MGLevel& C = c->lev[c->nlev - 1];
  double* mats = C.inv;
  double* work = C.inv + (size_t)kNH * C.n * C.n;
  if (c->nlev == 1) {
    Ptr4<const uint8_t> m;
    for (int h = 0; h < kNH; ++h) m.p[h] = C.mask[h];
    ::p4d::count_launch(), k_dense0<<<dim3(nblocks(C.n), kNH), kBlock, 0, c->stream>>>(c->g, c->Jst, c->sfix, svar, m, sf[0], sf[1], sf[2],
                                                                 mats);
  }
  // the inverse (into mats; work: the factors)
  const int n = (int)C.n;
  DenseRows dr{};
  dr.d = dims(C);
  Ptr4<const double> F{};
  Ptr4<const TV> V{};
  for (int h = 0; h < kNH; ++h) {
    dr.sc[h] = sch[h];
    if (c->nlev > 1) {
      F.p[h] = C.Ffix + (size_t)h * 27 * C.n;
      V.p[h] = (const TV*)C.Vvar + (size_t)h * 27 * C.n;
    }
  }
  if (n <= kLuMax) {
    const double* dense = c->nlev == 1 ? mats : nullptr;
    const dim3 gi((n + kLuCols - 1) / kLuCols, kNH);
    auto k = n <= 64 ? k_lu_inverse<2> : n <= 128 ? k_lu_inverse<4> : k_lu_inverse<8>;
    ::p4d::count_launch(), k_lu_factor<TV><<<kNH * kLuBlocks, lu_threads(n), lu_smem(n), c->stream>>>(n, dr, F, V, dense, work, C.perm);
    ::p4d::count_launch(), k<<<gi, 32 * kLuCols, 0, c->stream>>>(n, work, C.perm, mats);
  } else {
    if (c->nlev > 1)
      ::p4d::count_launch(), k_dense<TV><<<dim3(nblocks(C.n), kNH), kBlock, 0, c->stream>>>(dims(C), F, V, sch[0], sch[1], sch[2], sch[3], mats);
    ::p4d::count_launch(), k_gauss_jordan<<<kNH, 256, 0, c->stream>>>(n, mats, work);
  }
  P4D_TRY(cudaGetLastError());
  return P4D_OK;
}

p4d_status mg_update(p4d_ctx* c) {
  const int prec = c->prm.precision;
  const int64_t nn = c->g.nn;
  const double tau = (1.0 - c->prm.tplus) / c->prm.F;
  const double* sf = c->scale_f;
  const double sch[kNH] = {sf[0], sf[0], sf[1], sf[2]};
  double* svar = c->tmp;   // [3][nn] scratch (Krylov scratch is idle during an update)
  P4D_TRY(cudaMemsetAsync(c->lev[0].lam, 0, kNH * sizeof(double) * c->nlev, c->stream));   // one array over the levels
  MGLevel& l0 = c->lev[0];
  if (prec == 0)
    ::p4d::count_launch(), k_level0_update<double, double><<<nblocks(nn), kBlock, 0, c->stream>>>(
        c->g, tau, c->sfix, c->offsum, c->absoff, c->label, c->eidx, c->Aj, c->ge, c->gc, c->zeta, sf[0], sf[1], sf[2],
        (double*)l0.st[0], (double*)l0.st[2], (double*)l0.st[3], (double*)l0.dinv[0], (double*)l0.dinv[2],
        (double*)l0.dinv[3], svar, l0.lam, (float2*)nullptr);
  else
    ::p4d::count_launch(), k_level0_update<float, float><<<nblocks(nn), kBlock, 0, c->stream>>>(
        c->g, tau, c->sfix, c->offsum, c->absoff, c->label, c->eidx, c->Aj, c->ge, c->gc, c->zeta, sf[0], sf[1], sf[2],
        (float*)l0.st[0], (float*)l0.st[2], (float*)l0.st[3], (float*)l0.dinv[0], (float*)l0.dinv[2],
        (float*)l0.dinv[3], svar, l0.lam, (float2*)c->mf_svs);
  if (prec == 0) P4D_TRYS(mg_update_levels<double>(c, svar, sch));
  else P4D_TRYS(mg_update_levels<float>(c, svar, sch));
  P4D_TRY(cudaGetLastError());
  return P4D_OK;
}

p4d_status mg_fetch_lam(p4d_ctx* c) {
  P4D_TRY(cudaMemcpyAsync(c->lam_pin, c->lev[0].lam, kNH * sizeof(double) * c->nlev, cudaMemcpyDeviceToHost, c->stream));
  P4D_TRYS(check_flags(c));   // (synchronizes the stream, once for both)
  for (int l = 0; l < c->nlev; ++l)
    for (int h = 0; h < kNH; ++h) c->lam_h[l][h] = c->lam_pin[l * kNH + h];
  return cheb_upload(c, true);
}

// Chebyshev(degree d) coefficients on [lam/ratio, lam] of D^-1 A for every
// level, step and hierarchy (three-term recurrence of the shifted Chebyshev
// polynomials), copied to the device table.
p4d_status cheb_upload(p4d_ctx* c, bool synced) {
  const double ratio = c->prm.cheb_ratio;
  double* t = c->cheb_pin;
  if (!synced) P4D_TRY(cudaStreamSynchronize(c->stream));   // the previous copy from t has completed
  for (int l = 0; l < c->nlev; ++l)
    for (int h = 0; h < kNH; ++h) {
      const double lm = c->lam_h[l][h] > 0 ? c->lam_h[l][h] : 1.0;
      const double alpha = lm / ratio, beta = lm;
      const double theta = 0.5 * (beta + alpha), delta = 0.5 * (beta - alpha);
      const double sigma = theta / delta;
      double rho = 1.0 / sigma, rho_new = rho;
      for (int st = 0; st < c->prm.cheb_degree && st < kMaxDeg; ++st) {
        if (st > 0) {
          rho = rho_new;
          rho_new = 1.0 / (2.0 * sigma - rho);
        }
        t[((l * kMaxDeg + st) * 3 + 0) * kNH + h] = 1.0 / theta;
        t[((l * kMaxDeg + st) * 3 + 1) * kNH + h] = rho_new * rho;
        t[((l * kMaxDeg + st) * 3 + 2) * kNH + h] = 2.0 * rho_new / delta;
      }
    }
  const size_t ne = (size_t)kMaxLevels * kMaxDeg * 3 * kNH;
  float* t32 = reinterpret_cast<float*>(t + ne);   // FP32 copy for the FP32 smoothers
  for (size_t q = 0; q < ne; ++q) t32[q] = (float)t[q];
  // the smoothers read the table in their own precision
  if (c->prm.precision == 0) P4D_TRY(cudaMemcpyAsync(c->cheb_dev, t, sizeof(double) * ne, cudaMemcpyHostToDevice, c->stream));
  else P4D_TRY(cudaMemcpyAsync(c->cheb_dev32, t32, sizeof(float) * ne, cudaMemcpyHostToDevice, c->stream));
  return P4D_OK;
}

// Block-Jacobi application of a cell whose V-cycles are one launch: load,
// V-cycles of all hierarchies and store in it (z = P^-1 s^-1 r in the macro
// layout).  The load and the store were 8 of 28 us per application at 2,025
// nodes.
p4d_status mg_apply_tail(p4d_ctx* c, VRef r, VRef z) {
  TailIO io;
  io.on = 1;
  io.r = r;
  io.z = z;
  io.sqd = c->sqd;
  io.sqd32 = c->sqd32;
  io.iwf = c->iwf;
  io.label = c->label;
  for (int f = 0; f < 3; ++f) io.sc[f] = c->scale_f[f];
  const int hs[kNH] = {0, 1, 2, 3};
  switch (c->prm.precision) {
    case 0: return vcycle_t<double, double, double>(c, hs, kNH, io);
    case 1: return vcycle_t<float, float, float>(c, hs, kNH, io);
    default: return vcycle_t<float, __nv_bfloat16, float>(c, hs, kNH, io);
  }
}

p4d_status mg_vcycle(p4d_ctx* c, const int* hs, int nhs) {
  switch (c->prm.precision) {
    case 0: return vcycle_t<double, double, double>(c, hs, nhs);
    case 1: return vcycle_t<float, float, float>(c, hs, nhs);
    default: return vcycle_t<float, __nv_bfloat16, float>(c, hs, nhs);
  }
}

}  // namespace p4d
