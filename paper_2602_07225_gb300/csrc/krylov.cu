// Right-preconditioned flexible GMRES(m) (Saad 1993) in FP64 on the scaled
// system s.J.s x^ = s.b (s_i = w_f / sqrt(J_ii)); the preconditioned
// directions are stored unscaled (z_k = P^-1 (s^-1 v_k)), so that
// x = x0 + sum_k y_k z_k and the operator is applied as s.(J z_k).
//
// Orthogonalisation: classical Gram-Schmidt; a second pass runs only when the
// first cancelled more than half of the vector ("twice is enough" with the
// Daniel-Gragg-Kaufman-Stewart test, decided on the device).  Each pass is a
// register-blocked multi-dot over the basis with a fixed-shape two-stage
// reduction (deterministic order).  The second stage, the reorthogonalisation
// test, the Hessenberg column, the Givens rotations and the residual estimate
// run in the last block of the kernel that produced their inputs (each is a
// few microseconds of latency as a launch of its own): an Arnoldi step
// without refinement is multi-dot, update and scaling, three launches.
#include <cmath>
#include <cstring>
#include "p4d_common.cuh"

namespace p4d {
namespace {

constexpr int kRedBlocks = 4 * 152;   // reduction grid: a multiple of the SM count
constexpr int kRedThreads = 256;

// Multi-dot, register blocked with a compile-time group size: each thread
// keeps one accumulator per dot of a group of NG dots (plus w.w) over all of
// its elements, so exactly NG FP64 FMAs run per element (a run-time group
// size with predicated FMAs issued all sixteen).  The warp stage is a
// transpose reduction: with P (a power of two >= NG + WW) values per lane,
// each butterfly step halves the values a lane keeps, P - 1 + log2(32/P)
// FP64 adds per lane instead of 5 per value (FP64 adds are as scarce as FP64
// FMAs on this GPU).
// partial[blk][g0 + i] = sum over the block's elements of V[g0 + i][n] * w[n];
// WW: partial[blk][kp1] = sum w[n]^2.
constexpr int kDotGroup = 16;

template <int X>
struct Pow2Up {
  static constexpr int v = X <= 1 ? 1 : (X <= 2 ? 2 : (X <= 4 ? 4 : (X <= 8 ? 8 : (X <= 16 ? 16 : 32))));
};
template <int X>
struct Log2 {
  static constexpr int v = X <= 1 ? 0 : 1 + Log2<X / 2>::v;
};
template <>
struct Log2<1> {
  static constexpr int v = 0;
};

// After the call, lane l holds in a[0] the warp total of value index
// l >> (5 - log2 P) (every lane of a group of 32/P lanes holds the same).
template <int P>
__device__ __forceinline__ void warp_transpose_reduce(double (&a)[P], int lane) {
#pragma unroll
  for (int c = P, o = 16; c > 1; c >>= 1, o >>= 1) {
    const bool upper = lane & o;
#pragma unroll
    for (int t = 0; t < c / 2; ++t) {
      const double send = upper ? a[t] : a[t + c / 2];
      const double keep = upper ? a[t + c / 2] : a[t];
      a[t] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
#pragma unroll
  for (int o = 16 >> Log2<P>::v; o > 0; o >>= 1) a[0] += __shfl_xor_sync(0xffffffffu, a[0], o);
}

// True in every thread of the block that finishes its kernel last, with the
// partial sums of the other blocks visible; it resets the counter for the
// next launch.  The partial sums are written by the first warp, which alone
// orders its writes (a fence in every warp held the blocks of an update back
// by several microseconds).
__device__ __forceinline__ bool last_block(unsigned* cnt) {
  __shared__ bool last;
  if (threadIdx.x < 32) __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    last = atomicAdd(cnt, 1u) == gridDim.x - 1;
    if (last) *cnt = 0;
  }
  __syncthreads();
  if (last) __threadfence();
  return last;
}

// Sum of p[0..n) by one warp (fixed order: lanes stride, then a butterfly).
__device__ __forceinline__ double warp_sum(const double* p, int n, int lane) {
  double s = 0.0;
#pragma unroll 4
  for (int b = lane; b < n; b += 32) s += __ldcg(p + b);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

// Sum of p[0..n) by one warp in the order of a 256-thread block (thread t
// sums p[t], p[t + 256], ..., then a halving tree): lane l holds threads l,
// l + 32, ..., l + 224.  Lane 0 has the result.
__device__ __forceinline__ double warp_tree_sum(const double* p, int n, int lane) {
  if (n <= 32) {   // one partial per lane at most: the tree above the lanes adds zeros
    double t = lane < n ? __ldcg(p + lane) : 0.0;
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    return t;
  }
  double s[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    s[q] = 0.0;
    for (int b = lane + 32 * q; b < n; b += 256) s[q] += __ldcg(p + b);
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) s[q] += s[q + 4];
  s[0] += s[2];
  s[1] += s[3];
  double t = s[0] + s[1];
  for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
  return t;
}

// out[g0 + i] = V_{g0+i} . w (i < NG), out[kp1] = w . w (WW), summed over the
// blocks by the last one.  flag (optional): skipped when *flag == 0, out
// then zeroed (zero_if_skipped) or left as it is.
template <int NG, bool WW>
__global__ void __launch_bounds__(kRedThreads) k_mdot(const double* __restrict__ V, int64_t ldv, int g0, int kp1,
                                                      const double* __restrict__ w, int64_t len,
                                                      double* __restrict__ partial, double* __restrict__ out,
                                                      unsigned* cnt, const double* __restrict__ flag,
                                                      int zero_if_skipped) {
  constexpr int NA = NG + (WW ? 1 : 0);
  constexpr int P = Pow2Up<NA>::v;
  if (flag && *flag == 0.0) {   // conditional pass not needed
    if (zero_if_skipped && blockIdx.x == 0 && threadIdx.x < NG) out[g0 + threadIdx.x] = 0.0;
    return;
  }
  __shared__ double red[kRedThreads / 32][P];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  double acc[P];
#pragma unroll
  for (int i = 0; i < P; ++i) acc[i] = 0.0;
  const double* Vg = V + (int64_t)g0 * ldv;
  int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  // two elements per trip, all their loads issued before the FMAs (twice the
  // loads in flight); each accumulator still takes n, n + stride, ... in order
  for (; n + stride < len; n += 2 * stride) {
    const double w0 = w[n], w1 = w[n + stride];
    double a0[NG > 0 ? NG : 1], a1[NG > 0 ? NG : 1];
#pragma unroll
    for (int i = 0; i < NG; ++i) {
      a0[i] = Vg[(int64_t)i * ldv + n];
      a1[i] = Vg[(int64_t)i * ldv + n + stride];
    }
#pragma unroll
    for (int i = 0; i < NG; ++i) {
      acc[i] = fma(a0[i], w0, acc[i]);
      acc[i] = fma(a1[i], w1, acc[i]);
    }
    if (WW) {
      acc[NG] = fma(w0, w0, acc[NG]);
      acc[NG] = fma(w1, w1, acc[NG]);
    }
  }
  for (; n < len; n += stride) {
    const double wn = w[n];
#pragma unroll
    for (int i = 0; i < NG; ++i) acc[i] = fma(Vg[(int64_t)i * ldv + n], wn, acc[i]);
    if (WW) acc[NG] = fma(wn, wn, acc[NG]);
  }
  warp_transpose_reduce<P>(acc, lane);
  constexpr int span = 32 / P;
  if ((lane & (span - 1)) == 0) red[warp][lane / span] = acc[0];
  __syncthreads();
  if (threadIdx.x < NA) {
    const int i = threadIdx.x;
    double sum = 0.0;
#pragma unroll
    for (int wv = 0; wv < kRedThreads / 32; ++wv) sum += red[wv][i];
    partial[(int64_t)i * kRedBlocks + blockIdx.x] = sum;
  }
  if (!last_block(cnt)) return;
  for (int i = warp; i < NA; i += kRedThreads / 32) {
    const double sum = warp_tree_sum(partial + (int64_t)i * kRedBlocks, gridDim.x, lane);
    if (lane == 0) out[i < NG ? g0 + i : kp1] = sum;
  }
}

// Hessenberg layout in hs: H[(m+1) x m] column-major, cs[m], sn[m], g[m+1], y[m], misc
struct HLay {
  int m;
  int H, cs, sn, g, y, misc;
};
HLay hlay(int m) {
  HLay L;
  L.m = m;
  L.H = 0;
  L.cs = (m + 1) * m;
  L.sn = L.cs + m;
  L.g = L.sn + m;
  L.y = L.g + m + 1;
  L.misc = L.y + m;
  return L;
}
// misc: [0] h1 (m+1) ... we keep separate small arrays after misc:
//   misc+0 .. misc+m       : h1 (first-pass coefficients, then column)
//   misc+m+1 .. misc+2m+1  : h2 (second pass)
//   misc+2m+2              : ||w||^2 after the second pass (or first pass)
//   misc+2m+3              : residual estimate |g_{k+1}|
//   misc+2m+4              : status (0 ok, 1 breakdown, 2 nonfinite)
//   misc+2m+5              : beta (initial residual norm)

// Column k: h = h1 + h2, h_{k+1,k} = ||w||, previous rotations, new rotation.
// refine = 0: no second Gram-Schmidt pass ran, h2 is not read.  All threads
// of one block: the loads side by side, the rotations (a dependent chain) by
// thread 0 in shared memory.
__device__ void givens_block(double* hs, const HLay& L, int k, int* kdev, int refine) {
  __shared__ double col[130], c_[130], s_[130];
  const int m = L.m;
  const double* h1 = hs + L.misc;
  const double* h2 = hs + L.misc + m + 1;
  for (int i = threadIdx.x; i <= k; i += blockDim.x) {
    col[i] = refine ? __ldcg(h1 + i) + __ldcg(h2 + i) : __ldcg(h1 + i);
    c_[i] = i < k ? hs[L.cs + i] : 0.0;
    s_[i] = i < k ? hs[L.sn + i] : 0.0;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    *kdev = k + 1;
    double* g = hs + L.g;
    const double gk = g[k];
    const double nw = sqrt(__ldcg(hs + L.misc + 2 * m + 2));
    for (int i = 0; i < k; ++i) {
      const double t = c_[i] * col[i] + s_[i] * col[i + 1];
      col[i + 1] = -s_[i] * col[i] + c_[i] * col[i + 1];
      col[i] = t;
    }
    const double den = hypot(col[k], nw);
    double status = 0.0, ck = 1.0, sk = 0.0, last = nw;
    if (!(den > 0.0) || !isfinite(den)) {
      status = isfinite(den) ? 1.0 : 2.0;
    } else {
      ck = col[k] / den;
      sk = nw / den;
      col[k] = den;
      last = 0.0;
    }
    hs[L.cs + k] = ck;
    hs[L.sn + k] = sk;
    hs[L.H + (int64_t)k * (m + 1) + k + 1] = last;
    const double gn = -sk * gk;
    g[k + 1] = gn;
    g[k] = ck * gk;
    hs[L.misc + 2 * m + 3] = fabs(gn);
    if (nw == 0.0 && status == 0.0) status = 1.0;   // happy breakdown: exact solution in the space
    if (!isfinite(gn)) status = 2.0;
    hs[L.misc + 2 * m + 4] = status;
  }
  __syncthreads();
  for (int i = threadIdx.x; i <= k; i += blockDim.x) hs[L.H + (int64_t)k * (m + 1) + i] = col[i];
}

// Reorthogonalise only when the first Gram-Schmidt pass cancelled more than
// half of the vector (||w_after|| < 0.7 ||w_before||, Daniel-Gragg-Kaufman-
// Stewart); count the passes in misc+2m+7.
// eta2 = 0.49: a second pass when ||w|| fell below 0.7 ||w_0||; eta2 = 2:
// always (||w|| never grows in a pass).
__device__ void reorth_test(double* hs, const HLay& L, int k, double eta2) {
  double* misc = hs + L.misc;
  const double before = misc[k + 1];
  const double after = misc[2 * L.m + 2];
  const double f = (after < eta2 * before) ? 1.0 : 0.0;
  misc[2 * L.m + 6] = f;
  misc[2 * L.m + 7] += f;
}

// What the last block of an update does with ||w||^2.
enum : int {
  kFinNone = 0,     // no norm
  kFinNorm = 1,     // write it
  kFinReorth = 2,   // and decide on the second pass
  kFinGivens = 3,   // and update the Hessenberg column
};
struct Fin {
  int mode = kFinNone;
  double* norm = nullptr;    // ||w||^2
  int zero_if_skipped = 0;   // norm = 0 when the pass is skipped
  double* hs = nullptr;      // kFinReorth, kFinGivens
  HLay L{};
  int k = 0;
  double eta2 = 0.0;
  int* kdev = nullptr;
  int refine = 0;
};

// w[n] -= sum_i h[i] V[i][n] (h on the device), the products subtracted in
// order of i; the loads of eight basis vectors are in flight at a time (R:
// kp1 mod 8).  With fin.mode, the updated w[n]^2 are summed over nvb runs of
// 256 elements (grid-strided; the partition of the sums does not depend on
// the launch), four runs per block, and the last block finishes as fin says.
// With a block per run and every warp fencing, the arrival of 2,432 blocks at
// the counter took 10-15 of 25 us at 614 k elements.
template <int R>
__global__ void __launch_bounds__(kBlock) k_maxpy(const double* __restrict__ V, int64_t ldv, int kp1,
                                                  const double* __restrict__ h, double* __restrict__ w,
                                                  int64_t len, double sign, const double* __restrict__ flag,
                                                  double* __restrict__ partial, unsigned* cnt, int nvb, Fin fin) {
  if (flag && *flag == 0.0) {
    if (blockIdx.x == 0) {
      if (fin.mode == kFinGivens) givens_block(fin.hs, fin.L, fin.k, fin.kdev, fin.refine);
      else if (fin.zero_if_skipped && threadIdx.x == 0) *fin.norm = 0.0;
    }
    return;
  }
  __shared__ double hs[130];
  __shared__ double red[2][kBlock / 32];
  for (int i = threadIdx.x; i < kp1; i += blockDim.x) hs[i] = sign * h[i];
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int vb = blockIdx.x, it = 0; vb < nvb; vb += gridDim.x, ++it) {
    double ss = 0.0;
    for (int64_t n = vb * (int64_t)kBlock + threadIdx.x; n < len; n += (int64_t)nvb * kBlock) {
      double acc = w[n];
      const double* v = V + n;
      int i = 0;
      for (; i + 8 <= kp1; i += 8) {
        double a[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) a[q] = v[(int64_t)(i + q) * ldv];
#pragma unroll
        for (int q = 0; q < 8; ++q) acc -= hs[i + q] * a[q];
      }
      if (R > 0) {
        double a[R > 0 ? R : 1];
#pragma unroll
        for (int q = 0; q < R; ++q) a[q] = v[(int64_t)(i + q) * ldv];
#pragma unroll
        for (int q = 0; q < R; ++q) acc -= hs[i + q] * a[q];
      }
      w[n] = acc;
      if (fin.mode) ss = fma(acc, acc, ss);
    }
    if (!fin.mode) continue;
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    if (lane == 0) red[it & 1][warp] = ss;   // two buffers: one barrier per run
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int i = 0; i < kBlock / 32; ++i) t += red[it & 1][i];
      partial[vb] = t;
    }
  }
  if (!fin.mode) return;
  if (!last_block(cnt)) return;
  // strided sums per thread, then a halving tree over the 256 threads
  double t = 0.0;
  for (int b = threadIdx.x; b < nvb; b += kBlock) t += __ldcg(partial + b);
  __shared__ double tree[kBlock];
  tree[threadIdx.x] = t;
  __syncthreads();
  for (int off = kBlock / 2; off >= 32; off >>= 1) {
    if ((int)threadIdx.x < off) tree[threadIdx.x] += tree[threadIdx.x + off];
    __syncthreads();
  }
  if (threadIdx.x < 32) {
    t = tree[threadIdx.x];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
  }
  if (threadIdx.x == 0) {
    *fin.norm = t;
    if (fin.mode == kFinReorth) reorth_test(fin.hs, fin.L, fin.k, fin.eta2);
  }
  if (fin.mode != kFinGivens) return;
  __threadfence_block();
  __syncthreads();
  givens_block(fin.hs, fin.L, fin.k, fin.kdev, fin.refine);
}

// What block 0 of a scaling leaves behind.
struct Tail {
  int mode = 0;               // 1: start of a cycle (g, beta, kdev); 2: end of an Arnoldi step
  double* hs = nullptr;
  HLay L{};
  int* kdev = nullptr;
  double* stat = nullptr;     // mode 2: residual estimate and status of the step
  double* gate = nullptr;     // mode 2: gate of the cycle's graph (see kGateOff) ...
  int k = 0;                  // ... after step k
  int next = 0;               // ... with a step k + 1 in the same graph, run when `handle` is set
  cudaGraphConditionalHandle handle = 0;
  int nf = 0;                 // mode 1 with gate: fields of the Krylov vector, ...
  double limit = 0.0, rtol = 0.0;   // ... step limit and tolerance of the cycle
};

__device__ void init_cycle(const Tail& t) {
  double* hs = t.hs;
  const HLay& L = t.L;
  *t.kdev = 0;   // Krylov column of the next preconditioner application
  const double beta = sqrt(hs[L.misc + 2 * L.m + 2]);
  for (int i = 0; i <= L.m; ++i) hs[L.g + i] = 0.0;
  hs[L.g] = beta;
  hs[L.misc + 2 * L.m + 5] = beta;
  hs[L.misc + 2 * L.m + 3] = beta;
  if (!t.gate) return;
  // ||s.b_k|| and the tests the host makes before the first step (fg_bnorm,
  // fg_cycle_read): the same comparisons, so that a norm that is not a number
  // (squares that overflow) runs the step that the host waits for
  const double* bn2 = hs + L.misc + 2 * L.m + 8;
  const double* bk2 = hs + L.misc + 2 * L.m + 16;
  double bn = 0.0;
  for (int f = 0; f < t.nf; ++f) {
    const double wf = bn2[f] > 0 ? 1.0 / sqrt(bn2[f]) : 1.0;
    bn += wf * wf * bk2[f];
  }
  bn = sqrt(bn);
  t.gate[0] = bn == 0.0 || !isfinite(beta) || beta <= t.rtol * bn ? 1.0 : 0.0;
  t.gate[1] = t.gate[2] = t.gate[3] = 0.0;
  t.gate[4] = t.limit;
  t.gate[5] = bn;
  t.gate[6] = t.rtol;
}

// Condition of the first step of a segment of a cycle.
__global__ void k_gate(cudaGraphConditionalHandle h, const double* __restrict__ gate, int k) {
  if (threadIdx.x == 0) cudaGraphSetConditional(h, (gate[0] == 0.0 && (double)k < gate[4]) ? 1u : 0u);
}

// After Arnoldi step k: the cycle stops on a breakdown, a non-finite scalar
// or a converged estimate, the same tests the host applies to a step's
// status; otherwise the graph's next step runs (its conditional node's
// handle is 0 unless set here).
__device__ void step_done(const Tail& t) {
  const double est = t.hs[t.L.misc + 2 * t.L.m + 3], st = t.hs[t.L.misc + 2 * t.L.m + 4];
  if (t.stat) {
    t.stat[0] = est;
    t.stat[1] = st;
  }
  if (!t.gate) return;
  double* gate = t.gate;
  gate[1] = t.k + 1;
  gate[2] = est;
  gate[3] = st;
  const bool stop = st != 0.0 || est / gate[5] <= gate[6];
  if (stop) gate[0] = 1.0;
  if (t.next) cudaGraphSetConditional(t.handle, (!stop && (double)(t.k + 1) < gate[4]) ? 1u : 0u);
}

// y = x / sqrt(*sp) (0 if *sp == 0); x and y may be the same vector (no
// __restrict__ on them).
__global__ void k_scale(const double* x, double* y, int64_t len, const double* __restrict__ sp, Tail t) {
  // the factor once per block (an FP64 divide and square root per thread
  // cost more than the scaling itself on this GPU)
  __shared__ double sfac;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  // four elements in flight, the first four over the factor's latency
  double a[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) a[q] = n + q * stride < len ? x[n + q * stride] : 0.0;
  if (threadIdx.x == 0) {
    const double v = *sp;
    sfac = v != 0.0 ? 1.0 / sqrt(v) : 0.0;
  }
  __syncthreads();
  const double s = sfac;
  while (n < len) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (n + q * stride < len) y[n + q * stride] = a[q] * s;
    n += 4 * stride;
#pragma unroll
    for (int q = 0; q < 4; ++q) a[q] = n + q * stride < len ? x[n + q * stride] : 0.0;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    if (t.mode == 1) init_cycle(t);
    else if (t.mode == 2) step_done(t);
  }
}

// Field weights of the Krylov norm: w_f = 1 / max(||b~_f||, floor_f), b~ = b/sqrt(d).
// Forward solves: floor_f = (1e-14/rtol) ||(sqrt(d) u)_f|| with u the
// linearization state -- a field's right-hand side is balanced against the
// others unless it lies below the rounding level of the field's own terms
// (then FGMRES could never reduce its residual by rtol).  Adjoint solves:
// floor_f = 1e-2 ||b~|| (the adjoint variable has no state scale).
__device__ void weights_of(const double* s4, const double* __restrict__ unorm2, double floor_rel, int adjoint,
                           double* __restrict__ wf, double* __restrict__ iwf, double* bn2) {
  double all = 0.0;
  for (int f = 0; f < 4; ++f) all += s4[f];
  double tot = 0.0;
  for (int f = 0; f < 4; ++f) {
    const double fl = adjoint ? 1e-4 * all : floor_rel * floor_rel * unorm2[f];
    const double s = fmax(s4[f], fl);
    wf[f] = s > 0.0 ? 1.0 / sqrt(s) : 1.0;
    iwf[f] = s > 0.0 ? sqrt(s) : 1.0;
    bn2[f] = s;
    tot += s > 0.0 ? s4[f] / s : 0.0;
  }
  bn2[4] = tot;
}

// Block sums of NV per-thread values into partial[v][block] (fixed order).
template <int NV>
__device__ __forceinline__ void sum_partials(const double (&acc)[NV], double* partial) {
  __shared__ double red[NV][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int f = 0; f < NV; ++f) {
    double a = acc[f];
    for (int off = 16; off > 0; off >>= 1) a += __shfl_down_sync(0xffffffffu, a, off);
    if (lane == 0) red[f][warp] = a;
  }
  __syncthreads();
  if (threadIdx.x < NV) {
    double t = 0.0;
    for (int w = 0; w < nw; ++w) t += red[threadIdx.x][w];
    partial[(int64_t)threadIdx.x * kRedBlocks + blockIdx.x] = t;
  }
}

// Per-field squared norms of (b / sqrt(d)) over the 4 fields (c_s optional),
// one contiguous range per field: sums[0..3], or with wf the Krylov weights
// (see weights_of; bn2 is then sums[0..4]).
__global__ void __launch_bounds__(kRedThreads) k_field_norms(const double* __restrict__ b,
                                                             const double* __restrict__ rsqd, int64_t nn, int64_t len,
                                                             double* __restrict__ partial, unsigned* cnt,
                                                             const double* __restrict__ unorm2, double floor_rel,
                                                             int adjoint, double* __restrict__ wf,
                                                             double* __restrict__ iwf, double* __restrict__ sums) {
  double acc[4];
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    const int64_t lo = f * nn, hi = f < 3 ? (f + 1) * nn : len;
    acc[f] = hi > lo ? sumsq_share<true>(b + lo, rsqd + lo, hi - lo) : 0.0;
  }
  sum_partials<4>(acc, partial);
  if (!last_block(cnt)) return;
  __shared__ double s4[4];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp < 4) {
    const double t = warp_sum(partial + (int64_t)warp * kRedBlocks, gridDim.x, lane);
    if (lane == 0) s4[warp] = t;
  }
  __syncthreads();
  if (wf) {
    if (threadIdx.x == 0) weights_of(s4, unorm2, floor_rel, adjoint, wf, iwf, sums);
  } else if (threadIdx.x < 4) {
    sums[threadIdx.x] = s4[threadIdx.x];
  }
}

// The three sets of field norms of a finished solve in one pass over its
// vectors: out[0..3] = ||r_f||^2, out[8..11] = ||(sqd r)_f||^2, out[12..15] =
// ||b_f||^2.
__global__ void __launch_bounds__(kRedThreads) k_final_norms(const double* __restrict__ r,
                                                             const double* __restrict__ sqd,
                                                             const double* __restrict__ b, int64_t nn, int64_t len,
                                                             double* __restrict__ partial, unsigned* cnt,
                                                             double* __restrict__ out) {
  double acc[12];
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    const int64_t lo = f * nn, hi = f < 3 ? (f + 1) * nn : len, stride = (int64_t)gridDim.x * blockDim.x;
    double a0 = 0.0, a1 = 0.0, b0 = 0.0, b1 = 0.0, c0 = 0.0, c1 = 0.0;
    int64_t i = lo + blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    for (; i + stride < hi; i += 2 * stride) {   // two elements in flight
      const double r0 = r[i], r1 = r[i + stride], q0 = sqd[i], q1 = sqd[i + stride], v0 = b[i], v1 = b[i + stride];
      const double u0 = r0 * q0, u1 = r1 * q1;
      a0 = fma(r0, r0, a0);
      a1 = fma(r1, r1, a1);
      b0 = fma(u0, u0, b0);
      b1 = fma(u1, u1, b1);
      c0 = fma(v0, v0, c0);
      c1 = fma(v1, v1, c1);
    }
    if (i < hi) {
      const double r0 = r[i], u0 = r0 * sqd[i], v0 = b[i];
      a0 = fma(r0, r0, a0);
      b0 = fma(u0, u0, b0);
      c0 = fma(v0, v0, c0);
    }
    acc[f] = a0 + a1;
    acc[4 + f] = b0 + b1;
    acc[8 + f] = c0 + c1;
  }
  sum_partials<12>(acc, partial);
  if (!last_block(cnt)) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int v = warp; v < 12; v += kRedThreads / 32) {
    const double t = warp_sum(partial + (int64_t)v * kRedBlocks, gridDim.x, lane);
    if (lane == 0) out[v < 4 ? v : v + 4] = t;
  }
}

// The same from the four field sums already in sums[0..3] (bn2 may alias sums).
__global__ void k_weights_sums(const double* sums, const double* __restrict__ unorm2, double floor_rel,
                               double* __restrict__ wf, double* __restrict__ iwf, double* bn2) {
  if (threadIdx.x != 0) return;
  double s4[4];
  for (int f = 0; f < 4; ++f) s4[f] = sums[f];
  weights_of(s4, unorm2, floor_rel, 0, wf, iwf, bn2);
}

// dst = src when the second Gram-Schmidt pass ran (flag), else unchanged.
__global__ void k_take_if(double* dst, const double* __restrict__ src, const double* __restrict__ flag) {
  if (threadIdx.x == 0 && *flag != 0.0) *dst = *src;
}

// Launches of the above for the slab decomposition, whose sums pass through
// an allreduce between a kernel and its decision.
__global__ void k_givens(double* hs, HLay L, int k, int* kdev, int refine) { givens_block(hs, L, k, kdev, refine); }
__global__ void k_reorth_flag(double* hs, HLay L, int k, double eta2) {
  if (threadIdx.x == 0) reorth_test(hs, L, k, eta2);
}

// H y = g by one warp, row by row from the last: the lanes load the next row
// (strided: columns are contiguous) while lane 0 runs the current row's
// dependent chain out of shared memory.  With lane 0 loading for itself the
// substitution took 24 us at 13 columns.
__global__ void __launch_bounds__(32) k_backsolve(double* hs, HLay L, int kk) {
  __shared__ double row[2][130], y[130];
  const int lane = threadIdx.x, ld = L.m + 1;
  const double* H = hs + L.H;
  for (int j = kk - 1 + lane; j < kk; j += 32) row[(kk - 1) & 1][j] = H[(int64_t)j * ld + kk - 1];
  double gi = lane == 0 ? hs[L.g + kk - 1] : 0.0;
  __syncwarp();
  for (int i = kk - 1; i >= 0; --i) {
    double nx[4], gn = 0.0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int j = i - 1 + lane + 32 * q;
      nx[q] = i > 0 && j < kk ? H[(int64_t)j * ld + i - 1] : 0.0;
    }
    if (lane == 0) {
      if (i > 0) gn = hs[L.g + i - 1];
      const double* r = row[i & 1];
      double s = gi;
      for (int j = i + 1; j < kk; ++j) s -= r[j] * y[j];
      const double d = r[i];
      y[i] = d != 0.0 ? s / d : 0.0;
      gi = gn;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int j = i - 1 + lane + 32 * q;
      if (i > 0 && j < kk) row[(i - 1) & 1][j] = nx[q];
    }
    __syncwarp();
  }
  for (int i = lane; i < kk; i += 32) hs[L.y + i] = y[i];
}

// Reduced-mode condensation / back-substitution helpers (per node).
__global__ void k_condense(Grid g, int nc, double tau, const int32_t* __restrict__ eidx,
                           const uint8_t* __restrict__ label, const double* __restrict__ Aj,
                           const double* __restrict__ Mj, const double* __restrict__ betaj,
                           const double* __restrict__ ge, const double* __restrict__ gc,
                           const double* __restrict__ gs, const double* __restrict__ b,
                           const double* __restrict__ yc, double* __restrict__ bm, int trans) {
  const int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t nn = g.nn;
  if (n >= nn) return;
  const int32_t e = eidx[n];
  double r0 = b[n], r1 = b[nn + n], r2 = b[2 * nn + n];
  if (e >= 0) {
    const bool act = label[n] & kLabActive;
    const double A = Aj[e];
    const double yN = yc[(int64_t)e * nc + nc - 1];
    if (!trans) {
      const double gsv = gs[e];
      if (act) r0 -= A * gsv * yN;
      r1 -= -A * gsv * yN;
      r2 -= -tau * A * gsv * yN;
    } else {
      const double mb = Mj[e] * betaj[e];
      if (act) r0 -= mb * ge[e] * yN;
      r1 -= mb * (-ge[e]) * yN;
      r2 -= mb * gc[e] * yN;
    }
  }
  bm[n] = r0;
  bm[nn + n] = r1;
  bm[2 * nn + n] = r2;
}

__global__ void k_surface_coupling(int64_t NE, double tau, const int32_t* __restrict__ enode, int64_t nn,
                                   const uint8_t* __restrict__ label, const double* __restrict__ Aj,
                                   const double* __restrict__ Mj, const double* __restrict__ betaj,
                                   const double* __restrict__ ge, const double* __restrict__ gc,
                                   const double* __restrict__ gs, const double* __restrict__ xm,
                                   double* __restrict__ tN, int trans) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= NE) return;
  const int64_t n = enode[e];
  const bool act = label[n] & kLabActive;
  if (!trans) {
    tN[e] = Mj[e] * betaj[e] * ((act ? ge[e] * xm[n] : 0.0) - ge[e] * xm[nn + n] + gc[e] * xm[2 * nn + n]);
  } else {
    const double A = Aj[e];
    tN[e] = gs[e] * ((act ? A * xm[n] : 0.0) - A * xm[nn + n] - tau * A * xm[2 * nn + n]);
  }
}

// Vectors up to the size of a cell whose whole V-cycle is one launch (8,192
// nodes, three fields) are partitioned finer: their kernels are latency
// bound.  Above it the dots and norms of the Arnoldi process keep one partition
// at every size; the right-hand side's field norms do above 4 kSmallLen
// entries (norm_blocks).
constexpr int64_t kSmallLen = 3 * 8192;

struct Reducer {
  p4d_ctx* c;
  // eight elements per thread; on the smallest vectors one: a warp's FP64
  // instruction takes an SM's FP64 unit 20 clocks, so few elements per SM
  // count (6,075 elements, 12 dots: 14 us with 3 blocks, 10 us with 12)
  int nblk(int64_t len) const {
    const int64_t per = (int64_t)kRedThreads * (len <= kSmallLen ? 1 : 8);
    const int64_t want = (len + per - 1) / per;
    return (int)std::min<int64_t>(kRedBlocks, std::max<int64_t>(1, want));
  }
  // out[0..kp1) = V^T w, out[kp1] = w.w (optional)
  // flag (device, optional): the pass runs only if *flag != 0; otherwise out
  // is zeroed (zero_if_skipped) or left unchanged
  void mdot(const double* V, int64_t ldv, int kp1, const double* w, int64_t len, bool ww, double* out,
            const double* flag = nullptr, int zero_if_skipped = 0) {
    const int nb = nblk(len);
    if (kp1 == 0) launch_group<0>(ww, V, ldv, 0, kp1, w, len, nb, out, flag, zero_if_skipped);
    for (int g0 = 0; g0 < kp1; g0 += kDotGroup)
      dispatch(std::min(kDotGroup, kp1 - g0), ww && g0 == 0, V, ldv, g0, kp1, w, len, nb, out, flag, zero_if_skipped);
  }
  template <int NG>
  void launch_group(bool ww, const double* V, int64_t ldv, int g0, int kp1, const double* w, int64_t len, int nb,
                    double* out, const double* flag, int z) {
    if (ww) ::p4d::count_launch(), k_mdot<NG, true><<<nb, kRedThreads, 0, c->stream>>>(V, ldv, g0, kp1, w, len, c->part, out, c->red_cnt, flag, z);
    else ::p4d::count_launch(), k_mdot<NG, false><<<nb, kRedThreads, 0, c->stream>>>(V, ldv, g0, kp1, w, len, c->part, out, c->red_cnt, flag, z);
  }
  void dispatch(int ng, bool ww, const double* V, int64_t ldv, int g0, int kp1, const double* w, int64_t len, int nb,
                double* out, const double* flag, int z) {
    switch (ng) {
#define P4D_MDOT_CASE(K) \
  case K: launch_group<K>(ww, V, ldv, g0, kp1, w, len, nb, out, flag, z); break;
      P4D_MDOT_CASE(1) P4D_MDOT_CASE(2) P4D_MDOT_CASE(3) P4D_MDOT_CASE(4) P4D_MDOT_CASE(5) P4D_MDOT_CASE(6)
      P4D_MDOT_CASE(7) P4D_MDOT_CASE(8) P4D_MDOT_CASE(9) P4D_MDOT_CASE(10) P4D_MDOT_CASE(11) P4D_MDOT_CASE(12)
      P4D_MDOT_CASE(13) P4D_MDOT_CASE(14) P4D_MDOT_CASE(15) P4D_MDOT_CASE(16)
#undef P4D_MDOT_CASE
      default: break;
    }
  }
  // w -= V h over kp1 vectors, finished as fin says
  void maxpy(const double* V, int64_t ldv, int kp1, const double* h, double* w, int64_t len, double sign,
             const double* flag, const Fin& fin, unsigned gb) {
    switch (kp1 & 7) {
#define P4D_MAXPY_CASE(R) \
  case R: ::p4d::count_launch(), k_maxpy<R><<<std::min(gb, 4u * 152u), kBlock, 0, c->stream>>>(V, ldv, kp1, h, w, len, sign, flag, c->part, c->red_cnt, (int)gb, fin); break;
      P4D_MAXPY_CASE(0) P4D_MAXPY_CASE(1) P4D_MAXPY_CASE(2) P4D_MAXPY_CASE(3)
      P4D_MAXPY_CASE(4) P4D_MAXPY_CASE(5) P4D_MAXPY_CASE(6) P4D_MAXPY_CASE(7)
#undef P4D_MAXPY_CASE
    }
  }
  static Fin norm_to(double* out, int zero_if_skipped = 0) {
    Fin f;
    f.mode = kFinNorm;
    f.norm = out;
    f.zero_if_skipped = zero_if_skipped;
    return f;
  }
};

// Blocks of a sum over len entries: four per thread on the smallest vectors
// (608 blocks took 13 us for 24 k entries, mostly in the last sum).  Up to 4
// kSmallLen entries (32,768 nodes of three fields, about 14,000 nodes with
// their particles) the field norms, and with them the Krylov weights, depend
// on this partition in their last bits.
inline int norm_blocks(int64_t len) {
  return len <= 4 * kSmallLen ? (int)std::max<int64_t>(1, len / (4 * kRedThreads)) : kRedBlocks;
}

}  // namespace

namespace {

// ---------------------------------------------------------------- FGMRES driver
// One solve advanced in phases: a launch phase issues work on c->stream and
// returns; its read phase runs after that stream has been synchronized.  The
// single-cell driver (fgmres) synchronizes after each launch phase; the
// batched driver (fgmres_batched) runs every cell's launch phase, then one
// synchronization for all, then every cell's read phase, with the Arnoldi
// steps of all cells in one graph per Krylov column.

// Condition of a cell's conditional (IF) node in a batched step graph.
__global__ void k_set_active(cudaGraphConditionalHandle h, const int* __restrict__ active) {
  if (threadIdx.x == 0) cudaGraphSetConditional(h, *active ? 1u : 0u);
}

// Device gate of a graph-driven restart cycle (in hs after the misc scalars):
// [0] stop, [1] steps run, [2] residual estimate and [3] status of the last
// step, [4] step limit of the cycle, [5] ||s.b_k||, [6] rtol.
constexpr int kGateOff = 48;

// Pinned mirror (hs_h): [0..11] right-hand-side norms at the start, [0..32]
// the report at the end, [0..1] a step's status when stepped from the host,
// then
constexpr int kBetaOff = 40;   // beta of a cycle
constexpr int kTrueOff = 41;   // squared true residual at a cycle's end
constexpr int kGateRead = 44;  // gate[0..5] after a segment of a cycle

struct FgRun;
void fg_release(FgRun& r);

struct FgRun {
  p4d_ctx* c = nullptr;
  const double* b = nullptr;
  double* x = nullptr;
  int trans = 0;
  bool full = false;
  int64_t nn = 0, len = 0;
  int m = 0;
  HLay L{};
  unsigned gb = 0;
  double tau = 0.0;
  const double* bk = nullptr;   // Krylov right-hand side (unscaled)
  double bnorm = 0.0, est = 1.0;
  int iters = 0, restarts = 0, kk = 0;
  p4d_status st = P4D_ERR_NOT_CONVERGED;
  bool stop = false;            // the solve ended at the start of a restart cycle
  bool cycle_done = true;       // no further Arnoldi step in the current cycle
  cudaEvent_t ev0 = nullptr, ev1 = nullptr;
  double* misc() const { return c->hs + L.misc; }
  bool active() const { return !stop && st == P4D_ERR_NOT_CONVERGED && iters < c->prm.maxit; }
  FgRun() = default;
  FgRun(const FgRun&) = delete;
  FgRun& operator=(const FgRun&) = delete;
  ~FgRun() { fg_release(*this); }   // the timing events, also on an early error return
};

void fg_release(FgRun& r) {
  if (r.ev0) cudaEventDestroy(r.ev0);
  if (r.ev1) cudaEventDestroy(r.ev1);
  r.ev0 = r.ev1 = nullptr;
}

// Field weights of the right-hand side, the particle condensation (REDUCED)
// and the norms of the Krylov right-hand side.
p4d_status fg_begin(FgRun& r, p4d_ctx* c, const double* b, double* x, int trans) {
  r.c = c;
  r.b = b;
  r.x = x;
  r.trans = trans;
  r.nn = c->g.nn;
  r.full = c->prm.mode == 0;
  r.len = r.full ? c->ndof : 3 * r.nn;
  r.m = std::min(c->prm.restart, c->mcap);
  r.L = hlay(c->mcap);
  r.tau = (1.0 - c->prm.tplus) / c->prm.F;
  r.gb = (unsigned)std::min<int64_t>(4 * 152 * 4, (int64_t)nblocks(r.len));
  const HLay& L = r.L;
  double* hs = c->hs;
  prof_reset(c);
  P4D_TRY(cudaEventCreate(&r.ev0));
  P4D_TRY(cudaEventCreate(&r.ev1));
  P4D_TRY(cudaEventRecord(r.ev0, c->stream));
  // per-field weights from the full right-hand side
  {
    ::p4d::count_launch(), k_field_norms<<<norm_blocks(c->ndof), kRedThreads, 0, c->stream>>>(
        b, c->rsqd, r.nn, c->ndof, c->part, c->red_cnt, c->unorm2, 1e-14 / c->prm.rtol, trans, c->wf, c->iwf,
        hs + L.misc + 2 * L.m + 8);
  }
  r.bk = b;
  if (!r.full) {
    // b_m' = b_m - A_mc T^-1 b_c
    P4D_TRYS(particle_solve64(c, b + 3 * r.nn, c->tmp + 3 * r.nn, nullptr, trans));
    ::p4d::count_launch(), k_condense<<<nblocks(r.nn), kBlock, 0, c->stream>>>(
        c->g, c->nc, r.tau, c->eidx, c->label, c->Aj, c->Mj, c->betaj, c->ge, c->gc, c->gs, b, c->tmp + 3 * r.nn,
        c->bred, trans);
    r.bk = c->bred;
  }
  ::p4d::count_launch(), k_field_norms<<<norm_blocks(r.len), kRedThreads, 0, c->stream>>>(
      r.bk, c->rsqd, r.nn, r.len, c->part, c->red_cnt, nullptr, 0.0, 0, nullptr, nullptr, hs + L.misc + 2 * L.m + 16);
  P4D_TRY(cudaMemcpyAsync(c->hs_h, hs + L.misc + 2 * L.m + 8, sizeof(double) * 12, cudaMemcpyDeviceToHost, c->stream));
  P4D_TRY(cudaMemsetAsync(r.misc() + 2 * L.m + 7, 0, sizeof(double), c->stream));   // second passes
  return P4D_OK;
}

// ||s.b_k|| = sqrt(sum_f w_f^2 ||(b_k / sqrt(d))_f||^2); b_k = 0 gives x = 0.
p4d_status fg_bnorm(FgRun& r, bool gated = false) {
  p4d_ctx* c = r.c;
  const double* bn2 = c->hs_h;        // full-b field norms^2 (weights)
  const double* bk2 = c->hs_h + 8;    // Krylov-rhs field norms^2
  double bnorm = 0.0;
  for (int f = 0; f < (r.full ? 4 : 3); ++f) {
    const double wf = bn2[f] > 0 ? 1.0 / std::sqrt(bn2[f]) : 1.0;
    bnorm += wf * wf * bk2[f];
  }
  r.bnorm = std::sqrt(bnorm);
  if (gated) r.bnorm = c->hs_h[kGateRead + 5];   // the value the device gate tests with
  if (r.bnorm == 0.0) {
    P4D_TRY(cudaMemsetAsync(r.x, 0, sizeof(double) * c->ndof, c->stream));
    r.st = P4D_OK;
    r.est = 0.0;
  }
  return P4D_OK;
}

// Start of a restart cycle: V0 = s.(b_k - A x), beta = ||V0||, V0 /= beta.
// gate: also prepare the device gate of a graph-driven cycle.
p4d_status fg_cycle_launch(FgRun& r, bool gate = false) {
  p4d_ctx* c = r.c;
  Reducer R{c};
  double* misc = r.misc();
  const HLay& L = r.L;
  ++r.restarts;
  if (r.full) P4D_TRYS(jvp_full(c, r.x, c->V, r.trans, r.bk, true));
  else if (r.restarts == 1) P4D_TRYS(jvp_start(c, r.x, c->V, r.trans, r.bk));
  else P4D_TRYS(jvp_reduced(c, r.x, c->V, r.trans, r.bk, true));
  R.mdot(c->V, 0, 0, c->V, r.len, true, misc + 2 * L.m + 2);
  Tail t;
  t.mode = 1;
  t.hs = c->hs;
  t.L = L;
  t.kdev = c->kdev;
  if (gate) {
    t.gate = misc + 2 * L.m + kGateOff;
    t.nf = r.full ? 4 : 3;
    t.limit = (double)std::min(r.m, c->prm.maxit - r.iters);
    t.rtol = c->prm.rtol;
  }
  ::p4d::count_launch(), k_scale<<<std::min(r.gb, 4u * 152u), kBlock, 0, c->stream>>>(c->V, c->V, r.len, misc + 2 * L.m + 2, t);
  P4D_TRY(cudaMemcpyAsync(c->hs_h + kBetaOff, misc + 2 * L.m + 5, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
  return P4D_OK;
}

void fg_cycle_read(FgRun& r) {
  const double beta = r.c->hs_h[kBetaOff];
  r.est = beta / r.bnorm;
  r.kk = 0;
  r.cycle_done = false;
  if (!std::isfinite(beta)) {
    r.st = P4D_ERR_NONFINITE;
    r.stop = true;
  } else if (beta <= r.c->prm.rtol * r.bnorm) {
    r.st = P4D_OK;
    r.stop = true;
  }
  if (r.stop) r.cycle_done = true;
}

// Arnoldi step k: z_k = P^-1 (s^-1 v_k), w = s.J z_k, CGS (second pass only
// when needed), Givens, v_{k+1} = w / h_{k+1,k}; the residual estimate and
// status go where t says (batch status or cycle gate on the device), or to
// the host mirror.
p4d_status fg_step_body(FgRun& r, int k, bool graph_precond, Tail t) {
  p4d_ctx* c = r.c;
  Reducer R{c};
  double* misc = r.misc();
  const HLay& L = r.L;
  double* zk = c->Z + (int64_t)k * r.len;
  double* w = c->V + (int64_t)(k + 1) * r.len;
  prof_mark(c, 0);
  P4D_TRYS(precond_column(c, r.trans, graph_precond));   // k read from c->kdev
  prof_mark(c, 0);
  prof_mark(c, 1);
  const bool u = precond_leaves_u(c, r.trans);
  if (r.full) P4D_TRYS(jvp_full(c, zk, w, r.trans, nullptr, true, u));
  else P4D_TRYS(jvp_reduced(c, zk, w, r.trans, nullptr, true, u));
  prof_mark(c, 1);
  prof_mark(c, 2);
  const double* flag = misc + 2 * L.m + 6;
  const int refine = c->prm.cgs_refine;
  Fin fin = Reducer::norm_to(misc + 2 * L.m + 2);
  fin.hs = c->hs;
  fin.L = L;
  fin.k = k;
  fin.eta2 = refine == 2 ? 2.0 : 0.49;
  fin.kdev = c->kdev;
  fin.refine = refine;
  R.mdot(c->V, r.len, k + 1, w, r.len, true, misc);   // h1, ||w||^2 before
  fin.mode = refine > 0 ? kFinReorth : kFinGivens;
  R.maxpy(c->V, r.len, k + 1, misc, w, r.len, 1.0, nullptr, fin, r.gb);   // ||w||^2 after
  if (refine > 0) {
    R.mdot(c->V, r.len, k + 1, w, r.len, false, misc + L.m + 1, flag, 1);   // h2 (or 0)
    // ||w||^2 after the second pass (left unchanged when it is skipped)
    fin.mode = kFinGivens;
    R.maxpy(c->V, r.len, k + 1, misc + L.m + 1, w, r.len, 1.0, flag, fin, r.gb);
  }
  const bool host = !t.stat && !t.gate;
  t.mode = 2;
  t.hs = c->hs;
  t.L = L;
  t.k = k;
  ::p4d::count_launch(), k_scale<<<std::min(r.gb, 4u * 152u), kBlock, 0, c->stream>>>(w, w, r.len, misc + 2 * L.m + 2, t);
  prof_mark(c, 2);
  if (host) P4D_TRY(cudaMemcpyAsync(c->hs_h, misc + 2 * L.m + 3, 2 * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
  return P4D_OK;
}

// s2 = (residual estimate, status) of step k.
void fg_step_read(FgRun& r, int k, const double* s2) {
  ++r.iters;
  r.kk = k + 1;
  r.est = s2[0] / r.bnorm;
  const double stt = s2[1];
  if (stt == 2.0) r.st = P4D_ERR_NONFINITE;
  else if (r.est <= r.c->prm.rtol) r.st = P4D_OK;
  else if (stt == 1.0) r.st = P4D_OK;
  if (r.st != P4D_ERR_NOT_CONVERGED || r.kk >= r.m || r.iters >= r.c->prm.maxit) r.cycle_done = true;
}

// End of a cycle: x += Z y; when the estimate converged, the true residual.
p4d_status fg_cycle_end_launch(FgRun& r) {
  p4d_ctx* c = r.c;
  Reducer R{c};
  double* misc = r.misc();
  const HLay& L = r.L;
  if (r.kk > 0) {
    ::p4d::count_launch(), k_backsolve<<<1, 32, 0, c->stream>>>(c->hs, L, r.kk);
    // x += Z y  (k_maxpy computes w -= sum h_i V_i; use sign -1)
    R.maxpy(c->Z, r.len, r.kk, c->hs + L.y, r.x, r.len, -1.0, nullptr, Fin{}, r.gb);
  }
  if (r.st == P4D_OK) {
    if (r.full) P4D_TRYS(jvp_full(c, r.x, c->V, r.trans, r.bk, true));
    else P4D_TRYS(jvp_reduced(c, r.x, c->V, r.trans, r.bk, true));
    R.mdot(c->V, 0, 0, c->V, r.len, true, misc + 2 * L.m + 2);
    P4D_TRY(cudaMemcpyAsync(c->hs_h + kTrueOff, misc + 2 * L.m + 2, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
  }
  return P4D_OK;
}

// Confirmation by the true residual (only after st == OK was launched).
void fg_cycle_end_read(FgRun& r) {
  if (r.st != P4D_OK) return;
  r.est = std::sqrt(r.c->hs_h[kTrueOff]) / r.bnorm;
  if (!(r.est <= r.c->prm.rtol) && r.iters < r.c->prm.maxit) r.st = P4D_ERR_NOT_CONVERGED;
  if (!std::isfinite(r.est)) r.st = P4D_ERR_NONFINITE;
}

// Particle back-substitution (REDUCED) and the final true residual.
p4d_status fg_finish_launch(FgRun& r) {
  p4d_ctx* c = r.c;
  const HLay& L = r.L;
  const int64_t nn = r.nn;
  if (!r.full) {
    // x_c = T^-1 (b_c - A_cm x_m)
    ::p4d::count_launch(), k_surface_coupling<<<nblocks(std::max<int64_t>(1, c->NE)), kBlock, 0, c->stream>>>(
        c->NE, r.tau, c->enode, nn, c->label, c->Aj, c->Mj, c->betaj, c->ge, c->gc, c->gs, r.x, c->tloc, r.trans);
    P4D_TRYS(particle_solve64(c, r.b + 3 * nn, r.x + 3 * nn, c->tloc, r.trans));
  }
  // final true residual of the full system in the scaled norm
  P4D_TRYS(jvp_full(c, r.x, c->r0, r.trans, r.b, true));
  // and unscaled: ||(b - J x)_f||^2 = ||(sqrt(d) r0)_f||^2 / w_f^2, ||b_f||^2
  ::p4d::count_launch(), k_final_norms<<<norm_blocks(c->ndof), kRedThreads, 0, c->stream>>>(
      c->r0, c->sqd, r.b, nn, c->ndof, c->part, c->red_cnt, r.misc() + 2 * L.m + 24);
  P4D_TRY(cudaEventRecord(r.ev1, c->stream));
  P4D_TRY(cudaMemcpyAsync(c->hs_h, r.misc() + 2 * L.m + 7, sizeof(double) * 33, cudaMemcpyDeviceToHost, c->stream));
  return P4D_OK;
}

void fg_finish_read(FgRun& r, p4d_info* info) {
  p4d_ctx* c = r.c;
  float ms = 0.f;
  cudaEventElapsedTime(&ms, r.ev0, r.ev1);
  fg_release(r);
  if (!info) return;
  std::memset(info, 0, sizeof(*info));
  info->iters = r.iters;
  info->restarts = r.restarts;
  info->status = r.st;
  info->reorth = (int)c->hs_h[0];
  const double* bn2 = c->hs_h + 1;      // field norms^2 of b/sqd (weights: 1/sqrt)
  const double* rr = c->hs_h + 17;      // field norms^2 of s.(b - Jx)
  double tot_r = 0.0;
  const double tot_b = bn2[4];          // ||s.b||^2
  for (int f = 0; f < 4; ++f) {
    info->rel_res_block[f] = std::sqrt(rr[f]);   // relative to the field's (floored) rhs norm
    tot_r += rr[f];
  }
  info->rel_res = tot_b > 0 ? std::sqrt(tot_r / tot_b) : std::sqrt(tot_r);
  const double* ru = c->hs_h + 25;      // field norms^2 of sqrt(d) s.(b - Jx)
  const double* bu = c->hs_h + 29;      // field norms^2 of b
  double ur = 0.0, ub = 0.0;
  for (int f = 0; f < 4; ++f) {
    const double rf = ru[f] * (bn2[f] > 0 ? bn2[f] : 1.0);   // 1 / w_f^2
    info->rel_res_block_unscaled[f] = bu[f] > 0 ? std::sqrt(rf / bu[f]) : std::sqrt(rf);
    ur += rf;
    ub += bu[f];
  }
  info->rel_res_unscaled = ub > 0 ? std::sqrt(ur / ub) : std::sqrt(ur);
  info->nsolves = 1;
  info->iters_total = r.iters;
  info->ms_total = ms;
  if (c->prm.profile) {
    int n = 0;
    info->ms_precond = prof_sum(c, 0, nullptr);
    info->ms_jvp = prof_sum(c, 1, &n);
    info->n_jvp = n;
    info->ms_ortho = prof_sum(c, 2, nullptr);
    info->ms_smooth0 = prof_sum(c, 3, &n);
    info->n_smooth0 = n;
  }
}

// What body() launches on c->stream, captured into a new (not instantiated)
// graph; kernels = its kernel launches.
template <typename F>
p4d_status capture_body(p4d_ctx* c, cudaGraph_t* out, long long* kernels, F&& body) {
  cudaStream_t user = c->stream;
  c->stream = c->cap_stream;
  *kernels = 0;
  capture_counter(kernels);
  *out = nullptr;
  p4d_status st = P4D_OK;
  if (cudaStreamBeginCapture(c->cap_stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) st = P4D_ERR_CUDA;
  if (st == P4D_OK) {
    st = body();
    if (cudaStreamEndCapture(c->cap_stream, out) != cudaSuccess && st == P4D_OK) st = P4D_ERR_CUDA;
  }
  capture_counter(nullptr);
  c->stream = user;
  if (st != P4D_OK) {
    cudaGetLastError();
    if (*out) cudaGraphDestroy(*out);
    *out = nullptr;
  }
  return st;
}

// Steps [k0, k0 + kSegSteps) of a restart cycle as one graph: each Arnoldi
// step under a conditional (IF) node, the first one's condition set by
// k_gate from the device gate, the others' by the step before (default 0).
// A cycle is launched segment by segment: an IF node that is not taken costs
// 10 us, so the 17 idle steps of a 13-iteration solve in one graph of
// restart 30 cost 0.2 of 2.1 ms, while the host's check between segments
// costs about 15 us per eight steps; and only the segments in use are captured.
constexpr int kSegSteps = 8;

p4d_status segment_graph(FgRun& r, int k0, p4d_ctx::CycleGraph::Seg*& out) {
  p4d_ctx* c = r.c;
  p4d_ctx::CycleGraph& cg = c->cyc[r.trans ? 1 : 0][r.full ? 1 : 0];
  const size_t si = (size_t)(k0 / kSegSteps);
  if (cg.m != r.m) {   // another restart length: the last segment may end elsewhere
    for (auto& sg : cg.seg)
      if (sg.exec) cudaGraphExecDestroy(sg.exec);
    cg.seg.clear();
    cg.m = r.m;
  }
  if (cg.seg.size() <= si) cg.seg.resize(si + 1);
  p4d_ctx::CycleGraph::Seg& sg = cg.seg[si];
  out = &sg;
  if (sg.exec) return P4D_OK;
  const int n = std::min(kSegSteps, r.m - k0);
  sg.kernels.assign(n, 0);
  double* gate = r.misc() + 2 * r.L.m + kGateOff;
  cudaGraph_t G = nullptr;
  P4D_TRY(cudaGraphCreate(&G, 0));
  p4d_status st = P4D_OK;
  cudaGraphConditionalHandle h[kSegSteps];
  for (int q = 0; q < n && st == P4D_OK; ++q)
    if (cudaGraphConditionalHandleCreate(&h[q], G, 0, cudaGraphCondAssignDefault) != cudaSuccess) st = P4D_ERR_CUDA;
  cudaGraphNode_t prev = nullptr;
  if (st == P4D_OK) {
    const double* gc = gate;
    int kk = k0;
    void* args[] = {&h[0], &gc, &kk};
    cudaKernelNodeParams kp = {};
    kp.func = (void*)k_gate;
    kp.gridDim = dim3(1);
    kp.blockDim = dim3(32);
    kp.kernelParams = args;
    if (cudaGraphAddKernelNode(&prev, G, nullptr, 0, &kp) != cudaSuccess) st = P4D_ERR_CUDA;
  }
  for (int q = 0; q < n && st == P4D_OK; ++q) {
    cudaGraph_t step = nullptr;
    long long kc = 0;
    Tail t;
    t.gate = gate;
    t.next = q + 1 < n;
    if (t.next) t.handle = h[q + 1];
    st = capture_body(c, &step, &kc, [&]() { return fg_step_body(r, k0 + q, false, t); });
    if (st != P4D_OK) break;
    cudaGraphNode_t cn = nullptr, ch = nullptr;
    cudaGraphNodeParams cp = {};
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.type = cudaGraphCondTypeIf;
    cp.conditional.size = 1;
    cp.conditional.handle = h[q];
    if (cudaGraphAddNode(&cn, G, &prev, nullptr, 1, &cp) != cudaSuccess) st = P4D_ERR_CUDA;
    if (st == P4D_OK && cudaGraphAddChildGraphNode(&ch, cp.conditional.phGraph_out[0], nullptr, 0, step) != cudaSuccess)
      st = P4D_ERR_CUDA;
    cudaGraphDestroy(step);
    prev = cn;
    sg.kernels[q] = kc;
  }
  if (st == P4D_OK && cudaGraphInstantiate(&sg.exec, G, 0) != cudaSuccess) st = P4D_ERR_CUDA;
  cudaGraphDestroy(G);
  if (st != P4D_OK) {
    cudaGetLastError();
    sg.exec = nullptr;
  }
  return st;
}

// Launch the segment that starts at step k0, and read the gate after it.
p4d_status fg_segment_launch(FgRun& r, int k0) {
  p4d_ctx* c = r.c;
  p4d_ctx::CycleGraph::Seg* sg = nullptr;
  P4D_TRYS(segment_graph(r, k0, sg));
  P4D_TRY(cudaGraphLaunch(sg->exec, c->stream));
  P4D_TRY(cudaMemcpyAsync(c->hs_h + kGateRead, r.misc() + 2 * r.L.m + kGateOff, 6 * sizeof(double),
                          cudaMemcpyDeviceToHost, c->stream));
  return P4D_OK;
}

// After the synchronization: the steps the segment ran.
p4d_status fg_segment_read(FgRun& r, int k0) {
  p4d_ctx* c = r.c;
  const p4d_ctx::CycleGraph::Seg& sg = c->cyc[r.trans ? 1 : 0][r.full ? 1 : 0].seg[k0 / kSegSteps];
  const int nrun = (int)c->hs_h[kGateRead + 1] - k0;
  long long launched = 1;
  for (int q = 0; q < nrun && q < (int)sg.kernels.size(); ++q) launched += sg.kernels[q];
  count_launches(launched);
  if (nrun < 1 || nrun > (int)sg.kernels.size()) return P4D_ERR_CUDA;   // the first step always runs (limit > k0, no stop)
  r.iters += nrun - 1;
  fg_step_read(r, k0 + nrun - 1, c->hs_h + kGateRead + 2);
  return P4D_OK;
}

}  // namespace

p4d_status fgmres(p4d_ctx* c, const double* b, double* x, p4d_info* info, int trans) {
  FgRun r;
  const bool graph = !c->prm.profile;   // per-kernel events cannot sit inside a graph
  P4D_TRYS(fg_begin(r, c, b, x, trans));
  bool begun = false, finished = false;
  if (!graph) {
    P4D_TRY(cudaStreamSynchronize(c->stream));
    P4D_TRYS(fg_bnorm(r));
    begun = true;
  }
  while (r.active()) {
    // the first segment is launched before the host has seen the norms: the
    // device gate makes the same tests and lets none of its steps run
    // when there is nothing to solve
    P4D_TRYS(fg_cycle_launch(r, graph));
    if (graph) P4D_TRYS(fg_segment_launch(r, 0));
    P4D_TRY(cudaStreamSynchronize(c->stream));
    if (!begun) {
      P4D_TRYS(fg_bnorm(r, true));
      begun = true;
      if (r.st == P4D_OK) {   // b_k = 0
        r.restarts = 0;
        break;
      }
    }
    fg_cycle_read(r);
    if (r.stop) break;
    if (graph) {
      P4D_TRYS(fg_segment_read(r, 0));
      for (int k = kSegSteps; !r.cycle_done; k += kSegSteps) {
        P4D_TRYS(fg_segment_launch(r, k));
        P4D_TRY(cudaStreamSynchronize(c->stream));
        P4D_TRYS(fg_segment_read(r, k));
      }
    } else {
      for (int k = 0; !r.cycle_done; ++k) {
        P4D_TRYS(fg_step_body(r, k, true, Tail{}));
        P4D_TRY(cudaStreamSynchronize(c->stream));
        fg_step_read(r, k, c->hs_h);
      }
    }
    P4D_TRYS(fg_cycle_end_launch(r));
    if (r.st == P4D_ERR_NONFINITE) break;
    if (r.st == P4D_OK) {
      // the report's work runs with the confirmation (again when it fails)
      P4D_TRYS(fg_finish_launch(r));
      P4D_TRY(cudaStreamSynchronize(c->stream));
      fg_cycle_end_read(r);
      finished = r.st != P4D_ERR_NOT_CONVERGED;
    }
  }
  if (!finished) {
    P4D_TRYS(fg_finish_launch(r));
    P4D_TRY(cudaStreamSynchronize(c->stream));
  }
  fg_finish_read(r, info);
  return r.st;
}

// ---------------------------------------------------------------- batched driver
namespace {


// The batched graph of Krylov column k: for every cell whose restart length
// exceeds k, set_active(cell) -> IF(cell active) { Arnoldi step k of the
// cell }.  The cells' chains are independent nodes, so the GPU runs them
// concurrently.
p4d_status batch_step_graph(p4d_batch_ctx* B, std::vector<FgRun>& R, int k, int trans) {
  auto& vec = B->gk[trans ? 1 : 0];
  if ((int)vec.size() <= k) vec.resize(k + 1);
  p4d_batch_ctx::StepGraph& sg = vec[k];
  if (sg.exec) return P4D_OK;
  const int n = (int)B->cells.size();
  sg.kernels.assign(n, 0);
  cudaGraph_t G = nullptr;
  P4D_TRY(cudaGraphCreate(&G, 0));
  p4d_status st = P4D_OK;
  for (int i = 0; i < n && st == P4D_OK; ++i) {
    FgRun& r = R[i];
    if (k >= r.m) continue;
    cudaGraph_t step = nullptr;
    long long kc = 0;
    Tail t;
    t.stat = B->stat_dev + 2 * i;
    st = capture_body(r.c, &step, &kc, [&]() { return fg_step_body(r, k, false, t); });
    if (st != P4D_OK) break;
    cudaGraphConditionalHandle h;
    cudaGraphNode_t kn = nullptr, cn = nullptr, ch = nullptr;
    const int* act = B->active_dev + i;
    void* args[] = {&h, &act};
    cudaKernelNodeParams kp = {};
    kp.func = (void*)k_set_active;
    kp.gridDim = dim3(1);
    kp.blockDim = dim3(32);
    kp.kernelParams = args;
    cudaGraphNodeParams cp = {};
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.type = cudaGraphCondTypeIf;
    cp.conditional.size = 1;
    if (cudaGraphConditionalHandleCreate(&h, G, 0, cudaGraphCondAssignDefault) != cudaSuccess ||
        cudaGraphAddKernelNode(&kn, G, nullptr, 0, &kp) != cudaSuccess)
      st = P4D_ERR_CUDA;
    cp.conditional.handle = h;
    if (st == P4D_OK && cudaGraphAddNode(&cn, G, &kn, nullptr, 1, &cp) != cudaSuccess) st = P4D_ERR_CUDA;
    if (st == P4D_OK && cudaGraphAddChildGraphNode(&ch, cp.conditional.phGraph_out[0], nullptr, 0, step) != cudaSuccess)
      st = P4D_ERR_CUDA;
    cudaGraphDestroy(step);
    sg.kernels[i] = kc;
  }
  if (st == P4D_OK && cudaGraphInstantiate(&sg.exec, G, 0) != cudaSuccess) st = P4D_ERR_CUDA;
  cudaGraphDestroy(G);
  if (st != P4D_OK) {
    cudaGetLastError();
    sg.exec = nullptr;
  }
  return st;
}

p4d_status sync_cells(p4d_batch_ctx* B) {
  for (size_t i = 0; i < B->cells.size(); ++i) {
    bool seen = false;
    for (size_t j = 0; j < i && !seen; ++j) seen = B->cells[j]->stream == B->cells[i]->stream;
    if (!seen) P4D_TRY(cudaStreamSynchronize(B->cells[i]->stream));
  }
  return P4D_OK;
}

}  // namespace

void batch_drop_graphs(p4d_batch_ctx* B) {
  for (auto& v : B->gk) {
    for (auto& g : v)
      if (g.exec) cudaGraphExecDestroy(g.exec);
    v.clear();
  }
}

p4d_status fgmres_batched(p4d_batch_ctx* B, const double* const* b, double* const* x, p4d_info* info, int trans) {
  const int n = (int)B->cells.size();
  // step graphs captured before a cell's options changed are stale
  bool stale = (int)B->gen.size() != n;
  for (int i = 0; i < n && !stale; ++i) stale = B->gen[i] != B->cells[i]->graph_gen;
  if (stale) {
    batch_drop_graphs(B);
    B->gen.resize(n);
    for (int i = 0; i < n; ++i) B->gen[i] = B->cells[i]->graph_gen;
  }
  std::vector<FgRun> R(n);
  for (int i = 0; i < n; ++i) P4D_TRYS(fg_begin(R[i], B->cells[i], b[i], x[i], trans));
  P4D_TRYS(sync_cells(B));
  for (int i = 0; i < n; ++i) P4D_TRYS(fg_bnorm(R[i]));
  std::vector<int> cyc;
  while (true) {
    cyc.clear();
    for (int i = 0; i < n; ++i)
      if (R[i].active()) cyc.push_back(i);
    if (cyc.empty()) break;
    for (int i : cyc) P4D_TRYS(fg_cycle_launch(R[i]));
    P4D_TRYS(sync_cells(B));
    for (int i : cyc) fg_cycle_read(R[i]);
    // Arnoldi steps in lockstep; a cell leaves the cycle when its step says so
    for (int k = 0;; ++k) {
      bool any = false;
      for (int i = 0; i < n; ++i) {
        const bool a = !R[i].cycle_done && k < R[i].m;
        B->active_h[i] = a ? 1 : 0;
        any = any || a;
      }
      if (!any) break;
      P4D_TRYS(batch_step_graph(B, R, k, trans));
      const p4d_batch_ctx::StepGraph& sg = B->gk[trans ? 1 : 0][k];
      long long launched = 0;
      for (int i = 0; i < n; ++i)
        if (sg.kernels[i] > 0) launched += 1 + (B->active_h[i] ? sg.kernels[i] : 0);
      count_launches(launched);
      P4D_TRY(cudaMemcpyAsync(B->active_dev, B->active_h, sizeof(int) * n, cudaMemcpyHostToDevice, B->stream));
      P4D_TRY(cudaGraphLaunch(sg.exec, B->stream));
      P4D_TRY(cudaMemcpyAsync(B->stat_h, B->stat_dev, sizeof(double) * 2 * n, cudaMemcpyDeviceToHost, B->stream));
      P4D_TRY(cudaStreamSynchronize(B->stream));
      for (int i = 0; i < n; ++i)
        if (B->active_h[i]) fg_step_read(R[i], k, B->stat_h + 2 * i);
    }
    bool confirm = false;
    for (int i : cyc)
      if (!R[i].stop) {
        P4D_TRYS(fg_cycle_end_launch(R[i]));
        confirm = confirm || R[i].st == P4D_OK;
      }
    if (confirm) {
      P4D_TRYS(sync_cells(B));
      for (int i : cyc)
        if (!R[i].stop) fg_cycle_end_read(R[i]);
    }
  }
  for (int i = 0; i < n; ++i) P4D_TRYS(fg_finish_launch(R[i]));
  P4D_TRYS(sync_cells(B));
  p4d_status out = P4D_OK;
  for (int i = 0; i < n; ++i) {
    fg_finish_read(R[i], info ? info + i : nullptr);
    if (out == P4D_OK && R[i].st != P4D_OK) out = R[i].st;
  }
  return out;
}

// ---------------------------------------------------------------- slab-decomposed driver
// FGMRES over the z slabs of one cell (REDUCED mode, J x = b).  Every slab
// runs the single-cell steps on its own rows.  The Krylov vectors keep their
// ghost rows at zero, so an inner product is the allreduce of the slabs'
// partial sums, and every slab repeats the Givens update on the same reduced
// scalars (identical on all slabs).  The operator is the cell's J: before
// each application the ghost planes of its input receive the owners' values.
// The preconditioner of a slab is its own block preconditioner on the slab
// (block Jacobi across the slabs).
p4d_status fgmres_dd(p4d_dd_ctx* D, const double* const* b, double* const* x, p4d_info* info) {
  const int P = (int)D->parts.size();
  std::vector<FgRun> R(P);
  std::vector<double*> ptr(P), vec(P);
  auto reduce = [&](auto&& at, int n) -> p4d_status {
    for (int p = 0; p < P; ++p) ptr[p] = at(R[p]);
    return dd_allreduce(D, ptr.data(), n);
  };
  auto at_off = [](int64_t mult2m, int64_t add) {
    return [=](FgRun& r) { return r.misc() + mult2m * r.L.m + add; };
  };
  p4d_ctx* c0 = D->parts[0];
  FgRun& r0 = R[0];
  const int refine = c0->prm.cgs_refine;
  for (int p = 0; p < P; ++p) {
    FgRun& r = R[p];
    p4d_ctx* c = D->parts[p];
    r.c = c;
    r.b = D->bw[p];
    r.x = x[p];
    r.trans = 0;
    r.nn = c->g.nn;
    r.full = false;
    r.len = 3 * r.nn;
    r.m = std::min(c->prm.restart, c->mcap);
    r.L = hlay(c->mcap);
    r.tau = (1.0 - c->prm.tplus) / c->prm.F;
    r.gb = (unsigned)std::min<int64_t>(4 * 152 * 4, (int64_t)nblocks(r.len));
    prof_reset(c);
  }
  P4D_TRY(cudaEventCreate(&r0.ev0));
  P4D_TRY(cudaEventCreate(&r0.ev1));
  P4D_TRY(cudaEventRecord(r0.ev0, D->stream));
  // the right-hand side without its ghost rows
  for (int p = 0; p < P; ++p) {
    P4D_TRY(cudaMemcpyAsync(D->bw[p], b[p], sizeof(double) * D->parts[p]->ndof, cudaMemcpyDeviceToDevice, D->stream));
    P4D_TRYS(dd_zero_ghost(D, p, D->bw[p], true));
  }
  // field weights of the whole cell's right-hand side
  for (int p = 0; p < P; ++p) {
    p4d_ctx* c = D->parts[p];
    ::p4d::count_launch(), k_field_norms<<<norm_blocks(c->ndof), kRedThreads, 0, D->stream>>>(
        D->bw[p], c->rsqd, R[p].nn, c->ndof, c->part, c->red_cnt, nullptr, 0.0, 0, nullptr, nullptr,
        R[p].misc() + 2 * R[p].L.m + 8);
  }
  P4D_TRYS(reduce(at_off(2, 8), 4));
  for (int p = 0; p < P; ++p) {
    p4d_ctx* c = D->parts[p];
    double* s4 = R[p].misc() + 2 * R[p].L.m + 8;
    ::p4d::count_launch(), k_weights_sums<<<1, 32, 0, D->stream>>>(s4, c->unorm2, 1e-14 / c->prm.rtol, c->wf, c->iwf, s4);
  }
  // particle condensation (node-local) and the norms of the Krylov right-hand side
  for (int p = 0; p < P; ++p) {
    FgRun& r = R[p];
    p4d_ctx* c = r.c;
    P4D_TRYS(particle_solve64(c, r.b + 3 * r.nn, c->tmp + 3 * r.nn, nullptr, 0));
    ::p4d::count_launch(), k_condense<<<nblocks(r.nn), kBlock, 0, D->stream>>>(
        c->g, c->nc, r.tau, c->eidx, c->label, c->Aj, c->Mj, c->betaj, c->ge, c->gc, c->gs, r.b, c->tmp + 3 * r.nn,
        c->bred, 0);
    r.bk = c->bred;
    ::p4d::count_launch(), k_field_norms<<<norm_blocks(r.len), kRedThreads, 0, D->stream>>>(
        r.bk, c->rsqd, r.nn, r.len, c->part, c->red_cnt, nullptr, 0.0, 0, nullptr, nullptr, r.misc() + 2 * r.L.m + 16);
  }
  P4D_TRYS(reduce(at_off(2, 16), 4));
  P4D_TRY(cudaMemcpyAsync(c0->hs_h, r0.misc() + 2 * r0.L.m + 8, sizeof(double) * 12, cudaMemcpyDeviceToHost, D->stream));
  P4D_TRY(cudaStreamSynchronize(D->stream));
  for (int p = 0; p < P; ++p) {
    if (p > 0) std::memcpy(D->parts[p]->hs_h, c0->hs_h, sizeof(double) * 12);
    P4D_TRYS(fg_bnorm(R[p]));
    P4D_TRY(cudaMemsetAsync(R[p].misc() + 2 * R[p].L.m + 7, 0, sizeof(double), D->stream));
  }
  auto share_host = [&](int at) {
    for (int p = 1; p < P; ++p) D->parts[p]->hs_h[at] = c0->hs_h[at];
  };
  // V_0 = s.(b_k - J x), ||V_0|| and the true residual use the same sequence
  auto residual_norm = [&]() -> p4d_status {
    P4D_TRYS(dd_halo(D, x, false));
    for (int p = 0; p < P; ++p) {
      p4d_ctx* c = D->parts[p];
      P4D_TRYS(jvp_reduced(c, x[p], c->V, 0, R[p].bk, true));
      P4D_TRYS(dd_zero_ghost(D, p, c->V, false));
      Reducer{c}.mdot(c->V, 0, 0, c->V, R[p].len, true, R[p].misc() + 2 * R[p].L.m + 2);
    }
    return reduce(at_off(2, 2), 1);
  };
  while (r0.active()) {
    P4D_TRYS(residual_norm());
    for (int p = 0; p < P; ++p) {
      FgRun& r = R[p];
      p4d_ctx* c = r.c;
      ++r.restarts;
      Tail t;
      t.mode = 1;
      t.hs = c->hs;
      t.L = r.L;
      t.kdev = c->kdev;
      ::p4d::count_launch(), k_scale<<<std::min(r.gb, 4u * 152u), kBlock, 0, D->stream>>>(c->V, c->V, r.len, r.misc() + 2 * r.L.m + 2, t);
    }
    P4D_TRY(cudaMemcpyAsync(c0->hs_h + kBetaOff, r0.misc() + 2 * r0.L.m + 5, sizeof(double), cudaMemcpyDeviceToHost, D->stream));
    P4D_TRY(cudaStreamSynchronize(D->stream));
    share_host(kBetaOff);
    for (int p = 0; p < P; ++p) fg_cycle_read(R[p]);
    if (r0.stop) break;
    for (int k = 0; !r0.cycle_done; ++k) {
      // z_k = P_slab^-1 (s^-1 v_k), then the owners' values in its ghost planes
      // restricted additive Schwarz: every slab preconditions v_k on its
      // owned and ghost rows (the owners' values) and keeps its owned rows.
      // With a single ghost plane, whose rows miss the elements beyond the
      // slab, its rows stay zero (block Jacobi across the slabs): fed the
      // owners' residual there the iteration counts grow several times.
      for (int p = 0; p < P; ++p) {
        vec[p] = D->parts[p]->Z + (int64_t)k * R[p].len;
        ptr[p] = D->parts[p]->V + (int64_t)k * R[p].len;
      }
      if (D->ghosts > 1) P4D_TRYS(dd_halo(D, ptr.data(), true));
      for (int p = 0; p < P; ++p) {
        P4D_TRYS(precond_column(D->parts[p], 0, true));
        P4D_TRYS(dd_zero_ghost(D, p, ptr[p], false));
      }
      // two-level: z_k += Z A_c^-1 Z^T (s^-1 v_k)
      {
        std::vector<const double*> vk(ptr.begin(), ptr.end());
        P4D_TRYS(dd_coarse_correct(D, vk.data(), vec.data()));
      }
      P4D_TRYS(dd_halo(D, vec.data(), false));
      // w = s.J z_k on the owned rows; h = V^T w, ||w||^2
      for (int p = 0; p < P; ++p) {
        p4d_ctx* c = D->parts[p];
        double* w = c->V + (int64_t)(k + 1) * R[p].len;
        P4D_TRYS(jvp_reduced(c, vec[p], w, 0, nullptr, true));
        P4D_TRYS(dd_zero_ghost(D, p, w, false));
        Reducer{c}.mdot(c->V, R[p].len, k + 1, w, R[p].len, true, R[p].misc());
      }
      P4D_TRYS(reduce(at_off(0, 0), k + 2));
      for (int p = 0; p < P; ++p) {
        p4d_ctx* c = D->parts[p];
        FgRun& r = R[p];
        Reducer{c}.maxpy(c->V, r.len, k + 1, r.misc(), c->V + (int64_t)(k + 1) * r.len, r.len, 1.0, nullptr,
                         Reducer::norm_to(r.misc() + 2 * r.L.m + 2), r.gb);
      }
      P4D_TRYS(reduce(at_off(2, 2), 1));
      if (refine > 0) {
        // second pass, decided on every slab from the same reduced norms
        for (int p = 0; p < P; ++p) {
          p4d_ctx* c = D->parts[p];
          FgRun& r = R[p];
          const double* flag = r.misc() + 2 * r.L.m + 6;
          ::p4d::count_launch(), k_reorth_flag<<<1, 1, 0, D->stream>>>(c->hs, r.L, k, refine == 2 ? 2.0 : 0.49);
          Reducer{c}.mdot(c->V, r.len, k + 1, c->V + (int64_t)(k + 1) * r.len, r.len, false, r.misc() + r.L.m + 1,
                          flag, 1);
        }
        P4D_TRYS(reduce(at_off(1, 1), k + 1));
        for (int p = 0; p < P; ++p) {
          p4d_ctx* c = D->parts[p];
          FgRun& r = R[p];
          const double* flag = r.misc() + 2 * r.L.m + 6;
          Reducer{c}.maxpy(c->V, r.len, k + 1, r.misc() + r.L.m + 1, c->V + (int64_t)(k + 1) * r.len, r.len, 1.0, flag,
                           Reducer::norm_to(r.misc() + 2 * r.L.m + 44, 1), r.gb);
        }
        P4D_TRYS(reduce(at_off(2, 44), 1));
        for (int p = 0; p < P; ++p)
          ::p4d::count_launch(), k_take_if<<<1, 32, 0, D->stream>>>(R[p].misc() + 2 * R[p].L.m + 2,
                                                                    R[p].misc() + 2 * R[p].L.m + 44,
                                                                    R[p].misc() + 2 * R[p].L.m + 6);
      }
      for (int p = 0; p < P; ++p) {
        p4d_ctx* c = D->parts[p];
        FgRun& r = R[p];
        double* w = c->V + (int64_t)(k + 1) * r.len;
        ::p4d::count_launch(), k_givens<<<1, 32, 0, D->stream>>>(c->hs, r.L, k, c->kdev, refine);
        ::p4d::count_launch(), k_scale<<<std::min(r.gb, 4u * 152u), kBlock, 0, D->stream>>>(w, w, r.len, r.misc() + 2 * r.L.m + 2, Tail{});
      }
      P4D_TRY(cudaMemcpyAsync(c0->hs_h, r0.misc() + 2 * r0.L.m + 3, 2 * sizeof(double), cudaMemcpyDeviceToHost,
                              D->stream));
      P4D_TRY(cudaStreamSynchronize(D->stream));
      for (int p = 0; p < P; ++p) fg_step_read(R[p], k, c0->hs_h);
    }
    // x += Z y on every slab (the same y)
    for (int p = 0; p < P; ++p) {
      FgRun& r = R[p];
      p4d_ctx* c = r.c;
      if (r.kk > 0) {
        ::p4d::count_launch(), k_backsolve<<<1, 32, 0, D->stream>>>(c->hs, r.L, r.kk);
        Reducer{c}.maxpy(c->Z, r.len, r.kk, c->hs + r.L.y, r.x, r.len, -1.0, nullptr, Fin{}, r.gb);
      }
    }
    if (r0.st == P4D_ERR_NONFINITE) break;
    if (r0.st == P4D_OK) {
      P4D_TRYS(residual_norm());
      P4D_TRY(cudaMemcpyAsync(c0->hs_h + kTrueOff, r0.misc() + 2 * r0.L.m + 2, sizeof(double), cudaMemcpyDeviceToHost,
                              D->stream));
      P4D_TRY(cudaStreamSynchronize(D->stream));
      share_host(kTrueOff);
      for (int p = 0; p < P; ++p) fg_cycle_end_read(R[p]);
    }
  }
  // particle back-substitution, then the true residual of the full system
  for (int p = 0; p < P; ++p) {
    FgRun& r = R[p];
    p4d_ctx* c = r.c;
    ::p4d::count_launch(), k_surface_coupling<<<nblocks(std::max<int64_t>(1, c->NE)), kBlock, 0, D->stream>>>(
        c->NE, r.tau, c->enode, r.nn, c->label, c->Aj, c->Mj, c->betaj, c->ge, c->gc, c->gs, r.x, c->tloc, 0);
    P4D_TRYS(particle_solve64(c, r.b + 3 * r.nn, r.x + 3 * r.nn, c->tloc, 0));
  }
  P4D_TRYS(dd_halo(D, x, false));
  for (int p = 0; p < P; ++p) {
    FgRun& r = R[p];
    p4d_ctx* c = r.c;
    double* m = r.misc() + 2 * r.L.m;
    P4D_TRYS(jvp_full(c, r.x, c->r0, 0, r.b, true));
    P4D_TRYS(dd_zero_ghost(D, p, c->r0, true));
    ::p4d::count_launch(), k_final_norms<<<norm_blocks(c->ndof), kRedThreads, 0, D->stream>>>(
        c->r0, c->sqd, r.b, r.nn, c->ndof, c->part, c->red_cnt, m + 24);
  }
  P4D_TRYS(reduce(at_off(2, 24), 4));
  P4D_TRYS(reduce(at_off(2, 32), 8));
  P4D_TRY(cudaEventRecord(r0.ev1, D->stream));
  P4D_TRY(cudaMemcpyAsync(c0->hs_h, r0.misc() + 2 * r0.L.m + 7, sizeof(double) * 33, cudaMemcpyDeviceToHost, D->stream));
  P4D_TRY(cudaStreamSynchronize(D->stream));
  fg_finish_read(r0, info);
  return r0.st;
}

}  // namespace p4d
