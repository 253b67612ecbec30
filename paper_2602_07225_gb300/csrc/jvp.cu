// Coupled Jacobian-vector products (paper section 4, eq. blocks), FP64.
//
// Structure used: the electrode-level blocks are the fixed 27-point stencils
// K_sigma (lifted phi_s), K_kappa, C = M_eps/dt + K_D; the diffusion-potential
// block is K_kappa diag(gamma / c_e); every other coupling is node-local and,
// at electrode node j, of rank one:
//     L_j = u_j v_j^T,  u = (A act, -A, -tau A, M beta),  v = (g_eta act, -g_eta, g_c, g_s)
// over (phi_s, phi_e, c_e, c_s surface).  The particle rows add
// M (I/dt - kap Lref).  The reduced (Schur) operator replaces the local term by
// zeta_j u_m v_m^T with zeta_j = 1 - z_j g_s M_j beta_j.
//
// Output forms: y = sc .* (J x) or y = sc .* (b - J x), sc = w_f / sqrt(d) in
// the scaled Krylov space, 1 otherwise.
#include <algorithm>
#include <mutex>
#include "p4d_common.cuh"

namespace p4d {
namespace {

struct JvpArgs {
  Grid g;
  int64_t NE;
  int nc;
  double tau, dt, idt;
  const double* Jst;
  const uint8_t* label;
  const int32_t* eidx;
  const double *Aj, *Mj, *betaj, *kapj, *rref;
  const double *ge, *gc, *gs, *zeta, *gdc, *rsqd, *wf;
  double* tloc;
  const double* u;     // optional precombined phi_e + gamma/c_e * c_e of the input (non-transposed)
  const unsigned* nz;  // GATED: *nz == 0 says that the input is all zeros
};

__device__ __forceinline__ double outscale(const JvpArgs& a, bool scaled, int f, int64_t row) {
  return scaled ? a.wf[f] * a.rsqd[row] : 1.0;
}

// u = x_phie + (gamma / c_e) x_ce: the input of the K_kappa stencil in the
// phi_e rows, formed once per node instead of once per stencil neighbour.
__global__ void k_jvp_combine(int64_t nn, const double* __restrict__ x, const double* __restrict__ gdc,
                              double* __restrict__ u) {
  const int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (n >= nn) return;
  u[n] = fma(gdc[n], x[2 * nn + n], x[nn + n]);
}

// Node n's rows of the plain product with every neighbour tested (CHECK below).
template <bool TRANS>
__device__ __noinline__ void tested_rows(const JvpArgs& a, const double* x, double* y, int n) {
  const int64_t nn = a.g.nn;
  const int N = (int)nn;
  const double *xs = x, *xe = x + nn, *xc = x + 2 * nn;
  const bool act = a.label[n] & kLabActive;
  const int q = n / a.g.nnx, i = n - q * a.g.nnx, k = q / a.g.nny, j = q - k * a.g.nny;
  double ys = 0.0, ye = 0.0, yc = 0.0;
#pragma unroll 1
  for (int o = 0; o < 27; ++o) {
    const int dx = o % 3 - 1, dy = (o / 3) % 3 - 1, dz = o / 9 - 1;
    if ((unsigned)(i + dx) >= (unsigned)a.g.nnx || (unsigned)(j + dy) >= (unsigned)a.g.nny ||
        (unsigned)(k + dz) >= (unsigned)a.g.nnz)
      continue;
    const int m = n + dx + a.g.nnx * (dy + a.g.nny * dz);
    const double* J = a.Jst + o * N + n;
    if (act) ys += J[0] * xs[m];
    ye += J[27 * nn] * (TRANS ? xe[m] : (a.u ? a.u[m] : fma(a.gdc[m], xc[m], xe[m])));
    yc += J[2 * 27 * nn] * xc[m];
  }
  if (TRANS) yc += a.gdc[n] * ye;
  if (!act) ys = xs[n];
  const int32_t e = a.eidx[n];
  if (e >= 0) {
    const double t = a.tloc[e];   // left by the kernel
    if (act) ys += (TRANS ? a.ge[e] : a.Aj[e]) * t;
    ye -= (TRANS ? a.ge[e] : a.Aj[e]) * t;
    if (TRANS) yc += a.gc[e] * t;
    else yc -= a.tau * a.Aj[e] * t;
  }
  y[n] = ys;
  y[nn + n] = ye;
  y[2 * nn + n] = yc;
}

// Macro rows.  reduced: Schur operator on [phi_s | phi_e | c_e] only.
// Large cells are bound by the FP64 rate, small ones by the latency of the
// loads: every neighbour is loaded without a test (the stencils hold exact
// zeros in the slots of neighbours outside the grid, the index is clamped to
// the vector), one stencil line of three offsets at a time.
// CHECK: an entry that is not finite must not reach a row that it does not
// couple to (0 x Inf is NaN): a row of the plain product (b null, not scaled)
// that ends non-finite is summed again with the tests.  After the store and
// not inlined: inlined it held 96 registers a thread, and a product of
// 152,439 nodes took 58.0 us, 242,406 88.3, 1,614,177 470; at 64 registers
// (CHECK: blocks of 128 threads that an SM is to hold) 53.9, 80.8 and 449.
// Called before the coupling or the store, small products wait for it (42,439
// nodes 28.8 us instead of 26.8).  The Krylov solves, whose vectors are finite
// or end the solve, go without.
// GATED: see jvp_start.
template <bool TRANS, bool REDUCED, bool GATED = false, int CHECK = 0>
__global__ void __launch_bounds__(128, CHECK) k_jvp_macro(const __grid_constant__ JvpArgs a,
                                                          const double* __restrict__ x, const double* __restrict__ b,
                                                          double* __restrict__ y, bool scaled) {
  static_assert(!CHECK || (!REDUCED && !GATED), "tested_rows is the plain product");
  const int64_t nn = a.g.nn;
  const int n = blockIdx.x * blockDim.x + threadIdx.x;   // 27 nn < 2^31 (checked at setup)
  const int N = (int)nn;
  if (n >= N) return;
  if (GATED && *a.nz == 0) {
#pragma unroll
    for (int f = 0; f < 3; ++f) y[f * nn + n] = outscale(a, scaled, f, f * nn + n) * b[f * nn + n];
    return;
  }
  const double* xs = x;
  const double* xe = x + nn;
  const double* xc = x + 2 * nn;
  const double* Ks = a.Jst;
  const double* Kk = a.Jst + 27 * nn;
  const double* Cc = a.Jst + 2 * 27 * nn;
  double ys = 0.0, ye = 0.0, yc = 0.0;
  const bool act = a.label[n] & kLabActive;
  const double* ue = !TRANS && a.u ? a.u : xe;
  const bool comb = !TRANS && !a.u;
#pragma unroll
  for (int l = 0; l < 9; ++l) {
    const int mid = n + a.g.nnx * ((l % 3 - 1) + a.g.nny * (l / 3 - 1));
    double k0[3], k1[3], k2[3], v0[3], v1[3], v2[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int o = 3 * l + d;
      const int m = min(max(mid + d - 1, 0), N - 1);
      k1[d] = Kk[o * N + n];
      k2[d] = Cc[o * N + n];
      v1[d] = ue[m];
      v2[d] = xc[m];
      if (comb) v1[d] = fma(a.gdc[m], v2[d], v1[d]);
      if (act) {
        k0[d] = Ks[o * N + n];
        v0[d] = xs[m];
      }
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      if (act) ys += k0[d] * v0[d];
      ye += k1[d] * v1[d];
      yc += k2[d] * v2[d];
    }
  }
  auto couple = [&] {
    if (TRANS) yc += a.gdc[n] * ye;   // (K_kappa diag(gamma/c_e))^T = diag(gamma/c_e) K_kappa
    if (!act) ys = xs[n];
    const int32_t e = a.eidx[n];
    if (e >= 0) {
      const double A = a.Aj[e];
      const double ge = a.ge[e];
      if (!TRANS) {
        // t = v . x  (c_s surface value only in the full operator)
        double t = (act ? ge * xs[n] : 0.0) - ge * xe[n] + a.gc[e] * xc[n];
        if (REDUCED) t *= a.zeta[e];
        else t += a.gs[e] * x[3 * nn + (int64_t)e * a.nc + a.nc - 1];
        if (act) ys += A * t;
        ye -= A * t;
        yc -= a.tau * A * t;
        if (!REDUCED) a.tloc[e] = t;
      } else {
        // t = u . x
        double t = (act ? A * xs[n] : 0.0) - A * xe[n] - a.tau * A * xc[n];
        if (REDUCED) t *= a.zeta[e];
        else t += a.Mj[e] * a.betaj[e] * x[3 * nn + (int64_t)e * a.nc + a.nc - 1];
        if (act) ys += ge * t;
        ye -= ge * t;
        yc += a.gc[e] * t;
        if (!REDUCED) a.tloc[e] = t;
      }
    }
    if (b) {
      ys = b[n] - ys;
      ye = b[nn + n] - ye;
      yc = b[2 * nn + n] - yc;
    }
  };
  couple();
  y[n] = outscale(a, scaled, 0, n) * ys;
  y[nn + n] = outscale(a, scaled, 1, nn + n) * ye;
  y[2 * nn + n] = outscale(a, scaled, 2, 2 * nn + n) * yc;
  if (CHECK && !(finite_bits(ys) && finite_bits(ye) && finite_bits(yc))) tested_rows<TRANS>(a, x, y, n);
}

// Particle rows of the full operator (after k_jvp_macro wrote tloc).
template <bool TRANS>
__global__ void k_jvp_particle(JvpArgs a, const double* __restrict__ x, const double* __restrict__ b,
                               double* __restrict__ y, bool scaled) {
  const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int nc = a.nc;
  if (q >= a.NE * nc) return;
  const int64_t e = (uint32_t)q / (uint32_t)nc;   // NE nc < 2^31 (checked at setup)
  const int i = (int)(q - e * nc);
  const int64_t nn = a.g.nn;
  const double* xc = x + 3 * nn + e * nc;
  const double* lo = a.rref;
  const double* di = a.rref + nc;
  const double* up = a.rref + 2 * nc;
  double L = di[i] * xc[i];
  if (!TRANS) {
    if (i > 0) L += lo[i] * xc[i - 1];
    if (i < nc - 1) L += up[i] * xc[i + 1];
  } else {
    if (i > 0) L += up[i - 1] * xc[i - 1];
    if (i < nc - 1) L += lo[i + 1] * xc[i + 1];
  }
  double v = a.Mj[e] * (xc[i] * a.idt - a.kapj[e] * L);
  if (i == nc - 1) v += (TRANS ? a.gs[e] : a.Mj[e] * a.betaj[e]) * a.tloc[e];
  if (b) v = b[3 * nn + q] - v;
  y[3 * nn + q] = outscale(a, scaled, 3, 3 * nn + q) * v;
}

JvpArgs make_args(p4d_ctx* c) {
  JvpArgs a;
  a.g = c->g; a.NE = c->NE; a.nc = c->nc;
  a.tau = (1.0 - c->prm.tplus) / c->prm.F; a.dt = c->prm.dt; a.idt = 1.0 / c->prm.dt;
  a.Jst = c->Jst; a.label = c->label; a.eidx = c->eidx;
  a.Aj = c->Aj; a.Mj = c->Mj; a.betaj = c->betaj; a.kapj = c->kapj; a.rref = c->rref;
  a.ge = c->ge; a.gc = c->gc; a.gs = c->gs; a.zeta = c->zeta; a.gdc = c->gdc; a.rsqd = c->rsqd; a.wf = c->wf;
  a.tloc = c->tloc;
  a.u = nullptr;
  a.nz = nullptr;
  return a;
}

}  // namespace

// The input combination phi_e + gamma/c_e c_e: already in c->ujvp (u_ready:
// the preconditioner's store left it there), formed per node, or on small
// cells (latency: one launch less) inside the stencil loop; the values are
// the same.
static void jvp_input(p4d_ctx* c, JvpArgs& a, const double* x, bool u_ready) {
  const int64_t nn = c->g.nn;
  if (!u_ready && nn <= 8192) return;
  if (!u_ready)
    ::p4d::count_launch(), k_jvp_combine<<<nblocks(nn), kBlock, 0, c->stream>>>(nn, x, c->gdc, c->ujvp);
  a.u = c->ujvp;
}

// Macro rows of the plain product.
static auto jvp_checked(int transpose) {
  return transpose ? k_jvp_macro<true, false, false, 8> : k_jvp_macro<false, false, false, 8>;
}

p4d_status jvp_full(p4d_ctx* c, const double* x, double* y, int transpose, const double* b, bool scaled, bool u_ready) {
  JvpArgs a = make_args(c);
  const int64_t nn = c->g.nn;
  const int bt = row_threads(nn);
  if (!transpose) jvp_input(c, a, x, u_ready);
  auto k = transpose ? k_jvp_macro<true, false> : k_jvp_macro<false, false>;
  if (!scaled && !b) k = jvp_checked(transpose);
  ::p4d::count_launch(), k<<<nblocks(nn, bt), bt, 0, c->stream>>>(a, x, b, y, scaled);
  if (c->NE > 0) {
    const int64_t np = c->NE * c->nc;
    if (transpose) ::p4d::count_launch(), k_jvp_particle<true><<<nblocks(np), kBlock, 0, c->stream>>>(a, x, b, y, scaled);
    else ::p4d::count_launch(), k_jvp_particle<false><<<nblocks(np), kBlock, 0, c->stream>>>(a, x, b, y, scaled);
  }
  P4D_TRYS(transport_jvp(c, x, y, transpose, b, scaled));
  P4D_TRY(cudaGetLastError());
  return P4D_OK;
}

// Whether any entry of x[0..n) is not zero, into *nz (zeroed before).
__global__ void __launch_bounds__(kBlock) k_nonzero(const double* __restrict__ x, int64_t n, unsigned* __restrict__ nz) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  long long any = 0;
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  for (; i + 3 * stride < n; i += 4 * stride)
#pragma unroll
    for (int q = 0; q < 4; ++q) any |= __double_as_longlong(x[i + q * stride]);
  for (; i < n; i += stride) any |= __double_as_longlong(x[i]);
  if (__any_sync(0xffffffffu, any != 0) && (threadIdx.x & 31) == 0) atomicOr(nz, 1u);
}

// Residual of the first restart cycle in the reduced mode: y = sc (b - J x).
// Solves start from x = 0 as a rule; the product, FP64 bound, is then left
// out: one pass over x finds out (65 x 65 x 49 nodes 45.8 us of product
// against 4.5 us of pass and 5.8 us of y = sc b; 129 x 129 x 97 nodes 270
// against 12 and 23 us).  Up to 8,192 nodes the product takes 10 us, no more
// than the pass with its launch.
p4d_status jvp_start(p4d_ctx* c, const double* x, double* y, int transpose, const double* b) {
  const int64_t nn = c->g.nn;
  if (nn <= 8192 || c->prm.transport_model != 0) return jvp_reduced(c, x, y, transpose, b, true);
  P4D_TRY(cudaMemsetAsync(c->nzflag, 0, sizeof(unsigned), c->stream));
  ::p4d::count_launch(), k_nonzero<<<std::min<unsigned>(nblocks(3 * nn, 4 * kBlock), 8 * 152), kBlock, 0, c->stream>>>(x, 3 * nn, c->nzflag);
  JvpArgs a = make_args(c);
  a.nz = c->nzflag;
  const int bt = row_threads(nn);
  if (!transpose) jvp_input(c, a, x, false);
  if (transpose) ::p4d::count_launch(), k_jvp_macro<true, true, true><<<nblocks(nn, bt), bt, 0, c->stream>>>(a, x, b, y, true);
  else ::p4d::count_launch(), k_jvp_macro<false, true, true><<<nblocks(nn, bt), bt, 0, c->stream>>>(a, x, b, y, true);
  P4D_TRY(cudaGetLastError());
  return P4D_OK;
}

p4d_status jvp_reduced(p4d_ctx* c, const double* x, double* y, int transpose, const double* b, bool scaled,
                       bool u_ready) {
  JvpArgs a = make_args(c);
  const int64_t nn = c->g.nn;
  const int bt = row_threads(nn);
  if (!transpose) jvp_input(c, a, x, u_ready);
  if (transpose) ::p4d::count_launch(), k_jvp_macro<true, true><<<nblocks(nn, bt), bt, 0, c->stream>>>(a, x, b, y, scaled);
  else ::p4d::count_launch(), k_jvp_macro<false, true><<<nblocks(nn, bt), bt, 0, c->stream>>>(a, x, b, y, scaled);
  P4D_TRYS(transport_jvp(c, x, y, transpose, b, scaled));
  P4D_TRY(cudaGetLastError());
  return P4D_OK;
}

}  // namespace p4d

// ---------------------------------------------------------------------------
// p4d_jvp_noalloc: the full-layout coupled JVP with its one piece of scratch
// (the node-local coupling scalar per electrode node, written by the
// macro-row kernel and read by the particle-row kernel) kept in a fixed
// device array of this file instead of the handle's workspace.  Every GPU
// that loads the library holds this array until the process exits.
namespace p4d {

static __device__ __align__(256) double g_noalloc_tloc[P4D_NOALLOC_MAX_NELEC];

namespace {

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mu;
void* g_noalloc_ptr[kMaxDevices] = {};

// Device address of g_noalloc_tloc on the handle's device, looked up once per
// device with that device current (in host code the array's name is only a
// stand-in for the device symbol, never a device address).  The handle's
// kernels run on its stream, on the device it was set up on; a caller with
// another device current gets INVALID_ARG instead of another GPU's array.
p4d_status noalloc_scratch(const p4d_ctx* h, double** out) {
  int dev = -1;
  P4D_TRY(cudaGetDevice(&dev));
  if (dev != h->device) return P4D_ERR_INVALID_ARG;
  if (dev < 0 || dev >= kMaxDevices) return P4D_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (!g_noalloc_ptr[dev]) {
    void* ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_noalloc_tloc) != cudaSuccess || !ptr) {
      cudaGetLastError();
      return P4D_ERR_CUDA;
    }
    g_noalloc_ptr[dev] = ptr;
  }
  *out = static_cast<double*>(g_noalloc_ptr[dev]);
  return P4D_OK;
}

}  // namespace
}  // namespace p4d

extern "C" p4d_status p4d_jvp_noalloc(p4d_handle h, const double* x, double* y, int transpose) {
  using namespace p4d;
  if (!h || !x || !y || x == y || !h->linearized) return P4D_ERR_INVALID_ARG;
  if (h->NE > (int64_t)P4D_NOALLOC_MAX_NELEC || h->prm.transport_model != 0) return P4D_ERR_INVALID_ARG;
  double* tloc = nullptr;
  P4D_TRYS(noalloc_scratch(h, &tloc));
  JvpArgs a = make_args(h);
  a.tloc = tloc;   // each entry read by the particle rows is written first by the macro rows
  const int64_t nn = h->g.nn;
  const int bt = row_threads(nn);
  ::p4d::count_launch(), jvp_checked(transpose)<<<nblocks(nn, bt), bt, 0, h->stream>>>(a, x, nullptr, y, false);
  if (h->NE > 0) {
    const int64_t np = h->NE * h->nc;
    if (transpose) ::p4d::count_launch(), k_jvp_particle<true><<<nblocks(np), kBlock, 0, h->stream>>>(a, x, nullptr, y, false);
    else ::p4d::count_launch(), k_jvp_particle<false><<<nblocks(np), kBlock, 0, h->stream>>>(a, x, nullptr, y, false);
  }
  P4D_TRY(cudaGetLastError());
  return P4D_OK;
}
