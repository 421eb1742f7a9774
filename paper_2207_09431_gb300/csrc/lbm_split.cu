// Two-kernel form of the coupled D2Q9 step (arXiv 2207.09431, Sec. 2.2-2.3) for
// the mixed difference scheme and the open x boundaries:
//   k_fields_step   C_i = sum_a h_a^i (Eq. 22), rho, mu (Eq. 5), u (Eq. 23),
//                   p (Eq. 24/R3), new tau (Eq. 25-33)
//   k_collide_push  S_i + V_i (Eq. 6, 18, 21), collision of g (Eq. 14) and h (Eq.
//   k_collide_step  18), streaming with half-way bounce-back and (the latter) the open
//                   boundaries, the destination-side source term (R9)
// The fields between the two live in scratch planes carved from the caller's
// arena.  All arithmetic FP32.  Also the macro fields, the initial equilibria and
// the observables.
#include "lbm_device.cuh"
#include "lbm_internal.h"
#include "lbm_kernels.h"
#include "lbm_node.cuh"

namespace lbm {

namespace {

// Order parameter j (0..2) at node (x, y) of the scratch planes (C3 derived).
struct CReader {
  const float *C;
  long long plane;
  int nh;
  __device__ __forceinline__ void at(long long k, float out[3]) const {
    out[0] = C[k];
    out[1] = (nh == 2) ? C[plane + k] : 0.0f;
    out[2] = 1.0f - out[0] - out[1];
  }
};

__device__ __forceinline__ long long node_index(const DevParams &P, int x, int y) {
  return (long long)y * P.pitch + x;
}

// Column seen at x: periodic, or (open x) the mirror ghost columns beyond the
// inlet and outlet, for offsets of at most two columns.
__device__ __forceinline__ int column_of(const DevParams &P, int x) {
  if (!P.open_x) return wrap_x(x, P.nx);
  if (x < 0) x = -1 - x;
  if (x >= P.nx) x = 2 * P.nx - 1 - x;
  return x;
}

__device__ __forceinline__ long long shifted(const DevParams &P, int x, int y, int dx, int dy) {
  return node_index(P, column_of(P, x + dx), wrap_y(y + dy, P.ny, P.periodic_y));
}

// Directional derivative e_a . grad X from samples X(x - e), X(x), X(x + e),
// X(x + 2e) (R2; mixed = mean of central and second-order biased forms).
// The final scaling is a separate rounding (__fmul_rn), never fused into the
// caller's next addition, whether or not this is inlined.
__device__ __forceinline__ float dir_deriv(int scheme, float xm, float x0, float xp, float xpp) {
  if (scheme == 0) return __fmul_rn(0.5f, xp - xm);
  return __fmul_rn(0.25f, -xpp + 5.0f * xp - 3.0f * x0 - xm);
}

// Everything the forcing terms need at one node.
struct NodeCtx {
  float C[3], rho, ux, uy, p, mu[3];
  float gC[3][2], grho[2], gp[2], Fs[2], Fb[2];
  float dC[3][9], drho[9], dp[9];
};

// Gathers C (radius 1 or 2), rho (from C), p (radius 1 or 2) around a node.
// Inlined and unrolled, so that NodeCtx stays in registers.
template <typename Reader>
__device__ __forceinline__ void gather_gradients(int fd_scheme, const Reader &at, NodeCtx &n) {
  float Cn[9][3], rn[9], pn[9];
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    at.C(ex(a), ey(a), Cn[a]);
    rn[a] = at.rho(ex(a), ey(a), Cn[a]);
    pn[a] = at.p(ex(a), ey(a));
  }
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    n.C[j] = Cn[0][j];
    float sx = 0.f, sy = 0.f;
#pragma unroll
    for (int a = 0; a < 9; ++a) {
      sx += wt(a) * ex(a) * Cn[a][j];
      sy += wt(a) * ey(a) * Cn[a][j];
    }
    n.gC[j][0] = 3.0f * sx;
    n.gC[j][1] = 3.0f * sy;
  }
  n.rho = rn[0];
  n.p = pn[0];
  {
    float sx = 0.f, sy = 0.f, qx = 0.f, qy = 0.f;
#pragma unroll
    for (int a = 0; a < 9; ++a) {
      sx += wt(a) * ex(a) * rn[a];
      sy += wt(a) * ey(a) * rn[a];
      qx += wt(a) * ex(a) * pn[a];
      qy += wt(a) * ey(a) * pn[a];
    }
    n.grho[0] = 3.0f * sx;
    n.grho[1] = 3.0f * sy;
    n.gp[0] = 3.0f * qx;
    n.gp[1] = 3.0f * qy;
  }
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    const int o = opp(a);
    float C2e[3] = {0.f, 0.f, 0.f}, r2e = 0.f, p2e = 0.f;
    if (fd_scheme == 1) {
      at.C(2 * ex(a), 2 * ey(a), C2e);
      r2e = at.rho(2 * ex(a), 2 * ey(a), C2e);
      p2e = at.p(2 * ex(a), 2 * ey(a));
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) n.dC[j][a] = dir_deriv(fd_scheme, Cn[o][j], Cn[0][j], Cn[a][j], C2e[j]);
    n.drho[a] = dir_deriv(fd_scheme, rn[o], rn[0], rn[a], r2e);
    n.dp[a] = dir_deriv(fd_scheme, pn[o], pn[0], pn[a], p2e);
  }
}

// Forcing of Eq. 14 for direction a.
__device__ __forceinline__ float phi_g(const NodeCtx &n, int a, float G) {
  float e_rho = n.drho[a] - (n.ux * n.grho[0] + n.uy * n.grho[1]);
  float e_Fs = n.mu[0] * n.dC[0][a] + n.mu[1] * n.dC[1][a] + n.mu[2] * n.dC[2][a] -
               (n.ux * n.Fs[0] + n.uy * n.Fs[1]);
  float e_Fb = (ex(a) - n.ux) * n.Fb[0] + (ey(a) - n.uy) * n.Fb[1];
  return e_rho * kCs2 * (G - wt(a)) + (e_Fs + e_Fb) * G;
}

// Forcing of Eq. 18 for order parameter i, direction a.
__device__ __forceinline__ float phi_h(const NodeCtx &n, int i, int a, float G) {
  float e_C = n.dC[i][a] - (n.ux * n.gC[i][0] + n.uy * n.gC[i][1]);
  float e_p = n.dp[a] - (n.ux * n.gp[0] + n.uy * n.gp[1]);
  float e_Fs = n.mu[0] * n.dC[0][a] + n.mu[1] * n.dC[1][a] + n.mu[2] * n.dC[2][a] -
               (n.ux * n.Fs[0] + n.uy * n.Fs[1]);
  float e_Fb = (ex(a) - n.ux) * n.Fb[0] + (ey(a) - n.uy) * n.Fb[1];
  return (e_C - n.C[i] / (n.rho * kCs2) * (e_p - e_Fs - e_Fb)) * G;
}

__device__ __forceinline__ bool node_of_thread(const DevParams &P, int &x, int &y) {
  x = blockIdx.x * blockDim.x + threadIdx.x;
  y = blockIdx.y * blockDim.y + threadIdx.y;
  return x < P.nx && y < P.ny;
}

}  // namespace

__global__ void k_moments(DevParams P, const float *__restrict__ h, float *__restrict__ C) {
  int x, y;
  if (!node_of_thread(P, x, y)) return;
  const long long k = node_index(P, x, y);
  for (int i = 0; i < P.nh; ++i) {
    float s = 0.f;
    for (int a = 0; a < 9; ++a) s += h[pop_index(k, i * 9 + a, 9 * P.nh)];
    C[(long long)i * P.plane + k] = s;
  }
}

// The fields of a node from the order parameters around it and its g (Eq. 5,
// 22-24): grad C, lap C, grad rho, mu_1..3, the forces, the moments of g and u,
// from C and rho at the node and its neighbours.  Shared by every kernel that
// computes fields and the observables, so that all see the same velocity.
template <bool ROUND_FB>
__device__ __forceinline__ void fields_math(const DevParams &P, NodeCtx &n, const float (&Cn)[9][3],
                                            const float (&rn)[9], const float (&ga)[9], float &m0) {
  float lapC[3];
  for (int j = 0; j < 3; ++j) {
    n.C[j] = Cn[0][j];
    float sx = 0.f, sy = 0.f, lp = 0.f;
    for (int a = 0; a < 9; ++a) {
      sx += wt(a) * ex(a) * Cn[a][j];
      sy += wt(a) * ey(a) * Cn[a][j];
      lp += wt(a) * (Cn[a][j] - Cn[0][j]);
    }
    n.gC[j][0] = 3.0f * sx;
    n.gC[j][1] = 3.0f * sy;
    lapC[j] = 6.0f * lp;
  }
  n.rho = rn[0];
  {
    float sx = 0.f, sy = 0.f;
    for (int a = 0; a < 9; ++a) {
      sx += wt(a) * ex(a) * rn[a];
      sy += wt(a) * ey(a) * rn[a];
    }
    n.grho[0] = 3.0f * sx;
    n.grho[1] = 3.0f * sy;
  }
  chem_potentials(P, n.C, lapC, n.mu);
  n.Fs[0] = n.mu[0] * n.gC[0][0] + n.mu[1] * n.gC[1][0] + n.mu[2] * n.gC[2][0];
  n.Fs[1] = n.mu[0] * n.gC[0][1] + n.mu[1] * n.gC[1][1] + n.mu[2] * n.gC[2][1];
  n.Fb[0] = P.force_x;
  n.Fb[1] = ROUND_FB ? __fmul_rn(-n.rho, P.gravity) : -n.rho * P.gravity;
  m0 = 0.f;
  float mx = 0.f, my = 0.f;
  for (int a = 0; a < 9; ++a) {
    m0 += ga[a];
    mx += ex(a) * ga[a];
    my += ey(a) * ga[a];
  }
  n.ux = (3.0f * mx + 0.5f * (n.Fs[0] + n.Fb[0])) / n.rho;
  n.uy = (3.0f * my + 0.5f * (n.Fs[1] + n.Fb[1])) / n.rho;
}

// fields_math of node (x, y) from the C planes.
template <int NH, bool ROUND_FB>
__device__ __forceinline__ void fields_core(const DevParams &P, const float *__restrict__ Cf,
                                            const float *__restrict__ g, int x, int y, long long k, NodeCtx &n,
                                            float (&Cn)[9][3], float (&rn)[9], float (&ga)[9], float &m0) {
  CReader cr{Cf, P.plane, NH};
  for (int a = 0; a < 9; ++a) {
    long long kk = shifted(P, x, y, ex(a), ey(a));
    cr.at(kk, Cn[a]);
    rn[a] = rho_of(P, Cn[a][0], Cn[a][1], Cn[a][2]);
  }
  for (int a = 0; a < 9; ++a) ga[a] = g[pop_index(k, a, 9)];
  fields_math<ROUND_FB>(P, n, Cn, rn, ga, m0);
}

// mu_1..3, u, p of the current state (for lbm_get_field).
template <int NH>
__global__ void k_fields(DevParams P, const float *__restrict__ Cf, const float *__restrict__ g, float *__restrict__ mu,
                         float *__restrict__ pf, float *__restrict__ uxf, float *__restrict__ uyf) {
  int x, y;
  if (!node_of_thread(P, x, y)) return;
  const long long k = node_index(P, x, y);
  float Cn[9][3], rn[9], ga[9], m0;
  NodeCtx n;
  fields_core<NH, true>(P, Cf, g, x, y, k, n, Cn, rn, ga, m0);
  for (int j = 0; j < 3; ++j) mu[(long long)j * P.plane + k] = n.mu[j];
  pf[k] = m0 + 0.5f * kCs2 * (n.ux * n.grho[0] + n.uy * n.grho[1]);
  uxf[k] = n.ux;
  uyf[k] = n.uy;
}

// Row and column whose values stand at (x, y) of a tile and its rings: periodic, or
// the mirror ghost rows beyond walls and ghost columns beyond the open ends
// (slots far outside, of ragged tiles, hold some value that nothing reads).
__device__ __forceinline__ int tile_column(const DevParams &P, int x) {
  if (!P.open_x) return wrap_periodic(x, P.nx);
  const int xs = x < 0 ? -1 - x : (x >= P.nx ? 2 * P.nx - 1 - x : x);
  return xs < 0 ? 0 : (xs >= P.nx ? P.nx - 1 : xs);
}
__device__ __forceinline__ long long tile_node(const DevParams &P, int x, int y) {
  return node_index(P, tile_column(P, x), row_read(y, P.ny, P.periodic_y));
}

// Both step kernels take a tile of 32 x 4 output nodes per CTA and keep the
// stencil neighbourhoods in shared memory: one load and one density per node and
// ring slot, where a node's stencils of up to 25 points used to read the planes through
// L1 and form rho again at every point.  The kernels were four (moments, fields, sources,
// collision) and, with open ends, a fifth that walked the boundary rows: the
// sources and the open ends are now part of the collision kernel.  Bound by the latency of two
// short kernels on small lattices and by instruction issue on large ones.  Measured on a
// GB300, us per step of lbm_step calls of 65 steps, now and with four (five) kernels: mixed scheme
// 64 x 128 8.6 and 20.8, 200 x 400 12.4 and 28.0; open channel 240 x 60 9.3 and 28.5; mixed scheme
// 1024 x 2048 182 and 431.  Tiles of 8 rows (fewer collisions twice, fewer CTAs)
// ran 1 to 5 % slower above 400 x 800 at their best register budget and up to 10 % slower
// on small lattices.  The order of a node's operations is that of the earlier kernels.
constexpr int kTileX = 32, kTileY = 4;

// Whether a tile at (x0, y0) and R nodes around it lie inside the lattice: then a
// slot's node is at a fixed offset and nothing wraps or mirrors.
__device__ __forceinline__ bool tile_inside(const DevParams &P, int x0, int y0, int r) {
  return x0 >= r && y0 >= r && x0 + kTileX + r <= P.nx && y0 + kTileY + r <= P.ny;
}

// Shared-memory slots of a tile with a ring of R nodes.
template <int R>
struct Ring {
  static constexpr int W = kTileX + 2 * R, H = kTileY + 2 * R, N = W * H;
  static __device__ __forceinline__ int slot(int lx, int ly) { return (ly + R) * W + lx + R; }
};

// C_i, rho, mu_1..3, u, p, the new relaxation time and the strain rate.
// SCHEME 1: directional derivatives reach two nodes.
template <int NH, int SCHEME>
__global__ void __launch_bounds__(kTileX *kTileY)
    k_fields_step(DevParams P, const float *__restrict__ h, const float *__restrict__ g,
                  const float *__restrict__ tau_prev, float *__restrict__ Cf, float *__restrict__ mu,
                  float *__restrict__ pf, float *__restrict__ uxf, float *__restrict__ uyf,
                  float *__restrict__ tau_new, float *__restrict__ shear, unsigned *err) {
  using S = Ring<1 + SCHEME>;
  __shared__ float sC[NH][S::N], srho[S::N];
  const int t = threadIdx.x, x0 = blockIdx.x * kTileX, y0 = blockIdx.y * kTileY;
  const int tx = t % kTileX, ty = t / kTileX, x = x0 + tx, y = y0 + ty;
  const bool mine = x < P.nx && y < P.ny;
  const long long k = node_index(P, x, y);
  float ga[9], tp = 0.f;
  if (mine) {
#pragma unroll
    for (int a = 0; a < 9; ++a) ga[a] = g[pop_index(k, a, 9)];
    tp = tau_prev[k];
  }
  const bool inside = tile_inside(P, x0, y0, 1 + SCHEME);
  for (int q = t; q < S::N; q += kTileX * kTileY) {
    const int xq = x0 + q % S::W - (1 + SCHEME), yq = y0 + q / S::W - (1 + SCHEME);
    const long long kq = inside ? node_index(P, xq, yq) : tile_node(P, xq, yq);
    float c[2] = {0.f, 0.f};
#pragma unroll
    for (int i = 0; i < NH; ++i) {
      float s = 0.f;
#pragma unroll
      for (int a = 0; a < 9; ++a) s += h[pop_index(kq, i * 9 + a, 9 * NH)];
      sC[i][q] = c[i] = s;
    }
    srho[q] = rho_of(P, c[0], c[1], 1.0f - c[0] - c[1]);
  }
  __syncthreads();
  if (!mine) return;
  auto read = [&](int dx, int dy, float c[3]) {
    const int q = S::slot(tx + dx, ty + dy);
    c[0] = sC[0][q];
    c[1] = NH == 2 ? sC[NH - 1][q] : 0.0f;
    c[2] = 1.0f - c[0] - c[1];
    return srho[q];
  };
  NodeCtx n;
  float Cn[9][3], rn[9], m0;
#pragma unroll
  for (int a = 0; a < 9; ++a) rn[a] = read(ex(a), ey(a), Cn[a]);
  fields_math<true>(P, n, Cn, rn, ga, m0);
  n.p = m0 + 0.5f * kCs2 * (n.ux * n.grho[0] + n.uy * n.grho[1]);
#pragma unroll
  for (int i = 0; i < NH; ++i) Cf[(long long)i * P.plane + k] = n.C[i];
#pragma unroll
  for (int j = 0; j < 3; ++j) mu[(long long)j * P.plane + k] = n.mu[j];
  pf[k] = n.p;
  uxf[k] = n.ux;
  uyf[k] = n.uy;
  // directional derivatives of rho and C (the g forcing has no p derivative)
  for (int a = 0; a < 9; ++a) {
    const int o = opp(a);
    float C2e[3] = {0.f, 0.f, 0.f}, r2e = 0.f;
    if (SCHEME == 1) r2e = read(2 * ex(a), 2 * ey(a), C2e);
    for (int j = 0; j < 3; ++j) n.dC[j][a] = dir_deriv(SCHEME, Cn[o][j], Cn[0][j], Cn[a][j], C2e[j]);
    n.drho[a] = dir_deriv(SCHEME, rn[o], rn[0], rn[a], r2e);
  }
  // strain rate from the non-equilibrium part with the previous tau (R23)
  const float fac = 3.0f * (2.0f * tp / (2.0f * tp + 1.0f));
  float Pxx = 0.f, Pyy = 0.f, Pxy = 0.f;
  for (int a = 0; a < 9; ++a) {
    float G = gamma_a(a, n.ux, n.uy);
    float geq = wt(a) * n.p + n.rho * kCs2 * (G - wt(a)) - 0.5f * phi_g(n, a, G);
    float fneq = fac * (ga[a] - geq);
    Pxx += fneq * (float)(ex(a) * ex(a));
    Pyy += fneq * (float)(ey(a) * ey(a));
    Pxy += fneq * (float)(ex(a) * ey(a));
  }
  const float den = 2.0f * tp * n.rho * kCs2;
  const float Dxx = -Pxx / den, Dyy = -Pyy / den, Dxy = -Pxy / den;
  const float gd = sqrtf(2.0f * (Dxx * Dxx + Dyy * Dyy + 2.0f * Dxy * Dxy));
  const float tau1 = P.powerlaw ? tau_powerlaw(P, gd, 1.0f / n.rho) : P.tau[0];
  const float tn = tau_mix(P, n.C[0], n.C[1], n.C[2], tau1);
  tau_new[k] = tn;
  shear[k] = gd;
  if (!(isfinite(n.rho) && isfinite(n.p) && isfinite(n.ux) && isfinite(n.uy) && isfinite(tn))) atomicOr(err, 1u);
}

// S_i + V_i (Eq. 6, 18, 21; R8) from the stencils of C_i and mu_i around a node.
__device__ __forceinline__ float source_of(const DevParams &P, int i, const float (&cv)[9], const float (&mv)[9]) {
  float gcx = 0.f, gcy = 0.f, gmx = 0.f, gmy = 0.f, lm = 0.f;
  for (int a = 0; a < 9; ++a) {
    gcx += wt(a) * ex(a) * cv[a];
    gcy += wt(a) * ey(a) * cv[a];
    gmx += wt(a) * ex(a) * mv[a];
    gmy += wt(a) * ey(a) * mv[a];
    lm += wt(a) * (mv[a] - mv[0]);
  }
  const float lapmu = 6.0f * lm;
  const float C = cv[0];
  const float D0s = P.d0_sig[i];
  if (P.mobility == 1) {
    // mobility with C clipped to [0, 1] and its derivative (reading R8)
    const float cc = fminf(fmaxf(C, 0.0f), 1.0f);
    const float dv = (C >= 0.0f && C <= 1.0f)
                         ? D0s * (1.0f - 2.0f * C) * (3.0f * gcx * 3.0f * gmx + 3.0f * gcy * 3.0f * gmy)
                         : 0.0f;
    return D0s * cc * (1.0f - cc) * lapmu + dv;
  }
  return D0s * lapmu;
}

// Post-collision populations of a node whose u, mu and stencil values (at) are in place:
// sv its sources, gv its g, tn its new relaxation time; put(a, g*_a, h*) takes them.
// With tau_h = 1/2 the BGK step of Eq. 18 replaces h by its modified equilibrium:
// h* = C Gamma + Phi/2 + SV Gamma/2.
template <int NH, int SCHEME, typename Reader, typename Put>
__device__ __forceinline__ void collide_node(const DevParams &P, NodeCtx &n, const Reader &at, const float (&sv)[NH],
                                             const float (&gv)[9], float tn, const Put &put) {
  gather_gradients(SCHEME, at, n);
  n.Fs[0] = n.mu[0] * n.gC[0][0] + n.mu[1] * n.gC[1][0] + n.mu[2] * n.gC[2][0];
  n.Fs[1] = n.mu[0] * n.gC[0][1] + n.mu[1] * n.gC[1][1] + n.mu[2] * n.gC[2][1];
  n.Fb[0] = P.force_x;
  n.Fb[1] = -n.rho * P.gravity;
  const float omega = 1.0f / (tn + 0.5f);
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    const float G = gamma_a(a, n.ux, n.uy);
    // Which product of the equilibrium is rounded on its own is spelled out: left to the
    // compiler it changes with the code around it, and the results by rounding.  Either choice
    // is as accurate; this one, with its split at a = 5, is what the compiler made of an earlier
    // kernel, kept so that runs continue in the same bits.
    const float pg = phi_g(n, a, G), Gw = G - wt(a), rc = n.rho * kCs2;
    const float lin = a < 5 ? __fmaf_rn(wt(a), n.p, __fmul_rn(rc, Gw)) : __fmaf_rn(rc, Gw, __fmul_rn(wt(a), n.p));
    const float geq = lin - 0.5f * pg;
    float hs[NH];
#pragma unroll
    for (int i = 0; i < NH; ++i) {
      const float ph = phi_h(n, i, a, G);
      hs[i] = n.C[i] * G + 0.5f * ph + 0.5f * sv[i] * G;
    }
    put(a, gv[a] - omega * (gv[a] - geq) + pg, hs);
  }
}

// C, rho and p around node (lx, ly) of a tile.
template <int NH, typename S, typename RC>
struct StencilReader {
  const S &s;
  int lx, ly;
  __device__ __forceinline__ int q(int dx, int dy) const { return RC::slot(lx + dx, ly + dy); }
  __device__ __forceinline__ void C(int dx, int dy, float c[3]) const {
    c[0] = s.C[0][q(dx, dy)];
    c[1] = NH == 2 ? s.C[NH - 1][q(dx, dy)] : 0.0f;
    c[2] = 1.0f - c[0] - c[1];
  }
  __device__ __forceinline__ float rho(int dx, int dy, const float *) const { return s.rho[q(dx, dy)]; }
  __device__ __forceinline__ float p(int dx, int dy) const { return s.p[q(dx, dy)]; }
};

template <int NH, int SCHEME>
struct CollideSmem {
  using RC = Ring<2 + SCHEME>;
  using RM = Ring<2>;
  using R1 = Ring<1>;
  float C[NH][RC::N], rho[RC::N], p[RC::N], mu[NH][RM::N];
  float g[9][R1::N], h[NH][9][R1::N], sv[NH][R1::N], ux[R1::N], uy[R1::N];
};
// Threads: the collisions of the tile and its ring in one pass.
constexpr int kCollideThreads = (Ring<1>::N + 31) / 32 * 32;

// Sources, collision and streaming of a tile with open x boundaries: the populations of
// the tile and its ring meet in shared memory and are gathered by the node they arrive at
// (an outlet node needs all of its own at once).  Populations that would cross a wall return in
// the opposite direction.  At the inlet (x = 0, e_x = +1) g comes from a ghost
// column x = -1 whose post-collision g is the equilibrium w p + rho cs^2 (Gamma - w) at
// (u_in, 0) plus the non-equilibrium part of column 0's post-collision g, h the
// equilibrium c_in Gamma(u_in) plus the node's destination-side term; at the outlet
// (x = nx - 1, e_x = -1) the convective condition f(t+1) = (f(t) + U f_(nx-2)(t+1)) / (1 + U),
// U the node's x velocity clamped to [0, 1], then the shift (shared by weight among
// the entering g) that sets the node's pressure sum_a g_a to 0.  Wall rows keep bounce-back.
template <int NH, int SCHEME, int MINB>
__global__ void __launch_bounds__(kCollideThreads, MINB)
    k_collide_step(DevParams P, const float *__restrict__ g, const float *__restrict__ h_old,
                   const float *__restrict__ Cf, const float *__restrict__ mu, const float *__restrict__ pf,
                   const float *__restrict__ uxf, const float *__restrict__ uyf, const float *__restrict__ tau_new,
                   float *__restrict__ SV, float *__restrict__ g_out, float *__restrict__ h_out) {
  using S = CollideSmem<NH, SCHEME>;
  using RC = typename S::RC;
  using RM = typename S::RM;
  using R1 = typename S::R1;
  constexpr int NT = kCollideThreads;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  S &s = *reinterpret_cast<S *>(smem_raw);
  const int t = threadIdx.x, x0 = blockIdx.x * kTileX, y0 = blockIdx.y * kTileY;

  // this thread's node of the one-node ring (real rows, and columns of the lattice)
  const int lx = t % R1::W - 1, ly = t / R1::W - 1, xr = x0 + lx, yr = y0 + ly;
  const bool ring = t < R1::N && (P.periodic_y || (yr >= 0 && yr < P.ny)) && xr >= 0 && xr < P.nx;
  const bool inside = tile_inside(P, x0, y0, 2 + SCHEME);
  const long long kr = inside ? node_index(P, xr, yr) : tile_node(P, xr, yr);
  NodeCtx n;
  float gv[9], tn = 0.f;
  if (ring) {
#pragma unroll
    for (int a = 0; a < 9; ++a) gv[a] = g[pop_index(kr, a, 9)];
    tn = tau_new[kr];
    n.ux = uxf[kr];
    n.uy = uyf[kr];
#pragma unroll
    for (int j = 0; j < 3; ++j) n.mu[j] = mu[(long long)j * P.plane + kr];
  }
  for (int q = t; q < RC::N; q += NT) {
    const int cx = q % RC::W - (2 + SCHEME), cy = q / RC::W - (2 + SCHEME);
    const long long kq = inside ? node_index(P, x0 + cx, y0 + cy) : tile_node(P, x0 + cx, y0 + cy);
    const float c0 = Cf[kq], c1 = NH == 2 ? Cf[P.plane + kq] : 0.0f;
    s.C[0][q] = c0;
    if (NH == 2) s.C[NH - 1][q] = c1;
    s.rho[q] = rho_of(P, c0, c1, 1.0f - c0 - c1);
    s.p[q] = pf[kq];
    if (SCHEME == 0 || (cx >= -2 && cx < kTileX + 2 && cy >= -2 && cy < kTileY + 2)) {
#pragma unroll
      for (int i = 0; i < NH; ++i) s.mu[i][RM::slot(cx, cy)] = mu[(long long)i * P.plane + kq];
    }
  }
  __syncthreads();

  if (ring) {
    const StencilReader<NH, S, RC> at{s, lx, ly};
    float sv[NH];
#pragma unroll
    for (int i = 0; i < NH; ++i) {
      float cv[9], mv[9];
#pragma unroll
      for (int a = 0; a < 9; ++a) {
        cv[a] = s.C[i][RC::slot(lx + ex(a), ly + ey(a))];
        mv[a] = s.mu[i][RM::slot(lx + ex(a), ly + ey(a))];
      }
      sv[i] = source_of(P, i, cv, mv);
      s.sv[i][t] = sv[i];
    }
    s.ux[t] = n.ux;
    s.uy[t] = n.uy;
    collide_node<NH, SCHEME>(P, n, at, sv, gv, tn, [&](int a, float gs, const float (&hs)[NH]) {
      s.g[a][t] = gs;
#pragma unroll
      for (int i = 0; i < NH; ++i) s.h[i][a][t] = hs[i];
    });
  }
  __syncthreads();

  // streaming: the populations that arrive at output node (x, y)
  const int tx = t % kTileX, ty = t / kTileX, x = x0 + tx, y = y0 + ty;
  if (ty >= kTileY || x >= P.nx || y >= P.ny) return;
  const long long k = node_index(P, x, y);
  const int q0 = R1::slot(tx, ty);
  const float ux = s.ux[q0], uy = s.uy[q0];
  float gy[9];
  unsigned entered = 0;  // outlet: directions that enter there
  float wsum = 0.f, U = 0.f, inv = 1.f;
  const bool outlet = x == P.nx - 1;
  if (outlet) {
    U = fminf(fmaxf(ux, 0.0f), 1.0f);
    inv = 1.0f / (1.0f + U);
  }
#pragma unroll
  for (int i = 0; i < NH; ++i) SV[(long long)i * P.plane + k] = s.sv[i][q0];
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    const int sx = x - ex(a), sy = y - ey(a);
    const float G = gamma_a(a, ux, uy);
    if (!P.periodic_y && (sy < 0 || sy >= P.ny)) {  // returned by the wall
      gy[a] = s.g[opp(a)][q0];
#pragma unroll
      for (int i = 0; i < NH; ++i)
        h_out[pop_index(k, i * 9 + a, 9 * NH)] = s.h[i][opp(a)][q0] + 0.5f * s.sv[i][q0] * G;
    } else if (sx < 0) {
      const int q = R1::slot(tx, ty - ey(a));  // column 0 of the source row
      const int qc = RC::slot(tx, ty - ey(a));
      const float rho = s.rho[qc], p = s.p[qc], w = wt(a);
      const float Gin = gamma_a(a, P.u_in, 0.0f);
      const float rc = rho * kCs2, u0 = s.ux[q], v0 = s.uy[q];
      const float eu = ex(a) * u0 + ey(a) * v0, uu = u0 * u0 + v0 * v0;
      const float eq_in = __fmaf_rn(w, p, __fmul_rn(rc, __fsub_rn(Gin, w)));
      const float eq_0 = __fmaf_rn(w, p, __fmul_rn(rc, __fmaf_rn(w, 1.0f + 3.0f * eu + 4.5f * eu * eu - 1.5f * uu, -w)));
      gy[a] = eq_in + (s.g[a][q] - eq_0);
#pragma unroll
      for (int i = 0; i < NH; ++i)
        h_out[pop_index(k, i * 9 + a, 9 * NH)] = P.c_in[i] * Gin + 0.5f * s.sv[i][q0] * G;
    } else if (sx >= P.nx) {
      const int q = R1::slot(tx, ty - ey(a));       // column nx - 1 of the source row
      const int qi = R1::slot(tx - 1, ty);          // (nx - 2, y), where its population arrives
      entered |= 1u << a;
      wsum += wt(a);
      gy[a] = (g[pop_index(k, a, 9)] + U * s.g[a][q]) * inv;
      const float Gi = gamma_a(a, s.ux[qi], s.uy[qi]);
#pragma unroll
      for (int i = 0; i < NH; ++i) {
        const float arrives = s.h[i][a][q] + 0.5f * s.sv[i][qi] * Gi;
        const long long o = pop_index(k, i * 9 + a, 9 * NH);
        h_out[o] = (h_old[o] + U * arrives) * inv;
      }
    } else {
      const int q = R1::slot(tx - ex(a), ty - ey(a));
      gy[a] = s.g[a][q];
#pragma unroll
      for (int i = 0; i < NH; ++i)
        h_out[pop_index(k, i * 9 + a, 9 * NH)] = s.h[i][a][q] + 0.5f * s.sv[i][q0] * G;
    }
  }
  if (outlet && wsum > 0.f) {
    float p0 = 0.f;
#pragma unroll
    for (int a = 0; a < 9; ++a) p0 += gy[a];
#pragma unroll
    for (int a = 0; a < 9; ++a)
      if (entered >> a & 1u) gy[a] -= p0 * wt(a) / wsum;
  }
#pragma unroll
  for (int a = 0; a < 9; ++a) g_out[pop_index(k, a, 9)] = gy[a];
}

// Sources, collision and streaming of a tile where x is periodic: every node collides
// once and stores its populations at the nodes they arrive at, whose sources and
// velocity (for the term of R9) are in the tile's ring.  The gather form above
// collides the ring as well, 204 nodes for 128; here the ring costs its sources only, and the
// stencils of a node reach two nodes instead of three.  One row's stores stay
// together, shifted by a column in the six directions with e_x.  Bound by instruction issue.
// Against the gather form (which this scheme took as well), us per step, with the launches of the
// time (200 x 400 takes 12.4 with more of them in graphs): 200 x 400 18.0 -> 14.2,
// 1024 x 2048 225 -> 182 (157 -> 113 in this kernel), three components 256 x 256 18.3 -> 14.5.
// Five or six CTAs per SM (fewer registers) are within 2 % of the four asked for.
template <int NH>
struct PushSmem {
  using R2 = Ring<2>;
  using R1 = Ring<1>;
  float C[NH][R2::N], rho[R2::N], p[R2::N], mu[NH][R2::N];
  float sv[NH][R1::N], ux[R1::N], uy[R1::N];
};
template <int NH, int SCHEME, int MINB>
__global__ void __launch_bounds__(kTileX *kTileY, MINB)
    k_collide_push(DevParams P, const float *__restrict__ g, const float *__restrict__ Cf,
                   const float *__restrict__ mu, const float *__restrict__ pf, const float *__restrict__ uxf,
                   const float *__restrict__ uyf, const float *__restrict__ tau_new, float *__restrict__ SV,
                   float *__restrict__ g_out, float *__restrict__ h_out) {
  using S = PushSmem<NH>;
  using R2 = typename S::R2;
  using R1 = typename S::R1;
  constexpr int NT = kTileX * kTileY;
  __shared__ S s;
  const int t = threadIdx.x, x0 = blockIdx.x * kTileX, y0 = blockIdx.y * kTileY;
  const int tx = t % kTileX, ty = t / kTileX, x = x0 + tx, y = y0 + ty;
  const bool mine = x < P.nx && y < P.ny;
  const long long k = node_index(P, x, y);
  NodeCtx n;
  float gv[9], tn = 0.f;
  if (mine) {
#pragma unroll
    for (int a = 0; a < 9; ++a) gv[a] = g[pop_index(k, a, 9)];
    tn = tau_new[k];
#pragma unroll
    for (int j = 0; j < 3; ++j) n.mu[j] = mu[(long long)j * P.plane + k];
  }
  const bool inside = tile_inside(P, x0, y0, 2);
  for (int q = t; q < R2::N; q += NT) {
    const int cx = q % R2::W - 2, cy = q / R2::W - 2;
    const long long kq = inside ? node_index(P, x0 + cx, y0 + cy) : tile_node(P, x0 + cx, y0 + cy);
    const float c0 = Cf[kq], c1 = NH == 2 ? Cf[P.plane + kq] : 0.0f;
    s.C[0][q] = c0;
    if (NH == 2) s.C[NH - 1][q] = c1;
    s.rho[q] = rho_of(P, c0, c1, 1.0f - c0 - c1);
    s.p[q] = pf[kq];
#pragma unroll
    for (int i = 0; i < NH; ++i) s.mu[i][q] = mu[(long long)i * P.plane + kq];
    if (cx >= -1 && cx <= kTileX && cy >= -1 && cy <= kTileY) {
      s.ux[R1::slot(cx, cy)] = uxf[kq];
      s.uy[R1::slot(cx, cy)] = uyf[kq];
    }
  }
  __syncthreads();
  for (int q = t; q < R1::N; q += NT) {
    const int lx = q % R1::W - 1, ly = q / R1::W - 1;
    if (!P.periodic_y && (y0 + ly < 0 || y0 + ly >= P.ny)) continue;  // beyond a wall nothing arrives
#pragma unroll
    for (int i = 0; i < NH; ++i) {
      float cv[9], mv[9];
#pragma unroll
      for (int a = 0; a < 9; ++a) {
        cv[a] = s.C[i][R2::slot(lx + ex(a), ly + ey(a))];
        mv[a] = s.mu[i][R2::slot(lx + ex(a), ly + ey(a))];
      }
      s.sv[i][q] = source_of(P, i, cv, mv);
    }
  }
  __syncthreads();
  if (!mine) return;
  const int q0 = R1::slot(tx, ty);
  float sv[NH];
#pragma unroll
  for (int i = 0; i < NH; ++i) {
    sv[i] = s.sv[i][q0];
    SV[(long long)i * P.plane + k] = sv[i];
  }
  n.ux = s.ux[q0];
  n.uy = s.uy[q0];
  const StencilReader<NH, S, R2> at{s, tx, ty};
  const bool last_row = !P.periodic_y && y == P.ny - 1, first_row = !P.periodic_y && y == 0;
  collide_node<NH, SCHEME>(P, n, at, sv, gv, tn, [&](int a, float gs, const float (&hs)[NH]) {
    // half-way bounce-back: back to this node, in the opposite direction
    const bool back = (ey(a) > 0 && last_row) || (ey(a) < 0 && first_row);
    const int b = back ? opp(a) : a, q = back ? q0 : R1::slot(tx + ex(a), ty + ey(a));
    const long long kd = back ? k : node_index(P, wrap_x(x + ex(a), P.nx), wrap_y(y + ey(a), P.ny, 1));
    const float G = back ? gamma_a(opp(a), s.ux[q], s.uy[q]) : gamma_a(a, s.ux[q], s.uy[q]);
    g_out[pop_index(kd, b, 9)] = gs;
#pragma unroll
    for (int i = 0; i < NH; ++i) h_out[pop_index(kd, i * 9 + b, 9 * NH)] = hs[i] + 0.5f * s.sv[i][q] * G;
  });
}

// Modified equilibria (Eq. 16, 20) of given C, p, u, and tau at zero strain rate
// (reading R11), rows [y0, y1), into the stored form of the state.  The fields come as
// the host's dense FP64 planes and are rounded to FP32 (to nearest) as they enter the
// tile: C, rho and p of the 32 x 8 tile and its stencil ring in shared memory, g encoded
// and C stored by the same kernel in the C forms.  REST: p = u = 0 (the usual set-up),
// where Gamma_a = w_a and most terms of Phi vanish.  A conversion pass into FP32 planes, a
// pass that read them through L1 and, with FP16 storage, an encoding pass bound the set-up:
// lbm_set_fields of C from page-locked memory 815 -> 431 us at 2048 x 4096 (344 us of it the
// upload), 127 -> 68 us at 517 x 1031, 284 -> 137 us at 1024 x 2048 with FP16 storage (GB300).
struct InitFields {
  const double *C, *p, *ux, *uy;  // nh, 1, 1, 1 planes of ny x nx (p, ux, uy: NULL for zero)
};
template <int NH, int SCHEME, int FORM, bool REST>
__global__ void __launch_bounds__(256) k_init(DevParams P, InitFields in, float *__restrict__ g, float *__restrict__ h,
                                              float *__restrict__ tau, int row0, int row1) {
  constexpr int TX = 32, TY = 8, R = 1 + SCHEME, W = TX + 2 * R, N = W * (TY + 2 * R);
  __shared__ float sC[NH][N], srho[N], sp[REST ? 1 : N];
  const int t = threadIdx.x, tx = t % TX, ty = t / TX, x0 = blockIdx.x * TX, y0 = row0 + blockIdx.y * TY;
  const int x = x0 + tx, y = y0 + ty;
  const size_t dense = (size_t)P.nx * P.ny;
  const bool inside = x0 >= R && y0 >= R && x0 + TX + R <= P.nx && y0 + TY + R <= P.ny;
  for (int q = t; q < N; q += 256) {
    const int xq = x0 + q % W - R, yq = y0 + q / W - R;
    if (yq >= row1 + R) break;  // beyond what the rows below row1 read (it may not have arrived)
    const size_t d = inside ? (size_t)yq * P.nx + xq
                            : (size_t)row_read(yq, P.ny, P.periodic_y) * P.nx + tile_column(P, xq);
    const float c0 = (float)in.C[d], c1 = NH == 2 ? (float)in.C[dense + d] : 0.0f;
    sC[0][q] = c0;
    if (NH == 2) sC[NH - 1][q] = c1;
    srho[q] = rho_of(P, c0, c1, 1.0f - c0 - c1);
    if (!REST) sp[q] = in.p ? (float)in.p[d] : 0.0f;
  }
  __syncthreads();
  if (x >= P.nx || y >= row1) return;
  const long long k = node_index(P, x, y);
  struct {
    const float (&sC)[NH][N];
    const float (&srho)[N];
    const float *sp;
    int q0;
    __device__ __forceinline__ void C(int dx, int dy, float c[3]) const {
      const int q = q0 + dy * W + dx;
      c[0] = sC[0][q];
      c[1] = NH == 2 ? sC[NH - 1][q] : 0.0f;
      c[2] = 1.0f - c[0] - c[1];
    }
    __device__ __forceinline__ float rho(int dx, int dy, const float *) const { return srho[q0 + dy * W + dx]; }
    __device__ __forceinline__ float p(int dx, int dy) const { return REST ? 0.0f : sp[q0 + dy * W + dx]; }
  } at{sC, srho, sp, (ty + R) * W + tx + R};
  NodeCtx n;
  gather_gradients(SCHEME, at, n);
  float Cn[9][3], lapC[3];
#pragma unroll
  for (int a = 0; a < 9; ++a) at.C(ex(a), ey(a), Cn[a]);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    float lp = 0.f;
#pragma unroll
    for (int a = 0; a < 9; ++a) lp += wt(a) * (Cn[a][j] - Cn[0][j]);
    lapC[j] = 6.0f * lp;
  }
  chem_potentials(P, n.C, lapC, n.mu);
  const size_t d0 = (size_t)y * P.nx + x;
  n.ux = !REST && in.ux ? (float)in.ux[d0] : 0.0f;
  n.uy = !REST && in.uy ? (float)in.uy[d0] : 0.0f;
  n.Fs[0] = n.mu[0] * n.gC[0][0] + n.mu[1] * n.gC[1][0] + n.mu[2] * n.gC[2][0];
  n.Fs[1] = n.mu[0] * n.gC[0][1] + n.mu[1] * n.gC[1][1] + n.mu[2] * n.gC[2][1];
  n.Fb[0] = P.force_x;
  n.Fb[1] = -n.rho * P.gravity;
  // Which product is rounded on its own is spelled out, as in collide_node and for its reason: also the
  // dependence on the component count, below and in the test a < NH, is an earlier compilation's.
  auto h_eq = [](float C, float G, float ph) {
    return NH == 1 ? __fmaf_rn(C, G, -0.5f * ph) : __fmaf_rn(-0.5f, ph, __fmul_rn(C, G));
  };
  float ge[9];
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    if constexpr (REST) {
      const float w = wt(a);
      const float eF = (n.mu[0] * n.dC[0][a] + n.mu[1] * n.dC[1][a] + n.mu[2] * n.dC[2][a]) +
                       (ex(a) * n.Fb[0] + ey(a) * n.Fb[1]);
      ge[a] = 0.0f - 0.5f * (eF * w);  // subtracted from w p = 0, as below: no force gives +0
      if constexpr (FORM == 0) {
#pragma unroll
        for (int i = 0; i < NH; ++i) {
          const float ph = (n.dC[i][a] + n.C[i] / (n.rho * kCs2) * eF) * w;
          h[pop_index(k, i * 9 + a, 9 * NH)] = h_eq(n.C[i], w, ph);
        }
      }
    } else {
      const float G = gamma_a(a, n.ux, n.uy);
      const float pg = phi_g(n, a, G), Gw = G - wt(a), rc = n.rho * kCs2;
      const float lin = a < NH ? __fmaf_rn(wt(a), n.p, __fmul_rn(rc, Gw)) : __fmaf_rn(rc, Gw, __fmul_rn(wt(a), n.p));
      ge[a] = lin - 0.5f * pg;
      if constexpr (FORM == 0) {
#pragma unroll
        for (int i = 0; i < NH; ++i) h[pop_index(k, i * 9 + a, 9 * NH)] = h_eq(n.C[i], G, phi_h(n, i, a, G));
      }
    }
  }
  if constexpr (FORM == 2) {
    const float Pn = g16_reference(ge);
    g[(9 * P.plane) / 2 + k] = Pn;
    __half *gh = reinterpret_cast<__half *>(g) + pop_index(k, 0, 9);
#pragma unroll
    for (int a = 0; a < 9; ++a) gh[a * 32] = g16_encode(ge[a], Pn, a, P.g16_scale);
  } else {
#pragma unroll
    for (int a = 0; a < 9; ++a) g[pop_index(k, a, 9)] = ge[a];
  }
  if constexpr (FORM != 0) {
#pragma unroll
    for (int i = 0; i < NH; ++i) h[(long long)i * P.plane + k] = n.C[i];
  }
  const float tau1 = P.powerlaw ? tau_powerlaw(P, 0.0f, 1.0f / n.rho) : P.tau[0];
  tau[k] = tau_mix(P, n.C[0], n.C[1], n.C[2], tau1);
}

// Initial discs (Eq. 42) as dense FP64 planes of C_1 (and C_2), one thread per
// node: every disc adds 0.5 - 0.5 tanh((r - R) / (xi / 2)) to its component in
// the given order, then the noise, then the matrix takes the rest.  Discs come in groups
// of kDiscs per launch; between groups the planes hold the sums of components 3 and 2.
// Farther than 20 half widths from the interface the tanh is +-1 in FP64 (1 - 8.5e-18), so only
// the interface pays for it.  The host loop this replaces took 1.95 ms at 400 x 800 and 45.9 ms
// at 2048 x 4096 with its upload; on the device 0.06 and 0.87 ms with the equilibria (GB300).
__device__ __forceinline__ double noise_at(unsigned long long seed, unsigned long long i) {
  unsigned long long z = seed + (i + 1) * 0x9E3779B97F4A7C15ULL;  // SplitMix64 (Steele, Lea and Flood 2014)
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  z ^= z >> 31;
  return 2.0 * ((double)(z >> 11) * (1.0 / 9007199254740992.0)) - 1.0;
}
__global__ void __launch_bounds__(256) k_discs(int nx, int ny, int nh, int periodic_y, double xi, DiscGroup d,
                                               double *__restrict__ C) {
  const int x = blockIdx.x * 32 + threadIdx.x % 32, y = blockIdx.y * 8 + threadIdx.x / 32;
  if (x >= nx || y >= ny) return;
  const size_t n = (size_t)nx * ny, k = (size_t)y * nx + x;
  double gas = d.first ? 0.0 : C[k], second = d.first || nh == 1 ? 0.0 : C[n + k];  // components 3 and 2
  for (int b = 0; b < d.count; ++b) {
    double dx = fabs(x - d.disc[b].cx), dy = fabs(y - d.disc[b].cy);
    if (dx > 0.5 * nx) dx = nx - dx;
    if (periodic_y && dy > 0.5 * ny) dy = ny - dy;
    const double a = (sqrt(dx * dx + dy * dy) - d.disc[b].r) / (0.5 * xi);
    const double v = a > 20.0 ? 0.0 : (a < -20.0 ? 1.0 : 0.5 - 0.5 * tanh(a));
    if (d.disc[b].comp == 3) gas += v;
    else second += v;
  }
  if (!d.last) {
    C[k] = gas;
    if (nh == 2) C[n + k] = second;
    return;
  }
  if (d.noise[0] != 0.0) second += d.noise[0] * noise_at(d.seed, n + k);
  if (d.noise[1] != 0.0) gas += d.noise[1] * noise_at(d.seed, 2 * n + k);
  C[k] = 1.0 - second - gas;
  if (nh == 2) C[n + k] = second;
}

// Fields for the host, as dense FP64 planes: FP32 planes, C_3 or the density of the
// clipped mixture (R1) from the C planes, and planes [q0, q1) of a population array
// (g16: the FP16 form of g, decoded).  The host loops over FP32 copies that these replace
// took most of lbm_get_field: at 400 x 800 u_x 142 -> 58 us, rho 720 -> 68 us, g 2.7 -> 0.19 ms.
__global__ void __launch_bounds__(256) k_planes_to_f64(DevParams P, double3 rho, const float *__restrict__ src,
                                                       int kind, double *__restrict__ dst) {
  const int x = blockIdx.x * 32 + threadIdx.x % 32, y = blockIdx.y * 8 + threadIdx.x / 32, q = blockIdx.z;
  if (x >= P.nx || y >= P.ny) return;
  const long long k = node_index(P, x, y);
  const size_t o = ((size_t)q * P.ny + y) * P.nx + x;
  if (kind == kPlane) {
    dst[o] = (double)src[(long long)q * P.plane + k];
    return;
  }
  const float c1 = src[k], c2 = P.nh == 2 ? src[P.plane + k] : 0.0f, c3 = 1.0f - c1 - c2;
  if (kind == kThird) {
    dst[o] = (double)c3;
    return;
  }
  // (by comparisons: fmin and fmax would turn a NaN into a weight of 0 and hide it)
  auto clip = [](double v) { return v < 0.0 ? 0.0 : (v > 1.0 ? 1.0 : v); };
  const double w1 = clip((double)c1), w2 = clip((double)c2), w3 = clip((double)c3);
  dst[o] = (w1 * rho.x + w2 * rho.y + w3 * rho.z) / (w1 + w2 + w3);
}
__global__ void __launch_bounds__(256) k_pops_to_f64(DevParams P, const float *__restrict__ src, int q0, int nq, int g16,
                                                     double *__restrict__ dst) {
  const int x = blockIdx.x * 32 + threadIdx.x % 32, y = blockIdx.y * 8 + threadIdx.x / 32, q = q0 + blockIdx.z;
  if (x >= P.nx || y >= P.ny) return;
  const long long k = node_index(P, x, y);
  float v;
  if (g16)
    v = g16_decode(src[(9 * P.plane) / 2 + k], reinterpret_cast<const __half *>(src)[pop_index(k, q, 9)], q,
                   P.g16_inv_scale);
  else
    v = src[pop_index(k, q, nq)];
  dst[((size_t)blockIdx.z * P.ny + y) * P.nx + x] = (double)v;
}

// A running FP32 sum with Neumaier's compensation: c collects the rounding
// error of every addition (and, in add_prod, the exact error of the product,
// from fmaf), so s + c, taken in FP64, is the exact sum of a short run of
// terms up to a relative error of order n 2^-48.  Explicit _rn intrinsics keep
// the compiler from fusing a product into the next addition.
struct CompSum {
  float s, c;
  __device__ __forceinline__ void add(float v) {
    const float t = __fadd_rn(s, v);
    c = __fadd_rn(c, fabsf(s) >= fabsf(v) ? __fadd_rn(__fsub_rn(s, t), v) : __fadd_rn(__fsub_rn(v, t), s));
    s = t;
  }
  __device__ __forceinline__ void add_prod(float a, float b) {
    const float p = __fmul_rn(a, b);
    add(p);
    c = __fadd_rn(c, __fmaf_rn(a, b, -p));
  }
};

// Nodes a thread sums in FP32 (compensated) before it adds the run to its
// FP64 totals: GB300's FP64 pipe runs at a small fraction of its FP32 rate, so
// one FP64 addition per node and quantity bound the kernel.
constexpr int kObsRun = 16;

// Observable sums (Sec. 3.1; Eq. 43-44 inputs) in FP64: acc[0..10] = M1..3,
// M1..3 above 0.5, A, sum C_g x, sum C_g y, sum C_g ux, sum C_g uy; ext[0..3] =
// the largest nx - x, x + 1, ny - y, y + 1 of C_g > 0.5 (0: none).  Both zeroed before.
// Straight from the state in its stored form: a CTA walks tiles of 32 x 8 nodes
// with C and rho of the tile and its one-node ring in shared memory (two buffers, one
// barrier per tile), u computed per node by fields_math.  Each state value is read
// once (the ring's again, from L2), where a pass that wrote C planes and 9-point reads
// of them through L1 took 391 us at 2048 x 4096 per lbm_observables, and now 232 us (72 B/node at
// the measured HBM rate: 90 us; bound by the issue of a node's about 600
// instructions).  Sums: warp shuffles, one shared-memory pass per block, one atomic
// per block and quantity.
constexpr int kObsThreads = 256;
template <int NH, int FORM>
__global__ void __launch_bounds__(kObsThreads, 3) k_observe(DevParams P, FusedBuffers B, int gas_comp, double *acc,
                                                            int *ext) {
  constexpr int TX = 32, TY = 8, W = TX + 2, N = W * (TY + 2);
  static_assert(TX * TY == kObsThreads, "a thread per node");
  __shared__ float sC[2][NH][N], srho[2][N];
  const int t = threadIdx.x, tx = t % TX, ty = t / TX;
  // the FP64 totals are touched once per run of nodes and wait in shared memory
  __shared__ double total[11][kObsThreads];
  CompSum r[11];
#pragma unroll
  for (int q = 0; q < 11; ++q) {
    total[q][t] = 0.0;
    r[q] = {0.f, 0.f};
  }
  int run = 0;
  auto flush = [&]() {
#pragma unroll
    for (int q = 0; q < 11; ++q) {
      total[q][t] += (double)r[q].s + (double)r[q].c;
      r[q] = {0.f, 0.f};
    }
    run = 0;
  };
  int e[4] = {0, 0, 0, 0};
  const int cols = (P.nx + TX - 1) / TX, tiles = cols * ((P.ny + TY - 1) / TY);
  int buf = 0;
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x, buf ^= 1) {
    const int x0 = tile % cols * TX, y0 = tile / cols * TY, x = x0 + tx, y = y0 + ty;
    const bool mine = x < P.nx && y < P.ny;
    const bool inside = x0 >= 1 && y0 >= 1 && x0 + TX + 1 <= P.nx && y0 + TY + 1 <= P.ny;
    float ga[9];
    if (mine) load_populations<FORM>(P, B, P.plane, node_index(P, x, y), ga);
#pragma unroll
    for (int k = 0; k < (N + kObsThreads - 1) / kObsThreads; ++k) {
      const int q = t + k * kObsThreads;
      if (q < N) {
        const int xq = x0 + q % W - 1, yq = y0 + q / W - 1;
        float c[NH];
        load_order_parameters<NH, FORM>(B, P.plane, inside ? node_index(P, xq, yq) : tile_node(P, xq, yq), c);
#pragma unroll
        for (int i = 0; i < NH; ++i) sC[buf][i][q] = c[i];
        const float c1 = NH == 2 ? c[NH - 1] : 0.0f;
        srho[buf][q] = rho_of(P, c[0], c1, 1.0f - c[0] - c1);
      }
    }
    __syncthreads();
    if (!mine) continue;
    NodeCtx n;
    float Cn[9][3], rn[9], m0;
#pragma unroll
    for (int a = 0; a < 9; ++a) {
      const int q = (ty + 1 + ey(a)) * W + tx + 1 + ex(a);
      Cn[a][0] = sC[buf][0][q];
      Cn[a][1] = NH == 2 ? sC[buf][NH - 1][q] : 0.0f;
      Cn[a][2] = 1.0f - Cn[a][0] - Cn[a][1];
      rn[a] = srho[buf][q];
    }
    fields_math<false>(P, n, Cn, rn, ga, m0);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      r[i].add(n.C[i]);
      r[3 + i].add(n.C[i] > 0.5f ? n.C[i] : 0.0f);
    }
    // C of the gas component, selected without indexing (keeps n in registers)
    const float cg = gas_comp == 1 ? n.C[0] : (gas_comp == 2 ? n.C[1] : n.C[2]);
    r[6].add(cg);
    r[7].add_prod(cg, (float)x);  // x, y < 2^24: exact in FP32
    r[8].add_prod(cg, (float)y);
    r[9].add_prod(cg, n.ux);
    r[10].add_prod(cg, n.uy);
    if (++run == kObsRun) flush();
    if (cg > 0.5f) {
      e[0] = max(e[0], P.nx - x);
      e[1] = max(e[1], x + 1);
      e[2] = max(e[2], P.ny - y);
      e[3] = max(e[3], y + 1);
    }
  }
  flush();
  for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
    for (int q = 0; q < 4; ++q) e[q] = max(e[q], __shfl_down_sync(0xffffffffu, e[q], off));
  }
  __shared__ int se[kObsThreads / 32][4];
  const int lane = t & 31, warp = t >> 5;
  if (lane == 0) {
#pragma unroll
    for (int q = 0; q < 4; ++q) se[warp][q] = e[q];
  }
  __syncthreads();
  // the FP64 adder runs at a small fraction of the FP32 rate: a tree over shared memory
  // fills its lanes, where warp shuffles take five additions of every thread's eleven sums
  for (int w = kObsThreads / 2; w > 0; w >>= 1) {
    for (int i = t; i < 11 * w; i += kObsThreads) total[i / w][i & (w - 1)] += total[i / w][(i & (w - 1)) + w];
    __syncthreads();
  }
  if (t < 11) {
    atomicAdd(&acc[t], total[t][0]);
  } else if (t >= 32 && t < 36) {
    int m = 0;
    for (int w = 0; w < kObsThreads / 32; ++w) m = max(m, se[w][t - 32]);
    if (m > 0) atomicMax(&ext[t - 32], m);
  }
}

static dim3 node_grid(const DevParams &P, dim3 blk) {
  return dim3((P.nx + blk.x - 1) / blk.x, (P.ny + blk.y - 1) / blk.y);
}

template <int NH, int SCHEME>
static cudaError_t split_step(const DevParams &P, const StepBuffers &B, cudaStream_t s, cudaEvent_t *ev) {
  using S = CollideSmem<NH, SCHEME>;
  static_assert(sizeof(S) <= 48 * 1024, "no opt-in for more shared memory");
  const dim3 grd((P.nx + kTileX - 1) / kTileX, (P.ny + kTileY - 1) / kTileY);
  if (ev) cudaEventRecord(ev[0], s);
  k_fields_step<NH, SCHEME><<<grd, kTileX * kTileY, 0, s>>>(P, B.h_in, B.g_in, B.tau_in, B.C, B.mu, B.p, B.ux, B.uy,
                                                           B.tau_out, B.shear, B.err);
  if (ev) cudaEventRecord(ev[1], s);
  if (P.open_x)
    k_collide_step<NH, SCHEME, NH == 1 ? 4 : 2><<<grd, kCollideThreads, sizeof(S), s>>>(
        P, B.g_in, B.h_in, B.C, B.mu, B.p, B.ux, B.uy, B.tau_out, B.SV, B.g_out, B.h_out);
  else if constexpr (SCHEME == 1)  // (periodic x with central differences takes the one-kernel forms)
    k_collide_push<NH, SCHEME, NH == 1 ? 4 : 2><<<grd, kTileX * kTileY, 0, s>>>(P, B.g_in, B.C, B.mu, B.p, B.ux, B.uy, B.tau_out,
                                                                  B.SV, B.g_out, B.h_out);
  else
    return cudaErrorNotSupported;
  if (ev) cudaEventRecord(ev[2], s);
  return cudaGetLastError();
}

cudaError_t launch_split_step(const DevParams &P, const StepBuffers &B, cudaStream_t s, cudaEvent_t *ev) {
  if (P.nh == 1) return P.fd_scheme == 1 ? split_step<1, 1>(P, B, s, ev) : split_step<1, 0>(P, B, s, ev);
  return P.fd_scheme == 1 ? split_step<2, 1>(P, B, s, ev) : split_step<2, 0>(P, B, s, ev);
}

void launch_macros(const DevParams &P, const StepBuffers &B, cudaStream_t s) {
  const dim3 blk(32, 8);
  const dim3 grd = node_grid(P, blk);
  if (B.h_in) k_moments<<<grd, blk, 0, s>>>(P, B.h_in, B.C);  // null: the state holds C
  if (P.nh == 1)
    k_fields<1><<<grd, blk, 0, s>>>(P, B.C, B.g_in, B.mu, B.p, B.ux, B.uy);
  else
    k_fields<2><<<grd, blk, 0, s>>>(P, B.C, B.g_in, B.mu, B.p, B.ux, B.uy);
}

template <int NH, int SCHEME, int FORM>
static cudaError_t init_rows(const DevParams &P, const InitFields &in, float *g, float *h, float *tau, int y0, int y1,
                             cudaStream_t s) {
  const dim3 grd((P.nx + 31) / 32, (y1 - y0 + 7) / 8);
  if (!in.p && !in.ux && !in.uy)
    k_init<NH, SCHEME, FORM, true><<<grd, 256, 0, s>>>(P, in, g, h, tau, y0, y1);
  else
    k_init<NH, SCHEME, FORM, false><<<grd, 256, 0, s>>>(P, in, g, h, tau, y0, y1);
  return cudaGetLastError();
}

cudaError_t launch_init_rows(const DevParams &P, const double *C, const double *p, const double *ux, const double *uy,
                             float *g, float *h, float *tau, int y0, int y1, cudaStream_t s) {
  if (y1 <= y0) return cudaSuccess;
  const InitFields in{C, p, ux, uy};
  if (P.nh == 1) {
    if (P.g16) return init_rows<1, 0, 2>(P, in, g, h, tau, y0, y1, s);
    if (P.collapse_h) return init_rows<1, 0, 1>(P, in, g, h, tau, y0, y1, s);
    return P.fd_scheme == 1 ? init_rows<1, 1, 0>(P, in, g, h, tau, y0, y1, s)
                            : init_rows<1, 0, 0>(P, in, g, h, tau, y0, y1, s);
  }
  if (P.g16) return init_rows<2, 0, 2>(P, in, g, h, tau, y0, y1, s);
  if (P.collapse_h) return init_rows<2, 0, 1>(P, in, g, h, tau, y0, y1, s);
  return P.fd_scheme == 1 ? init_rows<2, 1, 0>(P, in, g, h, tau, y0, y1, s)
                          : init_rows<2, 0, 0>(P, in, g, h, tau, y0, y1, s);
}

cudaError_t launch_discs(const DevParams &P, double xi, const DiscGroup &d, double *C, cudaStream_t s) {
  k_discs<<<dim3((P.nx + 31) / 32, (P.ny + 7) / 8), 256, 0, s>>>(P.nx, P.ny, P.nh, P.periodic_y, xi, d, C);
  return cudaGetLastError();
}

cudaError_t launch_planes_to_f64(const DevParams &P, const double rho[3], const float *src, int kind, int nplanes,
                                 double *dst, cudaStream_t s) {
  k_planes_to_f64<<<dim3((P.nx + 31) / 32, (P.ny + 7) / 8, nplanes), 256, 0, s>>>(
      P, make_double3(rho[0], rho[1], rho[2]), src, kind, dst);
  return cudaGetLastError();
}

cudaError_t launch_pops_to_f64(const DevParams &P, const float *src, int q0, int q1, int nq, bool g16, double *dst,
                               cudaStream_t s) {
  k_pops_to_f64<<<dim3((P.nx + 31) / 32, (P.ny + 7) / 8, q1 - q0), 256, 0, s>>>(P, src, q0, nq, g16 ? 1 : 0, dst);
  return cudaGetLastError();
}

// C_i of the population form into the C planes.
void launch_moments(const DevParams &P, const float *h, float *C, cudaStream_t s) {
  const dim3 blk(32, 8);
  k_moments<<<node_grid(P, blk), blk, 0, s>>>(P, h, C);
}

cudaError_t launch_observe(const DevParams &P, const FusedBuffers &B, int gas_comp, double *acc, int *ext,
                           cudaStream_t s) {
  const long long tiles = (long long)((P.nx + 31) / 32) * ((P.ny + 7) / 8);
  const int cap = tiles < 912 ? 228 : 456;
  // three CTAs on each of the 152 SMs, half as many where each would have one tile or two
  const int blocks = tiles < cap ? (int)tiles : cap;
  const int form = P.g16 ? 2 : (P.collapse_h ? 1 : 0);
  if (P.nh == 1) {
    if (form == 2) k_observe<1, 2><<<blocks, kObsThreads, 0, s>>>(P, B, gas_comp, acc, ext);
    else if (form == 1) k_observe<1, 1><<<blocks, kObsThreads, 0, s>>>(P, B, gas_comp, acc, ext);
    else k_observe<1, 0><<<blocks, kObsThreads, 0, s>>>(P, B, gas_comp, acc, ext);
  } else {
    if (form == 2) k_observe<2, 2><<<blocks, kObsThreads, 0, s>>>(P, B, gas_comp, acc, ext);
    else if (form == 1) k_observe<2, 1><<<blocks, kObsThreads, 0, s>>>(P, B, gas_comp, acc, ext);
    else k_observe<2, 0><<<blocks, kObsThreads, 0, s>>>(P, B, gas_comp, acc, ext);
  }
  return cudaGetLastError();
}

}  // namespace lbm
