// Split form of the coupled step: node-parallel kernels over scratch planes.
//
// Binary32 arithmetic, three kernels:
//   k_macro    pull-stream + boundary closures; rho, j, T (moments), p_EOS -> psi and (dp/dT)_rho
//              (Eq. 56); optional per-block partial sums of rho for the buoyancy reference rho_ave.
//   k_force    psi stencil -> F = F_int + F_ads + F_b, v = (j + F/2)/rho, sigma term Q.
//   k_collide  pull again (same closures); isotropic grad T, lap T, grad rho, div v; source phi of
//              Eq. 28 and S0 of Eq. 46; flow MRT collide with forcing; thermal MRT collide with the
//              corrections of Eqs. 54-55; store post-collision f*, g* (pull scheme, A/B buffers).
// Binary64 and double-word arithmetic, two kernels: k_macro also leaves the flow moments and heat fluxes, and
// k_collide_tile takes the force and the collisions together.
//
// Each kernel reads its node's stencil straight from global memory (L1/L2 serve the reuse). With FP64
// arithmetic the step is bound by the FP64 pipe (84 % busy in both kernels), not by HBM, so its time is its
// count of FP64 instructions: 229 per node and step (k_macro 85, k_collide_tile 144). Three kernels that
// pulled f and g twice and rebuilt m* from all nine moments took 283. GB300, droplet evaporation 2048^2: 1.82 ms
// a step against 2.24 ms; 128^2 12 us against 20.6 us (with launch_pdl). Double-word arithmetic: 0.428 against
// 0.533 ms; there k_macro is at the measured HBM bandwidth (264 B per node in 164 us) and k_collide_tile at 64 % of
// it (280 B in 271 us) and bound by issue and latency.

#include <algorithm>
#include <type_traits>

#include "lbpc_device.cuh"
#include "lbpc_internal.h"

namespace lbpc {

constexpr int BLOCK = 64;  // small blocks spread small grids evenly over the 152 SMs

// Planes of the split path's scratch (type R, N nodes each).
enum { P_RHO = 0, P_T, P_PSI, P_JX, P_JY, P_DPDT, P_IRHO, P_VX, P_VY, P_FX, P_FY, P_Q, NPLANES };

template <class R> struct Planes {
  R* p[NPLANES];
};

__device__ __forceinline__ long long node_index(const DevParams& P, int x, int y) { return (long long)y * P.pitch + x; }

// Node i of the padded rows (i < 2^32, so the division is a 32-bit one).
struct Node {
  int x, y;
};
__device__ __forceinline__ Node node_at(const DevParams& P, long long i) {
  const unsigned y = (unsigned)i / (unsigned)P.pitch;
  return Node{(int)((unsigned)i - y * (unsigned)P.pitch), (int)y};
}

// Neighbour row for a stencil: wraps when y is periodic, else clamps to the edge row (ghost rows
// copy the edge row). out_lo/out_hi report a ghost beyond the lower / upper edge.
__device__ __forceinline__ int nb_row(const DevParams& P, int y, int dy, bool& ghost_lo, bool& ghost_hi) {
  int yy = y + dy;
  ghost_lo = ghost_hi = false;
  if (P.yper) return yy < 0 ? yy + P.ny : (yy >= P.ny ? yy - P.ny : yy);
  if (yy < 0) { ghost_lo = true; return 0; }
  if (yy >= P.ny) { ghost_hi = true; return P.ny - 1; }
  return yy;
}

// Gather the 3x3 neighbourhood c[dy+1][dx+1] of a plane with the copy-ghost rule.
template <class R> __device__ __forceinline__ void gather9(const R* __restrict__ X, const DevParams& P, int x, int y, R c[3][3]) {
  const int xm = wrapx(x - 1, P.nx), xp = wrapx(x + 1, P.nx);
#pragma unroll
  for (int dy = -1; dy <= 1; ++dy) {
    bool lo, hi;
    const long long row = (long long)nb_row(P, y, dy, lo, hi) * P.pitch;
    c[dy + 1][0] = ldgv(X + row + xm);
    c[dy + 1][1] = ldgv(X + row + x);
    c[dy + 1][2] = ldgv(X + row + xp);
  }
}

// Isotropic differences (reading of the paper's cited stencils): d_i X = 3 sum_a w_a X(x+e_a) e_ai,
// lap X = 6 sum_a w_a (X(x+e_a) - X(x)). c[1][1] is the centre, c[2][*] the row above.
template <class R> __device__ __forceinline__ R d_x(const R c[3][3]) {
  return (c[1][2] - c[1][0]) * R(1.0 / 3.0) + (c[2][2] - c[2][0] - c[0][0] + c[0][2]) * R(1.0 / 12.0);
}
template <class R> __device__ __forceinline__ R d_y(const R c[3][3]) {
  return (c[2][1] - c[0][1]) * R(1.0 / 3.0) + (c[2][2] + c[2][0] - c[0][0] - c[0][2]) * R(1.0 / 12.0);
}
template <class R> __device__ __forceinline__ R lap(const R c[3][3]) {
  const R ctr = c[1][1];
  return (c[1][2] + c[1][0] + c[2][1] + c[0][1] - ctr * 4) * R(2.0 / 3.0) +
         (c[2][2] + c[2][0] + c[0][0] + c[0][2] - ctr * 4) * R(1.0 / 6.0);
}

// STASH (binary64 and double-word steps): the flow moments and the heat fluxes n4, n6 go into the destination
// buffers (planes 0..5 of fdst, 0..1 of gdst), which nothing else uses until k_collide_tile overwrites the same
// entries of the same node with f*, g*.
template <class S, class R, bool STASH>
__global__ void __launch_bounds__(BLOCK) k_macro(PopBuf<S> fsrc, PopBuf<S> gsrc, S* __restrict__ fdst,
                                                 S* __restrict__ gdst, Planes<R> pl, DevParams P, long long step,
                                                 int do_partials, double* __restrict__ partials,
                                                 long long* __restrict__ status) {
  __shared__ double red[BLOCK / 32];
  const int t = pdl_wait<BLOCK>();
  const long long i = (long long)blockIdx.x * BLOCK + t;
  double rho_d = 0.0;
  const auto [x, y] = node_at(P, i);
  if (i < P.N && x < P.nx) {
    R f[9], g[9];
    if (sizeof(R) == 8 && x > 0 && x < P.nx - 1 && y > 0 && y < P.ny - 1) {
      const S *pf = fsrc.p + i, *pg = gsrc.p + i;  // no wrap, no closure
#pragma unroll
      for (int a = 0; a < 9; ++a) {
        const long long o = (long long)a * P.N - (long long)EY(a) * P.pitch - EX(a);
        f[a] = R(ldgv(pf + o));
        g[a] = R(ldgv(pg + o));
      }
    } else {
      pull_closed<S, R>(fsrc, gsrc, P, x, y, f, g);
    }
    R rho, jx, jy, Tlo, dpdT, inv_rho, psi2;
    const R T = heat_of(g, Tlo);
    if constexpr (sizeof(R) == 4) {
      rho = density_of(f);
      jx = f[1] - f[3] + f[5] - f[6] - f[7] + f[8];
      jy = f[2] - f[4] + f[5] + f[6] - f[7] - f[8];
      R p;
      eos(rho, T, P, p, dpdT, &inv_rho);
      psi2 = psi_squared(p, dpdT, Tlo, rho, coefs<R>(P));
    } else {
      R m[6];
      rho = flow_moments(f, jx, jy, m);
      psi2 = eos_psi_squared(rho, T, P, dpdT, inv_rho);
      if (STASH) {
#pragma unroll
        for (int a = 0; a < 6; ++a) fdst[(long long)a * P.N + i] = m[a];
        R n4, n6;
        heat_fluxes(g, n4, n6);
        gdst[i] = n4;
        gdst[P.N + i] = n6;
      }
    }
    check_node(rho, T, psi2, P, status, nullptr, step, x, y);
    pl.p[P_RHO][i] = rho;
    pl.p[P_T][i] = T;
    pl.p[P_PSI][i] = psi_of(psi2);
    pl.p[P_JX][i] = jx;
    pl.p[P_JY][i] = jy;
    pl.p[P_DPDT][i] = dpdT;
    pl.p[P_IRHO][i] = inv_rho;
    if (do_partials) rho_d = (double)rho;
  }
  if (do_partials) {
    const double s = block_sum<BLOCK>(rho_d, red);
    if (t == 0) partials[blockIdx.x] = s;
  }
}

template <class R>
__global__ void __launch_bounds__(BLOCK) k_force(Planes<R> pl, DevParams P, const double* __restrict__ rho_ave) {
  const int t = pdl_wait<BLOCK>();
  const Coefs<R>& C = coefs<R>(P);
  const long long i = (long long)blockIdx.x * BLOCK + t;
  if (i >= P.N) return;
  const auto [x, y] = node_at(P, i);
  if (x >= P.nx) return;
  const R* __restrict__ psi = pl.p[P_PSI];
  R c[3][3];
  gather9(psi, P, x, y, c);
  // F_int = -G psi(x) sum_a w(|e_a|^2) psi(x+e_a) e_a, w(1) = 1/3, w(2) = 1/12; ghost rows beyond a
  // non-periodic edge copy the edge row, so a wall with G_wall = 0 is neutral.
  const R pc = psi[i];
  const R sx = (c[1][2] - c[1][0]) * R(1.0 / 3.0) + (c[2][2] - c[2][0] - c[0][0] + c[0][2]) * R(1.0 / 12.0);
  const R sy = (c[2][1] - c[0][1]) * R(1.0 / 3.0) + (c[2][2] + c[2][0] - c[0][0] - c[0][2]) * R(1.0 / 12.0);
  const R Fix = -C.G * pc * sx, Fiy = -C.G * pc * sy;
  R Fx = Fix, Fy = Fiy;
  // F_ads = -G_w psi(x) sum_a w_a psi(x) s(x+e_a) e_a on the y- wall, whose solid ghost row gives the
  // sum (0, -1/2). A y+ wall is a neutral lid (the solid surfaces of Sec. IV are bottom walls).
  if (!P.yper && y == 0 && P.ybc_lo == BC_WALL) Fy += C.G_wall * 0.5f * pc * pc;
  const R rho = pl.p[P_RHO][i];
  if (P.buoyancy) {  // F_b = (rho - rho_ref) g: rho_ref = rho_ave (Sec. IV B) or the y+ edge's held density
    const R dr = rho - (P.buoyancy == 1 ? R(load_after_wait(rho_ave)) : C.rho_bc_hi);
    Fx += dr * C.gx;
    Fy += dr * C.gy;
  }
  const R inv_rho = pl.p[P_IRHO][i];
  pl.p[P_VX][i] = (pl.p[P_JX][i] + Fx * 0.5f) * inv_rho;
  pl.p[P_VY][i] = (pl.p[P_JY][i] + Fy * 0.5f) * inv_rho;
  pl.p[P_FX][i] = Fx;
  pl.p[P_FY][i] = Fy;
  // sigma term Q = qcoef |F_int|^2 / psi^2 = qcoef G^2 (sx^2 + sy^2): psi^2 cancels
  pl.p[P_Q][i] = C.qG2 * (sx * sx + sy * sy);
}

// Two warp-uniform roles per node: the first BLOCK threads of a block run the flow collision of
// BLOCK nodes, the next BLOCK threads run the source and thermal collision of the same nodes. The
// roles share no data (both read the scratch planes), so a node's work splits into two independent
// chains and twice as many warps hide the FP64 latency on small grids.
template <class S, class R>
__global__ void __launch_bounds__(2 * BLOCK)
    k_collide(PopBuf<S> fsrc, PopBuf<S> gsrc, PopBuf<S> fdst, PopBuf<S> gdst, Planes<R> pl, R* __restrict__ phi_prev,
              DevParams P, int first) {
  const Coefs<R>& C = coefs<R>(P);
  const int t = pdl_wait<2 * BLOCK>();
  const bool heat = t >= BLOCK;
  const long long i = (long long)blockIdx.x * BLOCK + (t - (heat ? BLOCK : 0));
  if (i >= P.N) return;
  const auto [x, y] = node_at(P, i);
  if (x >= P.nx) return;
  const R vx = pl.p[P_VX][i], vy = pl.p[P_VY][i];
  if (!heat) {
    R f[9];
    pull<S, R>(fsrc, C.wf, P, x, y, f);
    flow_closure(f, P, x, y, fsrc.wall);
    const R rho = pl.p[P_RHO][i];
    const R Fx = pl.p[P_FX][i], Fy = pl.p[P_FY][i];
    collide_flow(f, rho, vx, vy, Fx, Fy, pl.p[P_Q][i], P);
    pop_store<S, R>(fdst, P.N, i, f, rho, C.wf);
    wall_force_store(fdst.wall, P, x, y, Fx, Fy);
    return;
  }
  R g[9];
  pull<S, R>(gsrc, C.wg, P, x, y, g);
  heat_closure(g, P, x, y);
  const R rho = pl.p[P_RHO][i];
  const R T = pl.p[P_T][i];
  // gradients feeding the source (isotropic differences)
  R c[3][3];
  gather9(pl.p[P_T], P, x, y, c);
  const R gTx = d_x(c), gTy = d_y(c), lapT = lap(c);
  gather9(pl.p[P_VX], P, x, y, c);
  R divv = d_x(c);
  gather9(pl.p[P_VY], P, x, y, c);
  divv += d_y(c);
  const R rcv = rho * C.cV;
  const R inv_rcv = pl.p[P_IRHO][i] * C.inv_cV;
  R div_lam_gradT;
  if (P.lambda_mode == 0) {
    div_lam_gradT = C.lambda * lapT;
  } else {  // lambda = rho c_V chi: lambda lap T + c_V chi grad rho . grad T
    gather9(pl.p[P_RHO], P, x, y, c);
    div_lam_gradT = rcv * C.chi * lapT + C.cV_chi * (d_x(c) * gTx + d_y(c) * gTy);
  }
  const R compress = T * (R(1) - pl.p[P_DPDT][i] * inv_rcv) * divv;
  R phi, S0, tau_inv = R(0);
  if (P.model == 2) {
    // Gong-Cheng: the source is Eq. 13 alone; tau_g = lambda/(rho c_s^2 c_V) + 1/2 (Sec. IV A)
    phi = compress;
    S0 = phi;
    tau_inv = R(1) / ((P.lambda_mode == 0 ? C.lambda * 3 * inv_rcv : C.chi * 3) + R(0.5));
  } else {
    // phi: the underlined terms of Eq. 28 with k = (1/s_3 - 1/2) c_s^2
    phi = div_lam_gradT * inv_rcv - C.kdiff * lapT + compress;
    S0 = phi;
    if (P.model == 0) {  // S0 = phi + 0.5 dt d_t phi, d_t phi ~ [phi(t) - phi(t - dt)]/dt (Eq. 46)
      const R pp = first ? phi : phi_prev[i];
      S0 = phi + (phi - pp) * 0.5f;
    }
  }
  phi_prev[i] = phi;
  collide_heat(g, T, vx, vy, S0, P, tau_inv);
  pop_store<S, R>(gdst, P.N, i, g, T + S0, C.wg);
}

// Source offsets of the 3x3 neighbourhood of (x, y): rows below, at and above, columns left, at and right, as
// element offsets of a plane. interior: no neighbour lies beyond an edge.
struct Around {
  unsigned row[3], col[3];
};
__device__ __forceinline__ Around around(const DevParams& P, int x, int y, bool interior) {
  Around n;
  const unsigned nx = (unsigned)P.pitch;
  n.row[1] = (unsigned)y * nx;
  n.col[1] = (unsigned)x;
  if (interior) {
    n.row[0] = n.row[1] - nx;
    n.row[2] = n.row[1] + nx;
    n.col[0] = n.col[1] - 1u;
    n.col[2] = n.col[1] + 1u;
  } else {
    n.row[0] = y == 0 ? (P.yper ? (unsigned)(P.ny - 1) * nx : n.row[1]) : n.row[1] - nx;
    n.row[2] = y == P.ny - 1 ? (P.yper ? 0u : n.row[1]) : n.row[1] + nx;
    n.col[0] = x == 0 ? (unsigned)P.nx - 1u : n.col[1] - 1u;
    n.col[2] = x == P.nx - 1 ? 0u : n.col[1] + 1u;
  }
  return n;
}
template <class R> __device__ __forceinline__ void gather(const R* __restrict__ X, const Around& n, R c[3][3]) {
#pragma unroll
  for (int j = 0; j < 3; ++j)
#pragma unroll
    for (int k = 0; k < 3; ++k) c[j][k] = ldgv(X + (size_t)(n.row[j] + n.col[k]));
}

// Force and collision of the binary64 and double-word steps in one kernel over tiles of CX x CY nodes. The
// velocities of the tile and its 1-ring go to shared memory (the force of the ring is repeated: 15 of the 229
// binary64 instructions, 1.4 times), so the force, the velocity and the sigma term never visit device memory and the
// step is two launches. Then the two roles of
// k_collide: the first half of the block relaxes f from the moments that k_macro left in fdst, the second half
// evaluates the source and relaxes g from T, n4, n6 (or pulls g again where the rates are not all 1).
//
// The isotropic differences are taken without their common scale: d = (4 axis + diagonal)/12 and
// lap = (4 axes + diagonals - 20 centre)/6; the 1/12 and 1/6 join a coefficient that multiplies anyway.
template <class S, int CX, int CY>
__global__ void __launch_bounds__(2 * CX* CY)
    k_collide_tile(PopBuf<S> gsrc, PopBuf<S> fdst, PopBuf<S> gdst, Planes<S> pl, S* __restrict__ phi_prev, DevParams P,
                   int first, int tiles_x, const double* __restrict__ rho_ave) {
  using R = S;
  constexpr int CN = CX * CY, RING = 2 * (CX + 2) + 2 * CY;
  static_assert(RING <= CN, "one ring node per thread of the second half");
  __shared__ R s_vx[CY + 2][CX + 2], s_vy[CY + 2][CX + 2];
  const Coefs<R>& C = coefs<R>(P);
  const int t = pdl_wait<2 * CN>();
  const bool heat = t >= CN;
  const int x0 = (int)(blockIdx.x % (unsigned)tiles_x) * CX, y0 = (int)(blockIdx.x / (unsigned)tiles_x) * CY;
  const bool interior = x0 >= 2 && x0 + CX + 2 <= P.nx && y0 >= 2 && y0 + CY + 2 <= P.ny;
  // velocity node of this thread, in coordinates of the tile with its ring: the tile's own nodes, then the ring
  int hx, hy;
  const int q = heat ? t - CN : t;
  if (!heat) {
    hx = 1 + q % CX;
    hy = 1 + q / CX;
  } else if (q < 2 * (CX + 2)) {
    hx = q % (CX + 2);
    hy = q < CX + 2 ? 0 : CY + 1;
  } else {
    hx = (q & 1) ? CX + 1 : 0;
    hy = 1 + (q - 2 * (CX + 2)) / 2;
  }
  R Fx = R(0), Fy = R(0), Q = R(0), vx = R(0), vy = R(0), rho = R(0), jx = R(0), jy = R(0);
  // What the node's own role reads besides, asked for before the force so that its latency is hidden: the heat role's
  // values (double-word 2048^2 442 -> 430 us), and in binary64 the flow role's moments too; their 12 double-word
  // registers cost more there than they hide (459 us).
  constexpr bool kFlowFirst = !is_dw_t<S>::value;
  const int tx = q % CX, ty = q / CX;
  const bool active = x0 + tx < P.nx && y0 + ty < P.ny;
  const bool unit = P.model == 0 && P.heat_unit_rates;
  R m[6], n4 = R(0), n6 = R(0), pp = R(0), dpdT = R(0), inv_rho_own = R(0);
  auto pre_flow = [&]() {
    const S* pf = fdst.p + (size_t)(unsigned)(y0 + ty) * (unsigned)P.pitch + (unsigned)(x0 + tx);
#pragma unroll
    for (int a = 0; a < 6; ++a) m[a] = pf[(size_t)a * P.N];
  };
  auto pre_heat = [&]() {
    const size_t i = (size_t)(unsigned)(y0 + ty) * (unsigned)P.pitch + (unsigned)(x0 + tx);
    inv_rho_own = ldgv(pl.p[P_IRHO] + i);
    dpdT = ldgv(pl.p[P_DPDT] + i);
    if (P.model == 0 && !first) pp = phi_prev[i];
    if (unit) {
      n4 = gdst.p[i];
      n6 = gdst.p[P.N + i];
    }
  };
  if (kFlowFirst && !heat && active) pre_flow();
  if (heat && active) pre_heat();
  if (!heat || q < RING) {
    int x = x0 + hx - 1, y = y0 + hy - 1;
    if (!interior) {
      while (x < 0) x += P.nx;
      while (x >= P.nx) x -= P.nx;
      if (P.yper) {
        while (y < 0) y += P.ny;
        while (y >= P.ny) y -= P.ny;
      } else {  // a ghost row's velocity is the edge row's
        y = min(max(y, 0), P.ny - 1);
      }
    }
    const Around n = around(P, x, y, interior);
    const size_t i = n.row[1] + n.col[1];
    R c[3][3];
    gather(pl.p[P_PSI], n, c);
    rho = ldgv(pl.p[P_RHO] + i);
    const R inv_rho = ldgv(pl.p[P_IRHO] + i);
    jx = ldgv(pl.p[P_JX] + i);
    jy = ldgv(pl.p[P_JY] + i);
    const R pc = c[1][1];
    const R a = c[2][2] - c[0][0], b = c[0][2] - c[2][0];
    const R sx = (c[1][2] - c[1][0]) * 4 + (a + b);
    const R sy = (c[2][1] - c[0][1]) * 4 + (a - b);
    const R Gp = pc * C.flow.G12;
    Fx = Gp * sx;
    Fy = Gp * sy;
    if (!P.yper && y == 0 && P.ybc_lo == BC_WALL) Fy += C.G_wall * 0.5f * pc * pc;
    if (P.buoyancy) {
      const R dr = rho - (P.buoyancy == 1 ? R(load_after_wait(rho_ave)) : C.rho_bc_hi);
      Fx += dr * C.gx;
      Fy += dr * C.gy;
    }
    vx = (jx + Fx * 0.5f) * inv_rho;
    vy = (jy + Fy * 0.5f) * inv_rho;
    s_vx[hy][hx] = vx;
    s_vy[hy][hx] = vy;
    if (!heat) Q = C.flow.qG144 * (sx * sx + sy * sy);
  }
  __syncthreads();
  if (!active) return;
  const int x = x0 + tx, y = y0 + ty;
  if (!kFlowFirst && !heat) pre_flow();
  const Around n = around(P, x, y, interior);
  const size_t i = n.row[1] + n.col[1];
  if (!heat) {
    R f[9];
    S* pf = fdst.p + i;
    relax_flow(m, jx, jy, rho, vx, vy, Fx, Fy, Q, C, f);
#pragma unroll
    for (int a = 0; a < 9; ++a) pf[(size_t)a * P.N] = f[a];
    wall_force_store(fdst.wall, P, x, y, Fx, Fy);
    return;
  }
  hx = tx + 1;
  hy = ty + 1;
  R c[3][3];
  gather(pl.p[P_T], n, c);
  const R inv_rho = inv_rho_own;
  const R T = c[1][1];
  const R lap6 = (((c[1][2] + c[1][0]) + (c[2][1] + c[0][1])) * 4 + ((c[2][2] + c[2][0]) + (c[0][0] + c[0][2]))) - T * 20;
  const R gTa = c[2][2] - c[0][0], gTb = c[0][2] - c[2][0];
  const R gTx = (c[1][2] - c[1][0]) * 4 + (gTa + gTb), gTy = (c[2][1] - c[0][1]) * 4 + (gTa - gTb);  // 12 grad T
  // 12 div v: the diagonals of d_x vx and d_y vy share their weights
  const R dv1 = (s_vx[hy][hx + 1] - s_vx[hy][hx - 1]) + (s_vy[hy + 1][hx] - s_vy[hy - 1][hx]);
  const R dv2 = ((s_vx[hy + 1][hx + 1] + s_vy[hy + 1][hx + 1]) - (s_vx[hy - 1][hx - 1] + s_vy[hy - 1][hx - 1])) +
                ((s_vx[hy - 1][hx + 1] - s_vy[hy - 1][hx + 1]) - (s_vx[hy + 1][hx - 1] - s_vy[hy + 1][hx - 1]));
  const R div12 = dv1 * 4 + dv2;
  vx = s_vx[hy][hx];
  vy = s_vy[hy][hx];
  const R inv_rcv12 = inv_rho * C.flow.inv_cV12;  // 1 / (12 rho c_V)
  const R compress = (T * div12) * (R(1.0 / 12.0) - dpdT * inv_rcv12);
  R phi, S0, tau_inv = R(0);
  if (P.model == 2) {  // Gong-Cheng: Eq. 13 source, local tau_g (Sec. IV A)
    phi = compress;
    S0 = phi;
    tau_inv = R(1) / ((P.lambda_mode == 0 ? C.lambda * 36 * inv_rcv12 : C.chi * 3) + R(0.5));
  } else {
    // phi: the underlined terms of Eq. 28 with k = (1/s_3 - 1/2) c_s^2
    if (P.lambda_mode == 0) {
      phi = lap6 * (C.flow.lambda2 * inv_rcv12 - C.flow.kdiff6) + compress;
    } else {  // div(lambda grad T)/(rho c_V) = chi (lap T + grad rho . grad T / rho)
      gather(pl.p[P_RHO], n, c);
      const R gra = c[2][2] - c[0][0], grb = c[0][2] - c[2][0];
      const R grx = (c[1][2] - c[1][0]) * 4 + (gra + grb), gry = (c[2][1] - c[0][1]) * 4 + (gra - grb);
      phi = lap6 * C.flow.chi6 + ((C.flow.chi144 * inv_rho) * (grx * gTx + gry * gTy) + compress);
    }
    S0 = phi;
    if (P.model == 0) {  // S0 = phi + 0.5 dt d_t phi, d_t phi ~ [phi(t) - phi(t - dt)]/dt (Eq. 46)
      S0 = phi + (phi - (first ? phi : pp)) * 0.5f;
    }
  }
  phi_prev[i] = phi;
  R g[9];
  S* pg = gdst.p + i;
  if (unit) {
    relax_heat_unit(n4, n6, T, vx, vy, S0, g);
  } else {
    pull<S, R>(gsrc, C.wg, P, x, y, g);
    heat_closure(g, P, x, y);
    collide_heat(g, T, vx, vy, S0, P, tau_inv);
  }
#pragma unroll
  for (int a = 0; a < 9; ++a) pg[(size_t)a * P.N] = g[a];
}

// Fixed-order sums of the block partials, one block per sum: out[k] = sum(partials[k * stride + 0 .. n)) * scale.
// A thread adds every FINISH-th partial, four at a time so that four loads are in flight (the sum is one block's
// latency: with 64 threads and one load at a time it took 8 us of a 300 x 200 step's 30).
constexpr int FINISH = 512;
__global__ void __launch_bounds__(FINISH) k_finish(const double* __restrict__ partials, int n, int stride, double scale,
                                                   double* __restrict__ out, double* out2) {
  __shared__ double red[FINISH / 32];
  const int tid = pdl_wait<FINISH>();
  const double* p = partials + (long long)blockIdx.x * stride;
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  for (int j = tid; j < n; j += 4 * FINISH)
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (j + k * FINISH < n) s[k] += p[j + k * FINISH];
  const double t = block_sum<FINISH>((s[0] + s[1]) + (s[2] + s[3]), red);
  if (tid == 0) {
    out[blockIdx.x] = t * scale;
    if (out2) out2[blockIdx.x] = t * scale;  // the caller's copy, in device or pinned host memory
  }
}

// Equilibrium start: writes post-collision-layout buffers whose pull gives f = M^{-1} m_eq(rho, u),
// g = M^{-1} m_eq(T, u) at every node (the slot that node x pulls for direction a sits at x - e_a).
template <class S>
__global__ void __launch_bounds__(BLOCK) k_init(const double* __restrict__ rho_in, const double* __restrict__ T_in,
                                                const double* __restrict__ ux_in, const double* __restrict__ uy_in,
                                                PopBuf<S> f, PopBuf<S> g, DevParams P) {
  const long long i = (long long)blockIdx.x * BLOCK + pdl_wait<BLOCK>();
  if (i >= P.N) return;
  const auto [x, y] = node_at(P, i);
  if (x >= P.nx) return;
  double fv[9], gv[9];
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    // node whose pull reads slot (x, y) in direction a
    const int tx = wrapx(x + EX(a), P.nx);
    int ty = y + EY(a);
    if (ty < 0 || ty >= P.ny) {
      if (!P.yper) {  // no node pulls this slot; keep it finite
        fv[a] = 0.0;
        gv[a] = 0.0;
        continue;
      }
      ty = ty < 0 ? ty + P.ny : ty - P.ny;
    }
    const long long t = (long long)ty * P.nx + tx;
    const double rho = rho_in[t], T = T_in[t];
    const double vx = ux_in ? ux_in[t] : 0.0, vy = uy_in ? uy_in[t] : 0.0;
    const double v2 = vx * vx + vy * vy;
    double m[9], fe[9], ge[9];
    m[0] = rho; m[1] = rho * (-2.0 + 3.0 * v2); m[2] = rho * (1.0 - 3.0 * v2);
    m[3] = rho * vx; m[4] = -rho * vx; m[5] = rho * vy; m[6] = -rho * vy;
    m[7] = rho * (vx * vx - vy * vy); m[8] = rho * vx * vy;
    from_moments(m, fe);
    heat_meq(T, vx, vy, P.model, m);
    from_moments(m, ge);
    fv[a] = fe[a];
    gv[a] = ge[a];
  }
  // FP16 storage: deviations from the rest equilibrium of this slot's own node
  pop_store<S, double>(f, P.N, i, fv, rho_in[(long long)y * P.nx + x], P.cd.wf);
  pop_store<S, double>(g, P.N, i, gv, T_in[(long long)y * P.nx + x], P.cd.wg);
}

// Totals of two values over a block in block_sum's order, with half its additions: lanes 0 to 15 go on with the pairs'
// sums of a, lanes 16 to 31 with those of b. Valid in thread 0 (a) and thread 16 (b).
template <int NTH> __device__ __forceinline__ double block_sum_pair(int tid, double a, double b, double* smem) {
  const int lane = tid & 31, w = tid >> 5;
  const bool lo = lane < 16;
  const double other = __shfl_xor_sync(0xffffffffu, lo ? b : a, 16);
  double v = (lo ? a : b) + other;
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((lane & 15) == 0) smem[(lane >> 4) * (NTH / 32) + w] = v;
  __syncthreads();
  double s = 0.0;
  if (w == 0) {
    if ((lane & 15) < NTH / 32) s = smem[(lane >> 4) * (NTH / 32) + (lane & 15)];
#pragma unroll
    for (int o = NTH / 64; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  }
  __syncthreads();
  return s;
}

// Sums of rho and T over the current (post-boundary) state into per-block partials. Bound by the FP64 pipe
// (16 additions per node, and without BITS a conversion per population of a narrower storage), so a thread takes K nodes
// before the block's reduction, whose 7 instructions per warp K = 1 pays for every 32 nodes.
template <class S, int K, bool BITS>
__global__ void __launch_bounds__(BLOCK) k_sums(PopBuf<S> fsrc, PopBuf<S> gsrc, DevParams P,
                                                double* __restrict__ partials, int stride) {
  __shared__ double red[2 * (BLOCK / 32)];
  const int tid = pdl_wait<BLOCK>();
  double r = 0.0, t = 0.0;
#pragma unroll 2
  for (int k = 0; k < K; ++k) {
    const long long i = ((long long)blockIdx.x * K + k) * BLOCK + tid;
    if (i >= P.N) break;
    const auto [x, y] = node_at(P, i);
    if (x >= P.nx) continue;
    double f[9], g[9];
    pull_closed<S, double, long long, DevParams, BITS>(fsrc, gsrc, P, x, y, f, g);
    r += f[0] + f[1] + f[2] + f[3] + f[4] + f[5] + f[6] + f[7] + f[8];
    t += g[0] + g[1] + g[2] + g[3] + g[4] + g[5] + g[6] + g[7] + g[8];
  }
  const double s = block_sum_pair<BLOCK>(tid, r, t, red);
  if (tid == 0 || tid == 16) partials[(tid >> 4) * stride + blockIdx.x] = s;
}

// Post-boundary populations of the current state as FP64 [9][ny][nx] (which = 0: f, 1: g).
template <class S>
__global__ void __launch_bounds__(BLOCK) k_export_pops(PopBuf<S> fsrc, PopBuf<S> gsrc, DevParams P, int which,
                                                       int only, double* __restrict__ out) {
  const long long i = (long long)blockIdx.x * BLOCK + pdl_wait<BLOCK>();
  if (i >= P.N) return;
  const auto [x, y] = node_at(P, i);
  if (x >= P.nx) return;
  double f[9], g[9];
  pull_closed<S, double>(fsrc, gsrc, P, x, y, f, g);
  const long long o = (long long)y * P.nx + x;  // outputs have no padding
  if (only >= 0) {  // one population plane into out[ny][nx]
    out[o] = which ? g[only] : f[only];
    return;
  }
#pragma unroll
  for (int a = 0; a < 9; ++a) out[(long long)a * P.nx * P.ny + o] = which ? g[a] : f[a];
}

// Copy planes rho, vx, vy, T to FP64 outputs (any may be null).
template <class R>
__global__ void __launch_bounds__(BLOCK) k_export_fields(Planes<R> pl, DevParams P, double* rho, double* ux, double* uy,
                                                         double* T) {
  const long long i = (long long)blockIdx.x * BLOCK + pdl_wait<BLOCK>();
  if (i >= P.N) return;
  const auto [x, y] = node_at(P, i);
  if (x >= P.nx) return;
  const long long o = (long long)y * P.nx + x;  // outputs have no padding
  if (rho) rho[o] = (double)pl.p[P_RHO][i];
  if (ux) ux[o] = (double)pl.p[P_VX][i];
  if (uy) uy[o] = (double)pl.p[P_VY][i];
  if (T) T[o] = (double)pl.p[P_T][i];
}

// Rows of nx elements from one row stride to another, a warp per row: what packs the rows of a checkpoint and unpacks
// them. Bound by HBM, or by the link where one side is pinned host memory.
template <class E>
__device__ __forceinline__ void repack_row(E* __restrict__ d, const E* __restrict__ s, int lane, int nx) {
  int x = lane;
  for (; x + 7 * 32 < nx; x += 8 * 32) {  // eight loads in flight
    E v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = s[x + 32 * k];
#pragma unroll
    for (int k = 0; k < 8; ++k) d[x + 32 * k] = v[k];
  }
  for (; x < nx; x += 32) d[x] = s[x];
}
__global__ void __launch_bounds__(256) k_repack(const __grid_constant__ RowSets S) {
  const int t = pdl_wait<256>();
  long long r = (long long)blockIdx.x * 8 + (t >> 5);
#pragma unroll 1
  for (int k = 0; k < S.n; ++k) {
    const RowSet& q = S.set[k];
    for (; r < q.rows; r += (long long)gridDim.x * 8) {
      if (q.elem == 2)
        repack_row((unsigned short*)q.dst + r * q.dst_stride, (const unsigned short*)q.src + r * q.src_stride, t & 31, S.nx);
      else
        repack_row((unsigned*)q.dst + r * q.dst_stride, (const unsigned*)q.src + r * q.src_stride, t & 31, S.nx);
    }
    r -= q.rows;
  }
}

// ------------------------------------------------------------------------------------------------
// host launchers
// ------------------------------------------------------------------------------------------------
static inline unsigned blocks_for(long long N) { return (unsigned)((N + BLOCK - 1) / BLOCK); }

template <class S, class R> static Planes<R> planes_of(const SplitBuffers& b) {
  Planes<R> pl;
  for (int k = 0; k < NPLANES; ++k) pl.p[k] = (R*)b.planes[k];
  return pl;
}

template <class S> static PopBuf<S> fbuf(const SplitBuffers& b, int k) {
  return PopBuf<S>{(S*)b.f[k], b.ref_f[k], b.wall[k]};
}
template <class S> static PopBuf<S> gbuf(const SplitBuffers& b, int k) { return PopBuf<S>{(S*)b.g[k], b.ref_g[k]}; }

// The binary32 step as three kernels over scratch planes.
template <class S, class R>
static cudaError_t step_impl(const SplitBuffers& b, const DevParams& P, int cur, long long step, cudaStream_t st,
                             cudaEvent_t* ev) {
  const unsigned nb = blocks_for(P.N);
  Planes<R> pl = planes_of<S, R>(b);
  if (ev) cudaEventRecord(ev[0], st);
  launch_pdl(k_macro<S, R, false>, nb, BLOCK, 0, st, fbuf<S>(b, cur), gbuf<S>(b, cur), nullptr, nullptr, pl, P, step,
                                             P.buoyancy == 1, b.partials, b.status);
  if (ev) cudaEventRecord(ev[1], st);
  launch_pdl(k_force<R>, nb, BLOCK, 0, st, pl, P, b.scalars);
  if (ev) cudaEventRecord(ev[2], st);
  launch_pdl(k_collide<S, R>, nb, 2 * BLOCK, 0, st, fbuf<S>(b, cur), gbuf<S>(b, cur), fbuf<S>(b, cur ^ 1), gbuf<S>(b, cur ^ 1),
                                            pl, (R*)b.phi_prev, P, step == 0);
  if (ev) cudaEventRecord(ev[3], st);
  if (P.buoyancy == 1) {
    launch_pdl(k_finish, 1, FINISH, 0, st, b.partials, (int)nb, 0, 1.0 / node_count(P), b.scalars, nullptr);
    if (ev) cudaEventRecord(ev[4], st);
  }
  return cudaGetLastError();
}

// The binary64 and double-word steps as two kernels.
template <class S>
static cudaError_t step_wide(const SplitBuffers& b, const DevParams& P, int cur, long long step, cudaStream_t st,
                             cudaEvent_t* ev) {
  const unsigned nb = blocks_for(P.N);
  Planes<S> pl = planes_of<S, S>(b);
  const PopBuf<S> fd = fbuf<S>(b, cur ^ 1), gd = gbuf<S>(b, cur ^ 1);
  if (ev) cudaEventRecord(ev[0], st);
  launch_pdl(k_macro<S, S, true>, nb, BLOCK, 0, st, fbuf<S>(b, cur), gbuf<S>(b, cur), fd.p, gd.p, pl, P, step, P.buoyancy == 1,
                                            b.partials, b.status);
  if (ev) cudaEventRecord(ev[1], st);
  auto collide = [&](auto cx, auto cy) {
    constexpr int CX = decltype(cx)::value, CY = decltype(cy)::value;
    const int tiles_x = (P.nx + CX - 1) / CX;
    const unsigned tiles = (unsigned)((long long)tiles_x * ((P.ny + CY - 1) / CY));
    launch_pdl(k_collide_tile<S, CX, CY>, tiles, 2 * CX * CY, 0, st, gbuf<S>(b, cur), fd, gd, pl, (S*)b.phi_prev, P, step == 0,
                                                            tiles_x, b.scalars);
  };
  // 16 x 8 tiles; large binary64 grids take 32 x 8, whose ring repeats less of the force (1.33 instead of 1.41 times
  // the tile): 2048^2 1811 us a step against 1831. Below, more blocks matter more: 128^2 12.0 against 17.1 us,
  // 350^2 64 against 69 us. In double-word arithmetic 16 x 8 is the faster at every size (2048^2 467, 471 us).
  if (sizeof(S) == 8 && !is_dw_t<S>::value && P.N >= (1 << 20))
    collide(std::integral_constant<int, 32>(), std::integral_constant<int, 8>());
  else
    collide(std::integral_constant<int, 16>(), std::integral_constant<int, 8>());
  if (ev) cudaEventRecord(ev[2], st);
  if (P.buoyancy == 1) {
    launch_pdl(k_finish, 1, FINISH, 0, st, b.partials, (int)nb, 0, 1.0 / node_count(P), b.scalars, nullptr);
    if (ev) cudaEventRecord(ev[3], st);
  }
  return cudaGetLastError();
}

cudaError_t split_step(const SplitBuffers& b, const DevParams& P, int prec, int cur, long long step, cudaStream_t st,
                       cudaEvent_t* ev) {
  if (prec == 0) return step_wide<double>(b, P, cur, step, st, ev);
  if (prec == 1) return step_impl<float, float>(b, P, cur, step, st, ev);
  if (prec == 3) return step_wide<dw>(b, P, cur, step, st, ev);
  return step_impl<__half, float>(b, P, cur, step, st, ev);
}

static bool is_wide(int prec) { return prec == 0 || prec == 3; }  // 8-byte storage: two kernels

int split_kernel_count(const DevParams& P, int prec) { return (is_wide(prec) ? 2 : 3) + (P.buoyancy == 1); }

const char* split_kernel_name(int prec, int k) {
  static const char* names[] = {"k_macro", "k_force", "k_collide", "k_finish"};
  static const char* wide[] = {"k_macro", "k_collide_tile", "k_finish"};
  if (k < 0 || k >= (is_wide(prec) ? 3 : 4)) return "";
  return is_wide(prec) ? wide[k] : names[k];
}

// Enqueue k_sums; returns its number of blocks. Four nodes per thread on large grids (2048^2 with k_finish: binary64
// 264 us, 303 with one node), one where latency counts (256^2: 13.1 us, 15.4 with four; 11.7 with the paired reduction).
// Narrower storage is widened from its bits where the FP64 pipe sets the time. Converted and widened, us with k_finish:
// binary32 256^2 13.8, 15.2; 512^2 31.5, 27.3; 1000^2 91.9, 78.5; double-word 128^2 8.9, 12.8; 256^2 18.6, 15.7;
// 2048^2 652, 434; binary16 256^2 17.9, 15.9; 512^2 50.0, 32.0; 2048^2 657, 400.
template <class S> static int launch_sums(const SplitBuffers& b, const DevParams& P, int k, cudaStream_t st) {
  const int stride = (int)blocks_for(P.N);
  constexpr bool narrow = !std::is_same<S, double>::value;
  const int nb = P.N < (1 << 20) ? stride : (stride + 3) / 4;
  auto* kernel = k_sums<S, 1, false>;
  if (P.N >= (1 << 20))
    kernel = k_sums<S, 4, narrow>;
  else if (narrow && P.N >= (sizeof(S) == 4 ? 1 << 18 : 1 << 16))
    kernel = k_sums<S, 1, narrow>;
  launch_pdl(kernel, nb, BLOCK, 0, st, fbuf<S>(b, k), gbuf<S>(b, k), P, b.partials, stride);
  return nb;
}

template <class S>
static cudaError_t init_impl(const SplitBuffers& b, const DevParams& P, const double* rho, const double* T,
                             const double* ux, const double* uy, cudaStream_t st) {
  const unsigned nb = blocks_for(P.N);
  for (int k = 0; k < 2; ++k)  // no force before the first step: the initial closure takes j = 0 on walls
    if (b.wall[k]) {
      const cudaError_t e = cudaMemsetAsync(b.wall[k], 0, wall_doubles(P.nx) * sizeof(double), st);
      if (e != cudaSuccess) return e;
    }
  launch_pdl(k_init<S>, nb, BLOCK, 0, st, rho, T, ux, uy, fbuf<S>(b, 0), gbuf<S>(b, 0), P);
  // rho_ave of the initial (post-boundary) state
  const int ns = launch_sums<S>(b, P, 0, st);
  launch_pdl(k_finish, 1, FINISH, 0, st, b.partials, ns, 0, 1.0 / node_count(P), b.scalars, nullptr);
  return cudaGetLastError();
}

cudaError_t split_init(const SplitBuffers& b, const DevParams& P, int prec, const double* rho, const double* T,
                       const double* ux, const double* uy, cudaStream_t st) {
  if (prec == 0) return init_impl<double>(b, P, rho, T, ux, uy, st);
  if (prec == 1) return init_impl<float>(b, P, rho, T, ux, uy, st);
  if (prec == 3) return init_impl<dw>(b, P, rho, T, ux, uy, st);
  return init_impl<__half>(b, P, rho, T, ux, uy, st);
}

template <class S>
static cudaError_t sums_impl(const SplitBuffers& b, const DevParams& P, int cur, double* out, cudaStream_t st) {
  const int nb = launch_sums<S>(b, P, cur, st);
  launch_pdl(k_finish, 2, FINISH, 0, st, b.partials, nb, (int)blocks_for(P.N), 1.0, b.scalars + 1, out);
  return cudaGetLastError();
}

cudaError_t split_sums(const SplitBuffers& b, const DevParams& P, int prec, int cur, cudaStream_t st, double* out) {
  if (prec == 0) return sums_impl<double>(b, P, cur, out, st);
  if (prec == 1) return sums_impl<float>(b, P, cur, out, st);
  if (prec == 3) return sums_impl<dw>(b, P, cur, out, st);
  return sums_impl<__half>(b, P, cur, out, st);
}

template <class S, class R>
static cudaError_t fields_impl(const SplitBuffers& b, const DevParams& P, int cur, long long step, double* rho,
                               double* ux, double* uy, double* T, cudaStream_t st) {
  const unsigned nb = blocks_for(P.N);
  Planes<R> pl = planes_of<S, R>(b);
  launch_pdl(k_macro<S, R, false>, nb, BLOCK, 0, st, fbuf<S>(b, cur), gbuf<S>(b, cur), nullptr, nullptr, pl, P, step, 0,
                                             b.partials, b.status);
  launch_pdl(k_force<R>, nb, BLOCK, 0, st, pl, P, b.scalars);
  launch_pdl(k_export_fields<R>, nb, BLOCK, 0, st, pl, P, rho, ux, uy, T);
  return cudaGetLastError();
}

cudaError_t split_fields(const SplitBuffers& b, const DevParams& P, int prec, int cur, long long step, double* rho,
                         double* ux, double* uy, double* T, cudaStream_t st) {
  if (prec == 0) return fields_impl<double, double>(b, P, cur, step, rho, ux, uy, T, st);
  if (prec == 1) return fields_impl<float, float>(b, P, cur, step, rho, ux, uy, T, st);
  if (prec == 3) return fields_impl<dw, dw>(b, P, cur, step, rho, ux, uy, T, st);
  return fields_impl<__half, float>(b, P, cur, step, rho, ux, uy, T, st);
}

cudaError_t split_export_pops(const SplitBuffers& b, const DevParams& P, int prec, int cur, int which, int only,
                              double* out, cudaStream_t st) {
  const unsigned nb = blocks_for(P.N);
  if (prec == 0)
    launch_pdl(k_export_pops<double>, nb, BLOCK, 0, st, fbuf<double>(b, cur), gbuf<double>(b, cur), P, which, only, out);
  else if (prec == 1)
    launch_pdl(k_export_pops<float>, nb, BLOCK, 0, st, fbuf<float>(b, cur), gbuf<float>(b, cur), P, which, only, out);
  else if (prec == 3)
    launch_pdl(k_export_pops<dw>, nb, BLOCK, 0, st, fbuf<dw>(b, cur), gbuf<dw>(b, cur), P, which, only, out);
  else
    launch_pdl(k_export_pops<__half>, nb, BLOCK, 0, st, fbuf<__half>(b, cur), gbuf<__half>(b, cur), P, which, only, out);
  return cudaGetLastError();
}

cudaError_t repack_rows(const RowSets& s, cudaStream_t st) {
  long long rows = 0;
  for (int k = 0; k < s.n; ++k) rows += s.set[k].rows;
  if (rows == 0) return cudaSuccess;
  return launch_pdl(k_repack, (unsigned)std::min<long long>((rows + 7) / 8, 1 << 20), 256, 0, st, s);
}

void fused_finish(const SplitBuffers& b, const DevParams& P, int n, cudaStream_t st) {
  launch_pdl(k_finish, 1, FINISH, 0, st, b.partials, n, 0, 1.0 / node_count(P), b.scalars, nullptr);
}

int split_nplanes() { return NPLANES; }
int split_block() { return BLOCK; }

}  // namespace lbpc
