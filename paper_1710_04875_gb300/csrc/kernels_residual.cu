// Boundary ghosts, per-cell auxiliaries, the JST / thin-layer residual (section 2 of
// arXiv 1710.04875) and the Baldwin-Lomax closure, FP64.
#include "fasw_internal.cuh"
#include "fasw_roots.cuh"
#include "fasw_sweep.cuh"

namespace fasw {

namespace {

// Residual tile: TX x TY cells.  Warps 0..TY-1 compute the TX+1 = 32 i-faces of one tile row
// each, warps TY..2TY compute the TX j-faces of one row of j-faces each (lane 31 idle), so no
// warp mixes the two kinds of face and a j-face (with the viscous terms) is a thread of its
// own: on GB300 an SM sub-partition issues one FP64 warp-instruction every 64 clocks,
// so the FP64 work of a launch is spread over as many warps and SMs as the grid allows.  The cells'
// phase takes two components of a cell per thread, on tile height 1 (with a fourth warp) one.
//
// Tile height 4 where that still gives a block per SM of the GB300, else 1: a coarse level then spreads over four
// times as many SMs for 1.6 times the j-face work (its j-faces are computed by both neighbouring tiles).
// FP64, a finest level (with sensors), height 1 / 2 / 4 / 8: 64x16 7.9 / 10.2 / 14.7 / 23.4 us, 128x32 12.3 / 14.3 /
// 14.7 / 23.7, 256x64 (144 tiles of height 4) 20.0 / 25.4 / 24.0 / 23.5, 330x90 (253) 29.3 / 25.6 / 24.1 / 23.7,
// 512x128 54.7 / 49.2 / 46.5 / 47.8, 1024x256 201 / 170 / 168 / 190.  As coarse levels 64x16 takes 5.4 us, 128x32
// 8.8, 256x64 14.3 (8.5 and 10.1 on the first two before the cells' phase was split and its operands fetched ahead
// of the wait for the kernel before).  A case of a batch shares the chip, so the extra work of height 1 counts
// there: height 4 from half as many tiles, also with few cases (FP64 cycle, this rule / height 1 / height 4
// everywhere: 2 cases of 256x64 982 / 1,054 / 1,027 us, 4 of them 1,268 / 1,300 / 1,310, 16 2,598 / 2,703 / 2,606;
// at its worst 2 cases of 192x48 692 / 678 / 716).
constexpr int TX = 31;
constexpr int SMS = 152;
constexpr int res_threads(int ty) { return ty == 1 ? 128 : 32 * (2 * ty + 1); }
// Tile height: the level's setting (1, 2, 4 or 8, chosen by the batch autotuner or the caller), else
// by the rule above.
inline int res_ty(const LevelDev& L) {
  if (L.res_ty > 0) return L.res_ty;
  return ((L.ni + TX - 1) / TX) * ((L.nj + 3) / 4) >= (L.shared ? SMS / 2 : SMS) ? 4 : 1;
}

__device__ __forceinline__ int gidx(const LevelDev& L, int i, int j) { return (j + 2) * L.P + (i + 2); }
__device__ __forceinline__ bool on_cut(const LevelDev& L, int i) { return L.nw > 0 && (i < L.nw || i >= L.ni - L.nw); }

__device__ __forceinline__ void load4(const LevelDev& L, int g, double w[4]) {
#pragma unroll
  for (int k = 0; k < 4; ++k) w[k] = L.u[k * L.Gn + g];
}
__device__ __forceinline__ void store4(const LevelDev& L, int g, const double w[4]) {
#pragma unroll
  for (int k = 0; k < 4; ++k) L.u[k * L.Gn + g] = w[k];
}

__device__ __forceinline__ double pressure(const double w[4]) {
  return (GAM - 1.0) * (w[3] - 0.5 * (w[1] * w[1] + w[2] * w[2]) / w[0]);
}

// Far-field boundary state by 1-D Riemann invariants along the outward unit normal (nx, ny).
// vb: normal velocity of the (moving) boundary; in/outflow is decided on the relative velocity.
// The density follows from the entropy of the upwind side: with s = p/rho^gamma fixed,
// rho_b = (a_b^2 / (gamma s))^(1/(gamma-1)) = rho_up (a_b / a_up)^(2/(gamma-1)), and for
// gamma = 1.4 the exponent is the integer 5 (FP64 pow costs about a hundred FP64 instructions
// on a part whose FP64 issue rate is the bound of this kernel).
static_assert(GAM == 1.4, "far-field density uses 2/(gamma-1) = 5");
// The free stream's primitives (u, v, p, a) come from the host (PhysParams::finf).
__device__ void farfield(const double wi[4], const PhysParams& ph, double nx, double ny, double vb, double out[4]) {
  const double* wf = ph.uinf;
  const double ri = wi[0], rri = ph.fast ? rcp64(ri) : 1.0 / ri, ui = wi[1] * rri, vi = wi[2] * rri;
  const double pi = (GAM - 1.0) * (wi[3] - 0.5 * (wi[1] * ui + wi[2] * vi));
  const double rf = wf[0], uf = ph.finf[0], vf = ph.finf[1], af = ph.finf[3];
  const double ai = sqrt(GAM * pi * rri);
  const double vni = ui * nx + vi * ny, vnf = uf * nx + vf * ny;
  if (fabs(vni - vb) >= ai) {
    const double* src = vni - vb > 0.0 ? wi : wf;
#pragma unroll
    for (int k = 0; k < 4; ++k) out[k] = src[k];
    return;
  }
  constexpr double k2 = 2.0 / (GAM - 1.0);
  const double Rp = vni + k2 * ai;
  const double Rm = vnf - k2 * af;
  const double vnb = 0.5 * (Rp + Rm);
  const double ab = 0.25 * (GAM - 1.0) * (Rp - Rm);
  double rup, aup, ut, vt;
  if (vnb - vb > 0.0) {
    rup = ri;
    aup = ai;
    ut = ui - vni * nx;
    vt = vi - vni * ny;
  } else {
    rup = rf;
    aup = af;
    ut = uf - vnf * nx;
    vt = vf - vnf * ny;
  }
  const double ra = ph.fast ? div64(ab, aup, rcp64(aup)) : ab / aup, ra2 = ra * ra;
  const double rho = rup * (ra2 * ra2 * ra);
  const double p = rho * ab * ab * (1.0 / GAM);
  const double u = ut + vnb * nx, v = vt + vnb * ny;
  out[0] = rho;
  out[1] = rho * u;
  out[2] = rho * v;
  out[3] = p * (1.0 / (GAM - 1.0)) + 0.5 * rho * (u * u + v * v);
}

// State of an interior cell, the pending stage update made.
__device__ __forceinline__ void cell_u(const LevelDev& L, const WsPending& up, int i, int j, double w[4]) {
  if (up.z0)
    ws_updated(L, up, i, j, w);
  else
    load4(L, gidx(L, i, j), w);
}

// Where the boundary value of ghost cell (gi, gj) comes from (two layers on every side; corners
// excluded): j < 0: wake-cut copy of the mirror cell or wall reflection (slip / no-slip, moving wall);
// j >= nj, i < 0, i >= ni: Riemann far-field state (section 2, G9).  (i, j): the interior cell that it
// is formed from; (nx, ny): the unit normal; (vx, vy): the wall's velocity, vx: the far boundary's normal
// velocity.
enum GhostKind { GHOST_COPY, GHOST_WALL, GHOST_FAR };
struct GhostFrom {
  int kind, i, j;
  double nx, ny, vx, vy;
};

__device__ __forceinline__ GhostFrom ghost_from(const LevelDev& L, const PhysParams& ph, int gi, int gj) {
  const int ni = L.ni, nj = L.nj;
  GhostFrom f{};
  if (gj < 0) {
    f.j = -1 - gj;  // source row 0 or 1
    f.i = gi;
    f.kind = GHOST_WALL;
    if (on_cut(L, gi)) {
      f.i = ni - 1 - gi;
      f.kind = GHOST_COPY;
    } else if (!ph.viscous) {
      const double sx = L.seta[gi], sy = L.seta[L.nfe + gi];
      const double len = sqrt(sx * sx + sy * sy);
      f.nx = sx / len;
      f.ny = sy / len;
    }
    if (ph.moving) {
      f.vx = L.wvx[gi];
      f.vy = L.wvy[gi];
    }
    return f;
  }
  // One evaluation for the three outer sides, so that a warp with ghosts of several sides runs it once.
  // Outward is +S_eta at j = nj and +S_xi at i = ni, -S_xi at i = 0.
  const bool top = gj >= nj, left = !top && gi < 0;
  const int e = top ? nj * ni + gi : gj * (ni + 1) + (left ? 0 : ni);
  double sx, sy, vb;
  if (top) {
    sx = L.seta[e];
    sy = L.seta[L.nfe + e];
    vb = L.vfe[e];
  } else {
    sx = L.sxi[e];
    sy = L.sxi[L.nfx + e];
    vb = L.vfx[e];
  }
  if (left) {
    sx = -sx;
    sy = -sy;
    vb = -vb;
  }
  const double il = 1.0 / sqrt(sx * sx + sy * sy);
  f.kind = GHOST_FAR;
  f.i = top ? gi : left ? 0 : ni - 1;
  f.j = top ? nj - 1 : gj;
  f.nx = sx * il;
  f.ny = sy * il;
  f.vx = vb * il;
  return f;
}

__device__ void ghost_value(const LevelDev& L, const PhysParams& ph, const WsPending& up, const GhostFrom& f,
                            double g[4]) {
  double w[4];
  cell_u(L, up, f.i, f.j, w);
  if (f.kind == GHOST_FAR) {
    farfield(w, ph, f.nx, f.ny, f.vx, g);
  } else if (f.kind == GHOST_COPY) {
#pragma unroll
    for (int k = 0; k < 4; ++k) g[k] = w[k];
  } else if (!ph.moving) {
    g[0] = w[0];
    g[3] = w[3];
    if (ph.viscous) {
      g[1] = -w[1];
      g[2] = -w[2];
    } else {
      const double mn = w[1] * f.nx + w[2] * f.ny;
      g[1] = w[1] - 2.0 * mn * f.nx;
      g[2] = w[2] - 2.0 * mn * f.ny;
    }
  } else {  // moving wall: velocity mirrored about the wall velocity, same rho and p
    const double rho = w[0], u = w[1] / rho, v = w[2] / rho, p = pressure(w);
    double ug, vg;
    if (ph.viscous) {
      ug = 2.0 * f.vx - u;
      vg = 2.0 * f.vy - v;
    } else {
      const double rn = (u - f.vx) * f.nx + (v - f.vy) * f.ny;
      ug = u - 2.0 * rn * f.nx;
      vg = v - 2.0 * rn * f.ny;
    }
    g[0] = rho;
    g[1] = rho * ug;
    g[2] = rho * vg;
    g[3] = p / (GAM - 1.0) + 0.5 * rho * (ug * ug + vg * vg);
  }
}

// Ghost cell t of the two layers around the domain (corners excluded): rows j = -1, -2, rows
// j = nj, nj+1, columns i = -1, -2, columns i = ni, ni+1; false past the last one.
__device__ __forceinline__ bool ghost_of(const LevelDev& L, int t, int& gi, int& gj) {
  const int ni = L.ni, nj = L.nj;
  if (t < 2 * ni) {
    gi = t % ni;
    gj = -1 - t / ni;
  } else if (t < 4 * ni) {
    gi = (t - 2 * ni) % ni;
    gj = nj + (t - 2 * ni) / ni;
  } else if (t < 4 * ni + 2 * nj) {
    gj = (t - 4 * ni) % nj;
    gi = -1 - (t - 4 * ni) / nj;
  } else if (t < 4 * ni + 4 * nj) {
    gj = (t - 4 * ni - 2 * nj) % nj;
    gi = ni + (t - 4 * ni - 2 * nj) / nj;
  } else {
    return false;
  }
  return true;
}

// Ghost fill alone: one thread per ghost cell of the two layers.
__global__ void k_bc(LevelDev L, PhysParams ph) {
  pdl_entry();
  int gi, gj;
  if (!ghost_of(L, blockIdx.x * blockDim.x + threadIdx.x, gi, gj)) return;
  double g[4];
  ghost_value(L, ph, WsPending{}, ghost_from(L, ph, gi, gj), g);
  store4(L, gidx(L, gi, gj), g);
}

// FP64 on this part issues one warp instruction per 64 clocks per scheduler (fasw_fp64.cuh), and the
// library pow() costs about 3.3 us of dependent chain per call (cbrt 0.54 us, a division 0.29 us, an
// FMA 32 ns): the per-cell auxiliaries are bound by that chain, not by memory.  The two powers
// they need are computed as roots of polynomial equations by Newton's method in FP64 from an
// FP32 estimate; both are checked against pow() and cbrt() by fasw_check_math.

// Pressure, 1/rho and (finest level only: the coarse levels' dissipation has no sensor) the
// sensor quantity of one (ghosted) cell.
__device__ __forceinline__ void cell_thermo(const LevelDev& L, const PhysParams& ph, int g, const double w[4],
                                            double& rr, double& u, double& v, double& p) {
  rr = ph.fast ? rcp64(w[0]) : 1.0 / w[0];
  u = w[1] * rr;
  v = w[2] * rr;
  p = (GAM - 1.0) * (w[3] - 0.5 * (w[1] * u + w[2] * v));
  L.p[g] = p;
  L.rinv[g] = rr;
  if (L.finest) L.q[g] = ph.sensor ? p * pow_neg_gamma(w[0]) : p;
}

// Auxiliaries: blocks [0, nbi) take the interior cells (pressure, 1/rho, sensor quantity,
// Martinelli radii, dt*), the blocks after them the ghost cells (with fill_ghosts their
// boundary value first, which depends on interior cells only; then pressure, 1/rho, sensor).
// Interior and ghost work never share a warp, so neither path waits on the other's FP64 chain.
// up: the stage update the sweep left (made here first: one launch and one pass over the state less;
// a ghost thread makes it again for the cell it reflects).
// early: the geometry is read, and what depends on it alone formed, before the wait for the kernel before
// (which must not be one that writes the metrics; a kernel lets its successor start only once its own
// predecessors have completed): a quarter of an interior cell's FP64 chain and a third of a ghost's.  With a
// stage update 32x8 5.4 -> 4.2 us, 64x16 5.3 -> 4.0, 128x32 5.8 -> 4.0, 256x64 6.0 -> 5.2.
__global__ void k_cell_aux(LevelDev L, PhysParams ph, double cfl, int want_dts, int fill_ghosts, int nbi,
                           WsPending up, int early) {
  if (!early) pdl_entry();
  if ((int)blockIdx.x >= nbi) {
    int gi, gj;
    const bool has = ghost_of(L, (blockIdx.x - nbi) * blockDim.x + threadIdx.x, gi, gj);
    GhostFrom from{};
    if (has && fill_ghosts) from = ghost_from(L, ph, gi, gj);
    if (early) pdl_entry();
    if (!has) return;
    const int g = gidx(L, gi, gj);
    double w[4];
    if (fill_ghosts) {
      ghost_value(L, ph, up, from, w);
      store4(L, g, w);
    } else {
      load4(L, g, w);
    }
    double rr, u, v, p;
    cell_thermo(L, ph, g, w, rr, u, v, p);
    return;
  }
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  const int ni = L.ni, i = c % ni, j = c / ni;
  double sx = 0.0, sy = 0.0, ex = 0.0, ey = 0.0, vx = 0.0, ve = 0.0, lx = 0.0, le = 0.0, cv = 0.0;
  if (c < L.n) {
    const int fw = j * (ni + 1) + i, fs = j * ni + i;
    sx = 0.5 * (L.sxi[fw] + L.sxi[fw + 1]);
    sy = 0.5 * (L.sxi[L.nfx + fw] + L.sxi[L.nfx + fw + 1]);
    ex = 0.5 * (L.seta[fs] + L.seta[fs + ni]);
    ey = 0.5 * (L.seta[L.nfe + fs] + L.seta[L.nfe + fs + ni]);
    if (ph.moving) {
      vx = 0.5 * (L.vfx[fw] + L.vfx[fw + 1]);
      ve = 0.5 * (L.vfe[fs] + L.vfe[fs + ni]);
    }
    lx = L.clen[c];
    le = L.clen[L.n + c];
    if (want_dts) cv = cfl * L.vol[c];
  }
  if (early) pdl_entry();
  if (c >= L.n) return;
  const int g = gidx(L, i, j);
  double w[4];
  cell_u(L, up, i, j, w);
  if (up.z0) store4(L, g, w);
  double rr, u, v, p;
  cell_thermo(L, ph, g, w, rr, u, v, p);
  const double a = sqrt(GAM * p * rr);
  double qx = u * sx + v * sy, qe = u * ex + v * ey;
  if (ph.moving) {
    qx -= vx;
    qe -= ve;
  }
  const double rxi = fabs(qx) + a * lx, reta = fabs(qe) + a * le;
  // Martinelli scaling: with cr = (r_eta/r_xi)^(1/3), r_xi (r_eta/r_xi)^(2/3) = r_xi cr^2 and
  // r_eta (r_xi/r_eta)^(2/3) = r_xi cr (one cube root, no division).
  const double cr = cbrt_ratio(reta, rxi);
  L.rt[c] = rxi + rxi * (cr * cr);
  L.rt[L.n + c] = reta + rxi * cr;
  if (want_dts) {
    const double r = rxi + reta;
    L.dts[c] = ph.fast ? div64(cv, r, rcp64(r)) : cv / r;
  }
}

// Martinelli radius of a possibly-ghost cell: ghosts take the adjacent interior cell's value,
// across the wake cut the mirror cell's.
__device__ __forceinline__ double rt_cell(const LevelDev& L, int i, int j, int dir) {
  if (j < 0) {
    int ic = min(max(i, 0), L.ni - 1);
    i = on_cut(L, ic) ? L.ni - 1 - ic : ic;
    j = 0;
  }
  i = min(max(i, 0), L.ni - 1);
  j = min(j, L.nj - 1);
  return L.rt[dir * L.n + j * L.ni + i];
}

template <bool FAST>
__device__ __forceinline__ double sensor_val(double qm, double q0, double qp) {
  const double d = fabs(qp - 2.0 * q0 + qm), s = qp + 2.0 * q0 + qm + 0.001;
  return FAST ? div64(d, s, rcp64(s)) : d / s;
}

// First-order flux-vector-split face flux (the discretization section 4.4 linearizes for the
// preconditioner): h = A+(u_bar) u_L + A-(u_bar) u_R at the mean state u_bar, with the cutoff
// eigenvalues of eq. (cutoff), split as the JST flux is (h = hc - hd): hc = A(u_bar)(u_L + u_R)/2,
// hd = (A+ - A-)(u_R - u_L)/2.  Each product uses the closed rank-2 form of R diag(l) R^-1 for
// the wave pattern (l1, l1, l3, l4): M(l) x = l1 x + r0 (g0 . x) + r1 (g1 . x) with
// r0 = (1, u, v, H), r1 = (0, nx, ny, vn), g0 = c1/a^2 dp + c2/a dvn, g1 = c2/a dp + c1 dvn,
// dp = (gamma-1)(q^2/2, -u, -v, 1), dvn = (-vn, nx, ny, 0), c1 = (l3+l4)/2 - l1, c2 = (l3-l4)/2.
__device__ __forceinline__ double fvs_cutabs(double lam, double a, double d) {
  const double al = fabs(lam), ad = a * d;
  return (d > 0.0 && al <= ad) ? 0.5 * (ad + lam * lam / ad) : al;
}

__device__ void fvs_face(const LevelDev& L, int gL, int gR, double sx, double sy, double vf, double dcut,
                         double hc[4], double hd[4]) {
  double uL[4], uR[4], ub[4], xs[4], xd[4];
  load4(L, gL, uL);
  load4(L, gR, uR);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    ub[k] = 0.5 * (uL[k] + uR[k]);
    xs[k] = uL[k] + uR[k];
    xd[k] = uR[k] - uL[k];
  }
  const double g1 = GAM - 1.0;
  const double len = sqrt(sx * sx + sy * sy), rl = 1.0 / len;
  const double nx = sx * rl, ny = sy * rl;
  const double rr = 1.0 / ub[0], u = ub[1] * rr, v = ub[2] * rr;
  const double q2 = u * u + v * v;
  const double p = g1 * (ub[3] - 0.5 * ub[0] * q2);
  const double a = sqrt(GAM * p * rr), ia = 1.0 / a;
  const double H = (ub[3] + p) * rr;
  const double vn = u * nx + v * ny, vr = vn - vf * rl;
  const double r0[4] = {1.0, u, v, H}, r1[4] = {0.0, nx, ny, vn};
  const double dp[4] = {0.5 * g1 * q2, -g1 * u, -g1 * v, g1}, dv[4] = {-vn, nx, ny, 0.0};
  // M(l) x for the eigenvalue triple (l1, l3, l4), times the face length
  auto apply = [&](double l1, double l3, double l4, const double x[4], double out[4]) {
    double dpx = 0.0, dvx = 0.0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      dpx += dp[k] * x[k];
      dvx += dv[k] * x[k];
    }
    const double c1 = 0.5 * (l3 + l4) - l1, c2 = 0.5 * (l3 - l4);
    const double s0 = c1 * ia * ia * dpx + c2 * ia * dvx, s1 = c2 * ia * dpx + c1 * dvx;
#pragma unroll
    for (int k = 0; k < 4; ++k) out[k] = len * (l1 * x[k] + r0[k] * s0 + r1[k] * s1);
  };
  apply(vr, vr + a, vr - a, xs, hc);
  apply(fvs_cutabs(vr, a, dcut), fvs_cutabs(vr + a, a, dcut), fvs_cutabs(vr - a, a, dcut), xd, hd);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    hc[k] *= 0.5;
    hd[k] *= 0.5;
  }
}

// JST flux through a face with area vector (sx, sy) from L to R; stencil LL, L, R, RR
// given as ghosted indices.  hc: central part; hd: dissipation d (section 2).
// On a moving face (grid volume flux vf) the convective flux is F . S - u vf.
// The factor 1/2 of the averages goes on the face vector, and on a fixed grid (moving 0) the terms in vf
// are left out: both leave every bit as it is.  FAST (PhysParams::fast) takes the grid's flux off the
// normal velocities once, sums the two cells' terms in chains, and forms the third difference as
// (w_RR - w_LL) - 3 dw, with one rounding (with it spread over (eps2 + 3 eps4) dw - eps4 (w_RR - w_LL) four
// instructions fewer, but the rounding is that of the first differences: 40 % more error in the density
// dissipation of 330x90 RANS).  About 70 FP64 instructions a face.  s: the larger of the two cells' sensors
// (finest level).
template <bool FAST>
__device__ __forceinline__ void jst_face(const LevelDev& L, int gLL, int gL, int gR, int gRR, double sx, double sy,
                                         double vf, int moving, double rtL, double rtR, double s, double s_coarse,
                                         double hc[4], double hd[4]) {
  double uL[4], uR[4];
  load4(L, gL, uL);
  load4(L, gR, uR);
  const double pL = L.p[gL], pR = L.p[gR];
  const double wL3 = uL[3] + pL, wR3 = uR[3] + pR;  // w = (rho, rho u, rho v, rho H)
  {
    const double hx = 0.5 * sx, hy = 0.5 * sy, hf = 0.5 * vf;
    const double qL = (uL[1] * hx + uL[2] * hy) * L.rinv[gL];
    const double qR = (uR[1] * hx + uR[2] * hy) * L.rinv[gR];
    if (FAST) {
      const double aL = moving ? qL - hf : qL, aR = moving ? qR - hf : qR;
      hc[0] = uL[0] * aL + uR[0] * aR;
      hc[1] = pR * hx + (pL * hx + (uL[1] * aL + uR[1] * aR));  // the pressure's part, the largest, last
      hc[2] = pR * hy + (pL * hy + (uL[2] * aL + uR[2] * aR));
      hc[3] = wL3 * qL + wR3 * qR;
      if (moving) hc[3] -= hf * (uL[3] + uR[3]);
    } else if (moving) {
      const double qnL = (uL[1] * sx + uL[2] * sy) * L.rinv[gL];
      const double qnR = (uR[1] * sx + uR[2] * sy) * L.rinv[gR];
      hc[0] = 0.5 * ((uL[0] * qnL - uL[0] * vf) + (uR[0] * qnR - uR[0] * vf));
      hc[1] = 0.5 * (((uL[1] * qnL + pL * sx) - uL[1] * vf) + ((uR[1] * qnR + pR * sx) - uR[1] * vf));
      hc[2] = 0.5 * (((uL[2] * qnL + pL * sy) - uL[2] * vf) + ((uR[2] * qnR + pR * sy) - uR[2] * vf));
      hc[3] = 0.5 * (((uL[3] + pL) * qnL - uL[3] * vf) + ((uR[3] + pR) * qnR - uR[3] * vf));
    } else {
      hc[0] = __dadd_rn(__dmul_rn(uL[0], qL), __dmul_rn(uR[0], qR));
      hc[1] = __dadd_rn(uL[1] * qL + pL * hx, uR[1] * qR + pR * hx);
      hc[2] = __dadd_rn(uL[2] * qL + pL * hy, uR[2] * qR + pR * hy);
      hc[3] = __dadd_rn(__dmul_rn(wL3, qL), __dmul_rn(wR3, qR));
    }
  }
  const double r = max_nn(rtL, rtR);
  uL[3] = wL3;
  uR[3] = wR3;
  double e2 = s_coarse * r, e4 = 0.0;
  if (L.finest) {
    e2 = min_pos(s, 0.25) * r;
    e4 = relu64(fma(-2.0, e2, r * (1.0 / 32.0)));
  }
  if (!is_zero(e4)) {
    double uLL[4], uRR[4];
    load4(L, gLL, uLL);
    load4(L, gRR, uRR);
    uLL[3] += L.p[gLL];
    uRR[3] += L.p[gRR];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const double dw0 = uR[k] - uL[k];
      if (FAST) {
        hd[k] = fma(-e4, fma(-3.0, dw0, uRR[k] - uLL[k]), e2 * dw0);
      } else {
        const double dwm = uL[k] - uLL[k], dwp = uRR[k] - uR[k];
        hd[k] = fma(-e4, fma(-2.0, dw0, dwp + dwm), __dmul_rn(e2, dw0));
      }
    }
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) hd[k] = e2 * (uR[k] - uL[k]);
  }
}

// Sensor of the cell at ghosted index g along stride d (1: along i, the pitch: along j).
template <bool FAST>
__device__ __forceinline__ double cell_sensor(const LevelDev& L, int g, int d) {
  return sensor_val<FAST>(L.q[g - d], L.q[g], L.q[g + d]);
}

// Thin-layer viscous flux through j-face (i, j): gradients = jump across the face times S over
// the mean volume of the two cells.  FAST: with gradients (du, dv) S / Omega_f the stress on the face
// is mu_eff / Omega_f times (du (4/3 Sx^2 + Sy^2) + dv Sx Sy / 3, dv (4/3 Sy^2 + Sx^2) + du Sx Sy / 3).
template <bool FAST>
__device__ __forceinline__ void visc_face(const LevelDev& L, const PhysParams& ph, int i, int j, double sx, double sy,
                                          double hv[4]) {
  const int ni = L.ni, nj = L.nj;
  double mutf;
  if (j == 0)
    mutf = on_cut(L, i) ? 0.5 * (L.mut[i] + L.mut[ni - 1 - i]) : 0.0;
  else if (j == nj)
    mutf = L.mut[(nj - 1) * ni + i];
  else
    mutf = 0.5 * (L.mut[(j - 1) * ni + i] + L.mut[j * ni + i]);
  const double rvf = L.rvf[j * ni + i];
  double wL[4], wR[4];
  const int gL = gidx(L, i, j - 1), gR = gidx(L, i, j);
  load4(L, gL, wL);
  load4(L, gR, wR);
  const double rL = L.rinv[gL], rR = L.rinv[gR];
  const double uL = wL[1] * rL, vL = wL[2] * rL, uR = wR[1] * rR, vR = wR[2] * rR;
  constexpr double cp = GAM / (GAM - 1.0);
  const double mu = ph.inv_re;
  const double mueff = mu + mutf;
  const double keff = mu * ph.inv_pr + mutf * ph.inv_prt;
  hv[0] = 0.0;
  if (FAST) {
    const double du = uR - uL, dv = vR - vL, dh = L.p[gR] * rR - L.p[gL] * rL;
    const double xx = sx * sx, yy = sy * sy, s2 = xx + yy, c3 = (1.0 / 3.0) * sx * sy, k = mueff * rvf;
    const double fx = k * (du * fma(1.0 / 3.0, xx, s2) + dv * c3);
    const double fy = k * (dv * fma(1.0 / 3.0, yy, s2) + du * c3);
    hv[1] = fx;
    hv[2] = fy;
    hv[3] = 0.5 * ((uL + uR) * fx + (vL + vR) * fy) + (cp * keff * rvf) * (dh * s2);
    return;
  }
  const double hL = cp * L.p[gL] * rL, hR = cp * L.p[gR] * rR;
  const double sxv = sx * rvf, syv = sy * rvf;
  const double gux = (uR - uL) * sxv, guy = (uR - uL) * syv;
  const double gvx = (vR - vL) * sxv, gvy = (vR - vL) * syv;
  const double ghx = (hR - hL) * sxv, ghy = (hR - hL) * syv;
  const double div = gux + gvy;
  const double txx = mueff * (2.0 * gux - 2.0 / 3.0 * div);
  const double tyy = mueff * (2.0 * gvy - 2.0 / 3.0 * div);
  const double txy = mueff * (guy + gvx);
  const double uf = 0.5 * (uL + uR), vf = 0.5 * (vL + vR);
  const double fx = txx * sx + txy * sy, fy = txy * sx + tyy * sy;
  hv[1] = fx;
  hv[2] = fy;
  hv[3] = uf * fx + vf * fy + keff * (ghx * sx + ghy * sy);
}

// Deterministic block sum of one double per thread (fixed shuffle tree, then warps in order).
__device__ double block_sum(double v, double* wsum) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if ((threadIdx.x & 31) == 0) wsum[w] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int k = 0; k < nw; ++k) s += wsum[k];
  return s;
}

// entry e of a cell's transfer blocks
__device__ __forceinline__ double tb_entry(const LevelDev& L, int tb32, int e, int c) {
  const size_t at = (size_t)e * L.n + c;
  return tb32 ? f2d(reinterpret_cast<const float*>(L.tb)[at]) : L.tb[at];
}

// a cell's part of the squared norm
__device__ __forceinline__ double norm_of(const double F[4], int all) {
  double s = F[0] * F[0];
  if (all) {
    s = 0.0;
#pragma unroll
    for (int k = 0; k < 4; ++k) s += F[k] * F[k];
  }
  return s;
}

// One tile of TX x TY cells: every face of the tile is computed once into shared memory,
// then each cell assembles F^c and F^v and writes what the mode asks for.
template <int TY, bool FAST>
__global__ void __launch_bounds__(res_threads(TY)) k_residual(LevelDev L, PhysParams ph, ResArgs a) {
  __shared__ double xc[4][TY][TX + 1], xd[4][TY][TX + 1];
  __shared__ double ec[4][TY + 1][TX], ed[4][TY + 1][TX];
  __shared__ double wsum[res_threads(TY) / 32];
  __shared__ double si[TY], sj[TY + 2][TX];  // sensors: along i of cell (i0 + TX, j0 + y), along j of rows j0 - 1 ..
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i0 = blockIdx.x * TX, j0 = blockIdx.y * TY;
  const int ni = L.ni, nj = L.nj, n = L.n;
  // Before the wait for the kernel before: face vectors, volumes, forcing, history and carried viscous
  // part.  Each was written two launches ago or earlier (between any of their kernels and a residual lies
  // at least k_cell_aux), and a kernel lets its successor start only once its own predecessors have
  // completed (pdl_entry).
  const bool iface = warp < TY;
  const int fi = i0 + lane, fj = j0 + (iface ? warp : warp - TY);  // this thread's face
  const bool face = iface ? fi <= ni && fj < nj : lane < TX && warp <= 2 * TY && fi < ni && fj <= nj;
  double sx = 0.0, sy = 0.0, fvol = 0.0;
  if (face) {
    const int f = iface ? fj * (ni + 1) + fi : fj * ni + fi;
    sx = iface ? L.sxi[f] : L.seta[f];
    sy = iface ? L.sxi[L.nfx + f] : L.seta[L.nfe + f];
    if (ph.moving || ph.flux) fvol = iface ? L.vfx[f] : L.vfe[f];
  }
  // this thread's cell: one component of it (tile height 1, four warps) or two (a warp pair per row)
  constexpr int NK = TY == 1 ? 1 : 2;
  const int k0 = NK * (warp / TY), cy = warp % TY, c = (j0 + cy) * ni + fi;
  const bool cell = k0 < 4 && lane < TX && fi < ni && j0 + cy < nj;
  double rvol = 0.0, src[NK] = {}, frc[NK] = {}, old[NK] = {};
  auto load_cell = [&] {
    rvol = L.rvol[c];
#pragma unroll
    for (int k = 0; k < NK; ++k) {
      const int e = (k0 + k) * n + c;
      if (L.finest) src[k] = L.src[e];  // coarse levels have no history source
      frc[k] = a.mode == RES_FORCING ? L.rhs[e] : L.s[e];
      if (a.mode == RES_STAGE && a.stage > 1) old[k] = L.fvc[e];
    }
  };
  if (TY == 1 && cell) load_cell();
  pdl_entry();
  // Each cell's pressure switch is formed once (finest level): an i-face warp's lane takes cell
  // i0 + lane - 1 of its row and passes it on, its last cell is the j-face warps' spare lane's; the
  // j-face warps take a row each (the last one two; tile height 1: the spare warp the last).
  double sl = 0.0;
  const bool sensors = L.finest && !ph.flux;
  if (sensors) {
    if (warp < TY) {
      if (i0 + lane <= ni + 1 && j0 + warp < nj) sl = cell_sensor<FAST>(L, gidx(L, i0 + lane - 1, j0 + warp), 1);
    } else {
      const int y = warp - TY;
      const int i = i0 + lane, j = j0 + (lane < TX ? y - 1 : y);
      if (lane < TX ? i < ni && j <= nj : y < TY && i < ni + 1 && j < nj)
        (lane < TX ? sj[y][lane] : si[y]) =
            cell_sensor<FAST>(L, gidx(L, i, j), lane < TX ? L.P : 1);
      if (TY > 1 && y == TY && lane < TX && i < ni && j0 + TY <= nj) sj[TY + 1][lane] = cell_sensor<FAST>(L, gidx(L, i, j0 + TY), L.P);
    }
    __syncthreads();
  }
  // tile height 1: this thread's row of D^-1 and dt* are on their way early.  On larger tiles, whose other
  // blocks hide the latency, the registers are worth more (64 cases, mixed: 9.2 ms a cycle early, 8.8 late).
  double row[4], dt = 1.0;
  if (TY == 1 && cell) {
    if (a.mode == RES_STAGE && a.aw) dt = L.dts[c];
    if (a.wsC) {
#pragma unroll
      for (int k = 0; k < 4; ++k) row[k] = tb_entry(L, a.tb32, 4 * k0 + k, c);
    }
  }
  if (iface) {
    const double sdn = __shfl_down_sync(0xffffffffu, sl, 1), sr = lane < TX ? sdn : si[warp];
    if (face) {
      const int i = fi, j = fj;
      double hc[4], hd[4];
      if (ph.flux)
        fvs_face(L, gidx(L, i - 1, j), gidx(L, i, j), sx, sy, fvol, ph.d_cut, hc, hd);
      else
        jst_face<FAST>(L, gidx(L, i - 2, j), gidx(L, i - 1, j), gidx(L, i, j), gidx(L, i + 1, j), sx, sy, fvol,
                       ph.moving, rt_cell(L, i - 1, j, 0), rt_cell(L, i, j, 0), fmax(sl, sr), ph.s_coarse, hc, hd);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        xc[k][warp][lane] = hc[k];
        xd[k][warp][lane] = hd[k];
      }
    }
  } else if (face) {
    const int i = fi, j = fj, ty = warp - TY;
    double hc[4], hd[4];
    if (ph.flux)
      fvs_face(L, gidx(L, i, j - 1), gidx(L, i, j), sx, sy, fvol, ph.d_cut, hc, hd);
    else
      jst_face<FAST>(L, gidx(L, i, j - 2), gidx(L, i, j - 1), gidx(L, i, j), gidx(L, i, j + 1), sx, sy, fvol,
                     ph.moving, rt_cell(L, i, j - 1, 1), rt_cell(L, i, j, 1),
                     sensors ? fmax(sj[ty][lane], sj[ty + 1][lane]) : 0.0, ph.s_coarse, hc, hd);
    if (ph.viscous) {
      double hv[4];
      visc_face<FAST>(L, ph, i, j, sx, sy, hv);
#pragma unroll
      for (int k = 1; k < 4; ++k) hd[k] += hv[k];
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      ec[k][ty][lane] = hc[k];
      ed[k][ty][lane] = hd[k];
    }
  }
  __syncthreads();
  double nacc = 0.0;
  double r[NK], F[NK];  // this thread's stage right-hand side and residual
  if (cell) {
    if (TY > 1) {
      load_cell();
      if (a.mode == RES_STAGE && a.aw) dt = L.dts[c];
    }
    const int tx = lane, ty = cy;
    const bool timed = !is_zero(L.a_t);
    const int g = gidx(L, fi, j0 + cy);
#pragma unroll
    for (int q = 0; q < NK; ++q) {
      const int k = k0 + q, e = k * n + c;
      const double fc = (xc[k][ty][tx + 1] - xc[k][ty][tx]) + (ec[k][ty + 1][tx] - ec[k][ty][tx]);
      const double fd = (xd[k][ty][tx] - xd[k][ty][tx + 1]) + (ed[k][ty][tx] - ed[k][ty + 1][tx]);
      double Fc = timed ? fma(fc, rvol, __dmul_rn(L.a_t, L.u[k * L.Gn + g])) : fc * rvol;
      if (L.finest) Fc += src[q];
      if (a.mode != RES_FORCING) Fc -= frc[q];
      const double Fv = fd * rvol;
      F[q] = a.want_norm ? Fc + Fv : 0.0;
      if (a.mode == RES_STAGE) {
        const double carry = a.stage == 1 ? Fv : a.beta * Fv + (1.0 - a.beta) * old[q];
        L.fvc[e] = carry;
        r[q] = dt * (Fc + carry);
        if (!a.wsC) L.rhs[e] = r[q];
      } else if (a.mode == RES_FULL) {
        if (a.F) a.F[e] = Fc + Fv;
        if (a.Fc) a.Fc[e] = Fc;
        if (a.Fv) a.Fv[e] = Fv;
      } else if (a.mode == RES_FORCING) {
        L.s[e] = (Fc + Fv) + frc[q];
      } else {  // RES_FASRES
        L.rhs[e] = -(Fc + Fv);
      }
    }
  }
  // The warp-strip sweep's right-hand side D^-1 r, where r is: a launch less, and D^-1 r of the defect
  // with it.  Measured with the update moved to k_cell_aux: 1024x256 W-cycle FP64 11.43 -> 11.20 ms, mixed
  // 7.18 -> 7.03; 64 cases of 64x16 ... 256x64 in a batch, mixed 10.7 -> 8.8 ms a cycle, FP64 17.9 -> 13.2.
  if (a.wsC || a.want_norm) {
    // each warp has read its components' faces of its row: xc holds the right-hand sides now, xd the residuals
    __syncwarp();
    if (cell) {
#pragma unroll
      for (int q = 0; q < NK; ++q) {
        xc[k0 + q][cy][lane] = r[q];
        if (a.want_norm) xd[k0 + q][cy][lane] = F[q];
      }
    }
    __syncthreads();
    if (cell && a.want_norm && k0 == 0) {
      const double f[4] = {xd[0][cy][lane], xd[1][cy][lane], xd[2][cy][lane], xd[3][cy][lane]};
      nacc = norm_of(f, a.norm_all);
    }
    if (cell && a.wsC) {
      float* out = reinterpret_cast<float*>(a.wsC + ws_fpos(fi, j0 + cy, ws_steps(ni, nj))) + k0;
#pragma unroll
      for (int q = 0; q < NK; ++q) {
        double b = 0.0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const double d = TY == 1 ? row[k] : tb_entry(L, a.tb32, 4 * (k0 + q) + k, c);
          b += d * xc[k][cy][lane];
        }
        if (!a.tb32) L.wsR[(size_t)(k0 + q) * n + c] = b;
        out[q] = d2f(b);
      }
    }
  }
  if (a.want_norm) {
    const double s = block_sum(nacc, wsum);
    if (threadIdx.x == 0) L.norm_part[blockIdx.y * gridDim.x + blockIdx.x] = s;
  }
}

// Force on the body through each wall face (j = 0 off the wake cut): the residual's own
// j-face flux (central part minus dissipation minus viscous part) with the opposite sign,
// since the face vector points into the fluid.  fx, fy: ni entries, zero on the cut.
__global__ void k_wall_force(LevelDev L, PhysParams ph, double* fx, double* fy) {
  pdl_entry();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= L.ni) return;
  if (on_cut(L, i)) {
    fx[i] = fy[i] = 0.0;
    return;
  }
  const double sx = L.seta[i], sy = L.seta[L.nfe + i];
  double hc[4], hd[4];
  if (ph.flux)
    fvs_face(L, gidx(L, i, -1), gidx(L, i, 0), sx, sy, L.vfe[i], ph.d_cut, hc, hd);
  else
    jst_face<false>(L, gidx(L, i, -2), gidx(L, i, -1), gidx(L, i, 0), gidx(L, i, 1), sx, sy, L.vfe[i], ph.moving,
             rt_cell(L, i, -1, 1), rt_cell(L, i, 0, 1),
             L.finest ? fmax(cell_sensor<false>(L, gidx(L, i, -1), L.P), cell_sensor<false>(L, gidx(L, i, 0), L.P)) : 0.0,
             ph.s_coarse, hc, hd);
  if (ph.viscous) {
    double hv[4];
    visc_face<false>(L, ph, i, 0, sx, sy, hv);
    for (int k = 0; k < 4; ++k) hd[k] += hv[k];
  }
  fx[i] = -(hc[1] - hd[1]);
  fy[i] = -(hc[2] - hd[2]);
}

__global__ void k_norm_final(const double* part, int nparts, double count, double* out) {
  pdl_entry();
  __shared__ double wsum[8];
  double s = 0.0;
  for (int k = threadIdx.x; k < nparts; k += blockDim.x) s += part[k];
  const double t = block_sum(s, wsum);
  if (threadIdx.x == 0) out[0] = sqrt(t / count);
}

// A cycle's norm and error word go to pinned host memory from kernels (k_norm_final, k_report_error) instead of
// by a copy each after the last kernel, and the word is cleared here instead of by a fill before the next
// cycle: 64x16, a residual with its norm 28.7 -> 24.1 us, a cycle 268 -> 265.
__global__ void k_report_error(int* err, int* host) {
  pdl_entry();
  *host = *err;
  *err = 0;
}

// ---- Baldwin-Lomax (finest level): vorticity by Green-Gauss, then one thread per i-line.
__global__ void k_vorticity(LevelDev L) {
  pdl_entry();
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= L.n) return;
  const int ni = L.ni, i = c % ni, j = c / ni;
  const int g0 = gidx(L, i, j);
  const double u0 = L.u[L.Gn + g0] * L.rinv[g0], v0 = L.u[2 * L.Gn + g0] * L.rinv[g0];
  double fu[4], fv[4];
  const int nb[4][2] = {{i + 1, j}, {i - 1, j}, {i, j + 1}, {i, j - 1}};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int g = gidx(L, nb[k][0], nb[k][1]);
    fu[k] = 0.5 * (u0 + L.u[L.Gn + g] * L.rinv[g]);
    fv[k] = 0.5 * (v0 + L.u[2 * L.Gn + g] * L.rinv[g]);
  }
  const int fe = j * (ni + 1) + i + 1, fw = j * (ni + 1) + i, fn = (j + 1) * ni + i, fs = j * ni + i;
  const double circ = (fv[0] * L.sxi[fe] - fu[0] * L.sxi[L.nfx + fe]) - (fv[1] * L.sxi[fw] - fu[1] * L.sxi[L.nfx + fw]) +
                      (fv[2] * L.seta[fn] - fu[2] * L.seta[L.nfe + fn]) - (fv[3] * L.seta[fs] - fu[3] * L.seta[L.nfe + fs]);
  L.omega[c] = fabs(circ / L.vol[c]);
}

// Baldwin-Lomax along each grid line i = const: one warp per line, lanes over j.  The search
// for F_max takes the first j of the largest F (as a sequential scan with a strict > would),
// and the inner/outer crossover is the first j where the inner value reaches the outer one.
__global__ void k_bl_lines(LevelDev L, PhysParams ph) {
  pdl_entry();
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (i >= L.ni) return;  // whole warps leave together
  const double Aplus = 26.0, Ccp = 1.6, Ckleb = 0.3, Cwk = 0.25, kap = 0.4, Kc = 0.0168;
  const int ni = L.ni, nj = L.nj;
  const double mu = ph.inv_re;
  const bool wake = on_cut(L, i);
  const double rhow = L.u[gidx(L, i, 0)];
  const double tauw = mu * L.omega[i];
  const double utr = sqrt(rhow * tauw);
  const double yplus_scale = utr * ph.re / Aplus;  // y+ / A+ = y * utr / (mu A+)
  const int jsearch = max(1, nj / 2);
  double Fmax = 0.0, smax = 0.0, smin = 1e300;
  int jmax = 1 << 30;
  for (int j = lane; j < jsearch; j += 32) {
    const int c = j * ni + i;
    const double y = L.wdist[c];
    const double damp = wake ? 1.0 : 1.0 - exp(-y * yplus_scale);
    const double F = y * L.omega[c] * damp;
    if (F > Fmax) {  // lanes scan increasing j: keeps the first j of the lane's largest F
      Fmax = F;
      jmax = j;
    }
    const int g = gidx(L, i, j);
    const double rr = L.rinv[g], uu = L.u[L.Gn + g] * rr, vv = L.u[2 * L.Gn + g] * rr;
    const double sp = sqrt(uu * uu + vv * vv);
    smax = fmax(smax, sp);
    smin = fmin(smin, sp);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double F2 = __shfl_xor_sync(0xffffffffu, Fmax, o);
    const int j2 = __shfl_xor_sync(0xffffffffu, jmax, o);
    if (F2 > Fmax || (F2 == Fmax && j2 < jmax)) {
      Fmax = F2;
      jmax = j2;
    }
    smax = fmax(smax, __shfl_xor_sync(0xffffffffu, smax, o));
    smin = fmin(smin, __shfl_xor_sync(0xffffffffu, smin, o));
  }
  const double ymax = Fmax > 0.0 ? L.wdist[jmax * ni + i] : 0.0;
  const double udif = wake ? smax - smin : smax;
  const double Fwake = Fmax > 0.0 ? fmin(ymax * Fmax, Cwk * ymax * udif * udif / Fmax) : 0.0;
  const double rym = ymax > 0.0 ? Ckleb / ymax : 0.0;
  int jcross = wake ? 0 : nj;
  for (int j0 = 0; j0 < nj; j0 += 32) {
    const int j = j0 + lane;
    double mo = 0.0, mi = 0.0;
    if (j < nj) {
      const int c = j * ni + i;
      const double y = L.wdist[c];
      const double rho = L.u[gidx(L, i, j)];
      const double x = y * rym, x2 = x * x;
      const double fk = ymax > 0.0 ? 1.0 / (1.0 + 5.5 * (x2 * x2 * x2)) : 0.0;
      mo = Kc * Ccp * rho * Fwake * fk;
      const double damp = wake ? 1.0 : 1.0 - exp(-y * yplus_scale);
      const double l = kap * y * damp;
      mi = rho * l * l * L.omega[c];
    }
    if (jcross == nj) {
      const unsigned hit = __ballot_sync(0xffffffffu, j < nj && mi >= mo);
      if (hit) jcross = j0 + __ffs(hit) - 1;
    }
    if (j < nj) L.mut[j * ni + i] = j >= jcross ? mo : mi;
  }
}

// The two powers of the auxiliaries beside the CUDA math library's: out[4 t ..] =
// (pow_neg_gamma(a), pow(a, -gamma), cbrt_ratio(a, b), cbrt(a / b)).
__global__ void k_check_math(int n, const double* __restrict__ a, const double* __restrict__ b, double* __restrict__ out) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  out[4 * t + 0] = pow_neg_gamma(a[t]);
  out[4 * t + 1] = pow(a[t], -GAM);
  out[4 * t + 2] = cbrt_ratio(a[t], b[t]);
  out[4 * t + 3] = cbrt(a[t] / b[t]);
}

// The FP64 helpers beside the instructions they stand for: out[4 t ..] = (rcp64(a), 1/a, d2f(a),
// f2d((float)a)).
__global__ void k_check_fp64(int n, const double* __restrict__ a, double* __restrict__ out) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  out[4 * t + 0] = rcp64(a[t]);
  out[4 * t + 1] = 1.0 / a[t];
  out[4 * t + 2] = (double)d2f(a[t]);
  out[4 * t + 3] = f2d((float)a[t]);
}

}  // namespace

void launch_check_fp64(int n, const double* a, double* out, cudaStream_t st) {
  if (n > 0) k_check_fp64<<<(n + 127) / 128, 128, 0, st>>>(n, a, out);
}

void launch_check_math(int n, const double* a, const double* b, double* out, cudaStream_t st) {
  if (n > 0) k_check_math<<<(n + 127) / 128, 128, 0, st>>>(n, a, b, out);
}

cudaError_t launch_bc(const LevelDev& L, const PhysParams& ph, cudaStream_t st) {
  const int nt = 4 * L.ni + 4 * L.nj;
  return launch_pdl(k_bc, (nt + 63) / 64, 64, 0, st, L, ph);
}

cudaError_t launch_cell_aux(const LevelDev& L, const PhysParams& ph, double cfl, int want_dts, cudaStream_t st) {
  const int nbi = (L.n + 63) / 64, nbg = (4 * (L.ni + L.nj) + 63) / 64;
  return launch_pdl(k_cell_aux, nbi + nbg, 64, 0, st, L, ph, cfl, want_dts, 0, nbi, WsPending{}, 0);
}

void launch_bc_aux(const LevelDev& L, const PhysParams& ph, double cfl, int want_dts, cudaStream_t st,
                   const WsPending* pending, int early) {
  const int nbi = (L.n + 63) / 64, nbg = (4 * (L.ni + L.nj) + 63) / 64;
  launch_pdl(k_cell_aux, nbi + nbg, 64, 0, st, L, ph, cfl, want_dts, 1, nbi,
             pending ? *pending : WsPending{}, early);
}

void launch_wall_force(const LevelDev& L, const PhysParams& ph, double* fx, double* fy, cudaStream_t st) {
  launch_pdl(k_wall_force, (L.ni + 63) / 64, 64, 0, st, L, ph, fx, fy);
}

int residual_blocks(const LevelDev& L) {
  const int ty = res_ty(L);
  return ((L.ni + TX - 1) / TX) * ((L.nj + ty - 1) / ty);
}

namespace {
template <bool FAST>
cudaError_t residual_ty(int ty, dim3 grid, cudaStream_t st, const LevelDev& L, const PhysParams& ph, const ResArgs& a) {
  switch (ty) {
    case 8: return launch_pdl(k_residual<8, FAST>, grid, res_threads(8), 0, st, L, ph, a);
    case 4: return launch_pdl(k_residual<4, FAST>, grid, res_threads(4), 0, st, L, ph, a);
    case 2: return launch_pdl(k_residual<2, FAST>, grid, res_threads(2), 0, st, L, ph, a);
    default: return launch_pdl(k_residual<1, FAST>, grid, res_threads(1), 0, st, L, ph, a);
  }
}
}  // namespace

cudaError_t launch_residual(const LevelDev& L, const PhysParams& ph, const ResArgs& a, cudaStream_t st) {
  const int ty = res_ty(L);
  const dim3 grid((L.ni + TX - 1) / TX, (L.nj + ty - 1) / ty);
  return ph.fast ? residual_ty<true>(ty, grid, st, L, ph, a) : residual_ty<false>(ty, grid, st, L, ph, a);
}

int residual_blocks_max(const LevelDev& L) { return ((L.ni + TX - 1) / TX) * L.nj; }

void launch_norm_final(const LevelDev& L, int nparts, int ncomp_cells, double* out, cudaStream_t st) {
  launch_pdl(k_norm_final, 1, 256, 0, st, L.norm_part, nparts, (double)ncomp_cells, out);
}

void launch_report_error(int* err, int* host, cudaStream_t st) { launch_pdl(k_report_error, 1, 1, 0, st, err, host); }

void launch_bl(const LevelDev& L, const PhysParams& ph, cudaStream_t st) {
  launch_pdl(k_vorticity, (L.n + 63) / 64, 64, 0, st, L);
  launch_pdl(k_bl_lines, (L.ni + 1) / 2, 64, 0, st, L, ph);
}

}  // namespace fasw
