// dg2_fv.cuh -- the MUSCL-FV2 and FV1 comparator schemes of Sec. 2.2 (Eqs. 8-10)
// on the FP64 state layout.  The FV schemes hold cell averages only (planes
// h0, qx0, qy0); the slope planes are never read or written.
//
// Per cell and face: MUSCL limits of eta = h + z, h, qx, qy (Eq. 9) with
// Sweby's limiter (beta = 1.25, Eq. 10, r = forward / backward difference, no
// reconstruction across a wet-dry front), the free-surface revision of
// Sec. 2.2.2 (z* = max of the two bed limits, h* = max(0, eta - z*), q* = h* u,
// the own-side lowering of z* behind a wall), the run's Riemann solver and
// Eq. 8's bed term (factor 2 / dx as in Eq. 4a).  Friction is the DG2 friction
// kernel, which on zero slopes acts on the averages alone.
//
// One block per 16 x 8 half of a tile of the step's lists, as the DG2 stage kernels:
// the averages of the tile and a 2-cell halo are staged in shared memory, each
// thread forms its cell's four limits, the tile's last threads form the limits
// beyond the tile, and every face flux is evaluated once.  Dry-tile skipping
// carries over unchanged: a still, dry cell among still, dry neighbours has zero
// fluxes, and the dry reset removes the discharge its bed term makes.  The same
// holds for single cells, so a cell whose input and four neighbours are still and
// dry (read off the staged averages, fv_moves) takes L = 0 and its faces are left out.
//
// The FP64 pipe bounds the kernels.  Divisions (Sweby's ratio, the velocities) and FP64
// comparisons used to make up most of their FP64 instructions, and every cell of a
// computed tile was evaluated: a pass of 70 FV2 steps of a 2000 x 1000 floodplain, 4 % wet,
// took 43.1 ms with the state in and out, 20.4 ms without them, and 12.8 ms with blocks of
// half a listed tile and exact flags of a state set.
#pragma once
#include "dg2_device.cuh"

namespace dg2 {
namespace fv {

constexpr int TX = 16, PARTS = TW / TX;  // a block takes half a tile
constexpr int HX = TX + 4, HY = TY + 4;  // staged region: tile + 2-cell halo

struct L4 {
  double eta, h, qx, qy;
};

// A face after the revision: its flux (in the face's frame, Flux) and the lower (west /
// south) side's revised depth.
struct Face {
  double h, n, t, dp, ha;
};

struct Smem {
  union {
    double A[4][HY][HX];  // eta, h, qx, qy of the staged region
    struct {
      Face fx[TY][TX + 1];  // fx[ty][tx] is the west face of column tx
      Face fy[TY + 1][TX];  // fy[ty][tx] is the south face of row ty
    } f;
  } u;
  L4 e[TY][TX];  // east limit of each cell
  L4 n[TY][TX];  // north limit of each cell
  L4 hw[TY], he[TY], hs[TX], hn[TX];  // limits beyond the tile (neighbour or ghost)
  double red[32];
  StageK k;
  unsigned char cls[TY][TX];  // 0 outside the grid, 1 L = 0, 2 computed
};

// Slope of Eq. 10 with Sweby's limiter (beta = 1.25) from the backward and forward
// differences: phi(fd / bd) bd without the division, max(min(beta |fd|, |bd|),
// min(|fd|, beta |bd|)) with their sign where they share one, else 0.
__device__ __forceinline__ double sweby_slope(double bd, double fd) {
  if (!((is_pos(bd) && is_pos(fd)) || (is_neg(bd) && is_neg(fd)))) return 0.0;
  const double a = fabs(fd), b = fabs(bd);
  const double m = max_nn(min_nn(1.25 * a, b), min_nn(a, 1.25 * b));
  return is_neg(bd) ? -m : m;
}

// Limited slopes (Eq. 10) of the four components of staged cell (a, b) along
// (da, db); zero for FV1, at the domain edge along that direction, and where
// the cell or one of its two neighbours along it is at or below tol_dry.
template <bool ORDER2>
__device__ __forceinline__ void slopes4(const double (*A)[HY][HX], int a, int b, int da, int db,
                                        bool edge, double tol, double s[4]) {
#pragma unroll
  for (int k = 0; k < 4; ++k) s[k] = 0.0;
  if (!ORDER2 || edge) return;
  if (!above(A[1][b - db][a - da], tol) || !above(A[1][b][a], tol) ||
      !above(A[1][b + db][a + da], tol))
    return;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const double vc = A[k][b][a];
    s[k] = sweby_slope(vc - A[k][b - db][a - da], A[k][b + db][a + da] - vc);
  }
}

// Limit of staged cell (a, b) at the face on side sg (+0.5 east / north,
// -0.5 west / south) of the slopes' direction (Eq. 9).
__device__ __forceinline__ L4 lim4(const double (*A)[HY][HX], int a, int b, const double s[4],
                                   double sg) {
  L4 r;
  r.eta = fma(sg, s[0], A[0][b][a]);
  r.h = fma(sg, s[1], A[1][b][a]);
  r.qx = fma(sg, s[2], A[2][b][a]);
  r.qy = fma(sg, s[3], A[3][b][a]);
  return r;
}

// Boundary ghost of the own limit `own` at `edge` (0 W, 1 E, 2 S, 3 N), over
// the same bed.
__device__ __forceinline__ L4 ghost4(const Dev& d, int edge, double s, double t, const L4& own) {
  double h = own.h, qx = own.qx, qy = own.qy;
  ghost(d, edge, s, t, h, qx, qy);
  L4 r;
  r.eta = h + (own.eta - own.h);
  r.h = h;
  r.qx = qx;
  r.qy = qy;
  return r;
}

// Revision of a face (Sec. 2.2.2) from its lower (a) and upper (b) limits and
// the flux across it; hb takes the upper side's revised depth.  h* + z* is the side's
// own free surface on either side (z* lowered where the free surface lies below it), so
// the update needs no bed levels (fv_tile).
__device__ __forceinline__ Face face(const L4& a, const L4& b, bool ydir, double g, double tol,
                                     int flux, double& hb) {
  const double zs = max2(a.eta - a.h, b.eta - b.h);
  const double ha = pos_part(a.eta - zs);
  hb = pos_part(b.eta - zs);
  // q* = h* u with u of the limit (tol rule on the limit's depth); the flux
  // then takes its velocities from the revised state by the same rule, so a
  // face depth h* at or below tol_dry moves no water by advection
  double una = 0.0, uta = 0.0, unb = 0.0, utb = 0.0;
  if (above(a.h, tol)) {
    const double ih = rcp64(a.h);
    una = (ydir ? a.qy : a.qx) * ih;
    uta = (ydir ? a.qx : a.qy) * ih;
  }
  if (above(b.h, tol)) {
    const double ih = rcp64(b.h);
    unb = (ydir ? b.qy : b.qx) * ih;
    utb = (ydir ? b.qx : b.qy) * ih;
  }
  const double qna = ha * una, qta = ha * uta, qnb = hb * unb, qtb = hb * utb;
  Flux F;
  if (flux == 1) {
    if (!above(ha, tol)) { una = 0.0; uta = 0.0; }
    if (!above(hb, tol)) { unb = 0.0; utb = 0.0; }
    F = roe(ha, qna, qta, una, uta, hb, qnb, qtb, unb, utb, g, tol);
  } else {
    F = hll(ha, qna, qta, una, uta, hb, qnb, qtb, unb, utb, g, tol);
  }
  return Face{F.h, F.n, F.t, F.dp, ha};
}

// One FV stage on the 16 x 8 part (bx, by) of tile `tile`.  Stage 1: T = S + dt L(S) (all
// of FV1's update); stage 2 (FV2): S = (S + T + dt L(T)) / 2.  A dry cell
// keeps no discharge.  Accumulates the boundary inflow rate, and in the last
// stage the Courant rate and the non-finite / non-quiescent flags, of the
// thread's cell.
template <bool ORDER2, int STAGE>
__device__ __forceinline__ void fv_tile(const Dev& d, Smem& sm, int bx, int by, int tile,
                                        double& brate, double& lam, bool& bad, bool& nonq) {
  const Scalars* sc = d.sc;
  const int tid = threadIdx.y * TX + threadIdx.x;
  int tx, ty;
  warp_cell<TX>(tx, ty);
  const int i0 = bx * TX, j0 = by * TY, i = i0 + tx, j = j0 + ty;
  const int nx = d.nx, ny = d.ny;
  const bool act = i < nx && j < ny;
  const long long P = d.plane, c = (long long)j * d.pitch + i;
  const double dt = sc->dt;
  const double ts = STAGE == 1 ? sc->t : sc->t + dt;
  const double* __restrict__ In = STAGE == 1 ? d.S : d.T;
  const double g = d.g, tol = d.tol;
  const bool every = !d.tiles.skip || d.tiles.all_forced || d.tiles.forced[tile];
  if (tid == 0) {
    const double k = STAGE == 1 ? dt : 0.5 * dt;
    sm.k = StageK{-k * d.inv_dx, -k * d.inv_dy, 0.0, 0.0, -0.5 * g * k * d.inv_dx,
                  -0.5 * g * k * d.inv_dy};
  }

  // averages of the tile and its 2-cell halo
  for (int q = tid; q < HX * HY; q += TX * TY) {
    const int a = q % HX, b = q / HX;
    const int gi = i0 - 2 + a, gj = j0 - 2 + b;
    double h = 0.0, z = 0.0, qx = 0.0, qy = 0.0;
    if (gi >= 0 && gi < nx && gj >= 0 && gj < ny) {
      const long long cc = (long long)gj * d.pitch + gi;
      h = In[H0 * P + cc]; z = d.Z[cc]; qx = In[QX0 * P + cc]; qy = In[QY0 * P + cc];
    }
    sm.u.A[0][b][a] = h + z;
    sm.u.A[1][b][a] = h;
    sm.u.A[2][b][a] = qx;
    sm.u.A[3][b][a] = qy;
  }
  __syncthreads();

  const int a = tx + 2, b = ty + 2;
  const double(*A)[HY][HX] = sm.u.A;
  bool b_me = act && every;
  if (act && !every) {
    auto moves = [&](int aa, int bb) {
      return fv_moves(A[0][bb][aa], A[1][bb][aa], A[2][bb][aa], A[3][bb][aa], tol);
    };
    b_me = moves(a, b) || moves(a - 1, b) || moves(a + 1, b) || moves(a, b - 1) || moves(a, b + 1);
  }
  sm.cls[ty][tx] = (unsigned char)(act ? (b_me ? 2 : 1) : 0);
  __syncthreads();
  const bool b_w = tx > 0 && sm.cls[ty][tx - 1] == 2, b_e = tx + 1 < TX && sm.cls[ty][tx + 1] == 2;
  const bool b_s = ty > 0 && sm.cls[ty - 1][tx] == 2, b_n = ty + 1 < TY && sm.cls[ty + 1][tx] == 2;

  // limits of the computed cells and of their neighbours; the steps of the own free
  // surface between opposite faces are the slopes of eta
  L4 W = {}, S = {};
  double ex = 0.0, ey = 0.0;
  if (act && (b_me || b_w || b_e || b_s || b_n)) {
    double s[4];
    slopes4<ORDER2>(A, a, b, 1, 0, i == 0 || i == nx - 1, tol, s);
    ex = s[0];
    sm.e[ty][tx] = lim4(A, a, b, s, 0.5);
    W = lim4(A, a, b, s, -0.5);
    slopes4<ORDER2>(A, a, b, 0, 1, j == 0 || j == ny - 1, tol, s);
    ey = s[0];
    sm.n[ty][tx] = lim4(A, a, b, s, 0.5);
    S = lim4(A, a, b, s, -0.5);
  }
  // the limits beyond the tile, one per thread of the last 2 (TX + TY) threads: west and
  // east columns, south and north rows, on one code path (as the DG2 stages)
  const int ni = nx - i0 < TX ? nx - i0 : TX, nj = ny - j0 < TY ? ny - j0 : TY;
  {
    const int t = TX * TY - 1 - tid;
    const int kind = t < TY ? 0 : t < 2 * TY ? 1 : t < 2 * TY + TX ? 2 : 3;
    const int q = kind == 0 ? t : kind == 1 ? t - TY : kind == 2 ? t - 2 * TY : t - 2 * TY - TX;
    const int ci = kind == 0 ? 0 : kind == 1 ? ni - 1 : q;
    const int cj = kind <= 1 ? q : kind == 2 ? 0 : nj - 1;
    if (t < 2 * (TX + TY) && q < (kind <= 1 ? nj : ni) && sm.cls[cj][ci] == 2) {
      const int dx = kind <= 1 ? 1 : 0, dy = 1 - dx, side = kind & 1;
      const int gi = i0 + ci, gj = j0 + cj;
      const bool at_edge = dx ? (side ? gi == nx - 1 : gi == 0) : (side ? gj == ny - 1 : gj == 0);
      // the neighbour across the face, or at an edge the tile cell itself
      const int st = at_edge ? 0 : (side ? 1 : -1);
      const int la = ci + 2 + dx * st, lb = cj + 2 + dy * st;
      const int li = gi + dx * st, lj = gj + dy * st;
      double s[4];
      slopes4<ORDER2>(A, la, lb, dx, dy, dx ? li == 0 || li == nx - 1 : lj == 0 || lj == ny - 1,
                      tol, s);
      L4 r = lim4(A, la, lb, s, (at_edge ? side != 0 : side == 0) ? 0.5 : -0.5);
      if (at_edge) r = ghost4(d, kind, dx ? (gj + 0.5) * d.dy : (gi + 0.5) * d.dx, ts, r);
      (kind == 0 ? sm.hw : kind == 1 ? sm.he : kind == 2 ? sm.hs : sm.hn)[q] = r;
    }
  }
  __syncthreads();  // the staged averages are dead past here (the faces reuse them)

  // one revision and one flux per face a computed cell uses: each thread its west and
  // south faces, then the tile's east and north edge faces one per thread
  double hW = 0.0, hS = 0.0;  // own revised depths there
  if (act && (b_me || b_w)) {
    const Face f = face(tx > 0 ? sm.e[ty][tx - 1] : sm.hw[ty], W, false, g, tol, d.flux, hW);
    sm.u.f.fx[ty][tx] = f;
    if (i == 0) brate += f.h * d.dy;
  }
  if (act && (b_me || b_s)) {
    const Face f = face(ty > 0 ? sm.n[ty - 1][tx] : sm.hs[tx], S, true, g, tol, d.flux, hS);
    sm.u.f.fy[ty][tx] = f;
    if (j == 0) brate += f.h * d.dx;
  }
  {
    const int t = TX * TY - 1 - tid;
    const bool yf = t >= TY;
    const int q = yf ? t - TY : t;
    if ((yf ? q < ni : q < nj) && (yf ? sm.cls[nj - 1][q] : sm.cls[q][ni - 1]) == 2) {
      double hb;
      const Face f = face(yf ? sm.n[nj - 1][q] : sm.e[q][ni - 1], yf ? sm.hn[q] : sm.he[q], yf, g,
                          tol, d.flux, hb);
      *(yf ? &sm.u.f.fy[nj][q] : &sm.u.f.fx[q][ni]) = f;
      if (yf ? j0 + nj == ny : i0 + ni == nx) brate -= f.h * (yf ? d.dx : d.dy);
    }
  }
  __syncthreads();

  if (act) {
    double h = d.S[H0 * P + c], qx = d.S[QX0 * P + c], qy = d.S[QY0 * P + c];
    if (STAGE == 2) {
      h = half64(h + d.T[H0 * P + c]);
      qx = half64(qx + d.T[QX0 * P + c]);
      qy = half64(qy + d.T[QY0 * P + c]);
    }
    if (b_me) {
      // Eq. 8 with the own pressures in the bed terms: g / 2 (hE + hW) times the step of
      // the own free surface between the faces (see Flux)
      const StageK K = sm.k;
      const Face &fw = sm.u.f.fx[ty][tx], &fe = sm.u.f.fx[ty][tx + 1];
      const Face &fs = sm.u.f.fy[ty][tx], &fn = sm.u.f.fy[ty + 1][tx];
      h += fma(K.dx, fe.h - fw.h, K.dy * (fn.h - fs.h));
      qx += fma(K.dx, fe.n - (fw.n + fw.dp), fma(K.dy, fn.t - fs.t, K.bx * ex * (fe.ha + hW)));
      qy += fma(K.dx, fe.t - fw.t, fma(K.dy, fn.n - (fs.n + fs.dp), K.by * ey * (fn.ha + hS)));
      const double k = STAGE == 1 ? dt : 0.5 * dt;
      if (d.rain != 0.0 && ts >= d.rain_t0 && ts < d.rain_t1) h += k * d.rain;
      if (c == d.src_idx) h += k * (d.qp * d.inv_dx * d.inv_dy);
    }
    if (!above(h, tol)) { qx = 0.0; qy = 0.0; }
    double* O = STAGE == 1 ? d.T : d.S;
    O[H0 * P + c] = h;
    O[QX0 * P + c] = qx;
    O[QY0 * P + c] = qy;
    if (STAGE == 2 || !ORDER2) {
      lam = cell_rate(d, h, qx, qy);
      bad = bad || !(isfinite(h) && isfinite(qx) && isfinite(qy)) || h < -1.0;
      nonq = above(h, tol) || nonzero(qx) || nonzero(qy);
    }
  }
}

// The FV stage kernels over the step's tile lists (one block per entry, as
// the DG2 stage kernels).  Stage 1 also copies the frontier tiles' averages
// into T for a computed neighbour's halo.  The last stage (FV2's second, FV1's
// only) writes the tiles' quiescence flags and the Courant rate; FV1's stage
// leaves its result in T for fv1_commit_kernel.
template <bool ORDER2, int STAGE>
static __global__ void __launch_bounds__(TX* TY, 4) fv_stage_kernel(Dev d) {
  __shared__ Smem sm;
  Scalars* sc = d.sc;
  if (sc->done) return;
  constexpr bool last = STAGE == 2 || !ORDER2;
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int ntx = d.tiles.ntx;
  const int n_act = sc->n_act;
  const bool all = sc->list_all != 0;
  double lam = 0.0;
  bool bad = false;
  const int e = blockIdx.x / PARTS, part = blockIdx.x % PARTS;
  if (STAGE == 2 && e >= n_act) return;
  if (e < n_act) {
    const int tile = all ? e : list_tile(d.tiles, sc, e);
    const int tbx = tile % ntx, by = tile / ntx, bx = tbx * PARTS + part;
    double brate = 0.0;
    bool nonq = false;
    if (bx * TX < d.nx) fv_tile<ORDER2, STAGE>(d, sm, bx, by, tile, brate, lam, bad, nonq);
    if (tbx == 0 || by == 0 || tbx == ntx - 1 || by == d.tiles.nty - 1) {
      const double bsum = block_sum<TX * TY>(brate, sm.red);
      if (tx == 0 && ty == 0) {
        d.bpart[((STAGE - 1) * d.tiles.ntiles + tile) * PARTS + part] = bsum;
        // FV1's one stage counts for both slots of the step's ledger average
        if (!ORDER2) d.bpart[(d.tiles.ntiles + tile) * PARTS + part] = bsum;
      }
    }
    if (last) {
      const int any_nonq = __syncthreads_or(nonq);
      if (tx == 0 && ty == 0) d.tiles.flag[tile * PARTS + part] = any_nonq ? 1 : 0;
    }
    __syncthreads();
  }
  if (STAGE == 1) {
    const int f = e - n_act;
    if (f >= 0 && f < sc->n_front) {
      const int tile = d.tiles.front[f];
      const int i = (tile % ntx * PARTS + part) * TX + tx, j = (tile / ntx) * TY + ty;
      if (i < d.nx && j < d.ny) {
        const long long P = d.plane, c = (long long)j * d.pitch + i;
        d.T[H0 * P + c] = d.S[H0 * P + c];
        d.T[QX0 * P + c] = d.S[QX0 * P + c];
        d.T[QY0 * P + c] = d.S[QY0 * P + c];
      }
    }
  }
  if (!last) return;
  if (__syncthreads_or(bad) && tx == 0 && ty == 0) sc->nonfinite = 1;
  const double bl = block_max<TX * TY>(lam, sm.red);
  if (tx == 0 && ty == 0 && bl > 0.0)
    atomicMax(&sc->lam_bits, (unsigned long long)__double_as_longlong(bl));
}

// FV1's end of step: S = T on the computed tiles.
static __global__ void __launch_bounds__(TX* TY) fv1_commit_kernel(Dev d) {
  const Scalars* sc = d.sc;
  if (sc->done) return;
  const int n_act = sc->n_act, e = blockIdx.x / PARTS, part = blockIdx.x % PARTS;
  if (e >= n_act) return;
  const int ntx = d.tiles.ntx;
  const int tile = sc->list_all ? e : list_tile(d.tiles, sc, e);
  const int i = (tile % ntx * PARTS + part) * TX + threadIdx.x, j = (tile / ntx) * TY + threadIdx.y;
  if (i >= d.nx || j >= d.ny) return;
  const long long P = d.plane, c = (long long)j * d.pitch + i;
  d.S[H0 * P + c] = d.T[H0 * P + c];
  d.S[QX0 * P + c] = d.T[QX0 * P + c];
  d.S[QY0 * P + c] = d.T[QY0 * P + c];
}

}  // namespace fv
}  // namespace dg2
