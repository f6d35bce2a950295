// sweep64.cu -- the transport / relaxation / moments sweep of FP64 cases on
// uniform grids (2D and 3D, with or without a body and domain walls).
//
// Same arithmetic as the FP32 sweeps (Sec. 2.2 Eqs. reconstruction and limiter,
// the Shakhov equilibria of Sec. 2.1 and Sec. 4, forward Euler, Eqs. moments1-3
// by quadrature).  What bounds it: GB300 has two FP64 lanes per SM and clock
// (1.06 TFLOP/s measured, an FMA as two), 64 times fewer than FP32 lanes, so the
// number of FP64 instructions per pair is the time, and integer work, loads
// and shuffles beside them are nearly free.  The layout follows from that:
//
//   * every face value is formed once.  A warp owns a tile of cells (2D: 16
//     columns, its two half-warps taking two rows of velocities; 3D: 8 x 4
//     columns), one cell per lane, and a group of up to eight velocities of one
//     x row of the velocity grid (one sign of xi_x).  It marches along the last
//     axis in the direction of the group's velocities: the inflow face and
//     the upwind difference of a row are the previous row's, kept in registers;
//     the inflow faces along x and y come from the upwind neighbour's lane by
//     shuffle, those of the tile's upwind edge are spread over the lanes (one
//     value per lane) once per row;
//   * the limiter's quotient takes the hardware's approximate reciprocal and
//     one third-order Householder step (error 2^-60 from the seed's 2^-20)
//     instead of a division, and is skipped where no lane of the warp has
//     slopes of one sign;
//   * the velocity grid is a tensor product, so the equilibrium's exponential is
//     a product of one exponential per axis: a small kernel tabulates, per cell
//     and axis node, that factor, the node's share of the heat-flux term and of
//     c^2 / T, and the powers of c for the sums (nvx + nvy + nvz exponentials per
//     cell instead of nvx nvy nvz);
//   * the moment sums of a lane run over x only (sums of w h c_x^j, j <= 3): the
//     factors of the other axes are constant along the group and enter once
//     per group and row;
//   * the four warps of a block take four groups of one march direction; their
//     sums are added in shared memory, row by row and in a fixed order, over all
//     the groups the block takes (a compensated sum).
//
// Measured per step, tables included, on a state with slopes everywhere: 128^2
// cells x 40^2 velocities between walls 3.12 ms (the sweep that formed every
// face twice and divided took 9.55), 24^3 cells x 12^3 velocities 2.60 ms (7.48),
// 48^2 x 24^2 0.193 ms (0.54).  2 to 4% of these go into roundings: f^{n+1} rounded
// once, compensated sums, the tables' exact products (without them the rms error
// of f against extended precision was 1.2 to 1.4 times that of the sweep that
// divided, of the sums up to 1.7 times; now 0.7 to 0.9 and 0.8 to 1.1).  Kept out, at
// 3.02 and 2.44 ms: three blocks per
// SM (168 registers, spills: 4.29 ms), in 2D the upwind difference along x by
// shuffle (3.18 ms; in 3D it pays, 2.43 against 2.65 ms), the faces of a velocity
// as parallel chains under one vote (3.21 ms: fewer are skipped).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>
#include <vector>

#include "ctx.h"

namespace ibdvm {
namespace {

constexpr int W64 = 4;        // warps of a block, one group of velocities each
constexpr int KG = 8;         // velocities of a group at most
constexpr int T0 = 6, TP = 4; // table entries per x node (E, C, t, w c, w c^2, w c^3), per other node (E, C, t, c)
constexpr unsigned kAll = 0xffffffffu;

template <int D> struct Cfg64 {
  static constexpr int NC = (D == 2) ? 2 : 1;
  static constexpr int NM = (D == 2) ? 9 : 14;
  static constexpr int CX = (D == 2) ? 16 : 8;    // columns of a tile along x
  static constexpr int CT = (D == 2) ? 16 : 32;   // columns of a tile
  static constexpr int NH = (D == 2) ? 4 : 12;    // upwind edge values of a tile per velocity (2D: 2 rows x 2 components)
  static constexpr int MAXROWS = (D == 2) ? 32 : 12;
  static size_t smem(int rows) {
    return (size_t)(rows * NM * CT + 2 * W64 * NM * 32 + 2 * W64 * NH * KG) * sizeof(double) +
           (size_t)rows * NM * CT * sizeof(int);
  }
};

// a group of velocities: cnt of one x row from natural index k[0], and in 2D the
// same nodes of a second y row from k[1] (-1: none); sgn: bit a when
// component a is negative
struct Grp64 {
  int k[2], cnt, kx, ky[2], kz, sgn;
};

struct Sweep64Args {
  const double *__restrict__ f;
  double *__restrict__ fn;
  const double *__restrict__ mac;
  double *__restrict__ tab0;       // [cell - cbase][nv_x][T0]
  double *__restrict__ tabp;       // [cell - cbase][nv_y (+ nv_z)][TP]
  const double *__restrict__ xi1;  // per axis node, the axes one after the other: the component,
  const double *__restrict__ av;   // dt |xi| / dx,
  const double *__restrict__ wv;   // and the node's width
  const Grp64 *__restrict__ grp;
  const uint8_t *__restrict__ cmask;
  const int *__restrict__ dslot, *__restrict__ dlinks;
  const double *__restrict__ lval, *__restrict__ finf, *__restrict__ whalo;
  double *__restrict__ part;       // [nchunk][NM][ncell]
  long long ncell, cbase, ccount;  // the slab's cells [cbase, cbase + ccount)
  long long woff[6];
  int n[3], no[3], nvx[3];
  int nvp, wmask, rows, r0, r1;    // the slab's rows [r0, r1) of the last axis
  int nbatch, per;                 // batches of W64 groups, per chunk
};

// ---------------------------------------------------------------------------
// the equilibrium's tables (one thread per cell and axis node)
// ---------------------------------------------------------------------------

// With c = xi - U: e = dt/tau rho/(pi T)^(..) exp(-c^2/T) is a product over the
// axes, C = 2 A c.q and t = c^2/T - 2 (2D) or - 5/2 (3D) are sums; then
// dt/tau H = e (1 + C t), dt/tau B = T/2 (e (1 + C t) + e C).
template <int D> __global__ void __launch_bounds__(256) eq64_table_kernel(Sweep64Args A) {
  const int nt = A.nvx[0] + A.nvx[1] + ((D == 3) ? A.nvx[2] : 0);
  const long long total = A.ccount * nt;
  for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < total;
       q += (long long)gridDim.x * blockDim.x) {
    const long long ci = q / nt;
    const int j = (int)(q % nt), a = (j < A.nvx[0]) ? 0 : (j < A.nvx[0] + A.nvx[1]) ? 1 : 2;
    const double *M = A.mac + (A.cbase + ci) * kMac;
    const double c = A.xi1[j] - M[kU0 + a], invT = M[kInvT], c2 = c * c, z = c2 * invT;
    double E = exp(-z);
    const double C = 2.0 * M[kShA] * M[kQ0 + a] * c;
    if (a == 0) {
      E *= M[kDtTau] * M[kPre];
      // w c, w c^2 and w c^3, rounded once each (every velocity of the node carries
      // that rounding, so it does not average out): c as c + cl (Knuth's TwoSum),
      // products with their errors (FMA)
      const double w = A.wv[j], U = M[kU0], cb = c - A.xi1[j], cl = (A.xi1[j] - (c - cb)) - (U + cb);
      const double c2l = fma(2.0 * c, cl, fma(c, c, -c2));
      const double h1 = w * c, w1 = h1 + fma(w, cl, fma(w, c, -h1));
      const double h2 = w * c2, e2 = fma(w, c2l, fma(w, c2, -h2)), w2 = h2 + e2;
      const double h3 = h2 * c, w3 = h3 + fma(h2, cl, fma(e2, c, fma(h2, c, -h3)));
      double2 *o = reinterpret_cast<double2 *>(A.tab0 + (ci * A.nvx[0] + j) * T0);
      o[0] = make_double2(E, C);
      o[1] = make_double2(z - ((D == 2) ? 2.0 : 2.5), w1);
      o[2] = make_double2(w2, w3);
    } else {
      double2 *o = reinterpret_cast<double2 *>(A.tabp + (ci * (nt - A.nvx[0]) + j - A.nvx[0]) * TP);
      o[0] = make_double2(E, C);
      o[1] = make_double2(z, c);
    }
  }
}

// ---------------------------------------------------------------------------
// the sweep
// ---------------------------------------------------------------------------

// the hardware's reciprocal approximation (about 20 bits; subnormals as zero)
__device__ __forceinline__ double rcp_seed(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  return r;
}

// Downwind face f + ab / (a + b) for one-sided differences a, b of one sign,
// else f (half the van Leer slope, Eq. limiter).  The sign and the range of
// ab are read from its high word, off the FP64 pipe: a product below 2^-1042 (a
// subnormal number whose high word is zero), an infinite one or a NaN counts as no
// slope.  Called by whole warps.
__device__ __forceinline__ double face64(double f, double a, double b) {
  const double p = a * b;
  const bool slope = (unsigned)(__double2hiint(p) - 1) < 0x7fefffffu;
  if (!__any_sync(kAll, slope)) return f;
  const double s = a + b;
  double r = rcp_seed(s);
  const double e = fma(-s, r, 1.0); // 1/s = r (1 + e + e^2 + ...)
  r = fma(r, fma(e, e, e), r);
  const double v = fma(p, r, f);
  return slope ? v : f;
}

// the row [nvp][NC] of the value that cell c at ijk with flags fl sees across its
// face (a, s): a ghost's link value, the domain halo, or the neighbour's f
template <int D>
__device__ __forceinline__ const double *seen_row(const Sweep64Args &A, long long c, const int *ijk, unsigned fl, int a,
                                                  int s) {
  constexpr int NC = Cfg64<D>::NC;
  const int i = 2 * a + (s > 0);
  const int q = ijk[a] + s;
  if (q < 0 || q >= A.n[a]) {
    if (!((A.wmask >> i) & 1)) return A.finf;
    const long long slot = (a == 0) ? ijk[1] + (long long)A.n[1] * ijk[2]
                           : (a == 1) ? ijk[0] + (long long)A.n[0] * ijk[2] : ijk[0] + (long long)A.n[0] * ijk[1];
    return A.whalo + (size_t)(A.woff[i] + slot) * A.nvp * NC;
  }
  if (!(fl & kNotFluidCell) && ((fl >> i) & 1u)) {
    const int sl = A.dslot[c];
    const int l = (sl >= 0) ? A.dlinks[sl * 6 + i] : -1;
    return (l >= 0) ? A.lval + (size_t)l * A.nvp * NC : A.finf;
  }
  const long long st = (a == 0) ? 1LL : (a == 1) ? (long long)A.n[0] : (long long)A.n[0] * A.n[1];
  return A.f + (size_t)(c + s * st) * A.nvp * NC;
}

template <int NC> __device__ __forceinline__ void ld(const double *p, double *v) {
  if constexpr (NC == 2) {
    const double2 t = __ldg(reinterpret_cast<const double2 *>(p));
    v[0] = t.x;
    v[1] = t.y;
  } else {
    v[0] = __ldg(p);
  }
}

template <int D> __global__ void __launch_bounds__(32 * W64, 2) sweep64_kernel(Sweep64Args A) {
  using C = Cfg64<D>;
  constexpr int NC = C::NC, NM = C::NM, CT = C::CT, CX = C::CX, LA = D - 1;
  extern __shared__ double smem[];
  double *acc = smem;                        // [row][NM][CT], owned by fixed threads
  double *red = acc + A.rows * NM * CT;      // [2][W64][NM][32]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double *hb = red + 2 * W64 * NM * 32 + warp * 2 * C::NH * KG; // inflow faces at this warp's tile's upwind edge,
  double *hd = hb + C::NH * KG;                                 // and the differences across them
  int *low = reinterpret_cast<int *>(red + 2 * W64 * NM * 32 + W64 * 2 * C::NH * KG); // of acc: the sums' errors
  const int nx = A.n[0], ny = (D == 3) ? A.n[1] : 1, nl = A.n[LA];
  const int ntx = (nx + CX - 1) / CX, nty = (D == 3) ? (ny + 3) / 4 : 1;
  const int tile = blockIdx.x % (ntx * nty), rr = blockIdx.x / (ntx * nty);
  const int x0 = (tile % ntx) * CX, y0 = (tile / ntx) * 4;
  const int ya = A.r0 + rr * A.rows, yb = min(A.r1, ya + A.rows), M = yb - ya;
  const int i = lane & (CX - 1), jy = (D == 3) ? lane >> 3 : 0, half = (D == 2) ? lane >> 4 : 0;
  const bool col = x0 + i < nx && y0 + jy < ny; // a column of the domain; the others repeat the last one's reads
  const int ie = min(CX - 1, nx - 1 - x0), je = (D == 3) ? min(3, ny - 1 - y0) : 0; // the tile's last column and row
  int ijk[3] = {min(x0 + i, nx - 1), (D == 3) ? min(y0 + jy, ny - 1) : 0, 0};
  const long long ps = (long long)nx * ny, col0 = ijk[0] + (long long)nx * ijk[1];
  const int npn = A.nvx[1] + ((D == 3) ? A.nvx[2] : 0); // nodes of the other axes

  for (int e = threadIdx.x; e < M * NM * CT; e += 32 * W64) {
    acc[e] = 0.0;
    low[e] = 0;
  }
  __syncthreads();
  int par = 0;
  const int b1 = min(A.nbatch, ((int)blockIdx.y + 1) * A.per);
  for (int bt = blockIdx.y * A.per; bt < b1; ++bt) {
    const Grp64 g = A.grp[bt * W64 + warp];
    const int cnt = g.cnt;
    const int sx = (g.sgn & 1) ? -1 : 1, sy = (g.sgn & 2) ? -1 : 1, d = ((g.sgn >> LA) & 1) ? -1 : 1;
    const bool own2 = half == 0 || g.k[1] >= 0;
    const int kb = (half && g.k[1] >= 0) ? g.k[1] : g.k[0];
    const int ky = (half && g.k[1] >= 0) ? g.ky[1] : g.ky[0];
    const int p0 = (d > 0) ? ya : yb - 1;
    const double ayv = A.av[A.no[1] + ky], azv = (D == 3) ? A.av[A.no[2] + g.kz] : 0.0;
    const double wrow = A.wv[A.no[1] + ky] * ((D == 3) ? A.wv[A.no[2] + g.kz] : 1.0);
    const double al = (D == 3) ? azv : ayv; // along the march

    // the march axis, per velocity: the value, the difference from the
    // previous row's, and the previous row's face value (this row's inflow)
    double F[KG][NC], Dd[KG][NC], P[KG][NC];
    if (cnt > 0) {
      const double *fo = A.f + (size_t)(col0 + ps * p0) * A.nvp * NC;
      const int r = p0 - d;
      ijk[LA] = p0;
      const double *fp = nullptr, *fpp = nullptr;
      const bool out = r < 0 || r >= nl;
      if (out) {
        fp = fpp = seen_row<D>(A, col0 + ps * p0, ijk, 0u, LA, -d);
      } else {
        const long long cr = col0 + ps * r;
        ijk[LA] = r;
        fp = A.f + (size_t)cr * A.nvp * NC;
        fpp = seen_row<D>(A, cr, ijk, A.cmask[cr], LA, -d);
      }
#pragma unroll
      for (int j = 0; j < KG; ++j)
        if (j < cnt) {
          double vp[NC], vpp[NC];
          ld<NC>(fo + (size_t)(kb + j) * NC, F[j]);
          ld<NC>(fp + (size_t)(kb + j) * NC, vp);
          ld<NC>(fpp + (size_t)(kb + j) * NC, vpp);
          // a halo row has its value and no slope (vp - vpp is zero there); a ghost in
          // row p0 takes no inflow, and the row after it replaces its own
#pragma unroll
          for (int m = 0; m < NC; ++m) {
            Dd[j][m] = F[j][m] - vp[m];
            P[j][m] = face64(vp[m], vp[m] - vpp[m], Dd[j][m]);
          }
        }
    }

    for (int m0 = 0; m0 < M; ++m0, par ^= 1) {
      const int p = p0 + d * m0;
      double *rw = red + (par * W64 + warp) * NM * 32 + lane;
      if (cnt > 0) {
        const long long c = col0 + ps * p;
        ijk[LA] = p;
        const unsigned fl = A.cmask[c];
        const bool fluid = col && !(fl & kNotFluidCell);
        const double *xd = seen_row<D>(A, c, ijk, fl, 0, sx), *yd = nullptr;
        if constexpr (D == 3) yd = seen_row<D>(A, c, ijk, fl, 1, sy);
        const double *zd = seen_row<D>(A, c, ijk, fl, LA, d);
        const unsigned gf = fluid ? fl : 0u;
        const bool gx = (gf >> (sx < 0)) & 1u, gy = (D == 3) && ((gf >> (2 + (sy < 0))) & 1u),
                   gz = (gf >> (2 * LA + (d < 0))) & 1u; // a ghost upwind
        const bool ghosts = __any_sync(kAll, gx || gy || gz);
        const double *xu = (gx || D == 2) ? seen_row<D>(A, c, ijk, fl, 0, -sx) : xd;
        const double *yu = gy ? seen_row<D>(A, c, ijk, fl, 1, -sy) : xd;
        const double *zu = gz ? seen_row<D>(A, c, ijk, fl, LA, -d) : zd;
        const bool ex = i == ((sx > 0) ? 0 : ie), ey = D == 3 && jy == ((sy > 0) ? 0 : je);

        // the faces of the cells upwind of the tile towards it and the
        // differences across them, one value per lane: beyond the domain edge the
        // halo's value and no slope; where a cell is not fluid they are not used
        {
          const int nhv = C::NH * cnt;
#pragma unroll
          for (int q0 = 0; q0 < C::NH * KG; q0 += 32)
            if (q0 < nhv) {
              const int q = q0 + lane;
              const int j = min(q / C::NH, cnt - 1), h = q % C::NH;
              int hi[3] = {0, 0, 0}, k, cm = 0, a = 0, s = sx; // the tile's edge cell
              hi[LA] = p;
              if constexpr (D == 2) { // h: half-warp row and component
                cm = h & 1;
                k = (((h >> 1) && g.k[1] >= 0) ? g.k[1] : g.k[0]) + j;
                hi[0] = x0 + ((sx > 0) ? 0 : ie);
              } else {
                k = g.k[0] + j;
                if (h < 4) { // an x face: row h of the tile
                  hi[0] = x0 + ((sx > 0) ? 0 : ie);
                  hi[1] = min(y0 + h, ny - 1);
                } else { // a y face: column h - 4
                  a = 1;
                  s = sy;
                  hi[0] = min(x0 + h - 4, nx - 1);
                  hi[1] = y0 + ((sy > 0) ? 0 : je);
                }
              }
              const size_t o = (size_t)k * NC + cm;
              const long long ec = hi[0] + (long long)nx * ((D == 2) ? p : hi[1] + (long long)ny * p);
              const double vd = __ldg(A.f + (size_t)ec * A.nvp * NC + o);
              const double *pv = seen_row<D>(A, ec, hi, 0u, a, -s), *pu = pv;
              hi[a] -= s;
              if (hi[a] >= 0 && hi[a] < A.n[a]) {
                const long long hc = ec - s * ((a == 0) ? 1LL : (long long)nx);
                pu = seen_row<D>(A, hc, hi, A.cmask[hc], a, -s);
              }
              const double v = __ldg(pv + o), vu = __ldg(pu + o), dv = vd - v;
              const double r = face64(v, v - vu, dv);
              if (q < C::NH * KG) {
                hb[q] = r;
                hd[q] = dv;
              }
            }
          __syncwarp();
        }

        // the cell's constants of this row
        const double *Mc = A.mac + c * kMac;
        const double mt = -Mc[kDtTau], hT = (D == 2) ? Mc[kHalfT] : 0.0;
        const size_t ci = (size_t)(c - A.cbase);
        const double2 *t0 = reinterpret_cast<const double2 *>(A.tab0 + (ci * A.nvx[0] + g.kx) * T0);
        const double2 *tp = reinterpret_cast<const double2 *>(A.tabp + (ci * npn + ky) * TP);
        const double2 y0v = tp[0], y1v = tp[1];
        double Er = y0v.x, Cr = y0v.y, tr = y1v.x, cz = 0.0;
        const double cy = y1v.y;
        if constexpr (D == 3) {
          const double2 *tz = reinterpret_cast<const double2 *>(A.tabp + (ci * npn + A.nvx[1] + g.kz) * TP);
          const double2 z0 = tz[0], z1 = tz[1];
          Er *= z0.x;
          Cr += z0.y;
          tr += z1.x;
          cz = z1.y;
        }
        double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0, sb = 0.0;
        double *fo = A.fn + (size_t)c * A.nvp * NC;
        // the velocities of the group, in two copies: GEN, where a lane of the
        // warp has a ghost upwind, and plain
        auto update = [&](auto gen) {
          constexpr bool GEN = decltype(gen)::value;
#pragma unroll
          for (int j = 0; j < KG; ++j)
            if (j < cnt) {
              const size_t o = (size_t)(kb + j) * NC;
              double vxd[NC], vyd[NC], vz[NC], n[NC], vxu[NC];
              if constexpr (D == 2) ld<NC>(xu + o, vxu);
              ld<NC>(xd + o, vxd);
              ld<NC>(zd + o, vz);
              if constexpr (D == 3) ld<NC>(yd + o, vyd);
              const double2 e0 = t0[j * 3], e1 = t0[j * 3 + 1], e2 = t0[j * 3 + 2];
              const double ax = A.av[g.kx + j], wx = A.wv[g.kx + j];
              // dt / tau times the equilibrium
              const double e = e0.x * Er, Cc = e0.y + Cr, t = e1.x + tr;
              const double H = fma(e, Cc * t, e);
              // the increments of relaxation and fluxes first; f joins them last, so
              // that f^{n+1} is rounded once at its own size
              n[0] = fma(mt, F[j][0], H);
              if constexpr (D == 2) n[1] = fma(hT, fma(e, Cc, H), mt * F[j][1]);
#pragma unroll
              for (int m = 0; m < NC; ++m) {
                const double f = F[j][m];
                const int hx = (D == 2) ? j * 4 + half * 2 + m : j * 12 + jy, hy = j * 12 + 4 + i;
                double zin = P[j][m], za = Dd[j][m];
                if constexpr (D == 2) {
                  const double xo = face64(f, f - vxu[m], vxd[m] - f);
                  double xin = __shfl_sync(kAll, xo, lane - sx);
                  if (ex) xin = hb[hx];
                  if (GEN && gx) xin = 0.5 * (vxu[m] + f); // a ghost upwind: the mean (one-sided slope)
                  n[m] = fma(ax, xin - xo, n[m]);
                } else {
                  // the upwind differences are the upwind neighbours' downwind ones
                  const double dxd = vxd[m] - f, dyd = vyd[m] - f;
                  double dxu = __shfl_sync(kAll, dxd, lane - sx), dyu = __shfl_sync(kAll, dyd, lane - 8 * sy);
                  if (ex) dxu = hd[hx];
                  if (ey) dyu = hd[hy];
                  double lx = f, ly = f;
                  if constexpr (GEN) {
                    if (gx) {
                      lx = __ldg(xu + o + m);
                      dxu = f - lx;
                    }
                    if (gy) {
                      ly = __ldg(yu + o + m);
                      dyu = f - ly;
                    }
                  }
                  const double xo = face64(f, dxu, dxd), yo = face64(f, dyu, dyd);
                  double xin = __shfl_sync(kAll, xo, lane - sx), yin = __shfl_sync(kAll, yo, lane - 8 * sy);
                  if (ex) xin = hb[hx];
                  if (ey) yin = hb[hy];
                  if constexpr (GEN) {
                    if (gx) xin = 0.5 * (lx + f);
                    if (gy) yin = 0.5 * (ly + f);
                  }
                  n[m] = fma(ax, xin - xo, n[m]);
                  n[m] = fma(ayv, yin - yo, n[m]);
                }
                const double b = vz[m] - f;
                if (GEN && gz) {
                  const double lz = __ldg(zu + o + m);
                  za = f - lz;
                  zin = 0.5 * (lz + f);
                }
                const double zo = face64(f, za, b);
                P[j][m] = zo;
                Dd[j][m] = b;
                F[j][m] = vz[m];
                n[m] = fma(al, zin - zo, n[m]) + f;
              }
              if (fluid && own2) {
                if constexpr (NC == 2)
                  *reinterpret_cast<double2 *>(fo + o) = make_double2(n[0], n[1]);
                else
                  fo[o] = n[0];
              }
              s0 = fma(wx, n[0], s0);
              s1 = fma(e1.y, n[0], s1);
              s2 = fma(e2.x, n[0], s2);
              s3 = fma(e2.y, n[0], s3);
              if constexpr (D == 2) { // the second component adds to the energy and its flux
                sb = fma(wx, n[1], sb);
                s3 = fma(e1.y, n[1], s3);
              }
            }
        };
        if (ghosts)
          update(std::true_type{});
        else
          update(std::false_type{});
        if (!own2) s0 = s1 = s2 = s3 = sb = 0.0;
        __syncwarp(); // the edge values are consumed
        // the sums about the bulk velocity in the order of the finalize kernel
        const double S0 = wrow * s0, Sx = wrow * s1, Sxx = wrow * s2, S3 = wrow * s3;
        const double Sy = cy * S0, Sxy = cy * Sx, Syy = cy * Sy;
        if constexpr (D == 2) {
          const double E = fma(wrow, sb, Sxx + Syy);
          rw[0 * 32] = S0;
          rw[1 * 32] = Sx;
          rw[2 * 32] = Sy;
          rw[3 * 32] = E;
          rw[4 * 32] = Sxx;
          rw[5 * 32] = Sxy;
          rw[6 * 32] = Syy;
          rw[7 * 32] = fma(cy, Sxy, S3);
          rw[8 * 32] = cy * E;
        } else {
          const double Sz = cz * S0, Syz = cz * Sy, Szz = cz * Sz, E = Sxx + (Syy + Szz);
          rw[0 * 32] = S0;
          rw[1 * 32] = Sx;
          rw[2 * 32] = Sy;
          rw[3 * 32] = Sz;
          rw[4 * 32] = E;
          rw[5 * 32] = Sxx;
          rw[6 * 32] = Sxy;
          rw[7 * 32] = cz * Sx;
          rw[8 * 32] = Syy;
          rw[9 * 32] = Syz;
          rw[10 * 32] = Szz;
          rw[11 * 32] = fma(fma(cy, cy, cz * cz), Sx, S3);
          rw[12 * 32] = cy * E;
          rw[13 * 32] = cz * E;
        }
      } else {
#pragma unroll
        for (int m = 0; m < NM; ++m) rw[m * 32] = 0.0;
      }
      __syncthreads();
      // add the block's sums of this row (a buffer is written again two barriers later)
      // and keep what the additions round away (Kahan's sum): one such sum takes all
      // the groups of the block, a chain long enough to show in the heat flux where it
      // has more than two.  The high word of the error is enough, and needs no conversion
      double *ar = acc + (p - ya) * NM * CT;
      int *lr = low + (p - ya) * NM * CT;
      for (int e = threadIdx.x; e < NM * CT; e += 32 * W64) {
        const double *q = red + par * W64 * NM * 32 + (e / CT) * 32 + e % CT;
        static_assert(W64 == 4, "the pairwise sum below");
        auto at = [&](int w) { return (D == 2) ? q[w * NM * 32] + q[w * NM * 32 + 16] : q[w * NM * 32]; };
        const double v = (at(0) + at(1)) + (at(2) + at(3));
        const double s = ar[e];
        const int m = e / CT; // (the second moments enter times the change of U only)
        if (A.per > 2 && (m < D + 2 || m >= NM - D)) {
          const double y = v - __hiloint2double(lr[e], 0), t = s + y;
          lr[e] = __double2hiint((t - s) - y);
          ar[e] = t;
        } else {
          ar[e] = s + v;
        }
      }
    }
  }
  __syncthreads();
  for (int e = threadIdx.x; e < M * NM * CT; e += 32 * W64) {
    const int q = e % CT, m = (e / CT) % NM, p = ya + e / (CT * NM);
    const int x = x0 + q % CX, y = (D == 3) ? y0 + q / CX : 0;
    if (x < nx && y < ny)
      A.part[((size_t)blockIdx.y * NM + m) * A.ncell + x + (long long)nx * y + ps * p] = acc[e] - __hiloint2double(low[e], 0);
  }
}

Sweep64Args args64(const ibdvm_ctx *ctx) {
  const Sweep64Plan &pl = ctx->plan64;
  Sweep64Args A{};
  A.f = static_cast<const double *>(ctx->f[ctx->cur]);
  A.fn = static_cast<double *>(ctx->f[1 - ctx->cur]);
  A.mac = static_cast<const double *>(ctx->mac);
  A.xi1 = pl.nodes;
  const int nn = pl.nnode;
  A.av = pl.nodes + nn;
  A.wv = pl.nodes + 2 * nn;
  A.grp = reinterpret_cast<const Grp64 *>(pl.grp);
  A.cmask = ctx->cmask;
  A.dslot = ctx->dslot;
  A.dlinks = ctx->dlinks;
  A.lval = static_cast<const double *>(ctx->lval);
  A.finf = static_cast<const double *>(ctx->finf);
  A.whalo = static_cast<const double *>(ctx->whalo);
  A.part = ctx->part;
  A.ncell = ctx->ncell;
  for (int i = 0; i < 6; ++i) A.woff[i] = ctx->wall_off[i];
  for (int a = 0, o = 0; a < 3; ++a) {
    A.n[a] = ctx->geom.n[a];
    A.nvx[a] = ctx->geom.nvx[a];
    A.no[a] = o;
    if (a < ctx->dim) o += A.nvx[a];
  }
  A.nvp = ctx->nvp;
  A.wmask = ctx->wall_mask;
  A.rows = pl.rows;
  A.nbatch = pl.nbatch;
  A.per = pl.per;
  return A;
}

template <int D> cudaError_t launch64(ibdvm_ctx *ctx) {
  using C = Cfg64<D>;
  const Sweep64Plan &pl = ctx->plan64;
  Sweep64Args A = args64(ctx);
  const int nl = A.n[D - 1];
  const long long ps = (D == 2) ? A.n[0] : (long long)A.n[0] * A.n[1];
  const int ntx = (A.n[0] + C::CX - 1) / C::CX, nty = (D == 3) ? (A.n[1] + 3) / 4 : 1;
  const int nt = pl.nnode;
  for (A.r0 = 0; A.r0 < nl; A.r0 = A.r1) {
    A.r1 = std::min(nl, A.r0 + pl.slab);
    A.cbase = A.r0 * ps;
    A.ccount = (A.r1 - A.r0) * ps;
    A.tab0 = pl.tab;
    A.tabp = pl.tab + A.ccount * A.nvx[0] * T0;
    const long long blocks = (A.ccount * nt + 255) / 256;
    eq64_table_kernel<D><<<(unsigned)std::min<long long>(blocks, 152 * 64), 256, 0, ctx->stream>>>(A);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)(ntx * nty * ((A.r1 - A.r0 + pl.rows - 1) / pl.rows)),
                    (unsigned)((pl.nbatch + pl.per - 1) / pl.per));
    sweep64_kernel<D><<<grid, 32 * W64, C::smem(pl.rows), ctx->stream>>>(A);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// table bytes of one row of the last axis
size_t row_bytes(const Geom &G) {
  const size_t plane = (G.dim == 2) ? G.n[0] : (size_t)G.n[0] * G.n[1];
  size_t other = G.nvx[1] + ((G.dim == 3) ? G.nvx[2] : 0);
  return plane * ((size_t)G.nvx[0] * T0 + other * TP) * sizeof(double);
}

// Tables of at most this size: a larger grid is swept slab by slab (rows of the
// last axis), with one table for all
constexpr size_t kTableBytes = size_t(256) << 20;
// and of at most this share of the memory that the rest of the case leaves free
constexpr size_t kTableShare = 64;

int slab_rows(const Geom &G) {
  return (int)std::min<size_t>(G.n[G.dim - 1], std::max<size_t>(1, kTableBytes / row_bytes(G)));
}

} // namespace

// Where the direct sweep (sweep_kernel: a thread per cell and velocity, every face
// twice) is the faster one.  Its blocks are four cells and 64 velocities: up to one
// per SM it takes 25 us whatever they hold, less than a row and a march's start here
// (sweep and moments of 4^2 cells x 24^2 velocities 58 us direct, 66 here, 12^2 x 16^2
// 59 / 67; in two rounds 6^3 x 6^3 93 / 77).  And 2D grids of four columns leave three
// lanes of four idle here (4 x 512 x 24^2: 522 / 603; of five columns 696 / 607).
bool sweep64_direct(const Geom &G) {
  const long long blocks = ((G.ncell + 3) / 4) * ((G.nv + 63) / 64);
  return blocks <= 152 || (G.dim == 2 && G.n[0] <= 4);
}

void sweep64_groups(const Geom &G, std::vector<int> &out) {
  // groups of at most KG nodes of one sign along x, as even as they go; in 2D
  // two y rows of one sign each; the groups of one march sign in one list, filled
  // up with empty ones to whole batches
  std::vector<Grp64> list[2], gs;
  const int nx = G.nvx[0], ny = G.nvx[1], nz = (G.dim == 3) ? G.nvx[2] : 1;
  auto xi = [&](int kx, int ky, int kz, int a) { return G.xi[3 * (kx + (size_t)nx * (ky + (size_t)ny * kz)) + a]; };
  int negx = 0;
  while (negx < nx && xi(negx, 0, 0, 0) < 0.0) ++negx;
  for (int march = 0; march < 2; ++march) {
    // rows of the velocity grid marched this way (2D: pairs of one sign)
    struct Row {
      int ky[2], kz, sgn;
    };
    std::vector<Row> rows;
    for (int kz = 0; kz < nz; ++kz)
      for (int ky = 0; ky < ny; ++ky) {
        const bool yneg = xi(0, ky, kz, 1) < 0.0, zneg = G.dim == 3 && xi(0, ky, kz, 2) < 0.0;
        if ((G.dim == 3 ? zneg : yneg) != (march == 1)) continue;
        Row r{{ky, -1}, kz, (yneg ? 2 : 0) | (zneg ? 4 : 0)};
        if (G.dim == 2 && ky + 1 < ny && (xi(0, ky + 1, kz, 1) < 0.0) == yneg) r.ky[1] = ++ky;
        rows.push_back(r);
      }
    if (march == 1) std::reverse(rows.begin(), rows.end()); // the opposite rows at the same places
    // x runs outermost, a row's group of negative x and its mirror image next to
    // each other: a batch adds them first, so that the sums of odd moments stay
    // small (heat flux along x of a 16^2 box with 24^2 velocities: rms error 3.3e-17,
    // 5.0e-17 with four groups of one sign to a batch)
    const int lo[2] = {0, negx}, n[2] = {negx, nx - negx}, ng[2] = {(n[0] + KG - 1) / KG, (n[1] + KG - 1) / KG};
    for (int i = 0; i < std::max(ng[0], ng[1]); ++i)
      for (const Row &r : rows)
        for (int part = 0; part < 2; ++part) {
          if (i >= ng[part]) continue;
          const int q = part ? ng[1] - 1 - i : i;
          const int a = lo[part] + (int)((long long)n[part] * q / ng[part]);
          const int b = lo[part] + (int)((long long)n[part] * (q + 1) / ng[part]);
          Grp64 g{};
          for (int h = 0; h < 2; ++h) {
            const int ky = r.ky[h] < 0 ? r.ky[0] : r.ky[h];
            g.ky[h] = ky;
            g.k[h] = (r.ky[h] < 0) ? -1 : a + nx * (ky + ny * r.kz);
          }
          g.cnt = b - a;
          g.kx = a;
          g.kz = r.kz;
          g.sgn = (part ? 0 : 1) | r.sgn;
          list[march].push_back(g);
        }
    const Grp64 none{{0, -1}, 0, 0, {0, 0}, 0, march ? (G.dim == 3 ? 4 : 2) : 0};
    list[march].insert(list[march].end(), (W64 - list[march].size() % W64) % W64, none);
  }
  // the batches of the two lists, which hold opposite velocities, in turn: the sums
  // of odd moments stay small as they grow, and so do their roundings
  const size_t nb[2] = {list[0].size() / W64, list[1].size() / W64};
  for (size_t b = 0; b < std::max(nb[0], nb[1]); ++b)
    for (int march = 0; march < 2; ++march)
      if (b < nb[march]) gs.insert(gs.end(), list[march].begin() + b * W64, list[march].begin() + (b + 1) * W64);
  out.resize(gs.size() * sizeof(Grp64) / sizeof(int));
  std::copy(reinterpret_cast<const int *>(gs.data()), reinterpret_cast<const int *>(gs.data()) + out.size(), out.begin());
}

// Rows per block and batches per block: the split of least time on 152 SMs with
// two blocks each.  A block's work is its rows and the march's start (about half
// a row) times its batches; two blocks of an SM keep its FP64 pipe 86% busy, one
// alone 65% (measured), so a last round of at most one block per SM counts its
// work once over 0.65 and any other round twice over 0.86.  A chunk costs the
// finalize kernel of a small grid 0.75 to 0.9 us, 0.08 rows of a batch.
void sweep64_tiling(const Geom &G, int nbatch, int &rows, int &per) {
  const int D = G.dim, nl = slab_rows(G);
  const long long tiles = (D == 2) ? (G.n[0] + 15) / 16 : (long long)((G.n[0] + 7) / 8) * ((G.n[1] + 3) / 4);
  const int maxr = (D == 2) ? Cfg64<2>::MAXROWS : Cfg64<3>::MAXROWS;
  double best = 1e300;
  for (int most = std::min(maxr, nl); most >= 1; --most) {
    const int r = (nl + (nl + most - 1) / most - 1) / ((nl + most - 1) / most);
    const long long tr = tiles * ((nl + r - 1) / r);
    for (int pb = nbatch; pb >= 1; --pb) {
      const int nch = (nbatch + pb - 1) / pb;
      if (nch > 64) break;
      const long long blocks = tr * nch;
      const long long full = blocks / 304, rem = blocks % 304;
      const double rounds = full * (2.0 / 0.86) + (rem == 0 ? 0.0 : rem <= 152 ? 1.0 / 0.65 : 2.0 / 0.86);
      const double cost = rounds * pb * (r + 0.5) + 0.08 * nch;
      if (cost < best * (1.0 - 1e-9)) {
        best = cost;
        rows = r;
        per = pb;
      }
      if (blocks > 152 * 64) break; // enough blocks: more chunks gain nothing
    }
  }
}

int sweep64_nchunk(const Geom &G) {
  std::vector<int> g;
  sweep64_groups(G, g);
  const int nbatch = (int)(g.size() * sizeof(int) / sizeof(Grp64)) / W64;
  int rows = 0, per = 0;
  sweep64_tiling(G, nbatch, rows, per);
  return (nbatch + per - 1) / per;
}

size_t sweep64_table_bytes(const Geom &G) { return row_bytes(G) * slab_rows(G); }
size_t sweep64_row_bytes(const Geom &G) { return row_bytes(G); }

// The tables of `slab` rows (one at least), fewer where memory is short, in place
// of those there are; no work of the stream may use them
cudaError_t sweep64_tables(ibdvm_ctx *ctx, int slab) {
  const Geom &G = ctx->geom;
  Sweep64Plan &pl = ctx->plan64;
  if (pl.tab) cudaFree(pl.tab);
  pl.tab = nullptr;
  pl.tab_bytes = 0;
  const size_t rb = row_bytes(G);
  cudaError_t e;
  for (slab = std::max(slab, 1);; slab = (slab + 1) / 2) {
    void *p = nullptr;
    e = cudaMalloc(&p, rb * slab);
    pl.tab = static_cast<double *>(p);
    if (e == cudaSuccess || slab == 1) break;
    cudaGetLastError();
  }
  pl.slab = slab;
  if (e != cudaSuccess) return e;
  pl.tab_bytes = rb * slab;
  pl.rows = std::min(pl.most, slab);
  return cudaSuccess;
}

cudaError_t sweep64_prepare(ibdvm_ctx *ctx, std::vector<int> &grp, std::vector<double> &nodes) {
  const Geom &G = ctx->geom;
  Sweep64Plan &pl = ctx->plan64;
  sweep64_groups(G, grp);
  pl.nbatch = (int)(grp.size() * sizeof(int) / sizeof(Grp64)) / W64;
  sweep64_tiling(G, pl.nbatch, pl.most, pl.per);
  // axis nodes: the component, dt |xi| / dx and the node's width
  pl.nnode = G.nvx[0] + G.nvx[1] + ((G.dim == 3) ? G.nvx[2] : 0);
  nodes.assign(3 * (size_t)pl.nnode, 0.0);
  for (int a = 0, o = 0; a < G.dim; ++a) {
    const size_t st = (a == 0) ? 1 : (a == 1) ? G.nvx[0] : (size_t)G.nvx[0] * G.nvx[1];
    for (int i = 0; i < G.nvx[a]; ++i, ++o) {
      const double x = G.xi[3 * (i * st) + a];
      nodes[o] = x;
      nodes[pl.nnode + o] = G.dt * ((x < 0.0) ? -x : x) / G.dx[a];
      nodes[2 * (size_t)pl.nnode + o] = G.bhi[3 * (i * st) + a] - G.blo[3 * (i * st) + a];
    }
  }
  size_t freeb = 0, totb = 0;
  cudaError_t e = cudaMemGetInfo(&freeb, &totb);
  if (e == cudaSuccess) e = sweep64_tables(ctx, (int)std::min<size_t>(slab_rows(G), freeb / kTableShare / row_bytes(G)));
  if (e != cudaSuccess) return e;
  e = (G.dim == 2) ? cudaFuncSetAttribute(sweep64_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)Cfg64<2>::smem(Cfg64<2>::MAXROWS))
                   : cudaFuncSetAttribute(sweep64_kernel<3>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)Cfg64<3>::smem(Cfg64<3>::MAXROWS));
  return e;
}

int sweep64_launches(const ibdvm_ctx *ctx) {
  const int nl = ctx->geom.n[ctx->dim - 1];
  return 2 * ((nl + ctx->plan64.slab - 1) / ctx->plan64.slab);
}

cudaError_t sweep64_launch(ibdvm_ctx *ctx) {
  if (!ctx->plan64.tab) return cudaErrorMemoryAllocation;
  return (ctx->dim == 2) ? launch64<2>(ctx) : launch64<3>(ctx);
}

} // namespace ibdvm
