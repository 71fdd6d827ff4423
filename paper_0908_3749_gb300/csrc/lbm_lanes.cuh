// lbm_lanes.cuh -- the FP64 step of small grids: four lanes per node.
//
// GB300 issues an FP64 instruction of a warp every 64 clocks at best, whatever
// its number of active lanes and however independent its instructions are (and
// one per SM every 19 clocks over all warps). A grid that gives every SM less than
// a few warps of the one-thread-per-node form (k_step) therefore takes the time
// of one thread's 224 FP64 instructions, 224 x 64 clocks. Here lane g of a
// node's four holds the populations of velocity group g: each lane transforms
// its group; then lanes 0, 1, 2, 3 take the S, X, Y and C values of all groups (the
// rows of the moment blocks have the same form with other coefficients), share
// the steps of the equilibria, and each relaxes, transforms back and advects its
// own group: 68 FP64 instructions of a warp. Every value is computed by the
// operations of collide64 and neighbour_terms, in some lane, so the results are
// those of k_step bit for bit (a sum a + b as fma(1, a, b), a product a b as fma(a,
// b, -0), which round alike).
//
// Bound by the latency of those instructions and of the loads from L2.
// Measured per step, one thread per node in plain launches / in overlapped ones (k_step) /
// this form:
//   nodes         800   4800   9600  14000  19200  20000  30000  45000
//   periodic (us) 13.7  13.7   13.7   15.2   15.2   21.2   26.5   35.1
//                 11.6  11.6   12.1   12.9   12.9   17.8   21.8   28.7
//                  6.0   6.1    8.1   11.7   13.1   21.4   23.2   34.1
//   walled (us)     -     -      -    21.6   22.9   29.4   34.3   49.9
//                   -     -      -    20.1   20.5   25.2   28.7   43.8
//                   -     -      -    21.1   23.1   27.8   30.4   41.8
// (200 x 4, 1200 x 4, 2400 x 4, 140 x 100, 160 x 120, 200 x 100, 200 x 150, 250 x 180; the
// first three with Dirichlet ends, walled ones with ghosts on all four sides.)
#pragma once

#include "lbm_step.cuh"

namespace lbmk {

// Threads and nodes per block: eight nodes of a row of one 32 x 2 tile of k_step,
// LANES_BLOCKS blocks per tile.
constexpr int LANES_T = 32, LANES_NODES = LANES_T / 4;
constexpr int LANES_ROW = Shape<double>::X / LANES_NODES, LANES_BLOCKS = LANES_ROW * Shape<double>::Y;

// Grids that take this form: at most LANES_MAX_NODES nodes (two blocks per partition of
// every SM; more share the FP64 units, of whose instructions this form has 1.27 times
// as many in all), and beyond LANES_THIN of
// them (one per partition) only where few are next to a side that is not
// periodic: such a node's ghosts cost a block as many instructions as its eight
// nodes' own update. (1800 x 4 nodes between reflecting walls: 25.7 us against 23.2.)
constexpr long long LANES_MAX_NODES = 9728, LANES_THIN = 4864;

__device__ __forceinline__ double lane_value(double v, int src) { return __shfl_sync(0xffffffffu, v, src, 4); }

// Audit of a step in this form: the conserved moments of every node are in
// cons[4][nodes]; of a tile's blocks the one that finished last sums them exactly as
// k_step's block does (audit_tile), then counts the tile (audit_block_done).
__device__ __forceinline__ void lanes_audit(const StepArgs<double>& A, int tile, unsigned long long step,
                                            int* s_list, int* s_n) {
  constexpr int BX = Shape<double>::X, BY = Shape<double>::Y;
  static_assert(BX == 32, "a warp per tile row");
  const int lane = threadIdx.x;
  const long long n = (long long)A.nx * A.ny;
  const int x = (tile % A.tiles_x) * BX + lane, y0 = (tile / A.tiles_x) * BY;
  double v[BY][4], s = 0.0;
#pragma unroll
  for (int r = 0; r < BY; ++r)
#pragma unroll
    for (int q = 0; q < 4; ++q)
      v[r][q] = x < A.nx && y0 + r < A.ny ? __ldcg(A.cons + q * n + (long long)(y0 + r) * A.nx + x) : 0.0;
#pragma unroll
  for (int r = 0; r < BY; ++r) s += warp_sum4(v[r], lane);  // lanes 0, 8, 16, 24: the row's sums 0 .. 3
  if ((lane & 7) == 0) A.partial[4 * tile + (lane >> 3)] = s;
  audit_block_done(A, tile, A.ntiles, step, s_list, s_n);
}

// Counts this block (a warp) among its tile's; the last one audits the tile.
__device__ __forceinline__ void lanes_arrive(const StepArgs<double>& A, int tile, unsigned long long step,
                                             int* s_list, int* s_n) {
  __threadfence();
  __syncwarp();
  int last = 0;
  if (threadIdx.x == 0) {
    last = atomicAdd(&A.tcount[tile], 1u) == LANES_BLOCKS - 1;
    if (last) A.tcount[tile] = 0u;
  }
  if (!__shfl_sync(0xffffffffu, last, 0)) return;
  __threadfence();
  lanes_audit(A, tile, step, s_list, s_n);
}

__global__ void __launch_bounds__(LANES_T)
    k_step_lanes(const double* fin, double* fout, const StepArgs<double> A) {
  __shared__ unsigned long long s_step;
  __shared__ int s_audit, s_alist[32], s_an;
  const int lane = threadIdx.x, g = lane & 3;
  wait_for_previous();
  if (lane == 0) s_step = read_step(A, &s_audit);
  const int tile = blockIdx.x / LANES_BLOCKS, sub = blockIdx.x % LANES_BLOCKS;
  const int xt = (tile % A.tiles_x) * Shape<double>::X + (sub % LANES_ROW) * LANES_NODES + (lane >> 2);
  const int yt = (tile / A.tiles_x) * Shape<double>::Y + sub / LANES_ROW;
  const bool act = xt < A.nx && yt < A.ny;
  const int x = min(xt, A.nx - 1), y = min(yt, A.ny - 1);  // lanes without a node follow an edge node
  const unsigned P = (unsigned)A.plane, pitch = (unsigned)A.pitch;
  const unsigned c = (unsigned)y * pitch + (unsigned)x;
  const bool axis = g < 2;
  // Neighbours inside the grid or across a periodic side; else (ghost) the
  // node itself, replaced below.
  const bool px = A.bc[0] == LBM_BC_PERIODIC, py = A.bc[2] == LBM_BC_PERIODIC;
  const bool gw = x == 0 && !px, ge = x == A.nx - 1 && !px, gs = y == 0 && !py, gn = y == A.ny - 1 && !py;
  const unsigned cw = x > 0 ? c - 1 : px ? c + (unsigned)(A.nx - 1) : c;
  const unsigned ce = x < A.nx - 1 ? c + 1 : px ? c - (unsigned)(A.nx - 1) : c;
  const unsigned cs = y > 0 ? c - pitch : py ? c + (unsigned)(A.ny - 1) * pitch : c;
  const unsigned cn = y < A.ny - 1 ? c + pitch : py ? c - (unsigned)(A.ny - 1) * pitch : c;
  if (!__any_sync(0xffffffffu, act)) {  // a block beyond the grid's edge: counts itself only
    __syncwarp();
    if (s_audit) lanes_arrive(A, tile, s_step, s_alist, &s_an);
    return;
  }
  double f[4], w[4], e[4], s[4], n[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const double* p = fin + (unsigned)(4 * g + k) * P;
    const bool hx = !axis || !(k & 1), hy = !axis || (k & 1);  // has_x, has_y of population 4 g + k
    f[k] = p[c];
    w[k] = hx ? p[cw] : 0.0;
    e[k] = hx ? p[ce] : 0.0;
    s[k] = hy ? p[cs] : 0.0;
    n[k] = hy ? p[cn] : 0.0;
  }
  __syncwarp();
  const unsigned long long step = s_step;
  const bool audit = s_audit != 0;

  // 4-point transform of group g (transform)
  const double tp = f[0] + f[2], tq = f[1] + f[3], ta = f[0] - f[2], tb = f[1] - f[3];
  const double Sg = tp + tq, Cg = tp - tq;
  const double xd = ta - tb, yd = ta + tb;
  const double Xg = axis ? ta : xd, Yg = axis ? tb : yd;
  // This lane's role r = g: S, X, Y or C of all four groups.
  double V[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const double vs = lane_value(Sg, j), vx = lane_value(Xg, j), vy = lane_value(Yg, j), vc = lane_value(Cg, j);
    V[j] = g == 0 ? vs : g == 1 ? vx : g == 2 ? vy : vc;
  }
  const bool rs = g == 0, rc = g == 3;
  // Rows of the moment blocks (collide64's names in brackets: S | X, Y | C)
  const double u = fma(rs ? 1296.0 : rc ? 36.0 : 216.0, V[1], V[0]);      // su | xu | d5
  const double v = fma(rs ? 5.0625 : rc ? 2.25 : 3.375, V[3], V[2]);      // sv | xv | d6
  const double cv = rs ? 16.0 : R2x4;
  const double pl = fma(cv, v, u), mi = fma(-cv, v, u);
  const double u2 = fma(rs ? 36.0 : rc ? 1296.0 : 7776.0, V[1], V[0]);    // 2 e.. | d15.. | d13
  const double v2 = fma(rc ? 5.0625 : 7.59375, V[3], V[2]);               //   -   | d15.. | d14
  const double t2 = fma(rs ? 4.0 : -R2x16, rs ? V[2] : v2, u2);           // 2 e.. | d15
  const double e2r = fma(9.0, V[3], t2);                                  // 2 e
  const double cons = fma(rs ? 1.0 : R2, fma(rs ? 1.0 : 1.5, V[3], V[2]), fma(rs ? 1.0 : 6.0, V[1], V[0]));
  const double rho = lane_value(cons, 0), jx = lane_value(cons, 1), jy = lane_value(cons, 2);
  const double e2 = lane_value(e2r, 0);
  // Equilibria: one instruction computes up to three values, in lanes 0, 1, 2
  const double r = recip(rho);
  const double uo = (g == 2 ? jy : jx) * r;
  const double ux = lane_value(uo, 1), uy = lane_value(uo, 2);
  const double o1 = jx * (rs ? ux : uy);
  const double a = lane_value(o1, 0), m6 = lane_value(o1, 1);
  const double o2 = fma(g == 0 ? jy : g == 1 ? -jy : 1.0, g < 2 ? uy : m6, g < 2 ? a : m6);
  const double k2 = lane_value(o2, 0), m5 = lane_value(o2, 1), m6x2 = lane_value(o2, 2);
  const double o3 = fma(g == 0 ? -1.0 : g == 1 ? e2 : k2, g == 0 ? k2 : r, g == 0 ? e2 : -0.0);
  const double p2 = lane_value(o3, 0), er2 = lane_value(o3, 1), usq = lane_value(o3, 2);
  const double o4 = (g == 1 ? usq : e2) + (g == 0 ? p2 : g == 1 ? usq : e2);
  const double h2 = lane_value(o4, 0), uu = lane_value(o4, 1), e4 = lane_value(o4, 2);
  const double nA = fma(-3.0, er2, uu);
  const double nA8 = __dmul_rn(0.125, nA);
  // Deviations: S d11 d12 | X, Y d7 d9 d15 (d8 d10 d16) | C d5 d13 d6 d14
  const double q1 = fma(rs ? -e4 : rc ? -1.0 : -h2, rs ? er2 : rc ? m5 : g == 1 ? ux : uy, rc ? u : pl);
  const double q2 = fma(rs ? k2 : rc ? nA : g == 1 ? -m5 : m5, rs ? usq : rc ? m5 : g == 1 ? ux : uy,
                        rs ? q1 : rc ? u2 : mi);
  const double q3 = fma(rc ? -0.5 : m6x2, rc ? m6 : g == 1 ? uy : ux, rc ? v : q2);
  const double q4 = fma(nA8, m6, v2);
  const double d11 = lane_value(q2, 0), d12 = lane_value(mi, 0);
  const double d7 = lane_value(q1, 1), d9 = lane_value(q3, 1), d15 = lane_value(t2, 1);
  const double d8 = lane_value(q1, 2), d10 = lane_value(q3, 2), d16 = lane_value(t2, 2);
  const double d5 = lane_value(q1, 3), d13 = lane_value(q2, 3), d6 = lane_value(q3, 3), d14 = lane_value(q4, 3);
  // Back-map of group g and inverse 4-point transform (inverse_transform)
  const double S = fma(A.K.K0[g][1], d12, __dmul_rn(A.K.K0[g][0], d11));
  const double X = fma(A.K.KX[g][2], d15, fma(A.K.KX[g][1], d9, __dmul_rn(A.K.KX[g][0], d7)));
  const double Y = fma(A.K.KY[g][2], d16, fma(A.K.KY[g][1], d10, __dmul_rn(A.K.KY[g][0], d8)));
  const double kc0 = axis ? A.K.KC[g & 1][0] : A.K.KS[g & 1][0];
  const double kc1 = axis ? A.K.KC[g & 1][1] : A.K.KS[g & 1][1];
  const double C = fma(kc1, axis ? d13 : d14, __dmul_rn(kc0, axis ? d5 : d6));
  const double Pp = S + C, Qq = S - C;
  const double ad = X + Y, bd = Y - X;
  const double Aa = axis ? X : ad, Bb = axis ? Y : bd;
  double acc[4] = {Pp + Aa, Qq + Bb, Pp - Aa, Qq - Bb};
#pragma unroll
  for (int k = 0; k < 4; ++k) acc[k] = fma(A.K.a0[4 * g + k], f[k], acc[k]);

  const bool bad = !positive64(rho) || !finite64(rho, jx, jy, e2);
  const bool negT = !bad && !positive64(p2);
  const Cons<double> m = {rho, jx, jy, 0.5 * e2};

  // Ghosts of the sides that are not periodic (every lane of the node takes
  // them, and uses its own group's)
  if (gw || ge || gs || gn) {
    const double t = A.dtr * double(step);
    auto put = [&](int side, int along, unsigned inward, bool has_inward, double (&to)[4]) {
      double G[16];
      ghost(A, fin, P, side, side_kind(A, side, along, t), m, inward, has_inward, G);
#pragma unroll
      for (int k = 0; k < 4; ++k) to[k] = g == 0 ? G[k] : g == 1 ? G[4 + k] : g == 2 ? G[8 + k] : G[12 + k];
    };
    if (gw) put(0, y, c + 1, A.nx > 1, w);
    if (ge) put(1, y, c - 1, A.nx > 1, e);
    if (gs) put(2, x, c + pitch, A.ny > 1, s);
    if (gn) put(3, x, c - pitch, A.ny > 1, n);
  }
  if (!audit) dependents_may_start();
  __syncwarp();
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int i = 4 * g + k;
    if (!axis || !(k & 1)) {
      acc[k] = fma(A.K.aW[i], w[k], acc[k]);
      acc[k] = fma(A.K.aE[i], e[k], acc[k]);
    }
    if (!axis || (k & 1)) {
      acc[k] = fma(A.K.aS[i], s[k], acc[k]);
      acc[k] = fma(A.K.aN[i], n[k], acc[k]);
    }
    if (act) fout[(unsigned)i * P + c] = acc[k];
  }
  __syncwarp();
  watchdog_flags(A.st, step, act && bad, act && negT);
  if (audit) {
    if (act) {
      const double mg = g == 0 ? m.rho : g == 1 ? m.jx : g == 2 ? m.jy : m.e;
      A.cons[((long long)g * A.ny + y) * A.nx + x] = mg;
    }
    lanes_arrive(A, tile, step, s_alist, &s_an);
  }
}

}  // namespace lbmk
