// rlb_adjoint.cu -- reverse-mode (adjoint) kernels of the fused step and the
// checkpointed driver rlb_adjoint (include/rlb_adjoint.h).
//
// Per step the forward map is g^{t+1} = C(h; omega), h = S g^t, with S the pull
// stream and C the per-node g collide of rlb_node.cuh (FP64).  The adjoint of step
// t computes, per node, mu^t = C_h^T lambda^{t+1} and omega_bar += C_omega^T
// lambda^{t+1} (the forward intermediates are recomputed from h, then the chain is
// walked backwards by hand), where lambda^{t+1} = S^T mu^{t+1} is gathered at the node
// inside the same kernel: the adjoint of "node x pulls link a from src(x)" is "node y
// collects link a from every x with src(x) = y" -- one node for a periodic axis, and
// for a zero-gradient axis also the edge node's own clamped pull.  Small quasi-1D lattices
// take several reverse steps per launch on integers (k_adj_tube_steps), other small ones
// run the reverse step with four threads per node in two warp roles (k_adj_step_ws),
// larger ones with one thread per node (k_adj_step).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <string>
#include <vector>

#include "../../include/rlb.h"
#include "../../include/rlb_adjoint.h"
#include "rlb_internal.h"
#include "rlb_launch.cuh"
#include "rlb_node.cuh"
#include "rlb_quad.cuh"

using namespace rlb;

namespace {

constexpr int kThreads = 128;

struct AGeo {
  int nx, ny, nz;
  int zgx, zgy, zgz;
  unsigned long long n;
};

__device__ __forceinline__ int pull_src(int i, int c, int n, int zg) {
  int s = i - c;
  if (s < 0) s = zg ? 0 : n - 1;
  if (s >= n) s = zg ? n - 1 : 0;
  return s;
}

// Nodes x of one axis whose pull with offset c lands on i (at most two).
__device__ __forceinline__ int preimages(int i, int c, int n, int zg, int (&x)[2]) {
  if (c == 0) { x[0] = i; return 1; }
  if (!zg) { int v = i + c; if (v < 0) v += n; if (v >= n) v -= n; x[0] = v; return 1; }
  int k = 0;
  if (i + c >= 0 && i + c < n) x[k++] = i + c;
  if ((c == 1 && i == 0) || (c == -1 && i == n - 1)) x[k++] = i;
  return k;
}

struct GFwd {
  double sp[9], dp[9], Sa, Sd, T00, Mx, My, Mz, MM, A, sA, sigma, is, ux, uy, uz, P, u2, su2, P3, kg, geq0;
  double n0, nA, nD, ne, np, cu[9];
};

__device__ __forceinline__ void gforward(const double (&h)[19], const StepConst& k, bool mrt, GFwd& F) {
#pragma unroll
  for (int p = 0; p < 9; ++p) {
    F.sp[p] = h[2 * p + 1] + h[2 * p + 2];
    F.dp[p] = h[2 * p + 1] - h[2 * p + 2];
  }
  F.Sa = (F.sp[0] + F.sp[1]) + F.sp[2];
  F.Sd = ((F.sp[3] + F.sp[4]) + (F.sp[5] + F.sp[6])) + (F.sp[7] + F.sp[8]);
  F.T00 = (h[0] + F.Sa) + F.Sd;
  F.Mx = ((F.dp[0] + F.dp[3]) + (F.dp[4] + F.dp[5])) + F.dp[6];
  F.My = ((F.dp[1] + F.dp[3]) - (F.dp[4] - F.dp[7])) + F.dp[8];
  F.Mz = ((F.dp[2] + F.dp[5]) - (F.dp[6] - F.dp[7])) - F.dp[8];
  F.MM = fma(F.Mx, F.Mx, fma(F.My, F.My, F.Mz * F.Mz));
  F.A = fma(4.0 * F.T00, F.T00, -3.0 * F.MM);
  // sqrt and reciprocal: FP32 seeds refined by Newton steps to the FP64 rounding level
  // (a lone warp per SM issues these on its FP64 pipe, so the short forms matter)
  F.sA = sqrt_seeded(F.A);
  F.sigma = fma(2.0, F.T00, F.sA) * (1.0 / 3.0);
  F.is = rcp_seeded(F.sigma);
  F.ux = F.Mx * F.is;
  F.uy = F.My * F.is;
  F.uz = F.Mz * F.is;
  F.P = F.sigma - F.T00;
  F.u2 = fma(F.ux, F.ux, fma(F.uy, F.uy, F.uz * F.uz));
  F.su2 = F.sigma * F.u2;
  F.P3 = 3.0 * F.P;
  F.kg = fma(-1.5, F.su2, F.P3);
  F.geq0 = fma(-0.5, F.su2, F.sigma - F.P3);
  pair_cu<double>(F.ux, F.uy, F.uz, F.cu);
  if (mrt) {
    F.n0 = h[0] - F.geq0;
    F.nA = F.Sa - F.P;
    F.nD = fma(-0.5, F.su2, F.Sd - F.P);
    F.ne = fma(8.0, F.nD, fma(-11.0, F.nA, -30.0 * F.n0));
    F.np = fma(-4.0, F.nA, fma(12.0, F.n0, F.nD));
  }
}

// Reverse of the recovery + moments given cotangents of (sigma, P via Pb, u, T00):
// accumulates into hb.
__device__ __forceinline__ void recovery_moments_reverse(const GFwd& F, double sigmab, double Pb, double uxb,
                                                         double uyb, double uzb, double T00b, double Sab, double Sdb,
                                                         double h0b_extra, double (&hb)[19]) {
  // P = sigma - T00
  sigmab += Pb;
  T00b -= Pb;
  // u = M * is
  double Mxb = F.is * uxb, Myb = F.is * uyb, Mzb = F.is * uzb;
  const double isb = F.Mx * uxb + F.My * uyb + F.Mz * uzb;
  // is = 1 / sigma
  sigmab -= F.is * F.is * isb;
  // sigma = (2 T00 + sA) / 3
  T00b += (2.0 / 3.0) * sigmab;
  const double sAb = sigmab * (1.0 / 3.0);
  // sA = sqrt(A)
  const double Ab = sAb * 0.5 * rcp_seeded(F.sA);
  // A = 4 T00^2 - 3 MM
  T00b += 8.0 * F.T00 * Ab;
  const double MMb = -3.0 * Ab;
  Mxb += 2.0 * F.Mx * MMb;
  Myb += 2.0 * F.My * MMb;
  Mzb += 2.0 * F.Mz * MMb;
  // T00 = h0 + Sa + Sd ; Sa, Sd from pair sums ; M from pair differences
  Sab += T00b;
  Sdb += T00b;
  hb[0] += T00b + h0b_extra;
  double dpb[9];
  dpb[0] = Mxb; dpb[1] = Myb; dpb[2] = Mzb;
  dpb[3] = Mxb + Myb; dpb[4] = Mxb - Myb;
  dpb[5] = Mxb + Mzb; dpb[6] = Mxb - Mzb;
  dpb[7] = Myb + Mzb; dpb[8] = Myb - Mzb;
#pragma unroll
  for (int p = 0; p < 9; ++p) {
    const double spb = p < 3 ? Sab : Sdb;
    hb[2 * p + 1] += spb + dpb[p];
    hb[2 * p + 2] += spb - dpb[p];
  }
}

// Vector-Jacobian product of the g collide: given h (pulled) and lo (cotangent of
// the post-collision g), returns hb = C_h^T lo and the omega cotangents.
template <bool MRT>
__device__ __forceinline__ void g_collide_vjp(const double (&h)[19], const double (&lo)[19], const StepConst& k,
                                              double (&hb)[19], double& wvb, double& web, double& wpb) {
  GFwd F;
  gforward(h, k, MRT, F);
  const double om = k.omv, om1 = k.omv1;
  const double wA = 1.0 / 18.0, wD = 1.0 / 36.0;
  double SAb = 0, SDb = 0, AAb = 0, ADb = 0, KAb = 0, KDb = 0, cub[9];
  const double SA = k.gA_s * F.sigma, SD = k.gD_s * F.sigma, AA = k.gA_a * F.sigma, AD = k.gD_a * F.sigma;
  wvb = 0;
  web = 0;
  wpb = 0;
#pragma unroll
  for (int p = 0; p < 9; ++p) {
    const double la = lo[2 * p + 1], lb = lo[2 * p + 2];
    hb[2 * p + 1] = om1 * la;
    hb[2 * p + 2] = om1 * lb;
    wvb -= h[2 * p + 1] * la + h[2 * p + 2] * lb;
    const double evb = la + lb, odb = la - lb;
    const double c = F.cu[p];
    if (p < 3) {
      SAb += evb * c * c; KAb += evb; AAb += odb * c;
      cub[p] = evb * 2.0 * SA * c + odb * AA;
    } else {
      SDb += evb * c * c; KDb += evb; ADb += odb * c;
      cub[p] = evb * 2.0 * SD * c + odb * AD;
    }
  }
  // rest link: out0 = (1 - om) h0 + om geq0 (+ 30 ae - 12 ap)
  const double l0 = lo[0];
  hb[0] = om1 * l0;
  wvb += (F.geq0 - h[0]) * l0;
  double geq0b = om * l0;
  double aeb = 30.0 * l0, apb = -12.0 * l0;
  // K_A = om wA kg + 11 ae + 4 ap ; K_D = om wD kg - 8 ae - ap
  aeb += 11.0 * KAb - 8.0 * KDb;
  apb += 4.0 * KAb - KDb;
  const double kgb = om * (wA * KAb + wD * KDb);
  wvb += F.kg * (wA * KAb + wD * KDb);
  // S = 4.5 om w sigma, A = 3 om w sigma
  double sigmab = om * (4.5 * (wA * SAb + wD * SDb) + 3.0 * (wA * AAb + wD * ADb));
  wvb += F.sigma * (4.5 * (wA * SAb + wD * SDb) + 3.0 * (wA * AAb + wD * ADb));
  double Sab = 0, Sdb = 0, Pb = 0, su2b = 0, h0x = 0;
  if (MRT) {
    const double neb = k.ce * aeb, npb = k.cp * apb;
    const double ceb = F.ne * aeb, cpb = F.np * apb;
    web += ceb / 2394.0;
    wpb += cpb / 252.0;
    wvb -= ceb / 2394.0 + cpb / 252.0;
    const double n0b = -30.0 * neb + 12.0 * npb;
    const double nAb = -11.0 * neb - 4.0 * npb;
    const double nDb = 8.0 * neb + npb;
    h0x += n0b;
    geq0b -= n0b;
    Sab += nAb;
    Pb -= nAb;
    Sdb += nDb;
    Pb -= nDb;
    su2b -= 0.5 * nDb;
  }
  // geq0 = sigma - P3 - 0.5 su2 ; kg = P3 - 1.5 su2 ; P3 = 3 P ; su2 = sigma u2
  sigmab += geq0b;
  double P3b = -geq0b + kgb;
  su2b += -0.5 * geq0b - 1.5 * kgb;
  Pb += 3.0 * P3b;
  sigmab += F.u2 * su2b;
  const double u2b = F.sigma * su2b;
  // cu_p = c_p . u ; u2 = |u|^2
  double uxb = ((cub[0] + cub[3]) + (cub[4] + cub[5])) + cub[6];
  double uyb = ((cub[1] + cub[3]) - (cub[4] - cub[7])) + cub[8];
  double uzb = ((cub[2] + cub[5]) - (cub[6] - cub[7])) - cub[8];
  uxb += 2.0 * F.ux * u2b;
  uyb += 2.0 * F.uy * u2b;
  uzb += 2.0 * F.uz * u2b;
  recovery_moments_reverse(F, sigmab, Pb, uxb, uyb, uzb, 0.0, Sab, Sdb, h0x, hb);
}

// lambda_a at node (x, y, z) from the adjoint of the pull stream: the sum of mu_a over
// the nodes whose pull of link a lands on (x, y, z) (at most two per axis: the
// neighbour, and at a zero-gradient end the node itself).  Loads are unrolled and
// predicated; the order of the sum is fixed.
// The same on a quasi-1D lattice (ny = nz = 1), where every pull's y and z source and
// preimage is the node's own row: only the x preimages are summed, in the same order.
__device__ __forceinline__ double gather_link_tube(const double* __restrict__ mu_a, int x, int cx, const AGeo& geo) {
  int px[2];
  const int nxp = preimages(x, cx, geo.nx, geo.zgx, px);
  double acc = 0.0;
#pragma unroll
  for (int ix = 0; ix < 2; ++ix)
    if (ix < nxp) acc += mu_a[px[ix]];
  return acc;
}
template <bool TUBE>
__device__ __forceinline__ double gather_any(const double* __restrict__ mu_a, int x, int y, int z, int cx, int cy,
                                             int cz, const AGeo& geo);
__device__ __forceinline__ double gather_link(const double* __restrict__ mu_a, int x, int y, int z, int cx, int cy,
                                              int cz, const AGeo& geo) {
  int px[2], py[2], pz[2];
  const int nxp = preimages(x, cx, geo.nx, geo.zgx, px);
  const int nyp = preimages(y, cy, geo.ny, geo.zgy, py);
  const int nzp = preimages(z, cz, geo.nz, geo.zgz, pz);
  double acc = 0.0;
#pragma unroll
  for (int iz = 0; iz < 2; ++iz)
#pragma unroll
    for (int iy = 0; iy < 2; ++iy)
#pragma unroll
      for (int ix = 0; ix < 2; ++ix)
        if (iz < nzp && iy < nyp && ix < nxp)
          acc += mu_a[((unsigned long long)pz[iz] * geo.ny + py[iy]) * geo.nx + px[ix]];
  return acc;
}
template <bool TUBE>
__device__ __forceinline__ double gather_any(const double* __restrict__ mu_a, int x, int y, int z, int cx, int cy,
                                             int cz, const AGeo& geo) {
  if constexpr (TUBE) return gather_link_tube(mu_a, x, cx, geo);
  else return gather_link(mu_a, x, y, z, cx, cy, cz, geo);
}

// One reverse step at node (x, y, z) of a (ceil(nx / blockDim), ny, nz) grid: lambda^{t+1}
// at the node (read directly for the last step, FIRST, else gathered from the mu of the
// step after it), then mu = C_h^T lambda^{t+1} and the omega contributions.
// TUBE: ny = nz = 1 (only x-neighbours exchange populations).
template <bool MRT, bool FIRST, bool TUBE = false>
__global__ void __launch_bounds__(kThreads) k_adj_step(const double* __restrict__ g, const double* __restrict__ in,
                                                      double* __restrict__ mu, double* __restrict__ tb, AGeo geo,
                                                      StepConst k, int lanes) {
  // `lanes` nodes per block along x
  const int x = blockIdx.x * lanes + threadIdx.x;
  if ((int)threadIdx.x >= lanes || x >= geo.nx) return;
  const int y = blockIdx.y, z = blockIdx.z;
  const unsigned long long i = ((unsigned long long)z * geo.ny + y) * geo.nx + x;
  double h[19], lo[19], hb[19];
#pragma unroll
  for (int a = 0; a < 19; ++a) {
    const int xs = pull_src(x, link_cx(a), geo.nx, geo.zgx);
    const int ys = TUBE ? 0 : pull_src(y, link_cy(a), geo.ny, geo.zgy);
    const int zs = TUBE ? 0 : pull_src(z, link_cz(a), geo.nz, geo.zgz);
    const unsigned long long s = ((unsigned long long)zs * geo.ny + ys) * geo.nx + xs;
    h[a] = g[(unsigned long long)a * geo.n + s];
    lo[a] = FIRST ? in[(unsigned long long)a * geo.n + i]
                  : gather_any<TUBE>(in + (unsigned long long)a * geo.n, x, y, z, link_cx(a), link_cy(a), link_cz(a),
                                     geo);
  }
  double wvb, web, wpb;
  g_collide_vjp<MRT>(h, lo, k, hb, wvb, web, wpb);
#pragma unroll
  for (int a = 0; a < 19; ++a) mu[(unsigned long long)a * geo.n + i] = hb[a];
  tb[i] += wvb;
  tb[geo.n + i] += web;
  tb[2 * geo.n + i] += wpb;
}

// ---- four threads per node (small lattices)
//
// On a lattice of a few thousand nodes one thread per node leaves each SM with a
// single warp whose reverse step is one long dependent chain.  The helpers below give
// each node four lanes of a warp: lane j takes link pairs j, j + 4 and j + 8 (the rest
// link is read by all four), the moments and the per-pair cotangents are summed over
// the four lanes with xor shuffles, and the short scalar chains (recovery forward and
// backward, MRT scalars) run in all four lanes.  The arithmetic is that of
// g_collide_vjp summed in another order.

// Direction of link pair p (link 2p + 1 moves along it, link 2p + 2 against it) for a
// pair index known only at run time, from bit masks over p: x is +1 for p in
// {0, 3, 4, 5, 6}; y is +1 for {1, 3, 7, 8} and -1 for 4; z is +1 for {2, 5, 7} and
// -1 for {6, 8}.
__device__ __forceinline__ void pair_dir(int p, int& cx, int& cy, int& cz) {
  cx = (0x079 >> p) & 1;
  cy = ((0x19a >> p) & 1) * (p == 4 ? -1 : 1);
  cz = ((0x1e4 >> p) & 1) * ((p == 6 || p == 8) ? -1 : 1);
}

// c * v for c in {-1, 0, 1}, without a multiply
__device__ __forceinline__ double sel(int c, double v) { return c == 0 ? 0.0 : (c > 0 ? v : -v); }

// sum over the four lanes of one node (lanes 4m .. 4m + 3), returned to all four
__device__ __forceinline__ double quad_sum(double v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  return v;
}

// The pulled g of lane j's three link pairs p = j, j + 4, j + 8 at node (x, y, z) (zeros
// for p > 8) and their directions.
__device__ __forceinline__ void quad_pull(const double* __restrict__ g, int x, int y, int z, int j, const AGeo& geo,
                                          double (&ha)[3], double (&hb)[3], int (&cd)[3][3]) {
  const unsigned long long n = geo.n;
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    const int p = j + 4 * s;
    int cx = 0, cy = 0, cz = 0;
    if (p <= 8) pair_dir(p, cx, cy, cz);
    cd[s][0] = cx;
    cd[s][1] = cy;
    cd[s][2] = cz;
    ha[s] = hb[s] = 0.0;
    if (p <= 8) {
      const unsigned long long a1 = 2 * p + 1, a2 = 2 * p + 2;
      const unsigned long long s1 =
          ((unsigned long long)pull_src(z, cz, geo.nz, geo.zgz) * geo.ny + pull_src(y, cy, geo.ny, geo.zgy)) * geo.nx +
          pull_src(x, cx, geo.nx, geo.zgx);
      const unsigned long long s2 =
          ((unsigned long long)pull_src(z, -cz, geo.nz, geo.zgz) * geo.ny + pull_src(y, -cy, geo.ny, geo.zgy)) * geo.nx +
          pull_src(x, -cx, geo.nx, geo.zgx);
      ha[s] = g[a1 * n + s1];
      hb[s] = g[a2 * n + s2];
    }
  }
}

// lambda of lane j's pairs at the node: read directly (FIRST, the last step) or
// gathered from the mu of the step after it.
template <bool FIRST>
__device__ __forceinline__ void quad_lambda(const double* __restrict__ in, int x, int y, int z, int j,
                                            unsigned long long i, const AGeo& geo, const int (&cd)[3][3],
                                            double (&la)[3], double (&lb)[3]) {
  const unsigned long long n = geo.n;
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    const int p = j + 4 * s;
    la[s] = lb[s] = 0.0;
    if (p <= 8) {
      const unsigned long long a1 = 2 * p + 1, a2 = 2 * p + 2;
      const int cx = cd[s][0], cy = cd[s][1], cz = cd[s][2];
      la[s] = FIRST ? in[a1 * n + i] : gather_link(in + a1 * n, x, y, z, cx, cy, cz, geo);
      lb[s] = FIRST ? in[a2 * n + i] : gather_link(in + a2 * n, x, y, z, -cx, -cy, -cz, geo);
    }
  }
}

// The forward intermediates of the g collide that a node's reverse step uses; none of
// them depends on lambda.  Per node: u, sigma, 1/sigma and its square, u^2, kg, g^eq_0
// minus the rest population, the MRT scalars scaled by the row norms (ne / 2394,
// np / 252), M, 1 / (6 sqrt(A)), 8 T00, 2 sigma and the odd weights 3 omega w sigma of
// the axis and diagonal classes (the pulled state, Eq. 10 and the recovery).  Per link
// pair p, with c = c_p . u and the class weight w: 4.5 w c^2, 3 w c and 2 (4.5 omega w
// sigma) c, the products that multiply the pair's cotangents.
struct QFwd {
  double ux, uy, uz, sigma, is, is2, u2, kg, dg0, ne, np, Mx, My, Mz, rsA6, T8, s2, AA, AD;
};
constexpr int kFwdFields = 19;
constexpr int kPairFields = 3;   // per link pair, stored at (3 p + f) n + i

// QFwd and the pair products of lane j's pairs from the rest link h0 and lane j's
// pulled pairs: moments summed over the node's four lanes, then the scalar chain in
// every lane.
template <bool MRT>
__device__ __forceinline__ void quad_forward(double h0, const double (&ha)[3], const double (&hb)[3],
                                             const int (&cd)[3][3], int j, const StepConst& k, QFwd& F,
                                             double (&pc)[3][kPairFields]) {
  double Sa = 0, Sd = 0, Mx = 0, My = 0, Mz = 0;
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    const int p = j + 4 * s;
    const double sp = ha[s] + hb[s], dp = ha[s] - hb[s];
    if (p < 3) Sa += sp;
    else Sd += sp;   // zero for p > 8
    Mx += sel(cd[s][0], dp);
    My += sel(cd[s][1], dp);
    Mz += sel(cd[s][2], dp);
  }
  Sa = quad_sum(Sa);
  Sd = quad_sum(Sd);
  Mx = quad_sum(Mx);
  My = quad_sum(My);
  Mz = quad_sum(Mz);
  const double T00 = (h0 + Sa) + Sd;
  const double MM = fma(Mx, Mx, fma(My, My, Mz * Mz));
  const double A = fma(4.0 * T00, T00, -3.0 * MM);
  const double sA = sqrt_seeded(A);
  const double sigma = fma(2.0, T00, sA) * (1.0 / 3.0);
  const double is = rcp_seeded(sigma);
  const double ux = Mx * is, uy = My * is, uz = Mz * is;
  const double P = sigma - T00;
  const double u2 = fma(ux, ux, fma(uy, uy, uz * uz));
  const double su2 = sigma * u2, P3 = 3.0 * P;
  const double geq0 = fma(-0.5, su2, sigma - P3);
  F.kg = fma(-1.5, su2, P3);
  F.dg0 = geq0 - h0;
  F.ne = F.np = 0.0;
  if (MRT) {
    const double n0 = h0 - geq0, nA = Sa - P, nD = fma(-0.5, su2, Sd - P);
    F.ne = fma(8.0, nD, fma(-11.0, nA, -30.0 * n0)) * (1.0 / 2394.0);
    F.np = fma(-4.0, nA, fma(12.0, n0, nD)) * (1.0 / 252.0);
  }
  F.ux = ux;
  F.uy = uy;
  F.uz = uz;
  F.sigma = sigma;
  F.is = is;
  F.is2 = is * is;
  F.u2 = u2;
  F.Mx = Mx;
  F.My = My;
  F.Mz = Mz;
  F.rsA6 = rcp_seeded(sA) * (1.0 / 6.0);
  F.T8 = 8.0 * T00;
  F.s2 = 2.0 * sigma;
  F.AA = k.gA_a * sigma;
  F.AD = k.gD_a * sigma;
  const double SA2 = 2.0 * k.gA_s * sigma, SD2 = 2.0 * k.gD_s * sigma;
  const double wA = 1.0 / 18.0, wD = 1.0 / 36.0;
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    const bool ax = j + 4 * s < 3;
    const double c = (sel(cd[s][0], ux) + sel(cd[s][1], uy)) + sel(cd[s][2], uz);
    const double w = ax ? wA : wD;
    pc[s][0] = (4.5 * w * c) * c;
    pc[s][1] = (3.0 * w) * c;
    pc[s][2] = (ax ? SA2 : SD2) * c;
  }
}

// Stored QFwd of node i (field q at q * n + i) and the pair products (pair p, field f
// at (kFwdFields + 3 p + f) * n + i).
__device__ __forceinline__ void store_fwd(double* __restrict__ fw, unsigned long long i, unsigned long long n,
                                          const QFwd& F, bool node_fields, int j, const double (&pc)[3][kPairFields]) {
  if (node_fields) {
    const double v[kFwdFields] = {F.ux, F.uy, F.uz, F.sigma, F.is, F.is2, F.u2, F.kg, F.dg0, F.ne,
                                  F.np, F.Mx, F.My, F.Mz, F.rsA6, F.T8, F.s2, F.AA, F.AD};
#pragma unroll
    for (int q = 0; q < kFwdFields; ++q) fw[q * n + i] = v[q];
  }
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    const int p = j + 4 * s;
    if (p > 8) continue;
#pragma unroll
    for (int f = 0; f < kPairFields; ++f) fw[(kFwdFields + kPairFields * p + f) * n + i] = pc[s][f];
  }
}
__device__ __forceinline__ void load_fwd(const double* __restrict__ fw, unsigned long long i, unsigned long long n,
                                         int j, QFwd& F, double (&pc)[3][kPairFields]) {
  double v[kFwdFields];
#pragma unroll
  for (int q = 0; q < kFwdFields; ++q) v[q] = fw[q * n + i];
  F.ux = v[0]; F.uy = v[1]; F.uz = v[2]; F.sigma = v[3]; F.is = v[4]; F.is2 = v[5]; F.u2 = v[6]; F.kg = v[7];
  F.dg0 = v[8]; F.ne = v[9]; F.np = v[10]; F.Mx = v[11]; F.My = v[12]; F.Mz = v[13]; F.rsA6 = v[14]; F.T8 = v[15];
  F.s2 = v[16]; F.AA = v[17]; F.AD = v[18];
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    const int p = j + 4 * s;
#pragma unroll
    for (int f = 0; f < kPairFields; ++f) pc[s][f] = p <= 8 ? fw[(kFwdFields + kPairFields * p + f) * n + i] : 0.0;
  }
}

// The reverse of the collide at one node in lane j: per-pair cotangents, sums over the
// node's four lanes, the scalar chain backwards (MRT scalars, equilibria, recovery,
// moments), then the stores of mu for lane j's pairs and, in lane 0, the rest link and
// the omega contributions.  An FP64 instruction holds its sub-partition's FP64 unit for
// about 64 cycles whatever its active lanes, so the chain is written for few of them:
// the forward-only products come stored, the four class sums of the shear/bulk term are
// combined before the lane sums, and the relaxations fold into fused multiply-adds.
template <bool MRT>
__device__ __forceinline__ void quad_backward(const QFwd& F, const double (&pc)[3][kPairFields], double l0,
                                              const double (&ha)[3], const double (&hb)[3], const double (&la)[3],
                                              const double (&lb)[3], const int (&cd)[3][3], int j, bool valid,
                                              unsigned long long i, const StepConst& k, double* __restrict__ mu,
                                              double* __restrict__ tb, unsigned long long n) {
  const double om = k.omv, om1 = k.omv1;
  const double wA = 1.0 / 18.0, wD = 1.0 / 36.0;
  double sw = 0, KAb = 0, KDb = 0, wvb = 0, uxb = 0, uyb = 0, uzb = 0;
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    const bool ax = j + 4 * s < 3;   // only slot 0 holds axis pairs; pairs past 8 are zero
    wvb = fma(-ha[s], la[s], fma(-hb[s], lb[s], wvb));
    const double evb = la[s] + lb[s], odb = la[s] - lb[s];
    sw = fma(evb, pc[s][0], fma(odb, pc[s][1], sw));
    if (s == 0) {
      KAb += ax ? evb : 0.0;
      KDb += ax ? 0.0 : evb;
    } else {
      KDb += evb;
    }
    const double cub = fma(evb, pc[s][2], odb * (ax ? F.AA : F.AD));
    uxb += sel(cd[s][0], cub);
    uyb += sel(cd[s][1], cub);
    uzb += sel(cd[s][2], cub);
  }
  sw = quad_sum(sw);
  KAb = quad_sum(KAb);
  KDb = quad_sum(KDb);
  wvb = quad_sum(wvb);
  uxb = quad_sum(uxb);
  uyb = quad_sum(uyb);
  uzb = quad_sum(uzb);
  // rest link: out0 = (1 - om) h0 + om geq0 (+ 30 ae - 12 ap)
  wvb = fma(F.dg0, l0, wvb);
  double geq0b = om * l0;
  const double aeb = fma(11.0, KAb, fma(-8.0, KDb, 30.0 * l0));
  const double apb = fma(-12.0, l0, fma(4.0, KAb, -KDb));
  const double t = fma(wA, KAb, wD * KDb);
  const double kgb = om * t;
  wvb = fma(F.kg, t, wvb);
  double sigmab = om * sw;
  wvb = fma(F.sigma, sw, wvb);
  double Sab = 0, Sdb = 0, Pb = 0, su2b = 0, h0x = 0, web = 0, wpb = 0;
  if (MRT) {
    const double neb = k.ce * aeb, npb = k.cp * apb;
    web = F.ne * aeb;
    wpb = F.np * apb;
    wvb = (wvb - web) - wpb;
    const double n0b = fma(-30.0, neb, 12.0 * npb);
    const double nAb = fma(-11.0, neb, -4.0 * npb);
    const double nDb = fma(8.0, neb, npb);
    h0x = n0b;
    geq0b -= n0b;
    Sab = nAb;
    Sdb = nDb;
    Pb = -nAb - nDb;
    su2b = -0.5 * nDb;
  }
  // geq0 = sigma - P3 - 0.5 su2 ; kg = P3 - 1.5 su2 ; P3 = 3 P ; su2 = sigma u2
  sigmab += geq0b;
  su2b = fma(-0.5, geq0b, fma(-1.5, kgb, su2b));
  Pb = fma(3.0, kgb - geq0b, Pb);
  sigmab = fma(F.u2, su2b, sigmab);
  const double u2b2 = F.s2 * su2b;   // 2 d/du2
  uxb = fma(F.ux, u2b2, uxb);
  uyb = fma(F.uy, u2b2, uyb);
  uzb = fma(F.uz, u2b2, uzb);
  // P = sigma - T00 ; u = M / sigma ; sigma = (2 T00 + sqrt(A)) / 3 ; A = 4 T00^2 - 3 |M|^2
  sigmab += Pb;
  double T00b = -Pb;
  double Mxb = F.is * uxb, Myb = F.is * uyb, Mzb = F.is * uzb;
  sigmab = fma(-F.is2, fma(F.Mx, uxb, fma(F.My, uyb, F.Mz * uzb)), sigmab);
  T00b = fma(2.0 / 3.0, sigmab, T00b);
  const double Ab = sigmab * F.rsA6;
  T00b = fma(F.T8, Ab, T00b);
  const double MMb = -6.0 * Ab;
  Mxb = fma(F.Mx, MMb, Mxb);
  Myb = fma(F.My, MMb, Myb);
  Mzb = fma(F.Mz, MMb, Mzb);
  // T00 = h0 + Sa + Sd
  Sab += T00b;
  Sdb += T00b;
  if (!valid) return;
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    const int p = j + 4 * s;
    if (p > 8) continue;
    const double spb = p < 3 ? Sab : Sdb;
    const double dpb = (sel(cd[s][0], Mxb) + sel(cd[s][1], Myb)) + sel(cd[s][2], Mzb);
    mu[(unsigned long long)(2 * p + 1) * n + i] = fma(om1, la[s], spb + dpb);
    mu[(unsigned long long)(2 * p + 2) * n + i] = fma(om1, lb[s], spb - dpb);
  }
  if (j == 0) {
    mu[i] = fma(om1, l0, T00b + h0x);
    tb[i] += wvb;
    tb[n + i] += web;
    tb[2 * n + i] += wpb;
  }
}

// ---- two warp roles (small lattices, the reverse sweep's chain)
//
// Nothing in QFwd or the pair products depends on lambda, only on the forward state,
// so the reverse step need not compute them on its own dependent chain.  k_adj_step_ws
// runs 8 nodes per 64-thread block: warp 0 walks the backward chain of step t from the
// values stored for step t (fw), and warp 1 computes and stores those of step t - 1
// (from g_prev, the state at step t - 1, into fw_prev) for the next launch.  The two
// warps run on different sub-partitions, so each has its own FP64 unit.  k_adj_fwd
// stores the values of one step on its own (the last step, where the sweep starts).
template <bool MRT>
__global__ void __launch_bounds__(64) k_adj_fwd(const double* __restrict__ g, double* __restrict__ fw, AGeo geo,
                                                StepConst k) {
  const int j = threadIdx.x & 3;
  const int xg = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 2);
  const bool valid = xg < geo.nx;
  const int x = valid ? xg : geo.nx - 1;
  const int y = blockIdx.y, z = blockIdx.z;
  const unsigned long long i = ((unsigned long long)z * geo.ny + y) * geo.nx + x;
  double ha[3], hb[3], pc[3][kPairFields];
  int cd[3][3];
  const double h0 = g[i];
  quad_pull(g, x, y, z, j, geo, ha, hb, cd);
  QFwd F;
  quad_forward<MRT>(h0, ha, hb, cd, j, k, F, pc);
  if (valid) store_fwd(fw, i, geo.n, F, j == 0, j, pc);
}

template <bool MRT, bool FIRST>
__global__ void __launch_bounds__(64) k_adj_step_ws(const double* __restrict__ g, const double* __restrict__ in,
                                                    double* __restrict__ mu, double* __restrict__ tb,
                                                    const double* __restrict__ fw, const double* __restrict__ g_prev,
                                                    double* __restrict__ fw_prev, AGeo geo, StepConst k) {
  const int lane = threadIdx.x & 31, j = lane & 3;
  const int xg = (int)(blockIdx.x * 8 + (lane >> 2));
  const bool valid = xg < geo.nx;
  const int x = valid ? xg : geo.nx - 1;
  const int y = blockIdx.y, z = blockIdx.z;
  const unsigned long long i = ((unsigned long long)z * geo.ny + y) * geo.nx + x;
  double ha[3], hb[3], pc[3][kPairFields];
  int cd[3][3];
  QFwd F;
  wait_for_grid(g, in);
  wait_for_grid(fw, g_prev);
  wait_for_grid(tb);
  if (threadIdx.x >= 32) {
    // step t - 1's forward values (none before step 0)
    if (g_prev == nullptr) return;
    const double h0 = g_prev[i];
    quad_pull(g_prev, x, y, z, j, geo, ha, hb, cd);
    quad_forward<MRT>(h0, ha, hb, cd, j, k, F, pc);
    if (valid) store_fwd(fw_prev, i, geo.n, F, j == 0, j, pc);
    return;
  }
  const double l0 = in[i];
  double la[3], lb[3];
  quad_pull(g, x, y, z, j, geo, ha, hb, cd);
  quad_lambda<FIRST>(in, x, y, z, j, i, geo, cd, la, lb);
  load_fwd(fw, i, geo.n, j, F, pc);
  quad_backward<MRT>(F, pc, l0, ha, hb, la, lb, cd, j, valid, i, k, mu, tb, geo.n);
}

// ---- several reverse steps per launch (quasi-1D lattices)
//
// mu = C_h^T lambda depends on the forward state through u alone: with the cotangents of u
// taken per sigma, every coefficient of the walk back through the collide is dimensionless
// (r = sigma / sqrt(A) = 2 / (3 - u^2), T00 / sigma = (3 + u^2) / 4).  The walk runs in 64-bit
// block fixed point on the grid of the node's largest |lambda| (unit 2^-55 to 2^-56 of it; every
// intermediate stays below 2^62.6 for any u and any admissible rates), where an addition costs
// two issue slots instead of the 64 cycles that an FP64 instruction holds its unit.  The omega
// cotangents, which do multiply g by lambda, leave this chain: the lambda of every step is
// stored, and k_adj_omega forms them for a whole segment at once.
//
// A block holds kTubeTile nodes as k_tube_steps does (tiles that overlap by one node per
// step): warps 0..3 hold lambda, four lanes per node, and warp 4 recovers u of the next
// step's state, one node per lane, while they walk back through this one.  1600 nodes: 7.8 ->
// 4.2 us per reverse step, 1600 nodes x 4000 steps 40.7 -> 26.4 ms per gradient; bound by the
// dependent integer chains of the two roles (issue 25 %, fixed-latency waits).
struct RevU {
  unsigned long long ax[kTubeTile], ay[kTubeTile], az[kTubeTile];
  unsigned sg[kTubeTile];
};
// a b / 2^64, to the nearest.  Rounded, the walk's error is 0.4 x 2^-53 of the node's largest
// |lambda| (rms over random lambda and u, MRT; FP64 arithmetic: 1.67) with no bias; products cut
// off below on a grid half as fine gave 2.5 with a bias of -1.9, which added up over the steps.
__device__ __forceinline__ long long mul_s(long long a, long long b) {
  const unsigned a0 = (unsigned)a, a1 = (unsigned)((unsigned long long)a >> 32), b0 = (unsigned)b,
                 b1 = (unsigned)((unsigned long long)b >> 32);
  const unsigned long long t = (unsigned long long)a0 * b1 + ((unsigned long long)__umulhi(a0, b0) + 0x80000000ull);
  const unsigned long long m = (unsigned long long)a1 * b0 + (unsigned)t;
  const unsigned long long hi = (unsigned long long)a1 * b1 + ((t >> 32) + (m >> 32));
  return (long long)(hi - ((unsigned long long)(a >> 63) & (unsigned long long)b) -
                     ((unsigned long long)(b >> 63) & (unsigned long long)a));
}
// x / 2^K, to the nearest
template <int K>
__device__ __forceinline__ long long half_up(long long x) { return (x + (1ll << (K - 1))) >> K; }

// x, or an infinity where its sum went beyond the format: the exponent has then passed 0x7ff into
// the sign bit.
__device__ __noinline__ double past_format(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), f = (hi >> 20) & 0x7ffu;
  const bool past = f < 16u && (hi | (unsigned)__double2loint(x)) != 0;
  if (!past && f != 0x7ffu) return x;
  return __hiloint2double((int)(((hi ^ (past ? 0x80000000u : 0u)) & 0x80000000u) | 0x7ff00000u), 0);
}

// Cotangents of one node's pulled populations from those of its relaxed ones (v, lane
// (m, j)'s six links; lane 3 the rest link), in place.  W62 = omega_v 2^62.
template <bool MRT>
__device__ __forceinline__ void quad_vjp(int lane, double (&v)[6], const RevU& ru, int i, long long W62,
                                         const StepConst& k) {
  using namespace fx;
  const int j = lane & 3, base = lane & ~3;
  unsigned me = 0;
#pragma unroll
  for (int sl = 0; sl < 6; ++sl) me = max(me, (unsigned)__double2hiint(v[sl]) & 0x7fffffffu);
  me = max(me, (unsigned)__shfl_xor_sync(0xffffffffu, (int)me, 1));
  me = max(me, (unsigned)__shfl_xor_sync(0xffffffffu, (int)me, 2));
  const int E = max((int)(me >> 20), 64);   // tiny weights: see rlb_adjoint
  long long L[6];
#pragma unroll
  for (int sl = 0; sl < 6; ++sl) L[sl] = to_fixed(v[sl], E + 8);   // |L| < 2^56
  const long long l0 = __shfl_sync(0xffffffffu, L[0], base + 3);
  // u_i 2^62 and the pairs' c.u at 2^61
  const unsigned sg = ru.sg[i];
  const long long ux = with_sign(ru.ax[i] >> 1, sg & 1u), uy = with_sign(ru.ay[i] >> 1, (sg >> 1) & 1u),
                  uz = with_sign(ru.az[i] >> 1, sg >> 2);
  const unsigned long long u2 = mulhi(ru.ax[i], ru.ax[i]) + mulhi(ru.ay[i], ru.ay[i]) + mulhi(ru.az[i], ru.az[i]);
  const bool pairs = j < 3;
  const long long ca = sel3(j, ux, uy, uz) >> 1;
  const long long cp = (sel3(j, ux, uy, ux) >> 1) + (sel3(j, uy, uz, uz) >> 1);
  const long long cm = (sel3(j, ux, uy, ux) >> 1) - (sel3(j, uy, uz, uz) >> 1);
  constexpr long long kT = 0x2aaaaaaaaaaaaaabll;   // 2^63 / 3
  long long S[3], Q[3];
  const long long ev[3] = {L[0] + L[1], L[2] + L[3], L[4] + L[5]};
  const long long od[3] = {L[0] - L[1], L[2] - L[3], L[4] - L[5]}, cc[3] = {ca, cp, cm};
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    const long long p1 = mul_s(ev[p] << 3, cc[p]), o3 = mul_s(od[p] << 1, kT);   // c ev, od / 3
    S[p] = mul_s((p1 + 2 * o3) << 3, cc[p]);                                     // c (c ev + 2 od / 3)
    Q[p] = p1 + o3;
  }
  const long long hS = Q[1] + Q[2], hD = Q[1] - Q[2];
  const long long KA = quad_sum64(pairs ? ev[0] : 0), KD = quad_sum64(pairs ? ev[1] + ev[2] : 0);
  const long long SW = quad_sum64(pairs ? 2 * S[0] + S[1] + S[2] : 0);           // 8 times the density's cotangent
  const long long Bx = quad_sum64(j == 0 ? 2 * Q[0] + hS : (j == 2 ? hS : 0));   // twice the momentum sums of quad_collide
  const long long By = quad_sum64(j == 0 ? hD : (j == 1 ? 2 * Q[0] + hS : 0));
  const long long Bz = quad_sum64(j == 1 ? hD : (j == 2 ? 2 * Q[0] + hD : 0));
  const auto om = [W62](long long x) { return mul_s(x << 2, W62); };             // omega x
  long long gq = om(l0);                                                         // of g^eq_0
  const long long kg = om(mul_s(2 * KA + KD, (long long)k36th));                 // of 3P - 1.5 sigma u^2
  long long sb = mul_s(SW, W62 >> 1), Sab = 0, Sdb = 0, Pb = 0, h0 = 0;
  if (MRT) {
    const long long a2 = 15 * l0 + 11 * (KA >> 1) - 4 * KD, p4 = KA - (KD >> 2) - 3 * l0;
    const long long e8 = half_up<5>(mul_s(a2, k.CE)), p8 = mul_s(p4, k.CP);      // 8 ce (..), 8 cp (..)
    h0 = half_up<3>(12 * p8 - 30 * e8);
    Sab = -half_up<3>(11 * e8 + 4 * p8);
    Sdb = half_up<3>(8 * e8 + p8);
    gq -= h0;
    Pb = -Sab - Sdb;
  }
  sb += gq;
  const long long s2 = -Sdb - (gq + 3 * kg);                                     // of sigma u^2, twice
  Pb += 3 * (kg - gq);
  sb += mul_s(s2 << 1, (long long)u2);
  const long long bx = mul_s(Bx, W62) + mul_s(s2 << 2, ux), by = mul_s(By, W62) + mul_s(s2 << 2, uy),
                  bz = mul_s(Bz, W62) + mul_s(s2 << 2, uz);                      // of u, per sigma
  sb += Pb;
  sb -= mul_s(bx << 2, ux) + mul_s(by << 2, uy) + mul_s(bz << 2, uz);
  const long long r = (long long)(rcp_fixed((3ull << 62) - u2) >> 1);            // 2 / (3 - u^2) 2^62
  const long long w = mul_s(sb << 2, r);
  const long long T = 2 * w - Pb;                                                // of T00
  const long long mx = bx - mul_s(w << 2, ux), my = by - mul_s(w << 2, uy), mz = bz - mul_s(w << 2, uz);
  if (pairs) {
    const long long da = sel3(j, mx, my, mz), a = sel3(j, mx, my, mx), b = sel3(j, my, mz, mz);
    const long long d[3] = {da, a + b, a - b};
#pragma unroll
    for (int p = 0; p < 3; ++p) {
      const long long t = (p == 0 ? Sab : Sdb) + T;
      long long ya = L[2 * p] - om(L[2 * p]) + t, yb = L[2 * p + 1] - om(L[2 * p + 1]) + t;
      asm("" : "+l"(ya), "+l"(yb));   // as fx::relax says
      v[2 * p] = from_fixed_rn(ya + d[p], E + 1);
      v[2 * p + 1] = from_fixed_rn(yb - d[p], E + 1);
    }
  } else {
    v[0] = from_fixed_rn(l0 - om(l0) + T + h0, E + 1);
#pragma unroll
    for (int sl = 1; sl < 6; ++sl) v[sl] = v[0];
  }
  // near the format's end, or (0x7ff) NaN or infinite: the node then comes out NaN.  One branch
  // for all that is rare (500 nodes x 300 steps BGK: 1 % less than selects at each value)
  if (E > 2032) {
#pragma unroll
    for (int sl = 0; sl < 6; ++sl)
      v[sl] = me < 0x7ff00000u ? past_format(v[sl]) : __longlong_as_double(0x7ff8000000000000ll);
  }
}

// `steps` reverse steps: the first works on the state g (one array of 19 nx), each later one
// on the array before it, and stores its lambda at lam, each later one in the array before.
// in: lambda of the first step itself (first), else the mu to gather it from; out: the last mu.
template <bool MRT>
__global__ void __launch_bounds__(32 * (kTubeWarps + 1))
    k_adj_tube_steps(const double* __restrict__ g, double* __restrict__ lam, const double* __restrict__ in,
                     double* __restrict__ out, int nx, int zg, StepConst k, int steps, int core, bool first) {
  __shared__ RevU ru[2];
  __shared__ double ex[2][2][6][kTubeTile];   // [parity][lane 0 / 2][slot][node]
  wait_for_grid(g, in);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool u_warp = warp == kTubeWarps;
  const int i = u_warp ? lane : warp * 8 + (lane >> 2), j = u_warp ? 0 : lane & 3;
  const int halo = (kTubeTile - core) >> 1;
  const int xg = (int)blockIdx.x * core - halo + i;
  const bool own = i >= halo && i < halo + core && xg < nx;
  const bool idle = zg && (xg < 0 || xg >= nx);                 // past an open end
  const int x = zg ? min(max(xg, 0), nx - 1) : (xg < 0 ? (xg % nx + nx) % nx : xg % nx);
  const bool whole = core == kTubeTile;
  const unsigned long long n = (unsigned long long)nx;
  if (u_warp) {
    const int xm = x > 0 ? x - 1 : (zg ? 0 : nx - 1), xp = x < nx - 1 ? x + 1 : (zg ? nx - 1 : 0);
    double h[19];
    const auto load = [&](const double* gs) {
#pragma unroll
      for (int a = 0; a < 19; ++a) h[a] = gs[(unsigned long long)a * n + (link_cx(a) > 0 ? xm : link_cx(a) < 0 ? xp : x)];
    };
    load(g);
    for (int s = 0; s < steps; ++s) {
      bool fast;
      const int E = fx::max_exponent(h, fast);
      long long X[19];
      if (__all_sync(0xffffffffu, fast)) {
#pragma unroll
        for (int a = 0; a < 19; ++a) X[a] = fx::to_fixed_pos(h[a], E + 7);
      } else {
#pragma unroll
        for (int a = 0; a < 19; ++a) X[a] = fx::to_fixed(h[a], E + 7);
      }
      if (s + 1 < steps) load(g - (unsigned long long)(s + 1) * 19ull * n);   // in flight during the recovery
      long long T = X[0], d[9];
#pragma unroll
      for (int p = 0; p < 9; ++p) {
        T += X[2 * p + 1] + X[2 * p + 2];
        d[p] = X[2 * p + 1] - X[2 * p + 2];
      }
      UFix u;
      bool br;
      fx_recover(T, d[0] + d[3] + d[4] + d[5] + d[6], d[1] + d[3] - d[4] + d[7] + d[8], d[2] + d[5] - d[6] + d[7] - d[8],
                 u, br);
      RevU& r = ru[s & 1];
      r.ax[i] = u.ax;
      r.ay[i] = u.ay;
      r.az[i] = u.az;
      r.sg[i] = u.sx | (u.sy << 1) | (u.sz << 2);
      __syncthreads();   // step s may start; step s - 1 has read the other buffer
    }
    return;
  }
  // lambda of the first step
  double v[6];
#pragma unroll
  for (int sl = 0; sl < 6; ++sl) {
    int cx, cy, cz;
    quad_dir(j, sl, cx, cy, cz);
    const double* at = in + (unsigned long long)quad_link(j, sl) * n;
    v[sl] = idle ? 0.0 : first ? at[x] : gather_link_tube(at, x, cx, AGeo{nx, 1, 1, zg, 0, 0, n});
  }
  const long long W62 = (long long)(k.Om_v >> 1);
  // preimages of the x-moving links: cx = +1 (even slots) node i + 1, cx = -1 node i - 1; at an
  // open end none beyond it, and the end node its own clamped pull
  const bool lo = xg == 0, hi = xg == nx - 1;
  const bool np = !(zg && hi), nm = !(zg && lo);
  const int ip = whole && hi ? 0 : min(i + 1, kTubeTile - 1), im = whole && lo ? nx - 1 : max(i - 1, 0);
  const bool axis_moves = j == 0, moves = j == 0 || j == 2;
  for (int s = 0; s < steps; ++s) {
    __syncthreads();
    if (s > 0 && moves) {
      auto& e = ex[s & 1][j >> 1];
#pragma unroll
      for (int sl = 0; sl < 6; ++sl)
        if (sl >= 2 || axis_moves) {
          const bool plus = (sl & 1) == 0;
          double t = (plus ? np : nm) ? e[sl][plus ? ip : im] : 0.0;
          if (zg && (plus ? lo : hi)) t += v[sl];
          v[sl] = idle ? 0.0 : t;
        }
    }
    if (own) {
      double* ls = lam - (unsigned long long)s * 19ull * n + (unsigned)x;
      ls[(unsigned long long)quad_link(j, 0) * n] = v[0];
      if (j < 3) {
#pragma unroll
        for (int sl = 1; sl < 6; ++sl) ls[(unsigned long long)quad_link(j, sl) * n] = v[sl];
      }
    }
    quad_vjp<MRT>(lane, v, ru[s & 1], i, W62, k);
    if (s == steps - 1) break;
    if (moves) {
      auto& e = ex[(s + 1) & 1][j >> 1];
#pragma unroll
      for (int sl = 0; sl < 6; ++sl)
        if (sl >= 2 || axis_moves) e[sl][i] = v[sl];
    }
  }
  if (own) {
    double* o = out + (unsigned)x;
    o[(unsigned long long)quad_link(j, 0) * n] = v[0];
    if (j < 3) {
#pragma unroll
      for (int sl = 1; sl < 6; ++sl) o[(unsigned long long)quad_link(j, sl) * n] = v[sl];
    }
  }
}

// The omega cotangents of every node and step of a segment (blockIdx.y: the step), from its
// states and stored lambdas, and their sum over the steps in the order of the sweep.  A node's
// three cotangents take the place of its first three lambdas, which this thread alone reads.
template <bool MRT>
__global__ void __launch_bounds__(kThreads) k_adj_omega(const double* __restrict__ g, double* __restrict__ lam, int nx,
                                                       int zg, StepConst k) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= nx) return;
  const unsigned long long n = (unsigned long long)nx, off = blockIdx.y * 19ull * n;
  double h[19], lo[19];
#pragma unroll
  for (int a = 0; a < 19; ++a) {
    h[a] = g[off + (unsigned long long)a * n + pull_src(x, link_cx(a), nx, zg)];
    lo[a] = lam[off + (unsigned long long)a * n + x];
  }
  // d/d omega_v = lambda . (g^eq - h) less the e and eps rows; the differences link by link,
  // before the product, keep what the sums over g^eq and h would cancel
  GFwd F;
  gforward(h, k, MRT, F);
  double wvb = (F.geq0 - h[0]) * lo[0], KAb = 0, KDb = 0;
#pragma unroll
  for (int p = 0; p < 9; ++p) {
    const double w = p < 3 ? 1.0 / 18.0 : 1.0 / 36.0, c = F.cu[p];
    const double e = w * fma(4.5 * F.sigma * c, c, F.kg), o = (3.0 * w) * F.sigma * c;
    const double la = lo[2 * p + 1], lb = lo[2 * p + 2];
    wvb = fma((e + o) - h[2 * p + 1], la, fma((e - o) - h[2 * p + 2], lb, wvb));
    if (p < 3) KAb += la + lb;
    else KDb += la + lb;
  }
  double web = 0, wpb = 0;
  if (MRT) {
    web = F.ne * fma(11.0, KAb, fma(-8.0, KDb, 30.0 * lo[0])) * (1.0 / 2394.0);
    wpb = F.np * (fma(4.0, KAb, -KDb) - 12.0 * lo[0]) * (1.0 / 252.0);
    wvb -= web + wpb;
  }
  double* p = lam + off + x;
  p[0] = wvb;
  p[n] = web;
  p[2 * n] = wpb;
}
__global__ void __launch_bounds__(kThreads) k_adj_omega_sum(const double* __restrict__ part, double* __restrict__ tb,
                                                           unsigned long long n, int steps) {
  const unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
  if (i >= 3 * n) return;
  double acc = tb[i];
  for (int s = steps - 1; s >= 0; --s) acc += part[(unsigned long long)s * 19ull * n + i];
  tb[i] = acc;
}

// lambda^T = dJ/dg^T and the per-node misfit.
__global__ void __launch_bounds__(kThreads) k_adj_loss(const double* __restrict__ g, const double* __restrict__ tP,
                                                      const double* __restrict__ tux, const double* __restrict__ tuy,
                                                      const double* __restrict__ tuz, double wP, double wu,
                                                      double* __restrict__ lam, double* __restrict__ lossn,
                                                      unsigned long long n) {
  const unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  double h[19], hb[19];
#pragma unroll
  for (int a = 0; a < 19; ++a) {
    h[a] = g[(unsigned long long)a * n + i];
    hb[a] = 0.0;
  }
  GFwd F;
  StepConst dummy{};
  gforward(h, dummy, false, F);
  const double rP = F.P - tP[i], rx = F.ux - tux[i], ry = F.uy - tuy[i], rz = F.uz - tuz[i];
  lossn[i] = wP * rP * rP + wu * (rx * rx + ry * ry + rz * rz);
  recovery_moments_reverse(F, 0.0, 2.0 * wP * rP, 2.0 * wu * rx, 2.0 * wu * ry, 2.0 * wu * rz, 0.0, 0.0, 0.0, 0.0,
                           hb);
#pragma unroll
  for (int a = 0; a < 19; ++a) lam[(unsigned long long)a * n + i] = hb[a];
}

// dJ/de0 of an equilibrium initial state: g^0 is linear in e0, so sum_a lambda_a g0_a / e0.
// dJ/de0 at node (x, y, z): lambda^0 = S^T mu^0 gathered at the node, contracted with
// dg^eq/de of the initial state (g^eq is homogeneous of degree 1 in e at fixed u).  unit: a power
// of two that the misfit weights were divided by.
__global__ void __launch_bounds__(kThreads) k_adj_e0(const double* __restrict__ g0, const double* __restrict__ mu,
                                                    double* __restrict__ de0, double unit, AGeo geo, int lanes) {
  const int x = blockIdx.x * lanes + threadIdx.x;
  if ((int)threadIdx.x >= lanes || x >= geo.nx) return;
  const int y = blockIdx.y, z = blockIdx.z;
  const unsigned long long i = ((unsigned long long)z * geo.ny + y) * geo.nx + x;
  double h[19];
  double acc = 0.0;
#pragma unroll
  for (int a = 0; a < 19; ++a) {
    h[a] = g0[(unsigned long long)a * geo.n + i];
    const double l = gather_link(mu + (unsigned long long)a * geo.n, x, y, z, link_cx(a), link_cy(a), link_cz(a), geo);
    acc = fma(l, h[a], acc);
  }
  GFwd F;
  StepConst dummy{};
  gforward(h, dummy, false, F);
  de0[i] = acc / (3.0 * F.P) * unit;
}

// Deterministic sums of `rows` arrays of length n (one block per row).
__global__ void __launch_bounds__(256) k_rowsum(const double* __restrict__ a, unsigned long long n,
                                                double* __restrict__ out) {
  __shared__ double sh[256];
  double acc = 0.0;
  const double* r = a + blockIdx.x * n;
  for (unsigned long long i = threadIdx.x; i < n; i += 256) acc += r[i];
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[blockIdx.x] = sh[0];
}

int afail(rlb_handle* h, int code, const std::string& m) {
  h->err = m;
  return code;
}

// Buffers of one (nsteps, checkpoint interval) shape and, where every step is a launch of
// its own, the captured CUDA graph, kept on the handle so repeated gradients replay instead
// of re-launching ~4 T kernels one by one.
struct AdjPlan {
  int nsteps = -1, K = 0, nseg = 0, start_cur = 0, end_cur = 0, threads = 128, lanes = 128;
  int most = 1, core = 0;                     // quasi-1D: steps per launch (tube_launch_steps)
  bool quad = false;                          // reverse steps with four threads per node
  double wP = 0.0, wu = 0.0;                  // misfit weights baked into the graph
  std::vector<void*> ckpt, owned;
  // g^{t0 + j} of a recomputed segment at seg[s & 1][j] (quasi-1D: one array of g after the
  // other, and the lambda of each step in lamseg likewise; else whole states)
  std::vector<void*> seg[2];
  double *lam = nullptr, *mu = nullptr, *tb = nullptr, *lossn = nullptr, *sums = nullptr, *dde0 = nullptr;
  double* fw[2] = {nullptr, nullptr};         // QFwd of alternate reverse steps (two warp roles)
  double* tgt = nullptr;
  double* lamseg[2] = {nullptr, nullptr};     // quasi-1D: stored lambdas, then omega cotangents per step
  cudaStream_t cap3 = nullptr;                // the omega cotangents beside the sweep of the next segment
  cudaStream_t cap = nullptr;
  cudaStream_t cap2 = nullptr;                // recompute of segment s - 1 beside the reverse sweep of s
  cudaEvent_t ev[7] = {};                     // fork, ready[2], free[2], swept[2]
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  int runs = 0;                               // gradients computed with this plan
};

void free_plan(void* p) {
  AdjPlan* a = (AdjPlan*)p;
  if (!a) return;
  if (a->exec) cudaGraphExecDestroy(a->exec);
  if (a->graph) cudaGraphDestroy(a->graph);
  if (a->cap) cudaStreamDestroy(a->cap);
  if (a->cap2) cudaStreamDestroy(a->cap2);
  if (a->cap3) cudaStreamDestroy(a->cap3);
  for (cudaEvent_t e : a->ev)
    if (e) cudaEventDestroy(e);
  for (void* q : a->owned) cudaFree(q);
  delete a;
}

// The plan's buffers come from one allocation (a gradient of 400 steps has about 60 of them):
// plan_alloc notes each, plan_commit allocates and hands out the addresses.
struct PlanWant {
  void** p;
  size_t offset;
};
void plan_alloc(std::vector<PlanWant>& want, size_t& total, void** p, size_t bytes) {
  want.push_back({p, total});
  total += (bytes + 255) & ~(size_t)255;
}
bool plan_commit(AdjPlan* a, const std::vector<PlanWant>& want, size_t total) {
  void* base = nullptr;
  if (cudaMalloc(&base, total) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  a->owned.push_back(base);
  for (const PlanWant& w : want) *w.p = (char*)base + w.offset;
  return true;
}

// One reverse step with the kernel variant for the lattice: two warp roles with four
// threads per node (quad; fw holds step t's QFwd, and step t - 1's goes from g_prev
// into fw_prev) or one thread per node; quasi-1D (ny = nz = 1) or general; BGK or MRT.
template <bool FIRST>
cudaError_t reverse_step(bool quad, bool tube, bool mrt, dim3 grid8, dim3 grid3, int th, cudaStream_t st, bool early,
                         const double* gt, const double* in, double* out, double* tb, const double* fw,
                         const double* g_prev, double* fw_prev, const AGeo& geo, const StepConst& k, int lanes) {
  if (quad) {
    if (mrt) launch_after(grid8, 64, st, early, k_adj_step_ws<true, FIRST>, gt, in, out, tb, fw, g_prev, fw_prev, geo, k);
    else launch_after(grid8, 64, st, early, k_adj_step_ws<false, FIRST>, gt, in, out, tb, fw, g_prev, fw_prev, geo, k);
  } else if (tube) {
    if (mrt) k_adj_step<true, FIRST, true><<<grid3, th, 0, st>>>(gt, in, out, tb, geo, k, lanes);
    else k_adj_step<false, FIRST, true><<<grid3, th, 0, st>>>(gt, in, out, tb, geo, k, lanes);
  } else {
    if (mrt) k_adj_step<true, FIRST><<<grid3, th, 0, st>>>(gt, in, out, tb, geo, k, lanes);
    else k_adj_step<false, FIRST><<<grid3, th, 0, st>>>(gt, in, out, tb, geo, k, lanes);
  }
  return cudaGetLastError();
}

// Enqueue the whole gradient computation on stream st (the handle's, or the plan's stream
// whose work is being captured).
cudaError_t enqueue_adjoint(rlb_handle* h, AdjPlan* a, double wP, double wu, double unit, bool mrt, cudaStream_t st) {
  const unsigned long long N = h->nodes;
  const size_t state_bytes = 38 * N * sizeof(double);
  const int T = a->nsteps, K = a->K, th = a->threads;
  const unsigned grid = (unsigned)((N + th - 1) / th);
  const int lanes = a->lanes;
  const dim3 grid3((unsigned)((h->cfg.nx + lanes - 1) / lanes), (unsigned)h->cfg.ny, (unsigned)h->cfg.nz);
  const dim3 grid8((unsigned)((h->cfg.nx + 7) / 8), (unsigned)h->cfg.ny, (unsigned)h->cfg.nz);
  double* mu_cur = nullptr;   // buffer holding the mu of the latest reverse step (lam / mu alternate)
  AGeo geo{h->cfg.nx, h->cfg.ny, h->cfg.nz, h->cfg.bc[0] == RLB_ZERO_GRADIENT, h->cfg.bc[1] == RLB_ZERO_GRADIENT,
           h->cfg.bc[2] == RLB_ZERO_GRADIENT, N};
  const bool tube = h->cfg.ny == 1 && h->cfg.nz == 1;
  const double* tP = a->tgt;
  cudaError_t e;
#define ENQ(call) do { e = (call); if (e != cudaSuccess) return e; } while (0)
  // Forward with checkpoints (of which the first is the initial state).  On a quasi-1D lattice
  // the forward run and the recompute take several steps per launch, the forward run writes
  // its checkpoints in place and the recompute advances g alone: 1600 nodes x 4000 steps
  // 46.9 -> 40.7 ms per gradient with single reverse steps.
  const bool many = a->most > 1;
  ENQ(cudaMemcpyAsync(a->ckpt[0], h->lat[h->cur], state_bytes, cudaMemcpyDeviceToDevice, st));
  if (many) {
    // launches of several steps, each ending at a checkpoint at the latest and writing it in place
    const double* from = (const double*)a->ckpt[0];
    for (int t = 0; t < T;) {
      const int n = std::min(std::min(a->most, T - t), K - t % K);
      double* to = (double*)h->lat[from == h->lat[0] ? 1 : 0];
      if (t + n < T && (t + n) % K == 0) to = (double*)a->ckpt[(t + n) / K];
      ENQ(enqueue_tube(h, from, to, n, a->core, false, t > 0, st));
      t += n;
      from = to;
    }
    h->cur = from == h->lat[0] ? 0 : 1;
  } else {
    for (int t = 0; t < T; ++t) {
      if (t && t % K == 0) ENQ(cudaMemcpyAsync(a->ckpt[t / K], h->lat[h->cur], state_bytes, cudaMemcpyDeviceToDevice, st));
      ENQ(enqueue_steps(h, 1, st));
    }
  }
  a->end_cur = h->cur;
  // misfit and lambda^T
  const double* gT = (const double*)h->lat[h->cur] + 19 * N;
  k_adj_loss<<<grid, th, 0, st>>>(gT, tP, tP + N, tP + 2 * N, tP + 3 * N, wP, wu, a->lam, a->lossn, N);
  ENQ(cudaGetLastError());
  ENQ(cudaMemsetAsync(a->tb, 0, 3 * N * sizeof(double), st));
  // reverse sweep, segment by segment.  Each segment is recomputed from its checkpoint
  // on the second stream into one of two state buffers (segment s into buffer s & 1),
  // so the recompute of segment s - 1 runs beside the reverse sweep of segment s; a
  // buffer is refilled only after the reverse sweep that read it.
  cudaStream_t cs = a->cap2;
  cudaEvent_t ev_fork = a->ev[0], ev_ready[2] = {a->ev[1], a->ev[2]}, ev_free[2] = {a->ev[3], a->ev[4]};
  ENQ(cudaEventRecord(ev_fork, st));
  ENQ(cudaStreamWaitEvent(cs, ev_fork, 0));
  void* saved[2] = {h->lat[0], h->lat[1]};
  const int saved_cur = h->cur;
  // g at step t0 + j of segment s
  auto g_at = [&](int s, int j) -> const double* {
    return (const double*)a->seg[s & 1][j] + (many ? 0 : 19 * N);
  };
  auto recompute = [&](int s) -> cudaError_t {
    const std::vector<void*>& b = a->seg[s & 1];
    const int t0 = s * K, t1 = std::min(T, t0 + K);
    cudaError_t r = cudaSuccess;
    if (many) {
      // g alone
      r = cudaMemcpyAsync(b[0], (const double*)a->ckpt[s] + 19 * N, 19 * N * sizeof(double), cudaMemcpyDeviceToDevice,
                          cs);
      for (int j = 0; r == cudaSuccess && j + 1 < t1 - t0;) {
        const int n = std::min(a->most, t1 - t0 - 1 - j);
        r = enqueue_tube(h, g_at(s, j), (double*)b[j + 1], n, a->core, true, j > 0, cs);
        j += n;
      }
    } else {
      r = cudaMemcpyAsync(b[0], a->ckpt[s], state_bytes, cudaMemcpyDeviceToDevice, cs);
      for (int j = 0; r == cudaSuccess && j + 1 < t1 - t0; ++j) {   // b[j] holds the state t0 + j
        h->lat[0] = b[j];
        h->lat[1] = b[j + 1];
        h->cur = 0;
        r = enqueue_steps(h, 1, cs);
      }
      h->lat[0] = saved[0];
      h->lat[1] = saved[1];
      h->cur = saved_cur;
    }
    if (r == cudaSuccess) r = cudaEventRecord(ev_ready[s & 1], cs);
    return r;
  };
  ENQ(recompute(a->nseg - 1));
  for (int s = a->nseg - 1; s >= 0; --s) {
    if (s >= 1) {
      if (s + 1 <= a->nseg - 1) ENQ(cudaStreamWaitEvent(cs, ev_free[(s + 1) & 1], 0));
      ENQ(recompute(s - 1));
    }
    ENQ(cudaStreamWaitEvent(st, ev_ready[s & 1], 0));
    const int t0 = s * K, t1 = std::min(T, t0 + K);
    if (many) {
      // the sweep, then its omega cotangents on the third stream, beside the next segment's
      for (int j = t1 - t0 - 1; j >= 0;) {
        const int c = std::min(a->most, j + 1);
        const bool first = t0 + j == T - 1;
        double* out = mu_cur == a->mu ? a->lam : a->mu;
        double* ls = a->lamseg[s & 1] + (size_t)j * 19 * N;
        launch_after(dim3((unsigned)((N + a->core - 1) / a->core)), 32 * (kTubeWarps + 1), st, j < t1 - t0 - 1,
                     mrt ? k_adj_tube_steps<true> : k_adj_tube_steps<false>, g_at(s, j), ls, first ? a->lam : mu_cur, out,
                     geo.nx, geo.zgx, h->k, c, a->core, first);
        ENQ(cudaGetLastError());
        mu_cur = out;
        j -= c;
      }
      cudaEvent_t swept = a->ev[5 + (s & 1)];
      ENQ(cudaEventRecord(swept, st));
      ENQ(cudaStreamWaitEvent(a->cap3, swept, 0));
      for (int j = 0; j < t1 - t0; j += 65535) {   // steps along the grid's y
        const dim3 go((unsigned)((N + kThreads - 1) / kThreads), (unsigned)std::min(t1 - t0 - j, 65535));
        double* lj = a->lamseg[s & 1] + (size_t)j * 19 * N;
        if (mrt) k_adj_omega<true><<<go, kThreads, 0, a->cap3>>>(g_at(s, j), lj, geo.nx, geo.zgx, h->k);
        else k_adj_omega<false><<<go, kThreads, 0, a->cap3>>>(g_at(s, j), lj, geo.nx, geo.zgx, h->k);
      }
      k_adj_omega_sum<<<(unsigned)((3 * N + kThreads - 1) / kThreads), kThreads, 0, a->cap3>>>(a->lamseg[s & 1], a->tb, N,
                                                                                               t1 - t0);
      ENQ(cudaGetLastError());
      ENQ(cudaEventRecord(ev_free[s & 1], a->cap3));
      continue;
    }
    if (a->quad && t1 == T) {   // the QFwd of the last step
      if (mrt) k_adj_fwd<true><<<grid8, 64, 0, st>>>(g_at(s, T - 1 - t0), a->fw[(T - 1) & 1], geo, h->k);
      else k_adj_fwd<false><<<grid8, 64, 0, st>>>(g_at(s, T - 1 - t0), a->fw[(T - 1) & 1], geo, h->k);
      ENQ(cudaGetLastError());
    }
    for (int t = t1 - 1; t >= t0; --t) {
      const double* gt = g_at(s, t - t0);
      // the state at step t - 1: in this segment, else the top of the one below, whose
      // recompute must have finished
      const double* g_prev = nullptr;
      bool early = a->quad && t < t1 - 1;   // no other stream waited for just before
      if (t > t0) {
        g_prev = g_at(s, t - 1 - t0);
      } else if (s >= 1) {
        ENQ(cudaStreamWaitEvent(st, ev_ready[(s - 1) & 1], 0));
        g_prev = g_at(s - 1, K - 1);
        early = false;
      }
      const double* fw = a->fw[t & 1];
      double* fw_prev = a->fw[(t + 1) & 1];
      // the last step reads lambda^T; later ones gather from the mu of the step after
      double* out = mu_cur == a->mu ? a->lam : a->mu;
      if (t == T - 1) {
        out = a->mu;
        ENQ(reverse_step<true>(a->quad, tube, mrt, grid8, grid3, th, st, early, gt, a->lam, out, a->tb, fw, g_prev, fw_prev,
                               geo, h->k, lanes));
      } else {
        ENQ(reverse_step<false>(a->quad, tube, mrt, grid8, grid3, th, st, early, gt, mu_cur, out, a->tb, fw, g_prev, fw_prev,
                                geo, h->k, lanes));
      }
      mu_cur = out;
    }
    ENQ(cudaEventRecord(ev_free[s & 1], st));
  }
  // join the second stream back into the capture
  ENQ(cudaEventRecord(ev_fork, cs));
  ENQ(cudaStreamWaitEvent(st, ev_fork, 0));
  if (many) ENQ(cudaStreamWaitEvent(st, ev_free[0], 0));   // segment 0's omega cotangents, the last of that stream
  ENQ(cudaGetLastError());
  k_adj_e0<<<grid3, th, 0, st>>>((const double*)a->ckpt[0] + 19 * N, mu_cur, a->dde0, unit, geo, lanes);
  k_rowsum<<<3, 256, 0, st>>>(a->tb, N, a->sums);
  k_rowsum<<<1, 256, 0, st>>>(a->lossn, N, a->sums + 3);
  ENQ(cudaGetLastError());
#undef ENQ
  return cudaSuccess;
}

}  // namespace

extern "C" int rlb_adjoint(rlb_handle* h, int nsteps, int checkpoint_every, const double* target_P,
                           const double* target_ux, const double* target_uy, const double* target_uz, double w_P,
                           double w_u, int where, double* loss, double* dtau, double* de0) {
  if (!h) return RLB_EINVAL;
  if (nsteps < 1) return afail(h, RLB_EINVAL, "nsteps must be >= 1");
  if (!target_P || !target_ux || !target_uy || !target_uz || !loss || !dtau)
    return afail(h, RLB_EINVAL, "null argument");
  if (where != RLB_HOST && where != RLB_DEVICE) return afail(h, RLB_EINVAL, "where must be RLB_HOST or RLB_DEVICE");
  if (h->esize != 8) return afail(h, RLB_EINVAL, "rlb_adjoint needs an RLB_FP64 lattice");
  if (h->Q != 19) return afail(h, RLB_EINVAL, "rlb_adjoint supports RLB_D3Q19 lattices");
  if (h->cfg.eta_over_s > 0) return afail(h, RLB_EINVAL, "rlb_adjoint needs constant relaxation times");
  if (h->cfg.collision == RLB_MRT && h->cfg.tau_q > 0 && h->cfg.tau_q != h->cfg.tau_v)
    return afail(h, RLB_EINVAL, "rlb_adjoint needs tau_q tied to tau_v (tau_q <= 0)");
  const bool mrt = h->cfg.collision == RLB_MRT;
  const unsigned long long N = h->nodes;
  const size_t state_bytes = 38 * N * sizeof(double), gbytes = 19 * N * sizeof(double);
  const int K = checkpoint_every > 0 ? checkpoint_every : std::max(1, (int)std::ceil(std::sqrt((double)nsteps)));
  cudaStream_t st = h->stream;

#define ACUDA(call)                                                                       \
  do {                                                                                    \
    cudaError_t e_ = (call);                                                              \
    if (e_ != cudaSuccess) return afail(h, RLB_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

  // ---- plan (buffers + graph) for this shape
  AdjPlan* a = (AdjPlan*)h->adj_plan;
  if (a && (a->nsteps != nsteps || a->K != std::min(K, nsteps))) {
    ACUDA(cudaStreamSynchronize(st));
    free_plan(a);
    h->adj_plan = nullptr;
    a = nullptr;
  }
  if (!a) {
    a = new AdjPlan();
    a->nsteps = nsteps;
    a->K = std::min(K, nsteps);
    a->nseg = (nsteps + a->K - 1) / a->K;
    a->threads = N <= 152ull * 128ull * 2ull ? 32 : 128;
    // one node per thread (blocks with fewer active lanes, spreading a small lattice
    // over more SMs, measured slower on GB300)
    a->lanes = a->threads;
    // below ~2 warps per SM the one-thread-per-node step is one thread's dependent
    // chain; four threads per node shorten it (the scalar chain is repeated, so on
    // larger lattices, where the FP64 pipe is the limit, one thread per node is kept).
    // 1600-node tube, 4000 steps: 109 -> 87 ms per gradient on GB300.
    a->quad = a->threads == 32;
    a->ckpt.assign(a->nseg, nullptr);
    a->most = tube_launch_steps(h, a->core);
    std::vector<PlanWant> want;
    size_t total = 0;
    const auto need = [&](void** p, size_t bytes) { plan_alloc(want, total, p, bytes); };
    for (int s = 0; s < a->nseg; ++s) need(&a->ckpt[s], state_bytes);
    void* all[2] = {nullptr, nullptr};
    for (int q = 0; q < 2; ++q) {
      a->seg[q].assign(a->K + 1, nullptr);
      if (a->most > 1) {
        need(&all[q], (size_t)a->K * gbytes);
        need((void**)&a->lamseg[q], (size_t)a->K * gbytes);
      } else {
        for (int j = 0; j <= a->K; ++j) need(&a->seg[q][j], state_bytes);
      }
    }
    need((void**)&a->lam, gbytes);
    need((void**)&a->mu, gbytes);
    need((void**)&a->tb, 3 * N * sizeof(double));
    need((void**)&a->lossn, N * sizeof(double));
    need((void**)&a->sums, 8 * sizeof(double));
    need((void**)&a->dde0, N * sizeof(double));
    need((void**)&a->tgt, 4 * N * sizeof(double));
    for (int i = 0; i < 2 && a->quad && a->most == 1; ++i)
      need((void**)&a->fw[i], (kFwdFields + 9 * kPairFields) * N * sizeof(double));
    bool ok = plan_commit(a, want, total);
    for (int q = 0; q < 2 && a->most > 1; ++q)
      for (int j = 0; j < a->K; ++j) a->seg[q][j] = (char*)all[q] + (size_t)j * gbytes;
    for (int i = 0; i < 7 && ok; ++i) ok = cudaEventCreateWithFlags(&a->ev[i], cudaEventDisableTiming) == cudaSuccess;
    ok = ok && cudaStreamCreateWithFlags(&a->cap2, cudaStreamNonBlocking) == cudaSuccess &&
         cudaStreamCreateWithFlags(&a->cap3, cudaStreamNonBlocking) == cudaSuccess;
    if (!ok || cudaStreamCreateWithFlags(&a->cap, cudaStreamNonBlocking) != cudaSuccess) {
      free_plan(a);
      return afail(h, RLB_ENOMEM, "cannot allocate adjoint checkpoints and buffers");
    }
    a->start_cur = h->cur;
    h->adj_plan = a;
    h->adj_free = free_plan;
  }
  // a refused call (a stream under capture: nothing has run) leaves the state where it was
  const long long steps_before = h->steps;
  struct Keep {
    rlb_handle* h;
    int cur;
    long long steps;
    ~Keep() {
      h->cur = cur;
      h->steps = steps;
    }
  } keep{h, h->cur, h->steps};
  // the graph's lattice pointers assume the state starts in lat[start_cur]
  if (h->cur != a->start_cur) {
    ACUDA(cudaMemcpyAsync(h->lat[a->start_cur], h->lat[h->cur], state_bytes, cudaMemcpyDeviceToDevice, st));
    h->cur = a->start_cur;
  }
  // targets into the plan's buffer (outside the graph)
  {
    const double* src[4] = {target_P, target_ux, target_uy, target_uz};
    for (int c = 0; c < 4; ++c)
      ACUDA(cudaMemcpyAsync(a->tgt + c * N, src[c], N * sizeof(double),
                            where == RLB_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice, st));
  }
  // Enqueued as it is, without a graph: every gradient with several steps per launch (its
  // launches are few enough for the host to keep ahead; 1600 nodes x 4000 steps took 27.3 ms
  // so and 27.2 from a graph), and the first gradient of any plan (a program that makes a new
  // lattice per gradient, as the autograd function does, would not use a graph twice: 800
  // nodes x 400 steps 5.1 -> 3.6 ms per call with the plan's buffers in one allocation).
  const bool direct = a->most > 1 || a->runs++ == 0;
  // The integer walk keeps cotangents down to 2^-959: tiny weights are brought near 1 by a power
  // of two (the gradient is linear in them) and the results taken back.
  int up = 0;
  if (a->most > 1) {
    const double big = std::max(std::fabs(w_P), std::fabs(w_u));
    if (big > 0.0 && big < 0x1p-400) up = -std::ilogb(big);
  }
  if (direct) {
    const cudaError_t de = enqueue_adjoint(h, a, std::ldexp(w_P, up), std::ldexp(w_u, up), std::ldexp(1.0, -up), mrt, st);
    if (de != cudaSuccess) return afail(h, RLB_ECUDA, std::string("adjoint launch: ") + cudaGetErrorString(de));
  }
  // capture once per plan (the misfit weights are kernel arguments: recapture if they change)
  if (!direct && (!a->exec || a->wP != w_P || a->wu != w_u)) {
    if (a->exec) { cudaGraphExecDestroy(a->exec); a->exec = nullptr; }
    if (a->graph) { cudaGraphDestroy(a->graph); a->graph = nullptr; }
    const long long steps0 = h->steps;
    ACUDA(cudaStreamBeginCapture(a->cap, cudaStreamCaptureModeThreadLocal));
    cudaError_t ce = enqueue_adjoint(h, a, w_P, w_u, 1.0, mrt, a->cap);
    cudaGraph_t g = nullptr;
    cudaError_t ee = cudaStreamEndCapture(a->cap, &g);
    h->cur = a->start_cur;   // nothing ran yet
    h->steps = steps0;
    if (ce != cudaSuccess || ee != cudaSuccess) {
      if (g) cudaGraphDestroy(g);
      return afail(h, RLB_ECUDA, std::string("adjoint graph capture: ") + cudaGetErrorString(ce != cudaSuccess ? ce : ee));
    }
    a->graph = g;
    ACUDA(cudaGraphInstantiate(&a->exec, a->graph, 0));
    a->wP = w_P;
    a->wu = w_u;
  }
  if (!direct) ACUDA(cudaGraphLaunch(a->exec, st));
  double hs[4];
  ACUDA(cudaMemcpyAsync(hs, a->sums, 4 * sizeof(double), cudaMemcpyDeviceToHost, st));
  if (de0)
    ACUDA(cudaMemcpyAsync(de0, a->dde0, N * sizeof(double),
                          where == RLB_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice, st));
  ACUDA(cudaStreamSynchronize(st));
  keep.cur = a->end_cur;
  keep.steps = steps_before + nsteps;
  {
    unsigned long long bad = ~0ull;
    ACUDA(cudaMemcpy(&bad, h->d_bad, sizeof bad, cudaMemcpyDeviceToHost));
    if (bad != ~0ull) {
      const unsigned long long none = ~0ull;
      ACUDA(cudaMemcpy(h->d_bad, &none, sizeof none, cudaMemcpyHostToDevice));
      char buf[128];
      std::snprintf(buf, sizeof buf, "non-physical state at node %llu during the forward run", bad);
      return afail(h, RLB_ENONPHYS, buf);
    }
  }
  // omega = 1 / tau  =>  dJ/dtau = -omega^2 dJ/domega
  const double wv = 1.0 / h->cfg.tau_v;
  *loss = std::ldexp(hs[3], -up);
  dtau[0] = std::ldexp(-wv * wv * hs[0], -up);
  if (mrt) {
    const double we = 1.0 / h->cfg.tau_e, wp = 1.0 / h->cfg.tau_eps;
    dtau[1] = std::ldexp(-we * we * hs[1], -up);
    dtau[2] = std::ldexp(-wp * wp * hs[2], -up);
  } else {
    dtau[1] = 0.0;
    dtau[2] = 0.0;
  }
  return RLB_OK;
#undef ACUDA
}
