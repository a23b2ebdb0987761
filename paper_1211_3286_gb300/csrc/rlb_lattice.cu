// rlb_lattice.cu -- the lattice handle of librlb: allocation, initial state,
// fused pull-stream + collide step kernels, field output, conserved totals and
// raw state I/O (the C ABI declared in include/rlb.h).
//
// Data layout in HBM: two lattices (read / write, swapped every step), each
// holding f[19][nz][ny][nx] followed by g[19][nz][ny][nx] in the storage
// precision (FP64, or FP32 for RLB_FP32_STORAGE).  Populations are pulled from
// x - e_a (x-adjacent threads read adjacent addresses, so every load is
// coalesced), collided in registers with the per-node arithmetic of rlb_node.cuh,
// and written to the node's own slots.
//   FP64 (k_step_ws): two threads per node -- g warps (sums, recovery, g update)
//     and f warps (f update) of the same nodes, u handed over in shared memory;
//   FP32 storage (k_step): one thread per node;
//   D2Q9 (k_step_d2q9): one thread per node on the same integers, with k_macro_d2q9 first
//     when the C7 correction needs gradients of the macroscopic fields.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/rlb.h"
#include "rlb_internal.h"
#include "rlb_io.cuh"
#include "rlb_launch.cuh"
#include "rlb_node.cuh"
#include "rlb_quad.cuh"

using namespace rlb;


namespace {

thread_local std::string g_create_error;

int fail(rlb_handle* h, int code, const std::string& msg) {
  if (h) h->err = msg;
  else g_create_error = msg;
  return code;
}

int cuda_fail(rlb_handle* h, cudaError_t e, const char* what) {
  return fail(h, RLB_ECUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

#define RLB_CUDA(h, call)                               \
  do {                                                  \
    cudaError_t e_ = (call);                            \
    if (e_ != cudaSuccess) return cuda_fail(h, e_, #call); \
  } while (0)

constexpr int kBlockX = 128;
constexpr unsigned long long kSmallNodes = 152ull * 128ull * 2ull;   // lattices that cannot fill the GPU
constexpr int kRedBlocks = 608;   // 4 x 152 SMs; fixed so the reduction order is fixed
constexpr int kRedThreads = 256;

struct Geo {
  int nx, ny, nz;
  int bcx, bcy, bcz;   // 1 = zero-gradient
  unsigned long long plane;   // nodes
  // floor(2^64 / n) + 1 (0 for n = 1): the high half of its product with i < 2^32 is i / n
  unsigned long long inv_nx, inv_ny;
};

__device__ __forceinline__ int src_minus(int i, int n, int zg) {  // source of a pull with c = +1
  return i > 0 ? i - 1 : (zg ? 0 : n - 1);
}
__device__ __forceinline__ int src_plus(int i, int n, int zg) {   // source of a pull with c = -1
  return i < n - 1 ? i + 1 : (zg ? n - 1 : 0);
}

// Population load, coherent: the grid before may still be writing when this one is resident
// (wait_for_grid).  FP64 populations are streamed past L1 (each value is read once per step
// from its plane; L2 serves the neighbouring rows' reuse), which leaves L1 to the FP64 step's
// register spills.  L2 prefetch size 256 B, the row segment a warp reads (512^3 FP32 step
// 6.763 -> 6.740 ms, 256^3 FP64 step 1.859 -> 1.856 ms).
template <typename S>
__device__ __forceinline__ S ld_pop(const S* p) {
  S v;
  if constexpr (sizeof(S) == 8) asm("ld.global.L1::no_allocate.L2::256B.f64 %0, [%1];" : "=d"(v) : "l"(p));
  else asm("ld.global.L2::256B.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}

// Gather the 19 populations of one distribution arriving at node (x, y, z):
// link a comes from (x - cx, y - cy, z - cz).
template <typename S>
__device__ __forceinline__ void pull19(const S* __restrict__ base, unsigned long long plane, const int (&xs)[3],
                                       const unsigned (&row)[3][3], S (&v)[19]) {
#pragma unroll
  for (int a = 0; a < 19; ++a) {
    const int cx = link_cx(a), cy = link_cy(a), cz = link_cz(a);
    const unsigned idx = row[1 - cz][1 - cy] + (unsigned)xs[1 - cx];
    v[a] = ld_pop(base + (unsigned long long)a * plane + idx);
  }
}

// The same with the node's index and the index offsets of its pulls (rows numbered one
// after the other, so a warp's lanes may lie in different rows).
struct Nbr3 {
  int xm, xp, ym, yp, zm, zp;   // a pull with c = +1 / -1 along each axis
};
__device__ __forceinline__ Nbr3 neighbours3(const Geo& geo, unsigned i) {
  const unsigned q = geo.inv_nx ? (unsigned)__umul64hi(i, geo.inv_nx) : i;       // y + ny z
  const unsigned z = geo.inv_ny ? (unsigned)__umul64hi(q, geo.inv_ny) : q;
  const int x = (int)(i - q * (unsigned)geo.nx), y = (int)(q - z * (unsigned)geo.ny);
  const int nxy = geo.nx * geo.ny, top = (int)geo.plane - nxy;
  Nbr3 b;
  b.xm = x > 0 ? -1 : (geo.bcx ? 0 : geo.nx - 1);
  b.xp = x < geo.nx - 1 ? 1 : (geo.bcx ? 0 : 1 - geo.nx);
  b.ym = y > 0 ? -geo.nx : (geo.bcy ? 0 : nxy - geo.nx);
  b.yp = y < geo.ny - 1 ? geo.nx : (geo.bcy ? 0 : geo.nx - nxy);
  b.zm = z > 0 ? -nxy : (geo.bcz ? 0 : top);
  b.zp = (int)z < geo.nz - 1 ? nxy : (geo.bcz ? 0 : -top);
  return b;
}
template <typename S>
__device__ __forceinline__ void pull19(const S* __restrict__ base, unsigned long long plane, unsigned i, const Nbr3& b,
                                       S (&v)[19]) {
#pragma unroll
  for (int a = 0; a < 19; ++a) {
    const int cx = link_cx(a), cy = link_cy(a), cz = link_cz(a);
    const unsigned idx = i + (unsigned)((cx > 0 ? b.xm : cx < 0 ? b.xp : 0) + (cy > 0 ? b.ym : cy < 0 ? b.yp : 0) +
                                        (cz > 0 ? b.zm : cz < 0 ? b.zp : 0));
    v[a] = ld_pop(base + (unsigned long long)a * plane + idx);
  }
}

// Resident 128-thread blocks per SM the FP32-storage step is compiled for (6: 80
// registers, none spilled)
#ifndef RLB_F32_BLOCKS_PER_SM
#define RLB_F32_BLOCKS_PER_SM 6
#endif

// FLAT: thread i of the grid takes node i, whatever the row length; else the grid's y and
// z are the lattice's and each row has its own blocks, with the row offsets the same for
// all lanes (flat_rows below says which).
template <typename S, bool MRT, bool QSEP, bool FLAT>
__global__ void __launch_bounds__(kBlockX, RLB_F32_BLOCKS_PER_SM) k_step(const S* __restrict__ src,
                                                                         S* __restrict__ dst, Geo geo, StepConst k,
                                                                         unsigned long long* __restrict__ bad) {
  S f[19], g[19];
  unsigned node;
  if constexpr (FLAT) {
    node = blockIdx.x * blockDim.x + threadIdx.x;
    if (node >= geo.plane) return;
    const Nbr3 nb = neighbours3(geo, node);
    wait_for_grid(src);
    pull19<S>(src, geo.plane, node, nb, f);
    pull19<S>(src + 19ull * geo.plane, geo.plane, node, nb, g);
  } else {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= geo.nx) return;
    const int y = blockIdx.y, z = blockIdx.z;
    // source coordinates for offsets c = +1, 0, -1 (index 0, 1, 2 = 1 - c)
    const int xs[3] = {src_minus(x, geo.nx, geo.bcx), x, src_plus(x, geo.nx, geo.bcx)};
    const int ys[3] = {src_minus(y, geo.ny, geo.bcy), y, src_plus(y, geo.ny, geo.bcy)};
    const int zs[3] = {src_minus(z, geo.nz, geo.bcz), z, src_plus(z, geo.nz, geo.bcz)};
    unsigned row[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j)
        row[i][j] = ((unsigned)zs[i] * (unsigned)geo.ny + (unsigned)ys[j]) * (unsigned)geo.nx;
    wait_for_grid(src);
    pull19<S>(src, geo.plane, xs, row, f);
    pull19<S>(src + 19ull * geo.plane, geo.plane, xs, row, g);
    node = row[1][1] + (unsigned)x;
  }
  const bool b = node_collide_f32s<MRT, QSEP>(f, g, k);
  if (b) atomicMin(bad, (unsigned long long)node);
#pragma unroll
  for (int a = 0; a < 19; ++a) {
    dst[(unsigned long long)a * geo.plane + node] = f[a];
    dst[(19ull + a) * geo.plane + node] = g[a];
  }
}

// FP64 step with warp roles (the integer-pipe collide of rlb_node.cuh).  A block of
// 2 W warps serves 32 W nodes along x: warps [0, W) pull and relax g, warps [W, 2W)
// pull and relax f of the same nodes.  The g warps recover u (Eq. 10 inverted) and
// hand it to the f warps through shared memory across one barrier per warp pair.  Each
// thread holds one distribution of one node, so twice as many warps fit in the
// registers the single-role kernel needs; out-of-range threads (x >= nx) pull the
// clamped node nx - 1, pass the barrier and store that node's values again.
// Resident warps per SM the launch bounds ask of the large-lattice blocks (the
// register cap follows: 24 warps -> 80 registers, 40 B spilled; 32 warps -> 64
// registers, 184 B spilled with the shift-free relaxation, which keeps X^eq live past
// the product); small lattices keep 14 64-thread blocks.
#ifndef RLB_WS_WARPS_PER_SM
#define RLB_WS_WARPS_PER_SM 24
#endif
// Output rounding route of the f and g warps, one bit per link pair and bit 9 for
// the rest link: set = FP64-pipe conversion, clear = integer bit assembly with the
// FP64 pipe only for negative or tiny values (fx::from_fixed_pos).
#ifndef RLB_WS_OUT_F
#define RLB_WS_OUT_F 0x3ff
#endif
#ifndef RLB_WS_OUT_G
#define RLB_WS_OUT_G 0x3ff
#endif
// warps per role in the blocks of large lattices (4: 256-thread blocks serving 128
// nodes along x)
#ifndef RLB_WS_WARPS
#define RLB_WS_WARPS 4
#endif

// ETA (RV = RF = 0): relaxation rates per node from a fixed eta/s.  The f warps hand N0 to
// the g warps, which form the rates (eta_rates) and hand omega_f back across a second
// barrier; a node outside that form's range is left to its g lane, which runs the FP64 form
// for both distributions.  128 x 96 x 80 MRT with its own tau_q: 598 -> 182 us per step (FP64
// arithmetic held the FP64 pipe 88 % busy with 329 instructions per node, now 46; the limit
// is the integer instruction stream, issue 57 %, of which 400 bytes of spills per thread in
// the tau_q form are part).
template <bool MRT, bool QSEP>
__device__ __noinline__ void step_eta_general(const double* __restrict__ src, double* __restrict__ dst, const Geo& geo,
                                              const StepConst& k, unsigned long long* __restrict__ bad, unsigned node) {
  double f[19], g[19];
  const Nbr3 nb = neighbours3(geo, node);
  pull19<double>(src, geo.plane, node, nb, f);
  pull19<double>(src + 19ull * geo.plane, geo.plane, node, nb, g);
  if (node_collide_f64<MRT, QSEP>(f, g, k)) atomicMin(bad, (unsigned long long)node);
#pragma unroll
  for (int a = 0; a < 19; ++a) {
    dst[(unsigned long long)a * geo.plane + node] = f[a];
    dst[(19ull + a) * geo.plane + node] = g[a];
  }
}

template <int W, bool MRT, bool QSEP, bool FLAT, int RV, int RF, bool ETA = false>
__global__ void __launch_bounds__(64 * W, W == 1 ? (ETA ? 8 : 14) : RLB_WS_WARPS_PER_SM / (2 * W))
    k_step_ws(const double* __restrict__ src, double* __restrict__ dst, const __grid_constant__ Geo geo,
              const __grid_constant__ StepConst k,
              unsigned long long* __restrict__ bad) {
  __shared__ unsigned long long s_ax[32 * W], s_ay[32 * W], s_az[32 * W];
  __shared__ unsigned s_sg[32 * W];
  __shared__ unsigned long long s_n[ETA ? 32 * W : 1];
  __shared__ int s_e[ETA ? 32 * W : 1];
  const int warp = threadIdx.x >> 5;
  const bool is_g = warp < W;
  const int slot = (is_g ? warp : warp - W) * 32 + (threadIdx.x & 31);
  const unsigned long long plane0 = is_g ? 19ull * geo.plane : 0ull;
  double v[19];
  unsigned node;
  bool valid;
  if constexpr (FLAT) {
    const unsigned i = blockIdx.x * (32 * W) + slot;
    valid = i < geo.plane;
    node = valid ? i : (unsigned)geo.plane - 1;
    const Nbr3 nb = neighbours3(geo, node);
    wait_for_grid(src);
    pull19<double>(src + plane0, geo.plane, node, nb, v);
  } else {
    const int x0 = blockIdx.x * (32 * W) + slot;
    valid = x0 < geo.nx;
    const int x = valid ? x0 : geo.nx - 1;
    const int y = blockIdx.y, z = blockIdx.z;
    const int xs[3] = {src_minus(x, geo.nx, geo.bcx), x, src_plus(x, geo.nx, geo.bcx)};
    const int ys[3] = {src_minus(y, geo.ny, geo.bcy), y, src_plus(y, geo.ny, geo.bcy)};
    const int zs[3] = {src_minus(z, geo.nz, geo.bcz), z, src_plus(z, geo.nz, geo.bcz)};
    unsigned row[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j)
        row[i][j] = ((unsigned)zs[i] * (unsigned)geo.ny + (unsigned)ys[j]) * (unsigned)geo.nx;
    wait_for_grid(src);
    pull19<double>(src + plane0, geo.plane, xs, row, v);
    node = row[1][1] + (unsigned)x;
  }

  using namespace fx;
  // both roles: block exponent and fixed-point values.  When every value of every
  // lane of the warp is positive, finite and within 2^24 of its node's largest (the
  // normal case), the conversion skips the sign and the long-shift handling.
  int hmax = __double2hiint(v[0]), hmin = hmax;
#pragma unroll
  for (int a = 1; a < 19; ++a) {
    const int h = __double2hiint(v[a]);
    hmax = max(hmax, h);
    hmin = min(hmin, h);
  }
  const bool fast = __all_sync(0xffffffffu, hmin > 0 && hmax < 0x7ff00000 && hmin >= (((hmax >> 20) - 24) << 20));
  int E;
  long long X[19];
  if (fast) {
    E = hmax >> 20;
#pragma unroll
    for (int a = 0; a < 19; ++a) X[a] = to_fixed_pos(v[a], E + 7);
  } else {
    unsigned me = 0;
#pragma unroll
    for (int a = 0; a < 19; ++a) me = max(me, (unsigned)__double2hiint(v[a]) & 0x7ff00000u);
    E = (int)(me >> 20);
#pragma unroll
    for (int a = 0; a < 19; ++a) X[a] = to_fixed(v[a], E + 7);
  }

  UFix u;
  long long Sa = 0, Sd = 0, T00 = 0, Mx = 0, My = 0, Mz = 0, Pf = 0, dp0 = 0, dp1 = 0, dp2 = 0, N0 = 0;
  unsigned long long sig = 0;
  bool b = (E < 64) | (E > 2046);
  if (is_g) {
    // conserved sums (Eq. 10) and the recovery on them, in fixed point
    long long sp[9], dp[9];
#pragma unroll
    for (int p = 0; p < 9; ++p) {
      sp[p] = X[2 * p + 1] + X[2 * p + 2];
      dp[p] = X[2 * p + 1] - X[2 * p + 2];
    }
    dp0 = dp[0]; dp1 = dp[1]; dp2 = dp[2];
    Sa = sp[0] + sp[1] + sp[2];
    Sd = ((sp[3] + sp[4]) + (sp[5] + sp[6])) + (sp[7] + sp[8]);
    T00 = X[0] + Sa + Sd;
    Mx = dp[0] + dp[3] + dp[4] + dp[5] + dp[6];
    My = dp[1] + dp[3] - dp[4] + dp[7] + dp[8];
    Mz = dp[2] + dp[5] - dp[6] + dp[7] - dp[8];
    bool br;
    sig = fx_recover(T00, Mx, My, Mz, u, br);
    Pf = (long long)sig - T00;
    s_ax[slot] = u.ax;
    s_ay[slot] = u.ay;
    s_az[slot] = u.az;
    s_sg[slot] = u.sx | (u.sy << 1) | (u.sz << 2);
    ufix_products(u);
    b |= br | (Pf <= 0) | (u.xx + u.yy + u.zz >= (1ull << 62));
  } else {
    N0 = X[0];
#pragma unroll
    for (int a = 1; a < 19; ++a) N0 += X[a];
    if (ETA) {
      s_n[slot] = (unsigned long long)N0;
      s_e[slot] = E;
    }
  }
  // g warp i hands u to f warp i only: one named barrier per warp pair (ids 1..W, 64
  // threads each), so a slow g warp holds back its own f warp, not the whole block
  asm volatile("bar.sync %0, 64;" ::"r"(1 + (is_g ? warp : warp - W)) : "memory");
  if (!is_g) {
    u.ax = s_ax[slot];
    u.ay = s_ay[slot];
    u.az = s_az[slot];
    const unsigned sg = s_sg[slot];
    u.sx = sg & 1u;
    u.sy = (sg >> 1) & 1u;
    u.sz = sg >> 2;
    ufix_products(u);
  }

  // equilibria (Eqs. 7-9) and the relaxation constants of this role
  EqPieces q;
  eq_pieces(is_g ? sig : (unsigned long long)N0, u, q);
  const long long SX = q.Xx + q.Xy + q.Xz;             // D u^2 / 4
  long long eq0;
  if (is_g) {
    q.KA = (long long)mulhi((unsigned long long)Pf, kSixth) - (long long)mulhi((unsigned long long)SX, kThird);
    eq0 = (long long)sig - 3 * Pf - 2 * SX;             // sigma - 3P - sigma u^2 / 2
  } else {
    q.KA = (long long)mulhi((unsigned long long)N0, kEighteenth) - (long long)mulhi((unsigned long long)SX, kThird);
    eq0 = (long long)mulhi((unsigned long long)N0, kThird) - 2 * SX;   // N0/3 - N0 u^2 / 2
  }
  long long hM[3] = {0, 0, 0};
  if (ETA) {
    // sums of the equilibrium equal to the populations' (relax_links_store, EXACT): the FP64
    // arithmetic of this mode's general form does not drift as truncated integers do
    const long long h = ((q.Xx + q.Xy) >> 1) + ((q.Xx + q.Xz) >> 1) + ((q.Xy + q.Xz) >> 1);
    eq0 = (is_g ? T00 : N0) - (6 * q.KA + 2 * SX + 12 * (q.KA >> 1) + 4 * h);
    if (is_g) {
      hM[0] = Mx >> 1;
      hM[1] = My >> 1;
      hM[2] = Mz >> 1;
    } else {   // N0 u / 2
      hM[0] = with_sign(mulhi((unsigned long long)N0, u.ax), u.sx);
      hM[1] = with_sign(mulhi((unsigned long long)N0, u.ay), u.sy);
      hM[2] = with_sign(mulhi((unsigned long long)N0, u.az), u.sz);
    }
  }
  // shift-free relaxation (fx::relax_r): RV / RF = 2 for omega >= 1, 1 below
  unsigned long long Om = is_g ? k.Om2_v : k.Om2_f;
  long long CE = k.CE, CP = k.CP, CQ = k.CQ;
  if constexpr (ETA) {
    bool gen = false;
    if (is_g) {
      Rates r;
      gen = !eta_rates<MRT, QSEP>((long long)s_n[slot], s_e[slot], sig, Pf, E, k, r) || b;
      // 1 for the FP64 form: no rate is odd (0 is one: tau_f above 2^62).  This lane alone reads N0
      s_n[slot] = gen ? 1ull : r.Omf;
      Om = r.Omv;
      CE = r.CE;
      CP = r.CP;
      CQ = r.CQ;
    }
    asm volatile("bar.sync %0, 64;" ::"r"(1 + (is_g ? warp : warp - W)) : "memory");
    if (!is_g) {
      Om = s_n[slot];
      gen = Om == 1;
    }
    if (gen) {
      if (is_g && valid) step_eta_general<MRT, QSEP>(src, dst, geo, k, bad, node);
      return;
    }
  }
  // 1: truncation of the product (none for omega = 0, a frozen distribution)
  long long c0 = (long long)(Om >> 1) - (ETA ? (long long)(Om != 0) : 0), cA = c0, cD = c0;
  long long aq[3] = {0, 0, 0};
  if (MRT && is_g) {
    // e and eps projections of g - g^eq from the class sums, at 1/8 scale
    const long long n0 = (X[0] - eq0) >> 3;
    const long long nA = (Sa - Pf) >> 3;
    const long long nD = (Sd - Pf - 2 * SX) >> 3;
    const long long ae = __mul64hi(8 * nD - 11 * nA - 30 * n0, CE) >> 6;
    const long long ap = __mul64hi(nD - 4 * nA + 12 * n0, CP) >> 2;
    c0 += 30 * ae - 12 * ap;
    cA += 11 * ae + 4 * ap;
    cD -= 8 * ae + ap;
    if (QSEP) {
      const unsigned long long h23 = kTwoThirds >> 1;
      const long long vx = ((Mx - 5 * dp0) >> 2) + (mulhi_su(Mx, kTwoThirds, h23) >> 2);
      const long long vy = ((My - 5 * dp1) >> 2) + (mulhi_su(My, kTwoThirds, h23) >> 2);
      const long long vz = ((Mz - 5 * dp2) >> 2) + (mulhi_su(Mz, kTwoThirds, h23) >> 2);
      aq[0] = __mul64hi(vx, CQ) >> 1;
      aq[1] = __mul64hi(vy, CQ) >> 1;
      aq[2] = __mul64hi(vz, CQ) >> 1;
    }
  }
  if (valid && b) atomicMin(bad, (unsigned long long)node);
  // Lanes past the row repeat node nx - 1 and compute its values bit for bit, so every
  // lane stores: those lanes write the same bytes to node nx - 1 again, and no branch
  // guards the 19 stores (1.8164 -> 1.7977 ms per 256^3 step).
  double* out = dst + plane0 + node;
  if (ETA) {   // RV = 0 for both roles
    relax_links_store<0, MRT && QSEP, 0, true>(X, q, Om, cA, cD, aq, E, out, geo.plane, true, hM, is_g ? T00 : N0);
  } else if (is_g) {
    out[0] = from_fixed<(RLB_WS_OUT_G >> 9) & 1>(relax_r<RV>(X[0], eq0, Om, c0), E);
    relax_links_store<RLB_WS_OUT_G, MRT && QSEP, RV>(X, q, Om, cA, cD, aq, E, out, geo.plane, true);
  } else {
    out[0] = from_fixed<(RLB_WS_OUT_F >> 9) & 1>(relax_r<RF>(X[0], eq0, Om, c0), E);
    relax_links_store<RLB_WS_OUT_F, false, RF>(X, q, Om, cA, cD, aq, E, out, geo.plane, true);
  }
}

// ---- FP64 steps of small lattices: four lanes per node and distribution
//
// A g warp holds the g of 8 nodes along x, an f warp their f.  Lane j = 0, 1, 2 of a node
// holds axis pair j (links 2j + 1, 2j + 2) and the two diagonal pairs of one plane, (a, b)
// = (x, y), (y, z), (x, z): the pairs e_a + e_b and e_a - e_b (pairs 3-4, 7-8, 5-6), six
// links each; lane 3 holds the rest link.  The block exponent, the exact integer sums and
// the rest value are combined over the node's lanes with shuffles, the recovery and the
// equilibrium pieces run in every lane, and each lane relaxes its own links: the
// arithmetic of k_step_ws, link for link, with a node's dependent chain about a third as
// long.  u goes to the f warp through shared memory across a named barrier of the warp
// pair.  No separate tau_q (QSEP) in this form.
// u of the 8 nodes of a warp pair
struct QuadU {
  unsigned long long ax[8], ay[8], az[8];
  unsigned sg[8];
};
// Collides the pulled values v of lane (m, j) and leaves the relaxed ones in v (lane 3:
// the rest link in v[0]); true if the node is non-physical (valid in every lane of a g
// warp; of an f warp: its own exponent).  PAIR: an f warp runs beside the g warp (named
// barrier bar_id); else g alone.
template <bool MRT, int RV, int RF, bool PAIR = true>
__device__ __forceinline__ bool quad_collide(bool is_g, int lane, double (&v)[6], const StepConst& k, QuadU& su,
                                             int bar_id) {
  using namespace fx;
  const int m = lane >> 2, j = lane & 3;
  const int ai = j < 3 ? j : 0, da = j == 1 ? 1 : 0, db = j == 0 ? 1 : 2;
  // block exponent over the node's 19 values (max over its four lanes)
  int hmax = __double2hiint(v[0]), hmin = hmax;
#pragma unroll
  for (int sl = 1; sl < 6; ++sl) {
    const int h = __double2hiint(v[sl]);
    hmax = max(hmax, h);
    hmin = min(hmin, h);
  }
  hmax = max(hmax, __shfl_xor_sync(0xffffffffu, hmax, 1));
  hmax = max(hmax, __shfl_xor_sync(0xffffffffu, hmax, 2));
  const bool fast = __all_sync(0xffffffffu, hmin > 0 && hmax < 0x7ff00000 && hmin >= (((hmax >> 20) - 24) << 20));
  int E;
  long long X[6];
  if (fast) {
    E = hmax >> 20;
#pragma unroll
    for (int sl = 0; sl < 6; ++sl) X[sl] = to_fixed_pos(v[sl], E + 7);
  } else {
    unsigned me = 0;
#pragma unroll
    for (int sl = 0; sl < 6; ++sl) me = max(me, (unsigned)__double2hiint(v[sl]) & 0x7ff00000u);
    me = max(me, (unsigned)__shfl_xor_sync(0xffffffffu, (int)me, 1));
    me = max(me, (unsigned)__shfl_xor_sync(0xffffffffu, (int)me, 2));
    E = (int)(me >> 20);
#pragma unroll
    for (int sl = 0; sl < 6; ++sl) X[sl] = to_fixed(v[sl], E + 7);
  }
  const int base = lane & ~3;
  const long long Xr = __shfl_sync(0xffffffffu, X[0], base + 3);   // the rest link's value
  const long long spa = X[0] + X[1], dpa = X[0] - X[1];
  const long long spp = X[2] + X[3], dpp = X[2] - X[3];
  const long long spm = X[4] + X[5], dpm = X[4] - X[5];
  const bool pairs = j < 3;
  UFix u;
  unsigned long long sig = 0;
  long long Pf = 0, Sa = 0, Sd = 0, N0 = 0;
  bool b = (E < 64) | (E > 2046);
  if (is_g) {
    Sa = quad_sum64(pairs ? spa : 0);
    Sd = quad_sum64(pairs ? spp + spm : 0);
    const long long T00 = Xr + Sa + Sd;
    // momentum: lane 0 adds dp(x) + pairs 3, 4 to M_x and 3 - 4 to M_y; lane 1 dp(y) +
    // pairs 7, 8 to M_y and 7 - 8 to M_z; lane 2 dp(z) and 5 - 6 to M_z, 5 + 6 to M_x
    const long long S2 = dpp + dpm, S3 = dpp - dpm;
    const long long Mx = quad_sum64(j == 0 ? dpa + S2 : (j == 2 ? S2 : 0));
    const long long My = quad_sum64(j == 0 ? S3 : (j == 1 ? dpa + S2 : 0));
    const long long Mz = quad_sum64(j == 1 ? S3 : (j == 2 ? dpa + S3 : 0));
    bool br;
    sig = fx_recover(T00, Mx, My, Mz, u, br);
    Pf = (long long)sig - T00;
    if (PAIR && j == 0) {
      su.ax[m] = u.ax;
      su.ay[m] = u.ay;
      su.az[m] = u.az;
      su.sg[m] = u.sx | (u.sy << 1) | (u.sz << 2);
    }
    ufix_products(u);
    b |= br | (Pf <= 0) | (u.xx + u.yy + u.zz >= (1ull << 62));
  } else {
    N0 = Xr + quad_sum64(pairs ? (spa + spp) + spm : 0);
  }
  if (PAIR) asm volatile("bar.sync %0, 64;" ::"r"(bar_id) : "memory");
  if (!is_g) {
    u.ax = su.ax[m];
    u.ay = su.ay[m];
    u.az = su.az[m];
    const unsigned sg = su.sg[m];
    u.sx = sg & 1u;
    u.sy = (sg >> 1) & 1u;
    u.sz = sg >> 2;
    ufix_products(u);
  }
  EqPieces q;
  eq_pieces(is_g ? sig : (unsigned long long)N0, u, q);
  const long long SX = q.Xx + q.Xy + q.Xz;
  long long eq0;
  if (is_g) {
    q.KA = (long long)mulhi((unsigned long long)Pf, kSixth) - (long long)mulhi((unsigned long long)SX, kThird);
    eq0 = (long long)sig - 3 * Pf - 2 * SX;
  } else {
    q.KA = (long long)mulhi((unsigned long long)N0, kEighteenth) - (long long)mulhi((unsigned long long)SX, kThird);
    eq0 = (long long)mulhi((unsigned long long)N0, kThird) - 2 * SX;
  }
  const unsigned long long Om = is_g ? k.Om2_v : k.Om2_f;   // relax_r forms, as in k_step_ws
  const auto rlx = [is_g](long long X, long long Xeq, unsigned long long O, long long c) {
    return is_g ? relax_r<RV>(X, Xeq, O, c) : relax_r<RF>(X, Xeq, O, c);
  };
  long long c0 = (long long)(Om >> 1), cA = c0, cD = c0;
  if (MRT && is_g) {
    const long long n0 = (Xr - eq0) >> 3;
    const long long nA = (Sa - Pf) >> 3;
    const long long nD = (Sd - Pf - 2 * SX) >> 3;
    const long long ae = __mul64hi(8 * nD - 11 * nA - 30 * n0, k.CE) >> 6;
    const long long ap = __mul64hi(nD - 4 * nA + 12 * n0, k.CP) >> 2;
    c0 += 30 * ae - 12 * ap;
    cA += 11 * ae + 4 * ap;
    cD -= 8 * ae + ap;
  }
  if (pairs) {
    // axis pair: ev = KA + X_i, od = Z_i; diagonal pairs: ev = KA/2 + (X_a + X_b)/2 +- Y_ab,
    // od = (Z_a +- Z_b)/2 (the pieces of relax_links_store)
    const long long Xi = sel3(ai, q.Xx, q.Xy, q.Xz), Zi = sel3(ai, q.Zx, q.Zy, q.Zz);
    const long long Xa = sel3(da, q.Xx, q.Xy, q.Xz), Xb = sel3(db, q.Xx, q.Xy, q.Xz);
    const long long Za = sel3(da, q.Zx, q.Zy, q.Zz), Zb = sel3(db, q.Zx, q.Zy, q.Zz);
    const long long Yab = j == 0 ? q.Yxy : (j == 1 ? q.Yyz : q.Yxz);
    const long long evA = q.KA + Xi, odA = Zi;
    const long long evD = (q.KA >> 1) + ((Xa + Xb) >> 1);
    const long long evP = evD + Yab, odP = (Za + Zb) >> 1;
    const long long evM = evD - Yab, odM = (Za - Zb) >> 1;
    const long long y0 = rlx(X[0], evA + odA, Om, cA), y1 = rlx(X[1], evA - odA, Om, cA);
    const long long y2 = rlx(X[2], evP + odP, Om, cD), y3 = rlx(X[3], evP - odP, Om, cD);
    const long long y4 = rlx(X[4], evM + odM, Om, cD), y5 = rlx(X[5], evM - odM, Om, cD);
    v[0] = from_fixed_dp(y0, E);
    v[1] = from_fixed_dp(y1, E);
    v[2] = from_fixed_dp(y2, E);
    v[3] = from_fixed_dp(y3, E);
    v[4] = from_fixed_dp(y4, E);
    v[5] = from_fixed_dp(y5, E);
  } else {
    v[0] = from_fixed_dp(rlx(X[0], eq0, Om, c0), E);
#pragma unroll
    for (int sl = 1; sl < 6; ++sl) v[sl] = v[0];   // the rest link in every slot, as pulled
  }
  return b;
}

// One step of a small lattice: a 64-thread block serves 8 nodes along x.
template <bool MRT, int RV, int RF>
__global__ void __launch_bounds__(64, 8) k_step_quad(const double* __restrict__ src, double* __restrict__ dst, Geo geo,
                                                     StepConst k, unsigned long long* __restrict__ bad) {
  __shared__ QuadU su;
  const int lane = threadIdx.x & 31;
  const bool is_g = threadIdx.x < 32;
  const int m = lane >> 2, j = lane & 3;
  const int xv = blockIdx.x * 8 + m;
  const bool valid = xv < geo.nx;
  const int x = valid ? xv : geo.nx - 1;
  const int y = blockIdx.y, z = blockIdx.z;
  const int xm = src_minus(x, geo.nx, geo.bcx), xp = src_plus(x, geo.nx, geo.bcx);
  const int ym = src_minus(y, geo.ny, geo.bcy), yp = src_plus(y, geo.ny, geo.bcy);
  const int zm = src_minus(z, geo.nz, geo.bcz), zp = src_plus(z, geo.nz, geo.bcz);
  const unsigned long long plane0 = is_g ? 19ull * geo.plane : 0ull;
  wait_for_grid(src);
  double v[6];
#pragma unroll
  for (int sl = 0; sl < 6; ++sl) {
    int cx, cy, cz;
    quad_dir(j, sl, cx, cy, cz);
    const int sx = cx > 0 ? xm : (cx < 0 ? xp : x);
    const int sy = cy > 0 ? ym : (cy < 0 ? yp : y);
    const int sz = cz > 0 ? zm : (cz < 0 ? zp : z);
    const unsigned idx = ((unsigned)sz * (unsigned)geo.ny + (unsigned)sy) * (unsigned)geo.nx + (unsigned)sx;
    v[sl] = ld_pop(src + plane0 + (unsigned long long)quad_link(j, sl) * geo.plane + idx);
  }
  const bool b = quad_collide<MRT, RV, RF>(is_g, lane, v, k, su, 1);
  const unsigned node = ((unsigned)z * (unsigned)geo.ny + (unsigned)y) * (unsigned)geo.nx + (unsigned)x;
  if (valid && b && j == 0) atomicMin(bad, (unsigned long long)node);
  double* out = dst + plane0 + node;
  // every lane stores (lanes past the row repeat node nx - 1 bit for bit)
  out[(unsigned long long)quad_link(j, 0) * geo.plane] = v[0];
  if (j < 3) {
#pragma unroll
    for (int sl = 1; sl < 6; ++sl) out[(unsigned long long)quad_link(j, sl) * geo.plane] = v[sl];
  }
}

// Several steps of a quasi-1D lattice (ny = nz = 1) per launch.  A block holds kTubeTile nodes
// in registers (four lanes per node and distribution) and advances them by `steps`: the
// first step pulls from src, later ones exchange the x-moving links through shared memory.
// What a block does not know of its neighbours grows inwards by one node per later step,
// so it stores the `core` nodes in its middle, core <= kTubeTile - 2 (steps - 1): neighbouring
// blocks advance the overlap as well, with the same arithmetic, instead of waiting for one
// another.  k_step_quad takes 6.2 us per step of a 1600-node tube, launched one after the
// other (4.7 with BGK): 4 of them are the launch and the loads' latency, 2.1 the dependent
// integer chain.  Here a launch of 10 steps takes 1.4 + 10 x 2.24 us; the bound is that chain
// (issue slots 66 % busy on the SMs that have a block).  1600 nodes: 6.17 -> 2.37 us per step,
// 6400: 6.18 -> 3.31, 38912: 16.5 -> 13.4.  Tried: 16- and 64-node tiles (2.58 and 3.7 us at
// 1600 nodes), the output rounding on the integer pipe (2.84 against 2.59 at 8 steps).
//   G_ONLY: g alone (it does not depend on f), src and dst hold g only, and every step's g
//   is stored, step s at dst + 19 nx s (the adjoint's recompute).
template <bool MRT, int RV, int RF, bool G_ONLY>
__global__ void __launch_bounds__((G_ONLY ? 32 : 64) * kTubeWarps)
    k_tube_steps(const double* __restrict__ src, double* __restrict__ dst, int nx, int bcx, StepConst k, int steps,
                 int core, unsigned long long* __restrict__ bad) {
  __shared__ QuadU su[kTubeWarps];
  __shared__ double ex[2][G_ONLY ? 1 : 2][2][6][kTubeTile];   // [parity][role][lane 0 / 2][slot][node]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, m = lane >> 2, j = lane & 3;
  const bool is_g = G_ONLY || warp < kTubeWarps;
  const int pair = is_g ? warp : warp - kTubeWarps;
  const int i = pair * 8 + m;                                   // node of the tile
  const int halo = (kTubeTile - core) >> 1;
  const int xg = (int)blockIdx.x * core - halo + i;             // its place in the lattice
  const bool own = i >= halo && i < halo + core && xg < nx;     // stored (and checked) by this block
  int x = xg;
  if (bcx) x = min(max(xg, 0), nx - 1);                         // past an open end: idle copies
  else x = xg < 0 ? (xg % nx + nx) % nx : xg % nx;
  const unsigned long long n = (unsigned long long)nx;
  const double* in = src + (is_g && !G_ONLY ? 19ull * n : 0ull);
  const double* at[6];
#pragma unroll
  for (int sl = 0; sl < 6; ++sl) {
    int cx, cy, cz;
    quad_dir(j, sl, cx, cy, cz);
    const int sx = cx > 0 ? src_minus(x, nx, bcx) : (cx < 0 ? src_plus(x, nx, bcx) : x);
    at[sl] = in + (unsigned long long)quad_link(j, sl) * n + (unsigned)sx;
  }
  double v[6];
  // as wait_for_grid: nothing is read or written until the grid before is complete
  asm volatile("griddepcontrol.wait;" ::: "memory");
#pragma unroll
  for (int sl = 0; sl < 6; ++sl) asm volatile("ld.global.cg.f64 %0, [%1];" : "=d"(v[sl]) : "l"(at[sl]));
  // sources of the exchange: the tile's neighbours, at an open end the node itself; a tile
  // that holds the whole lattice (core = kTubeTile, no overlap) wraps onto itself
  const bool whole = core == kTubeTile;
  const int im = xg == 0 && (bcx || whole) ? (bcx ? i : nx - 1) : max(i - 1, 0);
  const int ip = xg == nx - 1 && (bcx || whole) ? (bcx ? i : 0) : min(i + 1, kTubeTile - 1);
  const bool axis_moves = j == 0, moves = j == 0 || j == 2;     // slots 0-1; slots 2-5
  for (int s = 0;; ++s) {
    const bool b = quad_collide<MRT, RV, RF, !G_ONLY>(is_g, lane, v, k, su[pair], 1 + pair);
    if (own && b && j == 0) atomicMin(bad, (unsigned long long)x);
    if (G_ONLY || s == steps - 1) {
      if (own) {
        double* out = dst + (G_ONLY ? (unsigned)s * 19ull * n : (is_g ? 19ull * n : 0ull)) + (unsigned)x;
        out[(unsigned long long)quad_link(j, 0) * n] = v[0];
        if (j < 3) {
#pragma unroll
          for (int sl = 1; sl < 6; ++sl) out[(unsigned long long)quad_link(j, sl) * n] = v[sl];
        }
      }
      if (s == steps - 1) return;
    }
    auto& e = ex[s & 1][is_g ? 0 : 1][j >> 1];
    if (moves) {
#pragma unroll
      for (int sl = 0; sl < 6; ++sl)
        if (sl >= 2 || axis_moves) e[sl][i] = v[sl];
    }
    __syncthreads();
    if (moves) {
#pragma unroll
      for (int sl = 0; sl < 6; ++sl)
        if (sl >= 2 || axis_moves) v[sl] = e[sl][(sl & 1) ? ip : im];
    }
  }
}

// ---- D2Q9: nodes are numbered along the rows one after the other (thread i of the grid
// takes node i), so rows of any length fill their warps: the paper's 4 x 800 tube, whose
// rows have 4 nodes, keeps 32 of 32 lanes busy instead of 4.
struct NodeXY {
  unsigned node;
  int x, y;
};
__device__ __forceinline__ bool node_xy(const Geo& geo, NodeXY& n) {
  n.node = blockIdx.x * blockDim.x + threadIdx.x;
  n.y = (int)(geo.inv_nx ? (unsigned)__umul64hi(n.node, geo.inv_nx) : n.node);   // 0: nx = 1
  n.x = (int)(n.node - (unsigned)n.y * (unsigned)geo.nx);
  return n.node < geo.plane;
}
// Index offsets to the node's neighbours: a pull with c = +1 / -1 along each axis.
struct Nbr {
  int xm, xp, ym, yp;
};
__device__ __forceinline__ Nbr neighbours(const Geo& geo, const NodeXY& n) {
  Nbr b;
  b.xm = n.x > 0 ? -1 : (geo.bcx ? 0 : geo.nx - 1);
  b.xp = n.x < geo.nx - 1 ? 1 : (geo.bcx ? 0 : 1 - geo.nx);
  b.ym = n.y > 0 ? -geo.nx : (geo.bcy ? 0 : (int)geo.plane - geo.nx);
  b.yp = n.y < geo.ny - 1 ? geo.nx : (geo.bcy ? 0 : geo.nx - (int)geo.plane);
  return b;
}
__device__ __forceinline__ void pull9(const double* __restrict__ base, const Geo& geo, unsigned node, const Nbr& b,
                                      double (&v)[9]) {
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    const int cx = d2_cx(a), cy = d2_cy(a);
    const unsigned i = node + (unsigned)((cx > 0 ? b.xm : cx < 0 ? b.xp : 0) + (cy > 0 ? b.ym : cy < 0 ? b.yp : 0));
    v[a] = ld_pop(base + (unsigned long long)a * geo.plane + i);
  }
}

// The FP64 forms of the two kernels below, for nodes outside the integer grid's exponent
// range (and a negative number density, which the FP64 step lets pass).
__device__ __noinline__ void macro_d2q9_general(const double* __restrict__ src, double* __restrict__ q, const Geo& geo,
                                                const NodeXY& nd) {
  const Nbr b = neighbours(geo, nd);
  double f[9], g[9], dp[4], Sa, Sd;
  pull9(src, geo, nd.node, b, f);
  pull9(src + 9ull * geo.plane, geo, nd.node, b, g);
  NodeMacro m;
  node_moments_d2q9<double>(f, g, dp, Sa, Sd, m);
  node_recover_fast(m);
  const double a = fma(1.0 / 3.0, m.sigma, -m.P), sux = m.sigma * m.ux, suy = m.sigma * m.uy;
  double* o = q + nd.node;
  o[0] = fma(-sux, m.ux, a);
  o[geo.plane] = fma(-suy, m.uy, a);
  o[2 * geo.plane] = sux;
  o[3 * geo.plane] = suy;
  o[4 * geo.plane] = 1.0 / sqrt(1.0 - m.u2);
}
// C_7 = E_x - E_y of Eq. 38 from the neighbours' macroscopic fields (below), with the
// node's u, sigma / (3 gamma) and (k / 2) theta.  The neighbours are the pulls' sources: a
// zero-gradient end reuses the edge node.
__device__ __forceinline__ double c7_of(const double* __restrict__ qn, unsigned long long P, const Nbr& b, double ux,
                                        double uy, double sg, double kth) {
  const double dgx = qn[4 * P + b.xp] - qn[4 * P + b.xm], dgy = qn[4 * P + b.yp] - qn[4 * P + b.ym];
  const double ex = fma(kth * ux, qn[2 * P + b.xp] - qn[2 * P + b.xm], fma(-sg, dgx, qn[b.xp] - qn[b.xm]));
  const double ey = fma(kth * uy, qn[3 * P + b.yp] - qn[3 * P + b.ym], fma(-sg, dgy, qn[P + b.yp] - qn[P + b.ym]));
  return fma(ux, ex, -uy * ey);
}
template <bool MRT, bool QSEP, bool CORR>
__device__ __noinline__ void step_d2q9_general(const double* __restrict__ src, double* __restrict__ dst, const Geo& geo,
                                               const StepConst& k, unsigned long long* __restrict__ bad,
                                               const double* __restrict__ q, const NodeXY& nd) {
  const Nbr b = neighbours(geo, nd);
  double f[9], g[9];
  pull9(src, geo, nd.node, b, f);
  pull9(src + 9ull * geo.plane, geo, nd.node, b, g);
  NodeMacro m;
  if (node_collide_d2q9_f64<MRT, QSEP, false>(f, g, k, m)) atomicMin(bad, (unsigned long long)nd.node);
  if (CORR) {
    const double sg = m.sigma * (1.0 / 3.0) / q[4 * geo.plane + nd.node];
    const double dq = (0.25 * (1.0 - 0.5 * k.omv)) *
                      c7_of(q + nd.node, geo.plane, b, m.ux, m.uy, sg, 0.5 * k.c7_theta * (4.0 / (3.0 + m.u2)));
    g[1] += dq;
    g[2] += dq;
    g[3] -= dq;
    g[4] -= dq;
  }
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    dst[(unsigned long long)a * geo.plane + nd.node] = f[a];
    dst[(9ull + a) * geo.plane + nd.node] = g[a];
  }
}

// Fields of the pulled D2Q9 state for the C_7 gradients (Eq. 38): per node
// c_s^2 sigma - P - sigma u_x^2, the same with u_y, sigma u_x, sigma u_y and gamma.  From
// the node's integers: c_s^2 sigma - P = T00 - (2/3) sigma and sigma u = M, one FP64
// rounding each.
constexpr int kMacroD2Q9 = 5;
__global__ void __launch_bounds__(kBlockX) k_macro_d2q9(const double* __restrict__ src, double* __restrict__ q,
                                                        const __grid_constant__ Geo geo) {
  NodeXY nd;
  if (!node_xy(geo, nd)) return;
  double v[9];
  const Nbr b = neighbours(geo, nd);
  wait_for_grid(src);
  pull9(src + 9ull * geo.plane, geo, nd.node, b, v);
  D9State s;
  d9_load(v, s);
  if (s.out) {
    macro_d2q9_general(src, q, geo, nd);
    return;
  }
  UFix u;
  bool br;
  const unsigned long long sig = fx_recover(s.T00, s.Mx, s.My, 0, u, br);
  const unsigned long long xx = fx::mulhi(u.ax, u.ax), yy = fx::mulhi(u.ay, u.ay);   // u_i^2 2^62
  const long long a = s.T00 - (long long)fx::mulhi(sig, fx::kTwoThirds);
  const unsigned long long u2 = min(xx + yy, (1ull << 62) - 1);   // a non-physical node is flagged by the step
  const unsigned long long w = (1ull << 62) - u2;
  const int sh = fx::even_shift(w), U = s.E - 1079;
  const unsigned long long Y = fx::rsqrt_fixed(w << sh);          // gamma 2^(62 - sh / 2)
  double* o = q + nd.node;
  o[0] = scale_pow2(__ll2double_rn(a - 4 * (long long)fx::mulhi(sig, xx)), U);
  o[geo.plane] = scale_pow2(__ll2double_rn(a - 4 * (long long)fx::mulhi(sig, yy)), U);
  o[2 * geo.plane] = scale_pow2(__ll2double_rn(s.Mx), U);
  o[3 * geo.plane] = scale_pow2(__ll2double_rn(s.My), U);
  o[4 * geo.plane] = scale_pow2(__ll2double_rn((long long)Y), (sh >> 1) - 62);
}

// D2Q9 (FP64): node (x, y) pulls link a from (x - c_x, y - c_y).  With CORR the
// C_7 term of Eqs. 37-38, C_7 = E_x - E_y, is added to the m_7 = p_xx moment of the
// result: with differences D over the two neighbours along axis a,
//   E_a = u_a [D(c_s^2 sigma - P - sigma u_a^2) - (sigma / (3 gamma)) D gamma
//              + (k/2) theta u_a D(sigma u_a)],   theta = 4 / (3 + u^2).
// f is rounded on the integer pipe and g on the FP64 pipe, 9 FP64-pipe instructions per
// node (31 with C_7), and f is pulled only when g is stored, which lets 8 blocks per SM
// hold the launch's latency (64 registers; 5 blocks at 96 registers: 145 us with C_7).
// 1200 x 900: 295 -> 70 us per step, with C_7 561 -> 124 (k_macro_d2q9 alone 138 -> 30).  Bound by
// issue and fixed latencies (issue 65 %, ALU 66 %), with C_7 by the FP64 pipe (71 %) and the
// waits for the neighbours' fields.
template <bool MRT, bool QSEP, bool CORR>
__global__ void __launch_bounds__(kBlockX, 8) k_step_d2q9(const double* __restrict__ src, double* __restrict__ dst,
                                                       const __grid_constant__ Geo geo, const __grid_constant__ StepConst k,
                                                       unsigned long long* __restrict__ bad,
                                                       const double* __restrict__ q) {
  NodeXY nd;
  if (!node_xy(geo, nd)) return;
  const unsigned node = nd.node;
  const Nbr b = neighbours(geo, nd);
  double v[9];
  if (CORR) wait_for_grid(src, q);
  else wait_for_grid(src);
  pull9(src + 9ull * geo.plane, geo, node, b, v);
  D9State g;
  d9_load(v, g);
  UFix u;
  bool br;
  const unsigned long long sig = fx_recover(g.T00, g.Mx, g.My, 0, u, br);
  const long long Pf = (long long)sig - g.T00;
  u.xx = fx::mulhi(u.ax, u.ax);
  u.yy = fx::mulhi(u.ay, u.ay);
  u.xy = fx::mulhi(u.ax, u.ay);
  const unsigned long long u2 = u.xx + u.yy;
  const bool phys = !(br | (Pf <= 0) | (u2 >= (1ull << 62)));
  const Rates r = constant_rates_d2q9(k);
  d9_relax<true, MRT, QSEP, false>(g, sig, Pf, u, r, v);
  if (CORR) {
    // sigma / (3 gamma) on the grid of g, theta = R 2^-62, u_i 2^-63
    int h;
    const unsigned long long Sq = fx::sqrt_one_minus((1ull << 62) - (phys ? u2 : 0ull), h);
    const double sg = scale_pow2(__ll2double_rn((long long)(fx::mulhi(fx::mulhi(sig, fx::kThird), Sq) << 1 >> h)), g.E - 1079);
    const double th = scale_pow2(__ll2double_rn((long long)fx::rcp_fixed((3ull << 62) + (phys ? u2 : 0ull))), -62);
    const double ux = scale_pow2(__ll2double_rn(fx::with_sign(u.ax, u.sx)), -63);
    const double uy = scale_pow2(__ll2double_rn(fx::with_sign(u.ay, u.sy)), -63);
    // m_7 = p_xx (row c_x^2 - c_y^2, norm 4): (1 - s_7/2) C_7 spread over the axis links
    const double dq = (0.25 * (1.0 - 0.5 * k.omv)) * c7_of(q + node, geo.plane, b, ux, uy, sg, 0.5 * k.c7_theta * th);
    v[1] += dq;
    v[2] += dq;
    v[3] -= dq;
    v[4] -= dq;
  }
#pragma unroll
  for (int a = 0; a < 9; ++a) dst[(9ull + a) * geo.plane + node] = v[a];
  pull9(src, geo, node, b, v);
  D9State f;
  d9_load(v, f);
  if (g.out | f.out | (f.T00 < 0)) {
    step_d2q9_general<MRT, QSEP, CORR>(src, dst, geo, k, bad, q, nd);
    return;
  }
  if (!phys) atomicMin(bad, (unsigned long long)node);
  d9_relax<false, false, false, true>(f, (unsigned long long)f.T00, 0, u, r, v);
#pragma unroll
  for (int a = 0; a < 9; ++a) dst[(unsigned long long)a * geo.plane + node] = v[a];
}

// D2Q9 with relaxation times per node from a fixed eta/s, in FP64 arithmetic.
template <bool MRT, bool QSEP>
__global__ void __launch_bounds__(kBlockX) k_step_d2q9_eta(const double* __restrict__ src, double* __restrict__ dst,
                                                           Geo geo, StepConst k, unsigned long long* __restrict__ bad) {
  NodeXY nd;
  if (!node_xy(geo, nd)) return;
  const Nbr b = neighbours(geo, nd);
  double f[9], g[9];
  wait_for_grid(src);
  pull9(src, geo, nd.node, b, f);
  pull9(src + 9ull * geo.plane, geo, nd.node, b, g);
  NodeMacro m;
  if (node_collide_d2q9_f64<MRT, QSEP, true>(f, g, k, m)) atomicMin(bad, (unsigned long long)nd.node);
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    dst[(unsigned long long)a * geo.plane + nd.node] = f[a];
    dst[(9ull + a) * geo.plane + nd.node] = g[a];
  }
}

// Deterministic two-pass sum of (N0, T00, Mx, My, Mz) over all nodes.
template <typename S, int Q = 19>
__global__ void __launch_bounds__(kRedThreads) k_totals_part(const S* __restrict__ lat, unsigned long long nodes,
                                                             double* __restrict__ part) {
  double acc[5] = {0, 0, 0, 0, 0};
  for (unsigned long long i = blockIdx.x * (unsigned long long)kRedThreads + threadIdx.x; i < nodes;
       i += (unsigned long long)kRedBlocks * kRedThreads) {
    double t[5];
    stored_totals<S, Q>(lat, nodes, i, t);
#pragma unroll
    for (int c = 0; c < 5; ++c) acc[c] += t[c];
  }
  __shared__ double sh[5][kRedThreads];
#pragma unroll
  for (int c = 0; c < 5; ++c) sh[c][threadIdx.x] = acc[c];
  __syncthreads();
  for (int s = kRedThreads / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s)
#pragma unroll
      for (int c = 0; c < 5; ++c) sh[c][threadIdx.x] += sh[c][threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x < 5) part[blockIdx.x * 5 + threadIdx.x] = sh[threadIdx.x][0];
}

__global__ void __launch_bounds__(kRedThreads) k_totals_final(const double* __restrict__ part, double* __restrict__ out) {
  __shared__ double sh[5][kRedThreads];
  double acc[5] = {0, 0, 0, 0, 0};
  for (int b = threadIdx.x; b < kRedBlocks; b += kRedThreads)
#pragma unroll
    for (int c = 0; c < 5; ++c) acc[c] += part[b * 5 + c];
#pragma unroll
  for (int c = 0; c < 5; ++c) sh[c][threadIdx.x] = acc[c];
  __syncthreads();
  for (int s = kRedThreads / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s)
#pragma unroll
      for (int c = 0; c < 5; ++c) sh[c][threadIdx.x] += sh[c][threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x < 5) out[threadIdx.x] = sh[threadIdx.x][0];
}

Geo make_geo(const rlb_handle* h) {
  Geo g;
  g.nx = h->cfg.nx; g.ny = h->cfg.ny; g.nz = h->cfg.nz;
  g.bcx = h->cfg.bc[0] == RLB_ZERO_GRADIENT;
  g.bcy = h->cfg.bc[1] == RLB_ZERO_GRADIENT;
  g.bcz = h->cfg.bc[2] == RLB_ZERO_GRADIENT;
  g.plane = h->nodes;
  g.inv_nx = g.nx > 1 ? ~0ull / (unsigned long long)g.nx + 1 : 0;
  g.inv_ny = g.ny > 1 ? ~0ull / (unsigned long long)g.ny + 1 : 0;
  return g;
}

bool qsep(const rlb_config& c) {
  if (c.eta_over_s > 0) return c.collision == RLB_MRT && c.tau_q > 0 && c.tau_q != 1.0;   // tau_q is a ratio
  return c.collision == RLB_MRT && c.tau_q > 0 && c.tau_q != c.tau_v;
}

// The FP64 steps for the relaxation forms of omega_v and omega_f (1: omega < 1, 2: omega >= 1).
template <int W, bool MRT, bool QSEP, bool FLAT>
void launch_ws(int rv, int rf, dim3 grid, cudaStream_t st, const double* s, double* d, const Geo& geo,
               const StepConst& k, unsigned long long* bad) {
  if (rv == 2 && rf == 2) launch_after(grid, 64 * W, st, true, k_step_ws<W, MRT, QSEP, FLAT, 2, 2>, s, d, geo, k, bad);
  else if (rv == 2) launch_after(grid, 64 * W, st, true, k_step_ws<W, MRT, QSEP, FLAT, 2, 1>, s, d, geo, k, bad);
  else if (rf == 2) launch_after(grid, 64 * W, st, true, k_step_ws<W, MRT, QSEP, FLAT, 1, 2>, s, d, geo, k, bad);
  else launch_after(grid, 64 * W, st, true, k_step_ws<W, MRT, QSEP, FLAT, 1, 1>, s, d, geo, k, bad);
}
template <int W, bool FLAT>
void launch_ws_coll(bool mrt, bool q, int rv, int rf, dim3 grid, cudaStream_t st, const double* s, double* d,
                    const Geo& geo, const StepConst& k, unsigned long long* bad) {
  if (!mrt) launch_ws<W, false, false, FLAT>(rv, rf, grid, st, s, d, geo, k, bad);
  else if (!q) launch_ws<W, true, false, FLAT>(rv, rf, grid, st, s, d, geo, k, bad);
  else launch_ws<W, true, true, FLAT>(rv, rf, grid, st, s, d, geo, k, bad);
}
template <int W, bool FLAT>
void launch_eta(bool mrt, bool q, dim3 grid, cudaStream_t st, const double* s, double* d, const Geo& geo,
                const StepConst& k, unsigned long long* bad) {
  if (!mrt) launch_after(grid, 64 * W, st, true, k_step_ws<W, false, false, FLAT, 0, 0, true>, s, d, geo, k, bad);
  else if (!q) launch_after(grid, 64 * W, st, true, k_step_ws<W, true, false, FLAT, 0, 0, true>, s, d, geo, k, bad);
  else launch_after(grid, 64 * W, st, true, k_step_ws<W, true, true, FLAT, 0, 0, true>, s, d, geo, k, bad);
}
template <bool FLAT>
void launch_f32(bool mrt, bool q, dim3 grid, int bx, cudaStream_t st, const float* s, float* d, const Geo& geo,
                const StepConst& k, unsigned long long* bad) {
  if (!mrt) launch_after(grid, bx, st, true, k_step<float, false, false, FLAT>, s, d, geo, k, bad);
  else if (!q) launch_after(grid, bx, st, true, k_step<float, true, false, FLAT>, s, d, geo, k, bad);
  else launch_after(grid, bx, st, true, k_step<float, true, true, FLAT>, s, d, geo, k, bad);
}

// Whether nodes are numbered across rows: where blocks of b nodes per row would leave more
// than 1 lane in 32 idle.  Numbering them costs 2 % on a row that fills its blocks (256^3
// FP64 1.798 against 1.834 ms per step, FP32 0.828 against 0.844) and saves the idle lanes:
// 150 x 110 x 90 FP64 262 -> 175 us (with its own tau_q 313 -> 194), 120 x 128 x 128 233 ->
// 223, 40 x 120 x 200 309 -> 114; FP32 90 -> 78, 107 -> 103, 82 -> 54.
bool flat_rows(int nx, int b) {
  const long long lanes = (long long)((nx + b - 1) / b) * b;
  return (lanes - nx) * 32 > lanes;
}

template <bool MRT>
void launch_quad(int rv, int rf, dim3 grid, cudaStream_t st, const double* s, double* d, const Geo& geo,
                 const StepConst& k, unsigned long long* bad) {
  if (rv == 2 && rf == 2) launch_after(grid, 64, st, true, k_step_quad<MRT, 2, 2>, s, d, geo, k, bad);
  else if (rv == 2) launch_after(grid, 64, st, true, k_step_quad<MRT, 2, 1>, s, d, geo, k, bad);
  else if (rf == 2) launch_after(grid, 64, st, true, k_step_quad<MRT, 1, 2>, s, d, geo, k, bad);
  else launch_after(grid, 64, st, true, k_step_quad<MRT, 1, 1>, s, d, geo, k, bad);
}

template <bool MRT, int RV, int RF, bool G_ONLY>
void launch_tube_as(int grid, cudaStream_t st, bool early, const double* s, double* d, const Geo& geo,
                    const StepConst& k, int steps, int core, unsigned long long* bad) {
  launch_after(grid, (G_ONLY ? 32 : 64) * kTubeWarps, st, early, k_tube_steps<MRT, RV, RF, G_ONLY>, s, d, geo.nx,
               geo.bcx, k, steps, core, bad);
}
template <bool MRT, bool G_ONLY>
void launch_tube(int rv, int rf, int grid, cudaStream_t st, bool early, const double* s, double* d, const Geo& geo,
                 const StepConst& k, int steps, int core, unsigned long long* bad) {
  if (G_ONLY) rf = rv;   // f is not advanced
  if (rv == 2 && rf == 2) launch_tube_as<MRT, 2, 2, G_ONLY>(grid, st, early, s, d, geo, k, steps, core, bad);
  else if (rv == 2) launch_tube_as<MRT, 2, G_ONLY ? 2 : 1, G_ONLY>(grid, st, early, s, d, geo, k, steps, core, bad);
  else if (rf == 2) launch_tube_as<MRT, 1, G_ONLY ? 1 : 2, G_ONLY>(grid, st, early, s, d, geo, k, steps, core, bad);
  else launch_tube_as<MRT, 1, 1, G_ONLY>(grid, st, early, s, d, geo, k, steps, core, bad);
}

template <typename S>
cudaError_t launch_step(rlb_handle* h, const void* src, void* dst, cudaStream_t st) {
  const Geo geo = make_geo(h);
  if (h->Q == 9) {
    // small planes spread over more SMs with one warp per block
    const int bx = h->nodes <= kSmallNodes ? 32 : kBlockX;
    const unsigned gr = (unsigned)((h->nodes + bx - 1) / bx);
    const bool mrt2 = h->cfg.collision == RLB_MRT, q2 = qsep(h->cfg);
    const double* s2 = (const double*)src;
    double* d2 = (double*)dst;
    if (h->cfg.eta_over_s > 0) {
      if (!mrt2) launch_after(gr, bx, st, true, k_step_d2q9_eta<false, false>, s2, d2, geo, h->k, h->d_bad);
      else if (!q2) launch_after(gr, bx, st, true, k_step_d2q9_eta<true, false>, s2, d2, geo, h->k, h->d_bad);
      else launch_after(gr, bx, st, true, k_step_d2q9_eta<true, true>, s2, d2, geo, h->k, h->d_bad);
    } else if (h->cfg.correction != RLB_CORR_NONE) {
      launch_after(gr, bx, st, true, k_macro_d2q9, s2, h->d_macro, geo);
      if (!q2) launch_after(gr, bx, st, true, k_step_d2q9<true, false, true>, s2, d2, geo, h->k, h->d_bad, h->d_macro);
      else launch_after(gr, bx, st, true, k_step_d2q9<true, true, true>, s2, d2, geo, h->k, h->d_bad, h->d_macro);
    } else if (!mrt2) {
      launch_after(gr, bx, st, true, k_step_d2q9<false, false, false>, s2, d2, geo, h->k, h->d_bad, (const double*)nullptr);
    } else if (!q2) {
      launch_after(gr, bx, st, true, k_step_d2q9<true, false, false>, s2, d2, geo, h->k, h->d_bad, (const double*)nullptr);
    } else {
      launch_after(gr, bx, st, true, k_step_d2q9<true, true, false>, s2, d2, geo, h->k, h->d_bad, (const double*)nullptr);
    }
    return cudaGetLastError();
  }
  // Lattices that cannot fill the GPU go in one-warp blocks (one warp per role), which spread
  // over more SMs; quasi-1D FP64 ones with constant rates come here for single steps only
  // (enqueue_tube).
  // FP32 storage: 64-thread blocks, whose finer tail suits every size (64^3 14.9 -> 14.5 us per
  // step, 100^3 52.5 -> 52.3, 256^3 820 -> 815; 96 threads 14.9, 52.7, 839)
  const int bx = h->nodes <= kSmallNodes ? 32 : sizeof(S) == 4 ? kBlockX / 2 : kBlockX;
  const bool flat = flat_rows(geo.nx, bx);
  const dim3 grid = flat ? dim3((unsigned)((h->nodes + bx - 1) / bx))
                         : dim3((unsigned)((geo.nx + bx - 1) / bx), geo.ny, geo.nz);
  const bool mrt = h->cfg.collision == RLB_MRT, q = qsep(h->cfg);
  const S* s = (const S*)src;
  S* d = (S*)dst;
  if constexpr (sizeof(S) == 8) {
    const int rv = h->k.r_v, rf = h->k.r_f;
    if (h->cfg.eta_over_s > 0) {
      if (bx == 32) {
        if (flat) launch_eta<1, true>(mrt, q, grid, st, s, d, geo, h->k, h->d_bad);
        else launch_eta<1, false>(mrt, q, grid, st, s, d, geo, h->k, h->d_bad);
      } else {
        if (flat) launch_eta<RLB_WS_WARPS, true>(mrt, q, grid, st, s, d, geo, h->k, h->d_bad);
        else launch_eta<RLB_WS_WARPS, false>(mrt, q, grid, st, s, d, geo, h->k, h->d_bad);
      }
    } else if (bx == 32 && !q) {
      // small lattices, four lanes per node: 8 nodes per 64-thread block
      dim3 gq((geo.nx + 7) / 8, geo.ny, geo.nz);
      if (mrt) launch_quad<true>(rv, rf, gq, st, s, d, geo, h->k, h->d_bad);
      else launch_quad<false>(rv, rf, gq, st, s, d, geo, h->k, h->d_bad);
    } else if (bx == 32) {
      // warp roles, one g and one f warp per block (a block serves bx nodes)
      if (flat) launch_ws<1, true, true, true>(rv, rf, grid, st, s, d, geo, h->k, h->d_bad);
      else launch_ws<1, true, true, false>(rv, rf, grid, st, s, d, geo, h->k, h->d_bad);
    } else {
      static_assert(32 * RLB_WS_WARPS == kBlockX, "a block serves kBlockX nodes");
      if (flat) launch_ws_coll<RLB_WS_WARPS, true>(mrt, q, rv, rf, grid, st, s, d, geo, h->k, h->d_bad);
      else launch_ws_coll<RLB_WS_WARPS, false>(mrt, q, rv, rf, grid, st, s, d, geo, h->k, h->d_bad);
    }
  } else {
    if (flat) launch_f32<true>(mrt, q, grid, bx, st, s, d, geo, h->k, h->d_bad);
    else launch_f32<false>(mrt, q, grid, bx, st, s, d, geo, h->k, h->d_bad);
  }
  return cudaGetLastError();
}

int check_flag(rlb_handle* h) {
  RLB_CUDA(h, cudaStreamSynchronize(h->stream));
  unsigned long long bad = ULLONG_MAX;
  RLB_CUDA(h, cudaMemcpy(&bad, h->d_bad, sizeof(bad), cudaMemcpyDeviceToHost));
  if (bad != ULLONG_MAX) {
    const unsigned long long reset = ULLONG_MAX;
    RLB_CUDA(h, cudaMemcpy(h->d_bad, &reset, sizeof(reset), cudaMemcpyHostToDevice));
    char buf[160];
    std::snprintf(buf, sizeof buf, "non-physical state at node %llu (x=%llu, y=%llu, z=%llu)", bad,
                  bad % (unsigned long long)h->cfg.nx, (bad / h->cfg.nx) % (unsigned long long)h->cfg.ny,
                  bad / ((unsigned long long)h->cfg.nx * h->cfg.ny));
    return fail(h, RLB_ENONPHYS, buf);
  }
  return RLB_OK;
}

int ensure_stage(rlb_handle* h) {
  if (h->d_stage) return RLB_OK;
  cudaError_t e = cudaMalloc(&h->d_stage, 6 * h->nodes * sizeof(double));
  if (e != cudaSuccess) {
    h->d_stage = nullptr;
    return fail(h, RLB_ENOMEM, "cannot allocate field staging buffer");
  }
  return RLB_OK;
}


}  // namespace

// ----------------------------------------------------------------------------- internal helpers
namespace rlb {
void set_handleless_error(const std::string& msg) { g_create_error = msg; }

int tube_launch_steps(const rlb_handle* h, int& core) {
  const rlb_config& c = h->cfg;
  if (h->Q != 19 || h->esize != 8 || c.ny != 1 || c.nz != 1 || h->nodes > kSmallNodes || c.eta_over_s > 0 || qsep(c))
    return 1;
  if (c.nx <= kTubeTile) {   // one block holds the lattice: only the launch limits the steps (9 ms here)
    core = kTubeTile;
    return 4096;
  }
  // H steps per launch cost 1.4 us / H for the launch and, per step, the chain (2.24 us) times
  // what w blocks per SM slow it down (measured: 1 block 1.0, 2 1.4, 3 1.8, 6 3.6, 9 5.7);
  // more steps mean a smaller core and so more blocks
  float best = 1e30f;
  int H = 2;
  for (int t = 2; t <= 12; ++t) {
    const int c = kTubeTile - 2 * (t - 1);
    const int w = (((int)h->nodes + c - 1) / c + 151) / 152;
    const float cost = 1.4f / t + 2.24f * std::max(1.0f, 0.1f + 0.62f * w);
    if (cost < best) {
      best = cost;
      H = t;
    }
  }
  core = kTubeTile - 2 * (H - 1);
  return H;
}

cudaError_t enqueue_tube(const rlb_handle* h, const double* src, double* dst, int nsteps, int core, bool g_only,
                         bool early, cudaStream_t st) {
  const Geo geo = make_geo(h);
  const int grid = (geo.nx + core - 1) / core, rv = h->k.r_v, rf = h->k.r_f;
  const bool mrt = h->cfg.collision == RLB_MRT;
  if (g_only) {
    if (mrt) launch_tube<true, true>(rv, rf, grid, st, early, src, dst, geo, h->k, nsteps, core, h->d_bad);
    else launch_tube<false, true>(rv, rf, grid, st, early, src, dst, geo, h->k, nsteps, core, h->d_bad);
  } else {
    if (mrt) launch_tube<true, false>(rv, rf, grid, st, early, src, dst, geo, h->k, nsteps, core, h->d_bad);
    else launch_tube<false, false>(rv, rf, grid, st, early, src, dst, geo, h->k, nsteps, core, h->d_bad);
  }
  return cudaGetLastError();
}

cudaError_t enqueue_steps(rlb_handle* h, int nsteps, cudaStream_t st) {
  int core = 0;
  const int most = tube_launch_steps(h, core);
  if (most > 1 && nsteps > 1) {
    for (int s = 0; s < nsteps;) {
      const int n = std::min(most, nsteps - s);
      const cudaError_t e = enqueue_tube(h, (const double*)h->lat[h->cur], (double*)h->lat[1 - h->cur], n, core, false,
                                         true, st);
      if (e != cudaSuccess) return e;
      h->cur = 1 - h->cur;
      h->steps += n;
      s += n;
    }
    return cudaSuccess;
  }
  for (int s = 0; s < nsteps; ++s) {
    const void* src = h->lat[h->cur];
    void* dst = h->lat[1 - h->cur];
    cudaError_t e = h->esize == 8 ? launch_step<double>(h, src, dst, st) : launch_step<float>(h, src, dst, st);
    if (e != cudaSuccess) return e;
    h->cur = 1 - h->cur;
    ++h->steps;
  }
  return cudaSuccess;
}

int validate_taus(double tau_f, double tau_v, double tau_e, double tau_eps, double tau_q, int collision,
                  std::string& why) {
  if (!(tau_f > 0.5) || !(tau_v > 0.5)) { why = "tau_f and tau_v must be > 0.5"; return RLB_EINVAL; }
  if (collision == RLB_MRT) {
    if (!(tau_e > 0.5) || !(tau_eps > 0.5)) { why = "tau_e and tau_eps must be > 0.5"; return RLB_EINVAL; }
    if (tau_q > 0 && !(tau_q > 0.5)) { why = "tau_q must be > 0.5 (or <= 0 for tau_v)"; return RLB_EINVAL; }
  }
  return RLB_OK;
}
}  // namespace rlb

// ----------------------------------------------------------------------------- C ABI
extern "C" int rlb_create(const rlb_config* cfg, rlb_handle** out) {
  if (!cfg || !out) return fail(nullptr, RLB_EINVAL, "null argument");
  if (cfg->nx <= 0 || cfg->ny <= 0 || cfg->nz <= 0) return fail(nullptr, RLB_EINVAL, "lattice extents must be > 0");
  if (cfg->lattice != RLB_D3Q19 && cfg->lattice != RLB_D2Q9)
    return fail(nullptr, RLB_EINVAL, "lattice must be RLB_D3Q19 or RLB_D2Q9");
  if (cfg->lattice == RLB_D2Q9 && (cfg->nz != 1 || cfg->precision != RLB_FP64))
    return fail(nullptr, RLB_EINVAL, "RLB_D2Q9 needs nz == 1 and RLB_FP64");
  if (cfg->correction != RLB_CORR_NONE && cfg->correction != RLB_CORR_C7 && cfg->correction != RLB_CORR_C7_PRINTED)
    return fail(nullptr, RLB_EINVAL, "unknown correction");
  if (cfg->correction != RLB_CORR_NONE && (cfg->lattice != RLB_D2Q9 || cfg->collision != RLB_MRT))
    return fail(nullptr, RLB_EINVAL, "RLB_CORR_C7 needs RLB_D2Q9 and RLB_MRT");
  if (cfg->eos != RLB_EOS_ULTRAREL) return fail(nullptr, RLB_EINVAL, "only RLB_EOS_ULTRAREL (P = e/3) is supported");
  if (cfg->collision != RLB_BGK && cfg->collision != RLB_MRT) return fail(nullptr, RLB_EINVAL, "unknown collision");
  if (cfg->precision != RLB_FP64 && cfg->precision != RLB_FP32_STORAGE)
    return fail(nullptr, RLB_EINVAL, "unknown precision");
  for (int a = 0; a < 3; ++a)
    if (cfg->bc[a] != RLB_PERIODIC && cfg->bc[a] != RLB_ZERO_GRADIENT)
      return fail(nullptr, RLB_EINVAL, "unknown boundary type");
  std::string why;
  const bool eta_mode = cfg->eta_over_s > 0;
  if (eta_mode && (cfg->precision != RLB_FP64 || cfg->correction != RLB_CORR_NONE))
    return fail(nullptr, RLB_EINVAL, "eta_over_s needs RLB_FP64 and no correction term");
  if (eta_mode && cfg->collision == RLB_MRT && (!(cfg->tau_e > 0) || !(cfg->tau_eps > 0)))
    return fail(nullptr, RLB_EINVAL, "eta_over_s with RLB_MRT reads tau_e, tau_eps (and tau_q > 0) as ratios > 0");
  if (!(cfg->eta_over_s >= 0)) return fail(nullptr, RLB_EINVAL, "eta_over_s must be >= 0");
  if (!eta_mode &&
      rlb::validate_taus(cfg->tau_f, cfg->tau_v, cfg->tau_e, cfg->tau_eps, cfg->tau_q, cfg->collision, why))
    return fail(nullptr, RLB_EINVAL, why);
  if (eta_mode && cfg->tau_f > 0 && !(cfg->tau_f > 0.5))
    return fail(nullptr, RLB_EINVAL, "tau_f must be > 0.5 (or <= 0 for tau_f = tau_g)");
  const unsigned long long nodes = (unsigned long long)cfg->nx * cfg->ny * cfg->nz;
  if (nodes >= (1ull << 32) || (unsigned long long)cfg->ny * cfg->nz > 65535ull * 65535ull || cfg->ny > 65535 ||
      cfg->nz > 65535)
    return fail(nullptr, RLB_EINVAL, "lattice too large (nodes must be < 2^32, ny and nz <= 65535)");

  rlb_handle* h = new rlb_handle();
  h->cfg = *cfg;
  h->stream = (cudaStream_t)cfg->stream;
  h->nodes = nodes;
  h->esize = cfg->precision == RLB_FP64 ? 8 : 4;
  h->Q = cfg->lattice == RLB_D2Q9 ? 9 : 19;
  h->k = make_step_const(eta_mode && cfg->tau_f <= 0 ? 1.0 : cfg->tau_f, eta_mode ? 1.0 : cfg->tau_v, cfg->tau_e,
                         cfg->tau_eps, cfg->tau_q, cfg->collision == RLB_MRT, h->Q);
  h->k.eta_s = cfg->eta_over_s;
  h->k.eta3 = 3.0 * cfg->eta_over_s;
  h->k.tauf_local = eta_mode && cfg->tau_f <= 0;
  h->k.a_e = cfg->tau_e;
  h->k.a_p = cfg->tau_eps;
  h->k.a_q = cfg->tau_q > 0 ? cfg->tau_q : 1.0;
  h->k.c7_theta = cfg->correction == RLB_CORR_C7_PRINTED ? 2.0 : 1.0;
  cudaGetDevice(&h->device);
  const size_t bytes = 2 * (size_t)h->Q * h->nodes * h->esize;
  for (int i = 0; i < 2; ++i) {
    if (cudaMalloc(&h->lat[i], bytes) != cudaSuccess) {
      cudaGetLastError();
      rlb_destroy(h);
      return fail(nullptr, RLB_ENOMEM, "cannot allocate the two lattices");
    }
  }
  if (cfg->correction != RLB_CORR_NONE &&
      cudaMalloc(&h->d_macro, kMacroD2Q9 * h->nodes * sizeof(double)) != cudaSuccess) {
    cudaGetLastError();
    h->d_macro = nullptr;
    rlb_destroy(h);
    return fail(nullptr, RLB_ENOMEM, "cannot allocate the correction fields");
  }
  if (cudaMalloc(&h->d_bad, sizeof(unsigned long long)) != cudaSuccess ||
      cudaMalloc(&h->d_part, (kRedBlocks * 5 + 8) * sizeof(double)) != cudaSuccess) {
    cudaGetLastError();
    rlb_destroy(h);
    return fail(nullptr, RLB_ENOMEM, "cannot allocate small device buffers");
  }
  const unsigned long long none = ULLONG_MAX;
  if (cudaMemcpy(h->d_bad, &none, sizeof none, cudaMemcpyHostToDevice) != cudaSuccess) {
    rlb_destroy(h);
    return fail(nullptr, RLB_ECUDA, "cannot initialise device flag");
  }
  *out = h;
  return RLB_OK;
}

extern "C" void rlb_destroy(rlb_handle* h) {
  if (!h) return;
  cudaStreamSynchronize(h->stream);
  if (h->adj_plan && h->adj_free) h->adj_free(h->adj_plan);
  for (int i = 0; i < 2; ++i)
    if (h->lat[i]) cudaFree(h->lat[i]);
  if (h->d_bad) cudaFree(h->d_bad);
  if (h->d_part) cudaFree(h->d_part);
  if (h->d_stage) cudaFree(h->d_stage);
  if (h->d_macro) cudaFree(h->d_macro);
  delete h;
}

extern "C" const char* rlb_last_error(const rlb_handle* h) {
  return h ? h->err.c_str() : g_create_error.c_str();
}

extern "C" int rlb_set_fields(rlb_handle* h, const double* e, const double* ux, const double* uy, const double* uz,
                              const double* n, int where) {
  if (!h || !e || !ux || !uy || !uz || !n) return fail(h, RLB_EINVAL, "null argument");
  if (where != RLB_HOST && where != RLB_DEVICE) return fail(h, RLB_EINVAL, "where must be RLB_HOST or RLB_DEVICE");
  const size_t N = h->nodes;
  const double *de = e, *dx = ux, *dy = uy, *dz = uz, *dn = n;
  if (where == RLB_HOST) {
    // host fields go to the staging buffer; k_init validates both kinds of input on
    // the device (first bad node by atomicMin)
    int rc = ensure_stage(h);
    if (rc) return rc;
    double* s = h->d_stage;
    const double* src[5] = {e, ux, uy, uz, n};
    for (int c = 0; c < 5; ++c)
      RLB_CUDA(h, cudaMemcpyAsync(s + c * N, src[c], N * sizeof(double), cudaMemcpyHostToDevice, h->stream));
    de = s; dx = s + N; dy = s + 2 * N; dz = s + 3 * N; dn = s + 4 * N;
  }
  // validate on the device and build the equilibrium state in the spare lattice
  const int spare = 1 - h->cur;
  const unsigned long long none = ULLONG_MAX;
  RLB_CUDA(h, cudaMemcpyAsync(h->d_bad, &none, sizeof none, cudaMemcpyHostToDevice, h->stream));
  if (h->Q == 9)
    k_init<double, 9><<<grid_for(N), 256, 0, h->stream>>>((double*)h->lat[spare], N, de, dx, dy, dz, dn, h->d_bad);
  else if (h->esize == 8)
    k_init<double><<<grid_for(N), 256, 0, h->stream>>>((double*)h->lat[spare], N, de, dx, dy, dz, dn, h->d_bad);
  else
    k_init<float><<<grid_for(N), 256, 0, h->stream>>>((float*)h->lat[spare], N, de, dx, dy, dz, dn, h->d_bad);
  RLB_CUDA(h, cudaGetLastError());
  RLB_CUDA(h, cudaStreamSynchronize(h->stream));
  unsigned long long bad = ULLONG_MAX;
  RLB_CUDA(h, cudaMemcpy(&bad, h->d_bad, sizeof bad, cudaMemcpyDeviceToHost));
  if (bad != ULLONG_MAX) {
    RLB_CUDA(h, cudaMemcpy(h->d_bad, &none, sizeof none, cudaMemcpyHostToDevice));
    char buf[128];
    std::snprintf(buf, sizeof buf, "invalid field at node %llu (need e > 0, n > 0, |u| < 1)", bad);
    return fail(h, RLB_EINVAL, buf);
  }
  h->cur = spare;
  h->steps = 0;
  return RLB_OK;
}

extern "C" int rlb_step(rlb_handle* h, int nsteps) {
  if (!h) return fail(h, RLB_EINVAL, "null handle");
  if (nsteps < 0) return fail(h, RLB_EINVAL, "nsteps must be >= 0");
  cudaError_t e = rlb::enqueue_steps(h, nsteps, h->stream);
  if (e != cudaSuccess) return cuda_fail(h, e, "step kernel launch");
  return RLB_OK;
}

extern "C" int rlb_check(rlb_handle* h) {
  if (!h) return fail(h, RLB_EINVAL, "null handle");
  return check_flag(h);
}

extern "C" int rlb_get_fields(rlb_handle* h, double* e, double* P, double* ux, double* uy, double* uz, double* n,
                              int where) {
  if (!h) return fail(h, RLB_EINVAL, "null handle");
  if (where != RLB_HOST && where != RLB_DEVICE) return fail(h, RLB_EINVAL, "where must be RLB_HOST or RLB_DEVICE");
  int rc = ensure_stage(h);
  if (rc) return rc;
  const size_t N = h->nodes;
  double* s = h->d_stage;
  double* dev[6] = {s, s + N, s + 2 * N, s + 3 * N, s + 4 * N, s + 5 * N};
  double* want[6] = {e, P, ux, uy, uz, n};
  if (where == RLB_DEVICE)
    for (int c = 0; c < 6; ++c)
      if (want[c]) dev[c] = want[c];
  if (h->Q == 9)
    k_fields<double, 9><<<grid_for(N), 256, 0, h->stream>>>((const double*)h->lat[h->cur], N, dev[0], dev[1], dev[2],
                                                             dev[3], dev[4], dev[5], h->d_bad);
  else if (h->esize == 8)
    k_fields<double><<<grid_for(N), 256, 0, h->stream>>>((const double*)h->lat[h->cur], N, dev[0], dev[1], dev[2],
                                                          dev[3], dev[4], dev[5], h->d_bad);
  else
    k_fields<float><<<grid_for(N), 256, 0, h->stream>>>((const float*)h->lat[h->cur], N, dev[0], dev[1], dev[2],
                                                         dev[3], dev[4], dev[5], h->d_bad);
  RLB_CUDA(h, cudaGetLastError());
  if (where == RLB_HOST)
    for (int c = 0; c < 6; ++c)
      if (want[c])
        RLB_CUDA(h, cudaMemcpyAsync(want[c], dev[c], N * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
  return check_flag(h);
}

extern "C" int rlb_conserved_totals(rlb_handle* h, double out[5]) {
  if (!h || !out) return fail(h, RLB_EINVAL, "null argument");
  const size_t N = h->nodes;
  if (h->Q == 9)
    k_totals_part<double, 9><<<kRedBlocks, kRedThreads, 0, h->stream>>>((const double*)h->lat[h->cur], N, h->d_part);
  else if (h->esize == 8)
    k_totals_part<double><<<kRedBlocks, kRedThreads, 0, h->stream>>>((const double*)h->lat[h->cur], N, h->d_part);
  else
    k_totals_part<float><<<kRedBlocks, kRedThreads, 0, h->stream>>>((const float*)h->lat[h->cur], N, h->d_part);
  RLB_CUDA(h, cudaGetLastError());
  k_totals_final<<<1, kRedThreads, 0, h->stream>>>(h->d_part, h->d_part + kRedBlocks * 5);
  RLB_CUDA(h, cudaGetLastError());
  RLB_CUDA(h, cudaMemcpyAsync(out, h->d_part + kRedBlocks * 5, 5 * sizeof(double), cudaMemcpyDeviceToHost,
                              h->stream));
  RLB_CUDA(h, cudaStreamSynchronize(h->stream));
  return RLB_OK;
}

extern "C" size_t rlb_state_bytes(const rlb_handle* h) { return h ? 2 * (size_t)h->Q * h->nodes * h->esize : 0; }

extern "C" int rlb_save_state(rlb_handle* h, void* buf, int where) {
  if (!h || !buf) return fail(h, RLB_EINVAL, "null argument");
  if (where != RLB_HOST && where != RLB_DEVICE) return fail(h, RLB_EINVAL, "where must be RLB_HOST or RLB_DEVICE");
  RLB_CUDA(h, cudaMemcpyAsync(buf, h->lat[h->cur], rlb_state_bytes(h),
                              where == RLB_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice, h->stream));
  RLB_CUDA(h, cudaStreamSynchronize(h->stream));
  return RLB_OK;
}

extern "C" int rlb_load_state(rlb_handle* h, const void* buf, int where) {
  if (!h || !buf) return fail(h, RLB_EINVAL, "null argument");
  if (where != RLB_HOST && where != RLB_DEVICE) return fail(h, RLB_EINVAL, "where must be RLB_HOST or RLB_DEVICE");
  RLB_CUDA(h, cudaMemcpyAsync(h->lat[h->cur], buf, rlb_state_bytes(h),
                              where == RLB_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice, h->stream));
  RLB_CUDA(h, cudaStreamSynchronize(h->stream));
  h->steps = 0;
  return RLB_OK;
}

extern "C" long long rlb_steps_done(const rlb_handle* h) { return h ? h->steps : -1; }
