// rlb_io.cuh -- kernels shared by the lattice and batch handles of librlb:
// equilibrium initial state from FP64 fields (Eqs. 7-9; Eqs. 32-33 for D2Q9) and
// field output from a stored state (Eq. 10 plus the closed-form recovery).  Both
// treat the state as a flat list of `nodes` nodes with layout f[Q][nodes] then
// g[Q][nodes], Q = 19 (D3Q19) or 9 (D2Q9, u_z = 0).
//
// All three kernels run on 64-bit integers.  In FP64 arithmetic they were bound by the
// FP64 pipe, which retires 2 lanes per clock and SM (ncu: 82-87 % busy, DRAM 14-28 % of
// its peak); the integer forms leave 6 (fields), 10 (totals) and 19 (initial state)
// FP64-pipe instructions per node (totals hold 38 % of the pipe, the others 10 to 49 %).  FP32 states come out bit for bit as from the FP64
// form.  Nodes outside the range of the integer forms
// (exponents near the ends of the format, non-physical or invalid values) take the FP64
// forms, which define what is accepted and what such a node's output is.
#pragma once
#include <cuda_runtime.h>

#include <cstddef>

#include "rlb_node.cuh"

namespace {
using namespace rlb;

// each stored value is read once per call: past L1
template <typename S>
__device__ __forceinline__ S ld_once(const S* p) {
  S v;
  if constexpr (sizeof(S) == 8) asm("ld.global.nc.L1::no_allocate.L2::256B.f64 %0, [%1];" : "=d"(v) : "l"(p));
  else asm("ld.global.nc.L1::no_allocate.L2::256B.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}

// ---- FP64 forms: the definition for any input, used where the integer forms stop

// Equilibrium of node i in FP64; flags an invalid input node.
template <typename S, int Q>
__device__ __noinline__ void init_general(S* __restrict__ lat, unsigned long long nodes, unsigned long long i, double ei,
                                          double xi, double yi, double zi, double ni,
                                          unsigned long long* __restrict__ bad) {
  const double u2 = xi * xi + yi * yi + zi * zi;
  if (!(ei > 0.0) || !(ni > 0.0) || !(u2 < 1.0) || !isfinite(ei) || !isfinite(ni) || (Q == 9 && zi != 0.0)) {
    atomicMin(bad, i);
    return;
  }
  double f[Q], g[Q];
  if constexpr (Q == 19) node_equilibrium(ei, xi, yi, zi, ni, f, g);
  else node_equilibrium_d2q9(ei, xi, yi, ni, f, g);
#pragma unroll
  for (int a = 0; a < Q; ++a) {
    lat[(unsigned long long)a * nodes + i] = (S)f[a];
    lat[((unsigned long long)Q + a) * nodes + i] = (S)g[a];
  }
}

// Moments of the stored populations of node i (Eq. 10), FP64.
template <typename S, int Q>
__device__ __noinline__ void moments_general(const S* __restrict__ lat, unsigned long long nodes, unsigned long long i,
                                             NodeMacro& m) {
  S f[Q], g[Q];
#pragma unroll
  for (int a = 0; a < Q; ++a) {
    f[a] = lat[(unsigned long long)a * nodes + i];
    g[a] = lat[((unsigned long long)Q + a) * nodes + i];
  }
  if constexpr (Q == 19) {
    double sp[9], dp[9], Sa, Sd;
    node_moments<S>(f, g, sp, dp, Sa, Sd, m);
  } else {
    double dp[4], Sa, Sd;
    node_moments_d2q9<S>(f, g, dp, Sa, Sd, m);
  }
}

template <typename S, int Q>
__device__ __noinline__ void fields_general(const S* __restrict__ lat, unsigned long long nodes, unsigned long long i,
                                            double* __restrict__ e, double* __restrict__ P, double* __restrict__ ux,
                                            double* __restrict__ uy, double* __restrict__ uz, double* __restrict__ n,
                                            unsigned long long* __restrict__ bad) {
  NodeMacro m;
  moments_general<S, Q>(lat, nodes, i, m);
  node_recover(m);
  if (m.bad) atomicMin(bad, i);
  e[i] = 3.0 * m.P;
  P[i] = m.P;
  ux[i] = m.ux;
  uy[i] = m.uy;
  uz[i] = m.uz;
  n[i] = m.N0 * sqrt(1.0 - m.u2);
}

// ---- initial state

// f = f^eq, g = g^eq of the given FP64 fields; flags invalid input nodes.  FP64 storage
// takes the f conversions on the integer pipe and the g conversions on the FP64 pipe, which
// shares the work between them (ALU 45 %, FP64 pipe 49 %): 256^3 4.31 -> 1.19 ms per
// rlb_set_fields, 1.4 times its memory time, the rest fixed-latency waits at 24 % of the
// warps.  FP32 storage, 512^3: 43.1 -> 10.3 ms, 2.7 times its memory time: bound by the ALU (67 %,
// issue 56 %), whose work is the single rounding of 38 values with its test for ties.
template <typename S, int Q = 19>
__global__ void __launch_bounds__(256, 2) k_init(S* __restrict__ lat, unsigned long long nodes,
                                              const double* __restrict__ e, const double* __restrict__ ux,
                                              const double* __restrict__ uy, const double* __restrict__ uz,
                                              const double* __restrict__ n, unsigned long long* __restrict__ bad) {
  for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < nodes;
       i += (unsigned long long)gridDim.x * blockDim.x) {
    const double ei = e[i], xi = ux[i], yi = uy[i], zi = uz[i], ni = n[i];
    FxEquilibrium q;
    if (!fx_equilibrium_of<sizeof(S) == 4>(ei, xi, yi, zi, ni, q) || (Q == 9 && ((__double2hiint(zi) << 1) | __double2loint(zi)) != 0)) {
      init_general<S, Q>(lat, nodes, i, ei, xi, yi, zi, ni, bad);
      continue;
    }
    S* out = lat + i;
    const bool nf = fx_equilibrium_store<S, Q, false>(q, out, nodes);
    const bool ng = fx_equilibrium_store<S, Q, true>(q, out + (unsigned long long)Q * nodes, nodes);
    if (sizeof(S) == 4 && (nf | ng)) init_general<S, Q>(lat, nodes, i, ei, xi, yi, zi, ni, bad);
  }
}

// ---- sums and fields of a stored state

// Exact integer sums of node i's stored populations (Eq. 10) on the grids of its f and g
// (unit 2^(E - FxUnit<S>::bias) of that distribution's largest exponent E).
struct StoredSums {
  long long T00, Mx, My, Mz, N0;
  int Eg, Ef;
};
template <int Q, typename V>
__device__ __forceinline__ void g_sums(const V& value, StoredSums& s) {
  long long dp[Q / 2];
  s.T00 = value(0);
#pragma unroll
  for (int p = 0; p < Q / 2; ++p) {
    const long long a = value(2 * p + 1), b = value(2 * p + 2);
    s.T00 += a + b;
    dp[p] = a - b;
  }
  if constexpr (Q == 19) {
    s.Mx = dp[0] + dp[3] + dp[4] + dp[5] + dp[6];
    s.My = dp[1] + dp[3] - dp[4] + dp[7] + dp[8];
    s.Mz = dp[2] + dp[5] - dp[6] + dp[7] - dp[8];
  } else {
    s.Mx = dp[0] + dp[2] + dp[3];
    s.My = dp[1] + dp[2] - dp[3];
    s.Mz = 0;
  }
}
template <int Q, typename V>
__device__ __forceinline__ void f_sum(const V& value, StoredSums& s) {
  s.N0 = value(0);
#pragma unroll
  for (int a = 1; a < Q; ++a) s.N0 += value(a);
}
// False for an exponent range where the grids, or the FP64 results formed on them, could
// leave the normal range; the FP64 form is then used.
template <typename S, int Q>
__device__ __forceinline__ bool stored_sums(const S* __restrict__ lat, unsigned long long nodes, unsigned long long i,
                                            StoredSums& s) {
  S v[Q];
#pragma unroll
  for (int a = 0; a < Q; ++a) v[a] = ld_once(lat + ((unsigned long long)Q + a) * nodes + i);
  S w[Q];
#pragma unroll
  for (int a = 0; a < Q; ++a) w[a] = ld_once(lat + (unsigned long long)a * nodes + i);
  if constexpr (sizeof(S) == 4) {
    // FP32: the step's exact sums on the FP32 pipe where its two-level form is exact (the
    // same integers as the shifts below), else bit shifts
    s.Eg = max_exp19(v);
    s.Ef = max_exp19(w);
    const bool two = min_exp19(v) >= s.Eg - 13 && s.Eg >= 16 && s.Eg <= 240 && min_exp19(w) >= s.Ef - 13 &&
                     s.Ef >= 16 && s.Ef <= 240;
    if (two) {
      float sa, sd;
      exact_ints_g2(v, s.Eg, s.T00, s.Mx, s.My, s.Mz, sa, sd);
      s.N0 = exact_int_f2(w, s.Ef);
    } else {
      g_sums<Q>([&](int a) { return fx::grid_value(v[a], s.Eg); }, s);
      f_sum<Q>([&](int a) { return fx::grid_value(w[a], s.Ef); }, s);
    }
  } else {
    bool fast;
    s.Eg = fx::max_exponent(v, fast);
    if (fast) g_sums<Q>([&](int a) { return fx::to_fixed_pos(v[a], s.Eg + 6); }, s);
    else g_sums<Q>([&](int a) { return fx::grid_value(v[a], s.Eg); }, s);
    s.Ef = fx::max_exponent(w, fast);
    if (fast) f_sum<Q>([&](int a) { return fx::to_fixed_pos(w[a], s.Ef + 6); }, s);
    else f_sum<Q>([&](int a) { return fx::grid_value(w[a], s.Ef); }, s);
  }
  return fx::FxUnit<S>::in_range(s.Eg) && fx::FxUnit<S>::in_range(s.Ef);
}

// Macroscopic fields of the stored state.  One thread per node, bound by the memory it
// reads (FP64: 1.1 times its memory time, 256^3 3.21 -> 0.95 ms per rlb_get_fields) and by issue
// (FP32 storage: 67 %, 1.4 times, 512^3 34.4 -> 5.6 ms), against the FP64 form's 85 % busy
// FP64 pipe.
template <typename S, int Q = 19>
__global__ void __launch_bounds__(256) k_fields(const S* __restrict__ lat, unsigned long long nodes,
                                                double* __restrict__ e, double* __restrict__ P,
                                                double* __restrict__ ux, double* __restrict__ uy,
                                                double* __restrict__ uz, double* __restrict__ n,
                                                unsigned long long* __restrict__ bad) {
  for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < nodes;
       i += (unsigned long long)gridDim.x * blockDim.x) {
    StoredSums s;
    bool ok = stored_sums<S, Q>(lat, nodes, i, s);
    UFix u;
    bool br;
    unsigned long long R;
    int nsh;
    const unsigned long long sig = fx_recover(s.T00, s.Mx, s.My, s.Mz, u, br, R, nsh);
    const long long Pf = (long long)sig - s.T00;
    const unsigned long long u2 = fx::mulhi(u.ax, u.ax) + fx::mulhi(u.ay, u.ay) + fx::mulhi(u.az, u.az);   // u^2 2^62
    ok = ok && !br && Pf > 0 && u2 < (1ull << 62) - (1ull << 30);
    if (!ok) {   // non-physical, nearly so, or near the ends of the format
      fields_general<S, Q>(lat, nodes, i, e, P, ux, uy, uz, n, bad);
      continue;
    }
    constexpr int B = fx::FxUnit<S>::bias;
    const double Pd = scale_pow2(__ll2double_rn(Pf), s.Eg - B);
    e[i] = 3.0 * Pd;
    P[i] = Pd;
    ux[i] = fx_velocity(s.Mx, R, nsh);
    uy[i] = fx_velocity(s.My, R, nsh);
    uz[i] = fx_velocity(s.Mz, R, nsh);
    // n = N0 / gamma: 1/gamma = sqrt(1 - u^2) as Sq 2^(-63 - h)
    int h;
    const unsigned long long Sq = fx::sqrt_one_minus((1ull << 62) - u2, h);
    const unsigned neg = (unsigned)((unsigned long long)s.N0 >> 63);
    const unsigned long long a0 = (unsigned long long)(neg ? -s.N0 : s.N0);
    const int lz = __clzll((long long)(a0 | 1ull));
    const double nd = __ll2double_rn(fx::with_sign(fx::mulhi(a0 << lz, Sq) >> 1, neg));
    n[i] = scale_pow2(nd, s.Ef - B + 2 - lz - h);
  }
}

// (N0, T00, Mx, My, Mz) of node i, each exact sum rounded once to FP64 (a totals call at
// 256^3 FP64: 2.04 -> 0.76 ms, 512^3 FP32 storage: 24.8 -> 4.5 ms).
template <typename S, int Q = 19>
__device__ __forceinline__ void stored_totals(const S* __restrict__ lat, unsigned long long nodes,
                                              unsigned long long i, double (&t)[5]) {
  StoredSums s;
  if (stored_sums<S, Q>(lat, nodes, i, s)) {
    constexpr int B = fx::FxUnit<S>::bias;
    t[0] = scale_pow2(__ll2double_rn(s.N0), s.Ef - B);
    t[1] = scale_pow2(__ll2double_rn(s.T00), s.Eg - B);
    t[2] = scale_pow2(__ll2double_rn(s.Mx), s.Eg - B);
    t[3] = scale_pow2(__ll2double_rn(s.My), s.Eg - B);
    t[4] = scale_pow2(__ll2double_rn(s.Mz), s.Eg - B);
  } else {
    NodeMacro m;
    moments_general<S, Q>(lat, nodes, i, m);
    t[0] = m.N0; t[1] = m.T00; t[2] = m.Mx; t[3] = m.My; t[4] = m.Mz;
  }
}

inline int grid_for(size_t nodes) {
  size_t b = (nodes + 255) / 256;
  return (int)(b < 152 * 32 ? (b ? b : 1) : 152 * 32);
}

}  // namespace
