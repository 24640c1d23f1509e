// FP64 fused MLS fit + MHD right-hand side (Paper II Sec. 2), the plain
// double-precision GPU form.  It serves every particle when the precision is
// PHB_FP64, and the particles that the FP32-mixed kernel routed to FP64.
//
// What bounds it: GB300's FP64 pipe.  A warp's FP64 instruction takes 17-20 SM
// cycles when all four sub-partitions issue them (measured: 34 with two busy,
// 68 with one), about 80 times an FP32 one, so the kernel counts FP64
// instructions and keeps four warps per SM at them; shared-memory traffic,
// integer work and FP32 work disappear behind them.  A lattice fit (52
// neighbours) is 267 FP64 instructions per neighbour (80 moments, 7 x 19
// right-hand sides, 54 for offsets, weight and monomials) and ~3,900 for the
// factorisation and the solves, ~700 for the estimate: 19,200, or 8.6-9.9 ms for 262,144 particles.
// Comparisons and the test for a periodic wrap run on the integer pipe for that
// reason.  Measured: 12.0 ms (FP64 pipe 67% busy); with all sums in shared memory
// and two warps per SM it was 23.0 ms (35%).
//
// Two ways to fit a particle, bit-identical (each sum and each substitution
// takes its terms in the same order):
//   * thread per particle (fit_thread): the 80 moments in registers, the
//     right-hand sides in a shared-memory column that the factor takes over
//     afterwards (190 doubles per thread: 128 threads per SM);
//   * warp per particle (fit_warp): neighbours one per lane for the monomials,
//     the 232 sums spread over the lanes, the factorisation and the
//     substitutions by rows.  1.7 times the FP64 instructions, 1/20 of the
//     latency.
// Fits whose Jacobi-scaled conditioning estimate exceeds a threshold take one
// corrected semi-normal-equations step (Bjorck) in the warp form: residuals
// r_j = (U_j - U_i) - p(q_j).c are recomputed from the data, A^T W r is
// accumulated again and solved with the same factor, so the error follows
// cond(A) rather than cond(A^T W A) = cond(A)^2.
#include "phb_fit64.cuh"
#include "phb_mhd.cuh"

namespace phb {
namespace {

constexpr int kWarps = 4;  // per block, one block per SM: one warp per sub-partition
constexpr int kT = 32 * kWarps;

// Thread form: a warp's shared memory is [slot][32 lanes] doubles.
constexpr int kSlots = kNT;  // the factor: 190 doubles per thread, 190 KB per block

// Warp form: per warp, doubles.
constexpr int kRow = 39;                 // staged neighbour: w, w q^cubic (10), w dU (8), q^basis (19); odd stride
constexpr int kWL = 32 * kRow;           // factor (packed lower triangle)
constexpr int kWB = kWL + kNT;           // right-hand sides [field][19]
constexpr int kWC = kWB + kNF * kNB;     // coefficients [field][19]
constexpr int kWM = kWC + kNF * kNB;     // moments
constexpr int kWI = kWM + kNM;           // 1 / L_kk
constexpr int kWarpSlots = kWI + kNB;
static_assert(kWarpSlots <= kSlots * 32, "the warp form runs in the thread form's shared memory");

// sqrt(M_kk) of a positive pivot's diagonal entry.
__device__ __forceinline__ double root64(double m) { return __dmul_rn(m, rsqrt(m)); }

// Estimate of ||M_s^-1||_inf of the Jacobi-scaled matrix (as mls_inv_norm_est,
// the back substitution by columns) from the factor in a thread's column and the
// diagonal mkk of M; it picks the fits that take the corrected step.  (Formed in
// FP32 it saved 0.27 of 12.28 ms for 262,144 particles, but the entries of a
// tight cluster's M underflow there.)  The factor is read twice (volatile) rather
// than kept: 190 registers.
__device__ __forceinline__ double inv_norm_est(const double* my, const double (&mkk)[kNB]) {
  const volatile double* L = my;
  double y[kNB];
#pragma unroll
  for (int i = 0; i < kNB; ++i) {
    double t = 0.0;
#pragma unroll
    for (int k = 0; k < i; ++k) t = fma(L[(tri0(i) + k) * 32], y[k], t);
    const double sq = root64(mkk[i]);
    y[i] = ((t > 0.0 ? -sq : sq) - t) * L[(tri0(i) + i) * 32];
  }
  double mx = 0.0;
#pragma unroll
  for (int k = kNB - 1; k >= 0; --k) {
    y[k] *= L[(tri0(k) + k) * 32];
    mx = fmax(mx, fabs(y[k]) * root64(mkk[k]));
#pragma unroll
    for (int i = 0; i < k; ++i) y[i] = fma(-L[(tri0(k) + i) * 32], y[k], y[i]);
  }
  return mx;
}

__device__ __forceinline__ void write_derivs(const FitArgs& a, int f, int dst, const double (&g)[3],
                                             const double (&h)[6]) {
  const int64_t n = a.n;
  for (int c = 0; c < 3; ++c) a.grad[(f * 3 + c) * n + dst] = g[c];
  if (a.hess)
    for (int c = 0; c < 6; ++c) a.hess[(f * 6 + c) * n + dst] = h[c];
}

// Time derivatives of slot s.  Out of line: both forms then run the same code.
__device__ __noinline__ void write_rhs(const FitArgs& a, int s, int dst, const MhdDerivs<double>& D) {
  const int64_t n = a.n;
  double u[8];
  for (int f = 0; f < 8; ++f) u[f] = a.sU[f * n + s];
  const int src = a.perm_in ? a.perm_in[s] : s;
  double zeta = a.zeta ? a.zeta[src] : 0.0;
  double eta = a.eta ? a.eta[src] : 0.0;
  if (a.c_zeta_l != 0.0 || a.c_zeta_a != 0.0 || a.c_eta != 0.0)
    mhd_laws(u, D, a.gamma, a.slam[s], a.c_zeta_l, a.c_zeta_a, a.c_eta, zeta, eta);
  double out[8];
  mhd_rhs(u, D, a.gamma, zeta, eta, out);
  bool finite = true;
  for (int f = 0; f < 8; ++f) {
    finite &= finite64(out[f]);
    a.dudt[f * n + dst] = out[f];
  }
  if (!finite) raise_flag(a.status_word, PHB_FLAG_NONFINITE);
}

// One particle per lane (slot < 0: none); my: the lane's shared-memory column
// (stride 32).  All lanes call it.  Returns true, with nothing written, when
// the fit needs the corrected step.
template <FitMode MODE>
__device__ __forceinline__ bool fit_thread(const FitArgs& a, const Box64& bx, int slot, bool routed,
                                           double refine_above, double* my) {
  constexpr int f0 = MODE == FitMode::kRHS ? 1 : 0;  // the RHS never needs the density fit
  const int64_t n = a.n;
  const int s = slot < 0 ? 0 : slot;
  const double lam = a.slam[s];
  const double inv_l = 1.0 / lam;
  const double rf = a.g.rf_factor * lam;
  const int64_t beg = a.off[s];
  const int len = slot < 0 ? 0 : list_len64(a.off, a.g.capacity, s);
  double m[kNM];
  const int cnt = accum_thread<f0>(a.spos, a.sU, n, a.idx + beg, len, s, bx, a.weight_kind, inv_l,
                                   1.0 / (rf * rf), my, m);
  // the right-hand sides to local memory, the normal matrix in their place
  double b[kNF * kNB];
#pragma unroll 4
  for (int k = f0 * kNB; k < kNF * kNB; ++k) b[k] = my[k * 32];
  struct Col {
    double* p;
    __device__ __forceinline__ double& operator[](int k) const { return p[k * 32]; }
  };
  Col M{my};
  mls_assemble(m, M);
  bool singular = cnt < kNB;
  if (!singular) {
    double mkk[kNB];
    chol_panel<0, 4>(my, mkk, singular);
    chol_panel<4, 4>(my, mkk, singular);
    chol_panel<8, 5>(my, mkk, singular);
    chol_panel<13, 6>(my, mkk, singular);
    if (!singular && kNB * inv_norm_est(my, mkk) > refine_above) return true;
  }
  if (slot < 0) return false;
  const int dst = a.perm_out ? a.perm_out[s] : s;
  if (a.fit_status) a.fit_status[dst] = singular ? 1 : (routed ? 2 : 0);
  if (singular) raise_flag(a.status_word, PHB_FLAG_FIT_SINGULAR);
  const double il2 = inv_l * inv_l;
  MhdDerivs<double> D;
  mhd_zero(D);
  // fields f .. f + N - 1
  auto fields = [&](int f, auto group) {
    constexpr int N = decltype(group)::value;
    double c[N][kNB];
#pragma unroll
    for (int u = 0; u < N; ++u)
#pragma unroll
      for (int k = 0; k < kNB; ++k) c[u][k] = b[(f + u) * kNB + k];
    solve_thread<N, 0, kQuad0>(my, c);
#pragma unroll
    for (int u = 0; u < N; ++u) {
      double g[3] = {0, 0, 0}, h[6] = {0, 0, 0, 0, 0, 0};
      if (!singular) derivs_of([&](int k) { return c[u][k]; }, inv_l, il2, g, h);
      if (MODE == FitMode::kDerivs) write_derivs(a, f + u, dst, g, h);
      else mhd_collect(D, f + u, g, h);
    }
  };
  if (MODE == FitMode::kDerivs) {
#pragma unroll 1
    for (int f = 0; f < kNF; f += 4) fields(f, Num<4>{});
  } else {
    fields(1, Num<4>{});
    fields(5, Num<3>{});
    write_rhs(a, s, dst, D);
  }
  return false;
}

// What a lane does in the warp form: its sums (operands within a staged
// neighbour's row) and its entries of the normal matrix.
struct WarpTab {
  int sum[8];    // byte offsets: first | second << 16
  int entry[6];  // row | column << 8 | moment << 16; column -1 (0xff): none
};

template <FitMode MODE>
__device__ __forceinline__ void warp_tab(WarpTab& w, int lane) {
  constexpr int f0 = MODE == FitMode::kRHS ? 1 : 0;
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int t = lane + 32 * u;
    int x = 0, y = 0;
    if (t < kNM) {
      mls_moment_split(t, x, y);
      y += kNB;
    } else if (t < kNM + (kNF - f0) * kNB) {
      x = 11 + f0 + (t - kNM) / kNB;
      y = kNB + (t - kNM) % kNB;
    }
    w.sum[u] = x * 8 | (y * 8) << 16;
  }
  // entries from the bottom right corner, column by column: those right of
  // column j are a prefix
#pragma unroll
  for (int u = 0; u < 6; ++u) {
    const int t = lane + 32 * u;
    int k = 0;
    while (tri0(k + 1) <= t) ++k;
    const int col = kNB - 1 - k, row = kNB - 1 - (t - tri0(k));
    w.entry[u] = t < kNT ? row | col << 8 | mls_moment_index(row, col) << 16 : 0xff00;
  }
}

// Sums over the neighbours of slot s; with Res, of the residuals of the
// coefficients in W[kWC..] instead of the field differences.  Moments to
// W[kWM..], right-hand sides to W[kWB..].  Returns the neighbours within r_f.
template <FitMode MODE, bool Res>
__device__ __forceinline__ int warp_sums(const FitArgs& a, const Box64& bx, const WarpTab& tab, int s,
                                         double inv_l, double inv_rf2, double* W, int lane) {
  constexpr int f0 = MODE == FitMode::kRHS ? 1 : 0;
  constexpr int nsum = kNM + (kNF - f0) * kNB;
  constexpr int rounds = (nsum + 31) / 32;
  const int64_t n = a.n;
  const int64_t beg = a.off[s], end = beg + list_len64(a.off, a.g.capacity, s);
  const double xs = a.spos[s], ys = a.spos[n + s], zs = a.spos[2 * n + s];
  double acc[rounds];
#pragma unroll
  for (int u = 0; u < rounds; ++u) acc[u] = 0.0;
  int cnt = 0;
  for (int64_t c0 = beg; c0 < end; c0 += 32) {
    const int64_t e = c0 + lane;
    bool inside = false;
    double dx = 0, dy = 0, dz = 0, s2 = 0;
    double du[kNF];
    if (e < end) {
      const int t = a.idx[e];
#pragma unroll
      for (int f = f0; f < kNF; ++f) du[f] = a.sU[f * n + t] - a.sU[f * n + s];
      dx = wrap64(bx, 0, a.spos[t] - xs);
      dy = wrap64(bx, 1, a.spos[n + t] - ys);
      dz = wrap64(bx, 2, a.spos[2 * n + t] - zs);
      s2 = dist_rel(dx, dy, dz, inv_rf2, inside);
    }
    const unsigned in = __ballot_sync(0xffffffffu, inside);
    if (inside) {
      double* row = W + __popc(in & ((1u << lane) - 1u)) * kRow;
      const double wt = weight64(s2, a.weight_kind);
      double qg[kNB], wq[kNB + 1];
      mls_monomials_cubic_w(dx * inv_l, dy * inv_l, dz * inv_l, wt, qg, wq);
#pragma unroll
      for (int k = 0; k < 11; ++k) row[k] = wq[k];
#pragma unroll
      for (int k = 0; k < kNB; ++k) row[kNB + k] = qg[k];
#pragma unroll
      for (int f = f0; f < kNF; ++f) {
        double r = du[f];
        if (Res)
#pragma unroll
          for (int k = 0; k < kNB; ++k) r = fma(-qg[k], W[kWC + f * kNB + k], r);
        row[11 + f] = wt * r;
      }
    }
    __syncwarp();
    const int m = __popc(in);
    cnt += m;
    const char* row = reinterpret_cast<const char*>(W);
#pragma unroll 2
    for (int j = 0; j < m; ++j, row += kRow * 8)
#pragma unroll
      for (int u = 0; u < rounds; ++u)
        acc[u] = fma(*reinterpret_cast<const double*>(row + (tab.sum[u] & 0xffff)),
                     *reinterpret_cast<const double*>(row + (tab.sum[u] >> 16)), acc[u]);
    __syncwarp();
  }
#pragma unroll
  for (int u = 0; u < rounds; ++u) {
    const int t = lane + 32 * u;
    if (t < kNM) W[kWM + t] = acc[u];
    else if (t < nsum) W[kWB + f0 * kNB + t - kNM] = acc[u];
  }
  __syncwarp();
  return cnt;
}

// inv_norm_est with a row per lane (each sum in its order).
__device__ __forceinline__ double warp_inv_norm_est(const double* W, int lane) {
  const double* L = W + kWL;
  const int i = lane < kNB ? lane : kNB - 1;
  const double inv = W[kWI + i];
  const double sq = root64(W[kWM + mls_moment_index(i, i)]);
  double s = 0.0, y = 0.0;
#pragma unroll
  for (int k = 0; k < kNB; ++k) {
    if (lane == k) y = ((s > 0.0 ? -sq : sq) - s) * inv;
    const double yk = __shfl_sync(0xffffffffu, y, k);
    if (i > k) s = fma(L[tri0(i) + k], yk, s);
  }
#pragma unroll
  for (int k = kNB - 1; k >= 0; --k) {
    if (lane == k) y *= inv;
    const double xk = __shfl_sync(0xffffffffu, y, k);
    if (i < k) y = fma(-L[tri0(k) + i], xk, y);
  }
  double mx = lane < kNB ? fabs(y) * sq : 0.0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  return mx;
}

// Substitutions of all fields at once, four lanes per field (rows i = q mod 4);
// coefficients Lo .. 18 of each field to v (row q + 4 u).
template <int Lo>
__device__ __forceinline__ void warp_solve(const double* W, const double* rhs, int q, double (&v)[5]) {
  const double* L = W + kWL;
  const double* inv = W + kWI;
#pragma unroll
  for (int u = 0; u < 5; ++u) v[u] = q + 4 * u < kNB ? rhs[q + 4 * u] : 0.0;
#pragma unroll
  for (int k = 0; k < kNB; ++k) {
    const double y = __shfl_sync(0xffffffffu, v[k >> 2] * inv[k], k & 3, 4);
    if (q == (k & 3)) v[k >> 2] = y;
#pragma unroll
    for (int u = 0; u < 5; ++u) {
      const int i = q + 4 * u;
      if (4 * u + 3 > k && i > k && i < kNB) v[u] = fma(-L[tri0(i) + k], y, v[u]);
    }
  }
#pragma unroll
  for (int i = kNB - 1; i >= Lo; --i) {
    const double c = __shfl_sync(0xffffffffu, v[i >> 2] * inv[i], i & 3, 4);
    if (q == (i & 3)) v[i >> 2] = c;
#pragma unroll
    for (int u = 0; u < 5; ++u) {
      const int k = q + 4 * u;
      if (4 * u < i && 4 * u + 3 >= Lo && k >= Lo && k < i) v[u] = fma(-L[tri0(i) + k], c, v[u]);
    }
  }
}

// One particle by one warp (all lanes call it with the same s).
template <FitMode MODE>
__device__ __forceinline__ void fit_warp(const FitArgs& a, const Box64& bx, const WarpTab& tab, int s,
                                         bool routed, double refine_above, double* W) {
  constexpr int f0 = MODE == FitMode::kRHS ? 1 : 0;
  const int lane = threadIdx.x & 31;
  const double lam = a.slam[s];
  const double rf = a.g.rf_factor * lam;
  const double inv_l = 1.0 / lam, inv_rf2 = 1.0 / (rf * rf);
  const int cnt = warp_sums<MODE, false>(a, bx, tab, s, inv_l, inv_rf2, W, lane);
  bool singular = cnt < kNB;
  double* L = W + kWL;
  const int q = lane & 3, f = f0 + (lane >> 2);
  const bool mine = f < kNF;
  if (!singular) {
    // each lane keeps its entries of the matrix; per column: the owners write
    // it out, every lane forms 1 / L_jj, the rows below are scaled, and the
    // entries right of it are updated
    double e[6];
    int row[6], col[6];
#pragma unroll
    for (int u = 0; u < 6; ++u) {
      row[u] = tab.entry[u] & 0xff;
      col[u] = tab.entry[u] >> 8 & 0xff;
      e[u] = W[kWM + (tab.entry[u] >> 16)];
      if (row[u] == col[u]) W[kWI + row[u]] = e[u];  // M_jj until 1 / L_jj takes its place
    }
#pragma unroll 1
    for (int j = 0; j < kNB; ++j) {
#pragma unroll
      for (int u = 0; u < 6; ++u)
        if (col[u] == j) L[tri0(row[u]) + j] = e[u];
      __syncwarp();
      const double p = L[tri0(j) + j], d = W[kWI + j];
      const int below = tri0(j + 1 + lane) + j;
      const double v = j + 1 + lane < kNB ? L[below] : 0.0;
      singular |= !(p > 0.0) || !(p > 1e-12 * d);
      const double r = rsqrt(p > 0.0 ? p : 1.0);
      if (j + 1 + lane < kNB) L[below] = v * r;
      __syncwarp();
      if (lane == 0) W[kWI + j] = r;
#pragma unroll
      for (int u = 0; u < 6; ++u)
        if (col[u] > j && col[u] < kNB)
          e[u] = fma(-L[tri0(row[u]) + j], L[tri0(col[u]) + j], e[u]);
    }
    __syncwarp();
  }
  bool refine = false;
  if (!singular) {
    const double est = warp_inv_norm_est(W, lane);
    refine = kNB * est > refine_above;
    __syncwarp();
    double v[5];
    const double* rhs = W + kWB + (mine ? f : f0) * kNB;
    if (refine) {
      warp_solve<0>(W, rhs, q, v);
      if (mine)
#pragma unroll
        for (int u = 0; u < 5; ++u)
          if (q + 4 * u < kNB) W[kWC + f * kNB + q + 4 * u] = v[u];
      __syncwarp();
      warp_sums<MODE, true>(a, bx, tab, s, inv_l, inv_rf2, W, lane);
      warp_solve<kQuad0>(W, rhs, q, v);
      if (mine)
#pragma unroll
        for (int u = 2; u < 5; ++u)
          if (q + 4 * u >= kQuad0 && q + 4 * u < kNB) W[kWC + f * kNB + q + 4 * u] += v[u];
    } else {
      warp_solve<kQuad0>(W, rhs, q, v);
      if (mine)
#pragma unroll
        for (int u = 2; u < 5; ++u)
          if (q + 4 * u < kNB) W[kWC + f * kNB + q + 4 * u] = v[u];
    }
  }
  __syncwarp();
  const int dst = a.perm_out ? a.perm_out[s] : s;
  const double il2 = inv_l * inv_l;
  if (lane == 0) {
    if (a.fit_status) a.fit_status[dst] = singular ? 1 : (routed ? 2 : 0);
    if (singular) raise_flag(a.status_word, PHB_FLAG_FIT_SINGULAR);
  }
  if (MODE == FitMode::kDerivs) {
    if (q == 0) {
      double g[3] = {0, 0, 0}, h[6] = {0, 0, 0, 0, 0, 0};
      if (!singular) derivs_of([&](int k) { return W[kWC + f * kNB + k]; }, inv_l, il2, g, h);
      write_derivs(a, f, dst, g, h);
    }
  } else if (lane == 0) {
    MhdDerivs<double> D;
    mhd_zero(D);
#pragma unroll
    for (int k = f0; k < kNF; ++k) {
      double g[3] = {0, 0, 0}, h[6] = {0, 0, 0, 0, 0, 0};
      if (!singular) derivs_of([&](int c) { return W[kWC + k * kNB + c]; }, inv_l, il2, g, h);
      mhd_collect(D, k, g, h);
    }
    write_rhs(a, s, dst, D);
  }
  __syncwarp();  // the next particle takes the same shared memory
}

// Which form serves which part of the work: a pass of the thread form over
// the grid fits gridDim x 128 particles (19,456 on 152 SMs) in 0.65 ms
// whatever their number, the warp form gridDim x 4 particles in 34 us; so
// full passes go to the thread form and a remainder of up to kWarpPasses
// passes of the warp form (0.54 ms) to the warp form.
constexpr int kWarpPasses = 8;

// Particles: the slots of `list` (device count *list_len), or all, taken tile
// by tile in the order of tmap (longest lists first within a tile), so that
// a warp's loops are of similar length.
template <FitMode MODE>
__global__ void __launch_bounds__(kT, 1) k_fit_fp64(const __grid_constant__ FitArgs a, bool routed,
                                                    const int32_t* list, const int32_t* list_len,
                                                    const uint8_t* tmap) {
  extern __shared__ double sm[];
  const int total = list ? *list_len : static_cast<int>((a.n + a.g.tile - 1) / a.g.tile) * a.g.tile;
  const int pass = gridDim.x * kT, warp_pass = gridDim.x * kWarps;
  int full = total / pass * pass;
  if (total - full > kWarpPasses * warp_pass) full = total;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  // warps numbered across the SMs first: a last, partial pass spreads over them
  const int gw = wid * gridDim.x + blockIdx.x;
  if (full == 0 && gw >= total) return;  // an empty or short queue: no FP64 set-up
  const Box64 bx = make_box64(a.g);
  double* W = sm + wid * kSlots * 32;
  // fits routed from the FP32-mixed path need ~1e-5: FP64 normal equations
  // meet that up to cond(M) ~ 1e9; the FP64 path itself targets ~1e-12
  const double refine_above = routed ? 1e9 : 1e4;
  auto slot = [&](int w) {
    if (list) return w < total ? list[w] : -1;
    if (w >= total) return -1;
    const int s = w / a.g.tile * a.g.tile + tmap[w];
    return s < a.n ? s : -1;
  };
  for (int w0 = gw * 32; w0 < full; w0 += pass) {
    const int s = w0 + lane < full ? slot(w0 + lane) : -1;
    const bool refine = fit_thread<MODE>(a, bx, s, routed, refine_above, W + lane);
    __syncwarp();
    unsigned todo = __ballot_sync(0xffffffffu, refine);
    if (todo != 0u) {
      WarpTab tab;
      warp_tab<MODE>(tab, lane);
      for (; todo != 0u; todo &= todo - 1u)
        fit_warp<MODE>(a, bx, tab, __shfl_sync(0xffffffffu, s, __ffs(todo) - 1), routed, refine_above, W);
    }
  }
  if (full + gw < total) {
    WarpTab tab;
    warp_tab<MODE>(tab, lane);
    for (int w = full + gw; w < total; w += warp_pass) {
      const int s = slot(w);
      if (s >= 0) fit_warp<MODE>(a, bx, tab, s, routed, refine_above, W);
    }
  }
}

}  // namespace

cudaError_t launch_fit_fp64(const FitArgs& a, FitMode mode, const int32_t* list,
                            const int32_t* list_len, const uint8_t* tmap, cudaStream_t st, bool routed) {
  const size_t smem = size_t(kSlots) * kT * sizeof(double);
  const unsigned blocks = static_cast<unsigned>(num_sms());
  const auto kernel = mode == FitMode::kDerivs ? k_fit_fp64<FitMode::kDerivs> : k_fit_fp64<FitMode::kRHS>;
  cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  const int tr = trace_begin(list ? 3 : 2, st);
  kernel<<<blocks, kT, smem, st>>>(a, routed, list, list_len, tmap);
  note_launch();
  trace_end(tr, st);
  return cudaGetLastError();
}

}  // namespace phb
