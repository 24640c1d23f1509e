// Reverse-mode adjoint of the fused MLS fit + MHD right-hand side, FP64.
// (The paper has no adjoint; this differentiates the forward map of
// phb_mhd_rhs: Sec. 2 fit and App. A right-hand side, neighbour sets fixed,
// lambda constant.)
//
// Per particle i, with fitted fields f (V, B, sigma) and neighbours j:
//   forward   m_a = sum_j w_j q_j^a,  b_f = sum_j w_j p_j dU_fj,  M c_f = b_f,
//             derivatives from c_f, right-hand side from derivatives and U_i;
//   backward  cbar_f from the right-hand side's adjoint, bbar_f = M^-1 cbar_f,
//             Mbar = -sum_f bbar_f c_f^T folded onto the moments (mbar),
//             then per neighbour
//               dUbar_fj = w_j (p_j . bbar_f)
//               wbar_j   = sum_a mbar_a q_j^a + sum_f dU_fj (p_j . bbar_f)
//               qbar_j   = w_j grad_q[ sum_a mbar_a q^a + sum_f dU_fj p(q) . bbar_f ]
//               dbar_j   = qbar_j / lambda_i + wbar_j dw/dd,
//             whose negatives are particle i's own terms (U_i, x_i).
// k_adjoint takes a particle per thread through all of it: the fit as in
// phb_fit64.cuh, the seeds bbar_f and mbar in the shared memory that held the
// factor, then the neighbours, whose ten terms go to a buffer, one row per
// list entry.  k_adj_gather sums, for every particle j, the rows of the entries
// that name it, through a reverse list in ascending order of the entries, so
// the result does not depend on thread scheduling.  The buffer holds a bounded
// part of the entries: the particles are taken in chunks of consecutive slots.
//
// What bounds it: the FP64 pipe (see phb_fit_fp64.cu).  Per neighbour the fit
// takes 267 FP64 instructions and the backward pass ~500 (266 products with the
// seeds, 162 FMAs and 40 others for the degree-6 polynomial and its gradient by
// nested multiplication, the rest offsets and weights); forming every entry's terms once and passing them through
// memory (80 B written and read per entry, 0.3 ms per 262,144 particles) costs
// less than forming them a second time for the neighbour.  Four warps per SM
// (213 doubles of shared memory per thread).  Measured, 262,144 particles:
// gradient 62.3 -> 28.2 ms, with the lists of a step's skin 67 -> 31.7 (before: each entry's terms formed again in the gather, 84
// tabulated monomials, seeds in global memory).
//
// By default the factorisation is recomputed here (nothing is stored by the
// forward call); the stored variant records, per particle, the Cholesky
// factor and the fitted coefficients once (kRecord) and the adjoint then starts from that record (kStored) instead of
// re-accumulating the moments and right-hand sides.
#include <algorithm>

#include "phb_fit64.cuh"
#include "phb_mhd.cuh"

namespace phb {
namespace {

constexpr int kWarps = 4;  // per block, one block per SM: one warp per sub-partition
constexpr int kT = 32 * kWarps;
constexpr int kThreads = 256;
constexpr int kNFit = 7;  // fitted fields: U indices 1..7 (V, B, sigma)
// a lane's column: the fit, the factor, then bbar_f [field][19] and mbar [80]
constexpr int kSlotMbar = kNFit * kNB;
constexpr int kSlots = kSlotMbar + kNM;
static_assert(kSlots >= kNT && size_t(kSlots) * kT * 8 <= 227 * 1024, "shared memory of a block");
// record of one particle's forward fit, [k][n] layout: factor (190, 1 / L_kk on
// its diagonal), 19 words not used (they keep the record's size), coefficients
// c_f (7 x 19), then 1 = singular / 0 = regular
constexpr int kRecFac = 0, kRecCoef = kNT + kNB, kRecFlag = kRecCoef + kNFit * kNB;
constexpr int kRecWords = kRecFlag + 1;
constexpr int kTerms = 10;  // an entry's row: dUbar of fields 1..7, dbar
enum AdjMode { kRecompute = 0, kRecord = 1, kStored = 2 };

struct AdjArgs {
  Grid g;
  int32_t n;
  const int32_t* perm;   // slot -> caller index
  const uint8_t* tmap;   // per tile: its particles, longest list first
  const double* spos;
  const double* slam;
  const double* sU;
  const int64_t* off;
  const int32_t* idx;
  const double* gbar;    // caller order [8][n]
  double gamma;
  int32_t weight_kind;
  const double* zeta;    // caller order or null
  const double* eta;
  double c_zeta_l, c_zeta_a, c_eta;  // coefficient laws (phb_params), 0 = off
  double* terms;         // [entries of a chunk][kTerms]
  double* acc;           // [11][n] slot order: Ubar, xbar so far
  double* rec;           // [kRecWords][n] slot order (stored variant) or null
  int32_t* status_word;
  int64_t span;          // list entries per chunk (rows of `terms` less n)
  int32_t chunk, chunks;
};

// First slot whose list starts at entry e0 or later (a warp samples 32 points
// per step).
__device__ __forceinline__ int first_slot(const int64_t* off, int n, int64_t e0) {
  const int lane = threadIdx.x & 31;
  int lo = 0, hi = n;  // off[lo - 1] < e0 <= off[hi]
  while (lo < hi) {
    const int step = (hi - lo + 31) / 32;
    const int at = lo + lane * step;
    const unsigned below = __ballot_sync(0xffffffffu, at < hi && off[at] < e0);
    if (below == 0u) return lo;
    const int last = lo + (31 - __clz(below)) * step;  // off[last] < e0
    lo = last + 1;
    hi = min(hi, last + step);
  }
  return lo;
}

// Slots [first, last) of the chunk: those whose lists start in its part of the
// entries, which as few chunks as hold them share evenly (a list is shorter
// than n, so a chunk's entries fit span + n rows; the later chunks of a capacity
// that the lists do not need are empty).
__device__ __forceinline__ void chunk_slots(const AdjArgs& a, int& first, int& last) {
  const int64_t total = a.off[a.n] < a.g.capacity ? a.off[a.n] : a.g.capacity;
  const int64_t used = total > a.span ? (total + a.span - 1) / a.span : 1;
  const int64_t part = (total + used - 1) / used;
  first = a.chunk == 0 ? 0 : (a.chunk < used ? first_slot(a.off, a.n, a.chunk * part) : a.n);
  last = a.chunk + 1 < used ? first_slot(a.off, a.n, (a.chunk + 1) * part) : a.n;
}

// Adjoint of the right-hand side at one particle.  In: point values u, the
// derivatives D, the input coefficients zeta / eta and the coefficient laws
// (lam, cl, ca, ce as in mhd_laws), output adjoint o.  Out: ubar (point
// values) and the adjoints of each fitted field's gradient gb[f][3] and
// packed Hessian hb[f][6] (f = 0..6 for U indices 1..7).
__device__ void rhs_adjoint_point(const double (&u)[8], const MhdDerivs<double>& D, double gamma,
                                  double zeta, double eta, double lam, double cl, double ca,
                                  double ce, const double (&o)[8], double (&ubar)[8],
                                  double (&gb)[kNFit][3], double (&hb)[kNFit][6]) {
  const double rho = u[0], sig = u[7];
  const double B[3] = {u[4], u[5], u[6]};
  const double divV = D.gV[0][0] + D.gV[1][1] + D.gV[2][2];
  // the laws' totals (forward as mhd_laws): c = sqrt(q), q = (gamma P + |B|^2) / rho
  const bool laws = cl != 0.0 || ca != 0.0 || ce != 0.0;
  double q = 0.0, c = 0.0;
  if (laws) {
    q = (gamma * ((gamma - 1.0) * sig) + B[0] * B[0] + B[1] * B[1] + B[2] * B[2]) / rho;
    c = sqrt(q);
    zeta += cl * lam * c;
    if (divV < 0.0) zeta -= ca * lam * lam * divV;
    eta += ce * lam * c;
  }
  const double J[3] = {D.gB[2][1] - D.gB[1][2], D.gB[0][2] - D.gB[2][0], D.gB[1][0] - D.gB[0][1]};
  const double F[3] = {J[1] * B[2] - J[2] * B[1], J[2] * B[0] - J[0] * B[2], J[0] * B[1] - J[1] * B[0]};
  for (int k = 0; k < 8; ++k) ubar[k] = 0.0;
  for (int f = 0; f < kNFit; ++f) {
    for (int c = 0; c < 3; ++c) gb[f][c] = 0.0;
    for (int c = 0; c < 6; ++c) hb[f][c] = 0.0;
  }
  const double irho = 1.0 / rho;
  // out[1+a] = (F_a - (gamma-1) gs_a) / rho + zeta gdivV_a
  double Fb[3], divVb = 0.0;
  for (int a = 0; a < 3; ++a) {
    const double ob = o[1 + a];
    Fb[a] = ob * irho;
    gb[6][a] += -ob * (gamma - 1.0) * irho;                       // sigma gradient
    ubar[0] += -ob * (F[a] - (gamma - 1.0) * D.gs[a]) * irho * irho;
    // gdivV_a = sum_c h_{V_c}[a, c]
    for (int c = 0; c < 3; ++c) hb[c][hpack(a, c)] += ob * zeta;
  }
  // out[0] = -rho divV
  ubar[0] += -o[0] * divV;
  divVb += -o[0] * rho;
  // out[4+a] = sum_b B_b gV[a][b] - B_a divV + eta gdivB_a
  for (int a = 0; a < 3; ++a) {
    const double ob = o[4 + a];
    for (int b = 0; b < 3; ++b) {
      gb[a][b] += ob * B[b];                 // gV[a][b]
      ubar[4 + b] += ob * D.gV[a][b];
    }
    ubar[4 + a] += -ob * divV;
    divVb += -ob * B[a];
    for (int c = 0; c < 3; ++c) hb[3 + c][hpack(a, c)] += ob * eta;
  }
  // out[7] = -gamma sigma divV + rho zeta divV^2
  ubar[7] += -o[7] * gamma * divV;
  ubar[0] += o[7] * zeta * divV * divV;
  divVb += o[7] * (-gamma * sig + 2.0 * rho * zeta * divV);
  if (laws) {
    // zeta_bar and eta_bar, then through zeta = .. + cl lam c + ca lam^2
    // max(0, -div V) and eta = .. + ce lam c
    double zb = o[7] * rho * divV * divV, eb = 0.0;
    for (int a = 0; a < 3; ++a) {
      zb += o[1 + a] * D.gdivV[a];
      eb += o[4 + a] * D.gdivB[a];
    }
    if (divV < 0.0) divVb += -zb * ca * lam * lam;
    const double cb = (zb * cl + eb * ce) * lam;
    if (c > 0.0) {
      const double qb = cb / (2.0 * c);
      ubar[7] += qb * gamma * (gamma - 1.0) / rho;
      for (int b = 0; b < 3; ++b) ubar[4 + b] += qb * 2.0 * B[b] / rho;
      ubar[0] += -qb * q / rho;
    }
  }
  for (int a = 0; a < 3; ++a) gb[a][a] += divVb;
  // F = J x B:  Bbar += Fbar x J,  Jbar = B x Fbar
  ubar[4] += Fb[1] * J[2] - Fb[2] * J[1];
  ubar[5] += Fb[2] * J[0] - Fb[0] * J[2];
  ubar[6] += Fb[0] * J[1] - Fb[1] * J[0];
  const double Jb[3] = {B[1] * Fb[2] - B[2] * Fb[1], B[2] * Fb[0] - B[0] * Fb[2], B[0] * Fb[1] - B[1] * Fb[0]};
  // J = (gB[2][1] - gB[1][2], gB[0][2] - gB[2][0], gB[1][0] - gB[0][1]); B_c is field 3 + c
  gb[3 + 2][1] += Jb[0];
  gb[3 + 1][2] -= Jb[0];
  gb[3 + 0][2] += Jb[1];
  gb[3 + 2][0] -= Jb[1];
  gb[3 + 1][0] += Jb[2];
  gb[3 + 0][1] -= Jb[2];
}

template <int MODE>
__global__ void __launch_bounds__(kT, 1) k_adjoint(const __grid_constant__ AdjArgs a) {
  extern __shared__ double sm[];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  double* my = sm + wid * kSlots * 32 + lane;
  const int64_t N = a.n;
  int first = 0, last = a.n;
  if (MODE != kRecord) chunk_slots(a, first, last);
  if (first >= last) return;
  const int64_t row0 = MODE == kRecord ? 0 : a.off[first];
  const Box64 bx = make_box64(a.g);
  const int T = a.g.tile;
  const int w_end = (last + T - 1) / T * T;
  // warps numbered across the SMs first: a last, partial pass spreads over them
  for (int w0 = first / T * T + (wid * gridDim.x + blockIdx.x) * 32; w0 < w_end; w0 += gridDim.x * kT) {
    const int own = w0 / T * T + a.tmap[w0 + lane];
    const bool act = own >= first && own < last;
    const int s = act ? own : first;
    const double lam = a.slam[s];
    const double rf = a.g.rf_factor * lam;
    const double inv_rf2 = 1.0 / (rf * rf), il = 1.0 / lam, il2 = il * il;
    const int64_t beg = a.off[s];
    const int len = act ? list_len64(a.off, a.g.capacity, s) : 0;
    double c[kNFit * kNB];  // right-hand sides, then coefficients c_f
    bool singular;
    if (MODE == kStored) {
      singular = a.rec[kRecFlag * N + s] != 0.0;
      if (!singular) {
#pragma unroll 10
        for (int k = 0; k < kNT; ++k) my[k * 32] = a.rec[(kRecFac + k) * N + s];
#pragma unroll 10
        for (int k = 0; k < kNFit * kNB; ++k) c[k] = a.rec[(kRecCoef + k) * N + s];
      }
    } else {
      double m[kNM];
      const int cnt = accum_thread<1>(a.spos, a.sU, N, a.idx + beg, len, s, bx, a.weight_kind, il,
                                      inv_rf2, my, m);
#pragma unroll 4
      for (int k = 0; k < kNFit * kNB; ++k) c[k] = my[(kNB + k) * 32];
      struct Col {
        double* p;
        __device__ __forceinline__ double& operator[](int k) const { return p[k * 32]; }
      };
      Col M{my};
      mls_assemble(m, M);
      singular = cnt < kNB;
      if (!singular) {
        double mkk[kNB];
        chol_panel<0, 4>(my, mkk, singular);
        chol_panel<4, 4>(my, mkk, singular);
        chol_panel<8, 5>(my, mkk, singular);
        chol_panel<13, 6>(my, mkk, singular);
      }
      if (!singular) {
        auto solve = [&](int f, auto group) {
          constexpr int G = decltype(group)::value;
          double b[G][kNB];
#pragma unroll
          for (int u = 0; u < G; ++u)
#pragma unroll
            for (int k = 0; k < kNB; ++k) b[u][k] = c[(f + u) * kNB + k];
          solve_thread<G, 0, 0>(my, b);
#pragma unroll
          for (int u = 0; u < G; ++u)
#pragma unroll
            for (int k = 0; k < kNB; ++k) c[(f + u) * kNB + k] = b[u][k];
        };
        solve(0, Num<4>{});
        solve(4, Num<3>{});
      }
    }
    if (act && singular) raise_flag(a.status_word, PHB_FLAG_FIT_SINGULAR);
    if (MODE == kRecord) {
      if (act) {
        a.rec[kRecFlag * N + s] = singular ? 1.0 : 0.0;
        if (!singular) {
#pragma unroll 10
          for (int k = 0; k < kNT; ++k) a.rec[(kRecFac + k) * N + s] = my[k * 32];
#pragma unroll 10
          for (int k = 0; k < kNFit * kNB; ++k) a.rec[(kRecCoef + k) * N + s] = c[k];
        }
      }
      __syncwarp();
      continue;
    }
    // a singular fit's right-hand side is zero and does not depend on the
    // inputs: no own terms, and zero rows for the gather
    const bool live = act && !singular;
    double u[8], selfu[8], selfx[3] = {0.0, 0.0, 0.0};
    for (int f = 0; f < 8; ++f) {
      u[f] = a.sU[f * N + s];
      selfu[f] = 0.0;
    }
    if (live) {
      const int src = a.perm[s];
      double o[8];
      for (int f = 0; f < 8; ++f) o[f] = a.gbar[f * N + src];
      // derivatives, right-hand-side adjoint, cbar -> bbar = M^-1 cbar
      double bbar[kNFit * kNB];
      {
        MhdDerivs<double> D;
        mhd_zero(D);
#pragma unroll
        for (int f = 0; f < kNFit; ++f) {
          double g[3], h[6];
          derivs_of([&](int k) { return c[f * kNB + k]; }, il, il2, g, h);
          mhd_collect(D, f + 1, g, h);
        }
        double gb[kNFit][3], hb[kNFit][6];
        rhs_adjoint_point(u, D, a.gamma, a.zeta ? a.zeta[src] : 0.0, a.eta ? a.eta[src] : 0.0, lam,
                          a.c_zeta_l, a.c_zeta_a, a.c_eta, o, selfu, gb, hb);
        auto seeds = [&](auto from, auto group) {
          constexpr int F = decltype(from)::value, G = decltype(group)::value;
          double b[G][kNB];
#pragma unroll
          for (int v = 0; v < G; ++v) {
#pragma unroll
            for (int k = 0; k < kQuad0; ++k) b[v][k] = 0.0;
            b[v][kQuad0] = 2.0 * hb[F + v][0] * il2;
            b[v][kQuad0 + 1] = hb[F + v][1] * il2;
            b[v][kQuad0 + 2] = hb[F + v][2] * il2;
            b[v][kQuad0 + 3] = 2.0 * hb[F + v][3] * il2;
            b[v][kQuad0 + 4] = hb[F + v][4] * il2;
            b[v][kQuad0 + 5] = 2.0 * hb[F + v][5] * il2;
#pragma unroll
            for (int k = 0; k < 3; ++k) b[v][kLin0 + k] = gb[F + v][k] * il;
          }
          solve_thread<G, kQuad0, 0>(my, b);
#pragma unroll
          for (int v = 0; v < G; ++v)
#pragma unroll
            for (int k = 0; k < kNB; ++k) bbar[(F + v) * kNB + k] = b[v][k];
        };
        seeds(Num<0>{}, Num<4>{});
        seeds(Num<4>{}, Num<3>{});
      }
      // mbar = fold of -sum_f bbar_f c_f^T onto the moments; the factor is dead
      double mb[kNM];
#pragma unroll
      for (int k = 0; k < kNM; ++k) mb[k] = 0.0;
#pragma unroll 1
      for (int f = 0; f < kNFit; ++f) {
        double bb[kNB], cc[kNB];
#pragma unroll
        for (int k = 0; k < kNB; ++k) {
          bb[k] = bbar[f * kNB + k];
          cc[k] = c[f * kNB + k];
          my[(f * kNB + k) * 32] = bb[k];
        }
        mls_accum_mbar(bb, cc, mb);
      }
#pragma unroll
      for (int k = 0; k < kNM; ++k) my[(kSlotMbar + k) * 32] = mb[k];
    }
    // backward pass over the neighbours: an entry's terms to its row, their
    // negatives to particle i's own
    const double xs = a.spos[s], ys = a.spos[N + s], zs = a.spos[2 * N + s];
    const double dwd = a.weight_kind == 1 ? 0.0 : -4.0 * inv_rf2;
    const volatile double* seed = my;  // read again for each neighbour rather than kept
    const struct {
      const volatile double* p;
      __device__ __forceinline__ double operator[](int k) const { return p[k * 32]; }
    } mbar{my + kSlotMbar * 32};
    const int32_t* list = a.idx + beg;
    double2* row = reinterpret_cast<double2*>(a.terms + (beg - row0) * kTerms);
    const int longest = __reduce_max_sync(0xffffffffu, len);
    int t = len > 0 ? list[0] : s;
    double nx = a.spos[t], ny = a.spos[N + t], nz = a.spos[2 * N + t], nu[kNFit];
#pragma unroll
    for (int f = 0; f < kNFit; ++f) nu[f] = a.sU[(f + 1) * N + t];
    t = len > 1 ? list[1] : s;
#pragma unroll 1
    for (int e = 0; e < longest; ++e) {
      const double dx = wrap64(bx, 0, nx - xs), dy = wrap64(bx, 1, ny - ys), dz = wrap64(bx, 2, nz - zs);
      double du[kNFit];
#pragma unroll
      for (int f = 0; f < kNFit; ++f) du[f] = nu[f] - u[f + 1];
      // the next neighbour's values, a neighbour ahead
      nx = a.spos[t];
      ny = a.spos[N + t];
      nz = a.spos[2 * N + t];
#pragma unroll
      for (int f = 0; f < kNFit; ++f) nu[f] = a.sU[(f + 1) * N + t];
      t = e + 2 < len ? list[e + 2] : s;
      bool inside;
      const double s2 = dist_rel(dx, dy, dz, inv_rf2, inside);
      if (e < len) {
        double ub[kNFit], xb[3] = {0.0, 0.0, 0.0};
#pragma unroll
        for (int f = 0; f < kNFit; ++f) ub[f] = 0.0;
        if (inside && live) {
          const double sw = 1.0 - s2;
          const double wt = a.weight_kind == 1 ? 1.0 : sw * sw;
          const double x = dx * il, y = dy * il, z = dz * il;
          double p[kNB], Bt[kNB];
          mls_basis(x, y, z, p);
#pragma unroll
          for (int k = 0; k < kNB; ++k) Bt[k] = 0.0;
#pragma unroll
          for (int f = 0; f < kNFit; ++f) {
            double pb = 0.0;
#pragma unroll
            for (int k = 0; k < kNB; ++k) {
              const double bk = seed[(f * kNB + k) * 32];
              pb = fma(p[k], bk, pb);
              Bt[k] = fma(du[f], bk, Bt[k]);
            }
            ub[f] = wt * pb;
            selfu[f + 1] -= ub[f];
          }
          double P, Px, Py, Pz;
          mls_poly_grad(x, y, z, mbar, Bt, P, Px, Py, Pz);
          const double dw = P * dwd * sw;  // d w / d d = -4 (1 - s^2) d / r_f^2
          const double wl = wt * il;
          xb[0] = fma(wl, Px, dw * dx);
          xb[1] = fma(wl, Py, dw * dy);
          xb[2] = fma(wl, Pz, dw * dz);
#pragma unroll
          for (int k = 0; k < 3; ++k) selfx[k] -= xb[k];
        }
        double2* to = row + e * (kTerms / 2);
        to[0] = make_double2(ub[0], ub[1]);
        to[1] = make_double2(ub[2], ub[3]);
        to[2] = make_double2(ub[4], ub[5]);
        to[3] = make_double2(ub[6], xb[0]);
        to[4] = make_double2(xb[1], xb[2]);
      }
      __syncwarp();
    }
    if (act) {
      for (int k = 0; k < 8; ++k) a.acc[k * N + s] += selfu[k];
      for (int k = 0; k < 3; ++k) a.acc[(8 + k) * N + s] += selfx[k];
    }
    __syncwarp();
  }
}

// ---- reverse neighbour lists of a chunk: for every particle t, the chunk's
// entries that name t (numbered from the chunk's first).  A thread per entry.
template <bool FILL>
__global__ void __launch_bounds__(kThreads) k_rev(const __grid_constant__ AdjArgs a, int32_t* __restrict__ rcnt,
                                                  const int64_t* __restrict__ roff,
                                                  uint32_t* __restrict__ rsrc) {
  int first, last;
  chunk_slots(a, first, last);
  if (first >= last) return;
  const int64_t e0 = a.off[first];
  const int64_t e1 = a.off[last] < a.g.capacity ? a.off[last] : a.g.capacity;
  for (int64_t e = e0 + static_cast<int64_t>(blockIdx.x) * kThreads + threadIdx.x; e < e1;
       e += static_cast<int64_t>(gridDim.x) * kThreads) {
    const int t = a.idx[e];
    const int k = atomicAdd(&rcnt[t], 1);
    if (FILL) rsrc[roff[t] + k] = static_cast<uint32_t>(e - e0);
  }
}

// Puts a particle's m entries of the reverse list in ascending order in place,
// by one warp: bitonic merges whose first step mirrors, so that every exchange
// puts the smaller entry first and places beyond m need not exist.
__device__ __noinline__ void sort_entries(uint32_t* v, int m, int lane) {
  auto exchange = [&](int i, int p) {
    if (p < m) {
      const uint32_t a = v[i], b = v[p];
      if (a > b) {
        v[i] = b;
        v[p] = a;
      }
    }
  };
  int bits = 0;  // 2^bits >= m
  while ((1 << bits) < m) ++bits;
  for (int k = 1; k <= bits; ++k) {
    for (int t = lane; t < 1 << (bits - 1); t += 32) {
      const int at = t >> (k - 1) << k, o = t & ((1 << (k - 1)) - 1);
      exchange(at + o, at + (1 << k) - 1 - o);
    }
    __syncwarp();
    for (int d = k - 2; d >= 0; --d) {
      for (int t = lane; t < 1 << (bits - 1); t += 32) {
        const int at = (t >> d << (d + 1)) + (t & ((1 << d) - 1));
        exchange(at, at + (1 << d));
      }
      __syncwarp();
    }
  }
}

// Add the chunk's rows that name t to t's sums: a warp per particle.  The
// atomics left its entries in any order: each entry's rank among them (their
// number smaller than it) puts them in order in shared memory, 32 at a time
// (more than a warp's registers hold, kNear, are sorted where they lie: with
// ranks read anew for every 32 the gradient of 50,000 particles with a clump
// of 1,000 took 49 ms, of 3,000 419; it takes 35 and 175), then three groups of ten lanes sum every third row, a column per lane, so
// that a row is read as one piece.  With the last chunk the sums go out in
// caller order.
__global__ void __launch_bounds__(128) k_adj_gather(const __grid_constant__ AdjArgs a,
                                                    const int64_t* __restrict__ roff, uint32_t* rsrc,
                                                    double* __restrict__ Ubar,
                                                    double* __restrict__ xbar) {
  constexpr int kRegs = 4, kNear = 32 * kRegs;  // entries per lane kept in registers
  __shared__ uint32_t sorted[4][32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t w = static_cast<int64_t>(blockIdx.x) * 4 + wid;
  if (w >= a.n) return;
  const int t = static_cast<int>(w);
  const int64_t N = a.n;
  const int64_t r0 = roff[t];
  const int m = static_cast<int>(roff[t + 1] - r0);
  const int grp = lane / kTerms, col = lane - grp * kTerms;
  double acc = 0.0;
  // sums of up to 32 entries from `from` on
  auto add_rows = [&](const uint32_t* from, int cnt) {
    if (grp < 3)
#pragma unroll 4
      for (int j = grp; j < cnt; j += 3) acc += a.terms[static_cast<int64_t>(from[j]) * kTerms + col];
  };
  if (m > kNear) {
    sort_entries(rsrc + r0, m, lane);
    for (int base = 0; base < m; base += 32) add_rows(rsrc + r0 + base, m - base < 32 ? m - base : 32);
  } else {
    uint32_t v[kRegs];
    int rank[kRegs];
#pragma unroll
    for (int q = 0; q < kRegs; ++q) {
      v[q] = q * 32 + lane < m ? rsrc[r0 + q * 32 + lane] : 0xffffffffu;
      rank[q] = 0;
    }
#pragma unroll
    for (int q = 0; q < kRegs; ++q)
      for (int j = 0; j < 32 && q * 32 + j < m; ++j) {
        const uint32_t x = __shfl_sync(0xffffffffu, v[q], j);
#pragma unroll
        for (int k = 0; k < kRegs; ++k) rank[k] += x < v[k] ? 1 : 0;
      }
    for (int base = 0; base < m; base += 32) {
      __syncwarp();
#pragma unroll
      for (int q = 0; q < kRegs; ++q)
        if (q * 32 + lane < m && rank[q] >= base && rank[q] < base + 32) sorted[wid][rank[q] - base] = v[q];
      __syncwarp();
      add_rows(sorted[wid], m - base < 32 ? m - base : 32);
    }
  }
  const bool done = a.chunk == a.chunks - 1;
  if (m == 0 && !done) return;  // (of an empty chunk, all)
  const double s1 = __shfl_down_sync(0xffffffffu, acc, kTerms);
  const double s2 = __shfl_down_sync(0xffffffffu, acc, 2 * kTerms);
  acc += s1 + s2;
  // columns 0..6: Ubar of fields 1..7, 7..9: xbar; Ubar of field 0 has own terms only
  const int k = lane < kTerms ? lane + 1 : 0;
  if (lane > kTerms) return;
  double* sum = a.acc + k * N + t;
  const double total = lane < kTerms ? *sum + acc : *sum;
  if (!done) {
    *sum = total;
    return;
  }
  const int i = a.perm[t];
  if (k < 8) Ubar[k * N + i] = total;
  else xbar[(k - 8) * N + i] = total;
}

}  // namespace
}  // namespace phb

using namespace phb;

namespace {

phb_status adjoint_impl(int mode, const phb_plan* plan, const phb_params* prm, const double* pos,
                        const double* lambda, const double* U, const double* gbar, void* ws,
                        size_t ws_bytes, double* rec, size_t rec_bytes, double* Ubar, double* xbar,
                        int32_t* status_word, cudaStream_t st) {
  phb_status s = check_common(plan, ws, ws_bytes, plan ? plan->ws_off[R_END_ADJ] : 0);
  if (s != PHB_OK) return s;
  if (!prm || !pos || !lambda || !U) return PHB_ERR_INVALID_ARG;
  if (mode != kRecord && (!gbar || !Ubar || !xbar)) return PHB_ERR_INVALID_ARG;
  if (mode != kRecompute && (!rec || rec_bytes < size_t(kRecWords) * 8 * size_t(plan->n)))
    return PHB_ERR_INVALID_ARG;
  if (prm->weight_kind != 0 && prm->weight_kind != 1) return PHB_ERR_INVALID_ARG;
  if (!(prm->gamma > 1.0)) return PHB_ERR_INVALID_ARG;
  const Grid g = make_grid(plan);
  const int n = g.n;
  cudaError_t e = gather_sorted(plan, g, pos, lambda, U, ws, status_word, st);
  if (e) return launch_status(e);
  AdjArgs a;
  a.g = g;
  a.n = n;
  a.perm = region<int32_t>(plan, ws, R_PERM);
  a.tmap = region<uint8_t>(plan, ws, R_TMAP);
  a.spos = region<double>(plan, ws, R_SPOS);
  a.slam = region<double>(plan, ws, R_SLAM);
  a.sU = region<double>(plan, ws, R_SU);
  a.off = region<int64_t>(plan, ws, R_OFF);
  a.idx = region<int32_t>(plan, ws, R_IDX);
  a.gbar = gbar;
  a.gamma = prm->gamma;
  a.weight_kind = prm->weight_kind;
  a.zeta = prm->zeta;
  a.eta = prm->eta;
  a.c_zeta_l = prm->c_zeta_l;
  a.c_zeta_a = prm->c_zeta_a;
  a.c_eta = prm->c_eta;
  a.terms = region<double>(plan, ws, R_ADJ_TERMS);
  a.acc = region<double>(plan, ws, R_ADJ_ACC);
  a.rec = rec;
  a.status_word = status_word;
  a.span = adjoint_rows(plan) - n;
  a.chunk = 0;
  // (no more entries than the capacity, and than every particle naming every other)
  const int64_t most = std::min<int64_t>(plan->nbr_capacity, int64_t(n) * (n - 1));
  a.chunks = static_cast<int32_t>(std::max<int64_t>((most + a.span - 1) / a.span, 1));
  const size_t smem = size_t(kSlots) * kT * sizeof(double);
  const unsigned grid = static_cast<unsigned>(num_sms());
  const auto kernel = mode == kRecompute ? k_adjoint<kRecompute>
                      : mode == kRecord  ? k_adjoint<kRecord>
                                         : k_adjoint<kStored>;
  cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (mode == kRecord) {
    kernel<<<grid, kT, smem, st>>>(a);
    note_launch();
    return launch_status(cudaSuccess);
  }
  int32_t* rcnt = region<int32_t>(plan, ws, R_ADJ_RCNT);
  int64_t* roff = region<int64_t>(plan, ws, R_ADJ_ROFF);
  uint32_t* rsrc = region<uint32_t>(plan, ws, R_ADJ_RSRC);
  int64_t* bsum = region<int64_t>(plan, ws, R_SCAN);
  const size_t cnt_bytes = (size_t(n) + 1) * sizeof(int32_t);
  if ((e = cudaMemsetAsync(a.acc, 0, size_t(11) * n * sizeof(double), st))) return launch_status(e);
  for (a.chunk = 0; a.chunk < a.chunks; ++a.chunk) {
    if ((e = cudaMemsetAsync(rcnt, 0, cnt_bytes, st))) return launch_status(e);
    k_rev<false><<<grid * 8, kThreads, 0, st>>>(a, rcnt, nullptr, nullptr);
    note_launch();
    if ((e = scan_exclusive_i32_to_i64(rcnt, roff, n + 1, bsum, st))) return launch_status(e);
    if ((e = cudaMemsetAsync(rcnt, 0, cnt_bytes, st))) return launch_status(e);
    k_rev<true><<<grid * 8, kThreads, 0, st>>>(a, rcnt, roff, rsrc);
    note_launch();
    kernel<<<grid, kT, smem, st>>>(a);
    note_launch();
    k_adj_gather<<<static_cast<unsigned>((n + 3) / 4), 128, 0, st>>>(a, roff, rsrc, Ubar, xbar);
    note_launch();
  }
  return launch_status(cudaSuccess);
}

}  // namespace

extern "C" phb_status phb_rhs_adjoint(const phb_plan* plan, const phb_params* prm, const double* pos,
                                      const double* lambda, const double* U, const double* gbar,
                                      void* ws, size_t ws_bytes, double* Ubar, double* xbar,
                                      int32_t* status_word, phb_stream_t stream) {
  return adjoint_impl(kRecompute, plan, prm, pos, lambda, U, gbar, ws, ws_bytes, nullptr, 0, Ubar,
                      xbar, status_word, reinterpret_cast<cudaStream_t>(stream));
}

extern "C" size_t phb_adjoint_record_bytes(const phb_plan* plan) {
  return plan && plan->n > 0 ? size_t(kRecWords) * 8 * size_t(plan->n) : 0;
}

extern "C" phb_status phb_adjoint_record(const phb_plan* plan, const phb_params* prm,
                                         const double* pos, const double* lambda, const double* U,
                                         void* ws, size_t ws_bytes, double* record,
                                         size_t record_bytes, int32_t* status_word,
                                         phb_stream_t stream) {
  return adjoint_impl(kRecord, plan, prm, pos, lambda, U, nullptr, ws, ws_bytes, record,
                      record_bytes, nullptr, nullptr, status_word,
                      reinterpret_cast<cudaStream_t>(stream));
}

extern "C" phb_status phb_rhs_adjoint_stored(const phb_plan* plan, const phb_params* prm,
                                             const double* pos, const double* lambda,
                                             const double* U, const double* gbar, void* ws,
                                             size_t ws_bytes, const double* record,
                                             size_t record_bytes, double* Ubar, double* xbar,
                                             int32_t* status_word, phb_stream_t stream) {
  return adjoint_impl(kStored, plan, prm, pos, lambda, U, gbar, ws, ws_bytes,
                      const_cast<double*>(record), record_bytes, Ubar, xbar, status_word,
                      reinterpret_cast<cudaStream_t>(stream));
}
