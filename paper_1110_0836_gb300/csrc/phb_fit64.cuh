// FP64 fit of one particle by one thread: what the FP64 fit (phb_fit_fp64.cu)
// and the adjoint (phb_adjoint.cu) share.  The four warps of a block each have
// their own shared memory, [slot][32 lanes] doubles; `my` is a lane's column.
// Every sum and product is an explicit operation, so that files compiled with
// and without implicit contraction round alike.
#pragma once

#include "phb_internal.cuh"
#include "mls_gen.cuh"

namespace phb {

// While accumulating, above the right-hand sides [field][19]: x, y, z,
// 1/lambda, 1/r_f^2, U of the particle, and x, y, z, U of two neighbours, the
// next one on its way.
constexpr int kSlotOwn = kNF * kNB;
constexpr int kSlotNbr = kSlotOwn + 13;
static_assert(kSlotNbr + 2 * 11 <= kNT, "accumulators and values must fit below the factor's end");

__device__ __forceinline__ int tri0(int r) { return r * (r + 1) / 2; }

struct Box64 {
  double len[3], inv_len[3];
  int far[3];  // high word of a quarter box length: below it an offset is its minimum image
};

__device__ __forceinline__ Box64 make_box64(const Grid& g) {
  Box64 b;
  for (int c = 0; c < 3; ++c) {
    b.len[c] = g.len[c];
    b.inv_len[c] = g.periodic[c] ? 1.0 / g.len[c] : 0.0;
    b.far[c] = g.periodic[c] ? __double2hiint(0.25 * g.len[c]) : 0x7fffffff;
  }
  return b;
}

// d - len rint(d / len) (the wrap only where it changes something)
__device__ __forceinline__ double wrap64(const Box64& b, int c, double d) {
  if ((__double2hiint(d) & 0x7fffffff) >= b.far[c]) d = fma(-b.len[c], rint(d * b.inv_len[c]), d);
  return d;
}

// Squared distance over r_f^2; `inside` (s2 < 1) from the exponent bits: s2 >= 0
// or a NaN of either sign, whose high word lies above that of 1.
__device__ __forceinline__ double dist_rel(double dx, double dy, double dz, double inv_rf2, bool& inside) {
  const double s2 = fma(dz, dz, fma(dy, dy, __dmul_rn(dx, dx))) * inv_rf2;
  inside = static_cast<unsigned>(__double2hiint(s2)) < 0x3ff00000u;
  return s2;
}

__device__ __forceinline__ double weight64(double s2, int weight_kind) {
  const double sw = __dadd_rn(1.0, -s2);
  return weight_kind == 1 ? 1.0 : __dmul_rn(sw, sw);
}

template <int N>
struct Num {
  static constexpr int value = N;
};

// Cholesky of columns C0 .. C0 + W - 1 of the factor in a thread's column (my,
// stride 32), the columns before them done: the panel in registers, so that
// its independent FMAs cover the shared-memory loads (loops of dot products
// through shared memory took 290 cycles per FMA, this form ~90).  The diagonal
// slots take 1 / L_kk, mkk the diagonal of M.  A Jacobi-scaled pivot
// below 1e-12 (cond(M) above ~1e12) is treated as singular.
template <int C0, int W>
__device__ __forceinline__ void chol_panel(double* my, double (&mkk)[kNB], bool& singular) {
  constexpr int R = kNB - C0;
  double v[W][R];
  double d[W];
#pragma unroll
  for (int c = 0; c < W; ++c) {
#pragma unroll
    for (int r = c; r < R; ++r) v[c][r] = my[(tri0(C0 + r) + C0 + c) * 32];
    d[c] = v[c][c];
    mkk[C0 + c] = d[c];
  }
#pragma unroll 1
  for (int k = 0; k < C0; ++k) {
    double l[R];
#pragma unroll
    for (int r = 0; r < R; ++r) l[r] = my[(tri0(C0 + r) + k) * 32];
#pragma unroll
    for (int c = 0; c < W; ++c)
#pragma unroll
      for (int r = c; r < R; ++r) v[c][r] = fma(-l[r], l[c], v[c][r]);
  }
#pragma unroll
  for (int c = 0; c < W; ++c) {
    const double p = v[c][c];
    singular |= !(p > 0.0) || !(p > 1e-12 * d[c]);
    const double inv = rsqrt(p > 0.0 ? p : 1.0);
    my[(tri0(C0 + c) + C0 + c) * 32] = inv;
#pragma unroll
    for (int r = c + 1; r < R; ++r) {
      v[c][r] *= inv;
      my[(tri0(C0 + r) + C0 + c) * 32] = v[c][r];
    }
#pragma unroll
    for (int e = c + 1; e < W; ++e)
#pragma unroll
      for (int r = e; r < R; ++r) v[e][r] = fma(-v[c][r], v[c][e], v[e][r]);
  }
}

// Substitutions of NF right-hand sides at once in registers, with the factor
// in a thread's column.  First: the rows before it are zero on entry (and
// stay so in the forward substitution); the coefficients Last .. 18 are formed.
template <int NF, int First, int Last>
__device__ __forceinline__ void solve_thread(const double* factor, double (&b)[NF][kNB]) {
  const volatile double* my = factor;  // read again by each group of fields rather than kept
#pragma unroll
  for (int i = First; i < kNB; ++i) {
#pragma unroll
    for (int k = First; k < i; ++k) {
      const double l = my[(tri0(i) + k) * 32];
#pragma unroll
      for (int f = 0; f < NF; ++f) b[f][i] = fma(-l, b[f][k], b[f][i]);
    }
    const double inv = my[(tri0(i) + i) * 32];
#pragma unroll
    for (int f = 0; f < NF; ++f) b[f][i] *= inv;
  }
#pragma unroll
  for (int i = kNB - 1; i >= Last; --i) {
#pragma unroll
    for (int k = kNB - 1; k > i; --k) {
      const double l = my[(tri0(k) + i) * 32];
#pragma unroll
      for (int f = 0; f < NF; ++f) b[f][i] = fma(-l, b[f][k], b[f][i]);
    }
    const double inv = my[(tri0(i) + i) * 32];
#pragma unroll
    for (int f = 0; f < NF; ++f) b[f][i] *= inv;
  }
}

// Gradient and packed Hessian from a field's linear and quadratic coefficients.
template <class C>
__device__ __forceinline__ void derivs_of(C c, double il, double il2, double (&g)[3], double (&h)[6]) {
  for (int k = 0; k < 3; ++k) g[k] = c(kLin0 + k) * il;
  h[0] = 2.0 * c(kQuad0) * il2;
  h[1] = c(kQuad0 + 1) * il2;
  h[2] = c(kQuad0 + 2) * il2;
  h[3] = 2.0 * c(kQuad0 + 3) * il2;
  h[4] = c(kQuad0 + 4) * il2;
  h[5] = 2.0 * c(kQuad0 + 5) * il2;
}

// Moments (m, registers) and right-hand sides of the fields F0 .. 7 (my[f * 19
// + k], shared memory) of slot s over its list of len entries; returns the
// neighbours within r_f.  All lanes of the warp call it, and meet again after
// every neighbour: left to themselves the lanes of lists of different lengths
// ran the loop apart, in up to twice the time.
template <int F0>
__device__ __forceinline__ int accum_thread(const double* spos, const double* sU, int64_t n,
                                            const int32_t* list, int len, int s, const Box64& bx,
                                            int weight_kind, double inv_l, double inv_rf2, double* my,
                                            double (&m)[kNM]) {
  // the particle's own values in shared memory, read when used: registers
  // hold the 80 moments
  volatile double* own = my + kSlotOwn * 32;
  for (int c = 0; c < 3; ++c) own[c * 32] = spos[c * n + s];
  own[3 * 32] = inv_l;
  own[4 * 32] = inv_rf2;
  for (int f = F0; f < kNF; ++f) own[(5 + f) * 32] = sU[f * n + s];
  for (int k = F0 * kNB; k < kNF * kNB; ++k) my[k * 32] = 0.0;
#pragma unroll
  for (int k = 0; k < kNM; ++k) m[k] = 0.0;
  int cnt = 0;
  const int longest = __reduce_max_sync(0xffffffffu, len);
  // the next neighbour's values are copied to shared memory during this one's
  // sums (no registers, and their latency, ~1,400 cycles a neighbour, hidden)
  constexpr int kNbr = 3 + kNF - F0;
  volatile double* nbr = my + kSlotNbr * 32;
  auto fetch = [&](int t, int e) {
    const unsigned to = static_cast<unsigned>(__cvta_generic_to_shared(my + (kSlotNbr + (e & 1) * kNbr) * 32));
#pragma unroll
    for (int c = 0; c < kNbr; ++c) {
      const double* from = c < 3 ? spos + c * n + t : sU + (F0 + c - 3) * n + t;
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(to + c * 256), "l"(from) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  fetch(len > 0 ? list[0] : s, 0);
  int next = len > 1 ? list[1] : s;
#pragma unroll 1
  for (int e = 0; e < longest; ++e) {
    fetch(next, e + 1);
    next = e + 2 < len ? list[e + 2] : s;
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    const volatile double* at = nbr + (e & 1) * kNbr * 32;
    const double dx = wrap64(bx, 0, at[0] - own[0]);
    const double dy = wrap64(bx, 1, at[32] - own[32]);
    const double dz = wrap64(bx, 2, at[64] - own[64]);
    bool inside;
    const double s2 = dist_rel(dx, dy, dz, own[4 * 32], inside);
    if (inside && e < len) {
      ++cnt;
      const double wt = weight64(s2, weight_kind);
      double qg[kNB], wq[kNB + 1];
      const double il = own[3 * 32];
      mls_monomials_cubic_w(dx * il, dy * il, dz * il, wt, qg, wq);
      // the sums in shared memory are loaded two ahead: with the moments in
      // registers the compiler otherwise loads each just before its FMA
      // (123 instead of 70 cycles per FMA)
      volatile double* b = my + F0 * kNB * 32;
      constexpr int N = (kNF - F0) * kNB;
      double ahead[2] = {b[0], b[32]};
#pragma unroll
      for (int f = F0; f < kNF; ++f) {
        const double wdu = wt * (at[(3 + f - F0) * 32] - own[(5 + f) * 32]);
#pragma unroll
        for (int k = 0; k < kNB; ++k) {
          const int i = (f - F0) * kNB + k;
          const double v = ahead[i & 1];
          if (i + 2 < N) ahead[i & 1] = b[(i + 2) * 32];
          b[i * 32] = fma(qg[k], wdu, v);
        }
      }
      mls_accum_moments(qg, wq, m);
    }
    __syncwarp();
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  return cnt;
}

}  // namespace phb
