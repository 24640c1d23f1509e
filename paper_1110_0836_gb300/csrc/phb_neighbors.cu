// Cell binning (counting sort, stable by caller index) and the fixed-radius
// neighbour search of Paper II Sec. 2 / Sec. 2.1: strict, not mutual, radius
// of the gathering particle, no iteration.
//
// The search screens candidates in FP32 and decides the band of ambiguous
// candidates with the exact FP64 test, so every set equals the definition
// ((dx*dx + dy*dy) + dz*dz) < r*r evaluated in FP64 without contraction.
#include "phb_internal.cuh"
#include "phb_tile.cuh"

namespace phb {
namespace {

constexpr int kThreads = 256;
constexpr int kOwnerCap = 8192;  // list entries of a tile mapped to their particle in shared memory

inline unsigned blocks_for(int64_t n, int t = kThreads) { return static_cast<unsigned>((n + t - 1) / t); }

// The grid's bricks in the bitmap of the Hilbert cube, and the bricks per word
// (whose exclusive scan is Bricks::before).
__global__ void k_brick_mark(Grid g, uint32_t* __restrict__ bits) {
  const int64_t k = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const int nz = g.nbrick[2], ny = g.nbrick[1];
  if (k >= static_cast<int64_t>(g.nbrick[0]) * ny * nz) return;
  const uint32_t h = hilbert3(static_cast<uint32_t>(k / (static_cast<int64_t>(ny) * nz)),
                              static_cast<uint32_t>(k / nz % ny), static_cast<uint32_t>(k % nz), g.hbits);
  atomicOr(&bits[h >> 5], 1u << (h & 31u));
}

__global__ void k_brick_count(int64_t words, const uint32_t* __restrict__ bits, int32_t* __restrict__ before) {
  const int64_t w = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (w <= words) before[w] = w < words ? __popc(bits[w]) : 0;
}

// Cell keys and counts.  A particle without a finite position gets the key
// after the last cell: it has no neighbours and is nobody's, so it must not
// stand among a cell's candidates (157,000 of them in cell 0 made the search
// of a blown-up 200,000-particle set 74 ms).
__global__ void k_keys(Grid g, Bricks br, int32_t nkeys, const double* __restrict__ pos, const double* __restrict__ lam,
                       int32_t* __restrict__ keys, int32_t* __restrict__ counts,
                       int32_t* status_word) {
  const int n = g.n;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int c[3];
  bool finite = true;
  for (int a = 0; a < 3; ++a) {
    const double x = pos[a * n + i];
    const bool f = finite64(x);
    finite &= f;
    c[a] = f ? cell_coord(g, a, x) : 0;
  }
  const double l = lam[i];
  if (!finite || !finite64(l)) raise_flag(status_word, PHB_FLAG_NONFINITE);
  if (!lambda_in_range(g, l)) raise_flag(status_word, PHB_FLAG_LAMBDA_RANGE);
  const int32_t k = finite ? cell_key(g, br, c[0], c[1], c[2]) : nkeys;
  keys[i] = k;
  atomicAdd(&counts[k], 1);
}

__global__ void k_scatter(int n, const int32_t* __restrict__ keys, const int32_t* __restrict__ cell_start,
                          int32_t* __restrict__ cursor, int32_t* __restrict__ perm) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int32_t k = keys[i];
  perm[cell_start[k] + atomicAdd(&cursor[k], 1)] = i;
}

// Make the order inside each cell deterministic: ascending caller index.
// Thread per particle: its rank among the particles of its cell is the number
// of them with a smaller caller index (the cells' members come from the
// atomic scatter in arbitrary order).  That is quadratic in a cell's members
// (~12), so a crowded one - a clump, or the key of the particles without a
// finite position - is listed in one sweep over all n keys by the block that
// holds its first scattered member.  The sweep takes n x 2 ns (200,000
// particles 0.23 ms, 1M 1.05, 8M 16.2), the ranks 35 ns per member and up to 10 ps
// per pair of them (builds in ms, ranks / sweep: 8M with 8,000 members 7.8 / 23.4,
// 32,000: 15.0 / 23.4, 64,000: 30.1 / 23.4, 256,000: 200 / 23.2; 1M with 8,000: 1.38
// / 1.99, 16,000: 2.20 / 1.99; 200,000 with 4,000: 0.39 / 0.53, 8,000: 0.55 / 0.52).
__device__ __forceinline__ bool crowded(int members, int n) {
  return static_cast<int64_t>(members) * members > 256 * static_cast<int64_t>(n);
}

__global__ void __launch_bounds__(kThreads) k_rank_cells(int n, int32_t nkeys, const int32_t* __restrict__ keys,
                                                         const int32_t* __restrict__ cell_start,
                                                         const int32_t* __restrict__ scattered,
                                                         int32_t* __restrict__ perm) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  bool lead = false;
  int32_t k = -1;
  if (i < n) {
    k = keys[i];
    const int a = cell_start[k], b = k < nkeys ? cell_start[k + 1] : n;
    if (!crowded(b - a, n)) {
      int rank = 0;
      for (int t = a; t < b; ++t) rank += scattered[t] < i ? 1 : 0;
      perm[a + rank] = i;
    } else {
      lead = scattered[a] == i;
    }
  }
  if (!__syncthreads_or(lead)) return;
  __shared__ int cell;
  __shared__ int sums[kThreads / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  while (__syncthreads_or(lead)) {
    if (threadIdx.x == 0) cell = -1;
    __syncthreads();
    if (lead) atomicMax(&cell, k);
    __syncthreads();
    const int c = cell;
    if (k == c) lead = false;
    int at = cell_start[c];
    for (int j0 = 0; j0 < n; j0 += kThreads) {
      const int j = j0 + threadIdx.x;
      const bool in = j < n && keys[j] == c;
      const unsigned m = __ballot_sync(0xffffffffu, in);
      if (lane == 0) sums[wid] = __popc(m);
      __syncthreads();
      int before = 0, total = 0;
      for (int w = 0; w < kThreads / 32; ++w) {
        before += w < wid ? sums[w] : 0;
        total += sums[w];
      }
      if (in) perm[at + before + __popc(m & ((1u << lane) - 1u))] = j;
      at += total;
      __syncthreads();
    }
  }
}

// Slot-order copies of positions and lambda, the inverse permutation and the
// wrapped FP32 screen positions (wrapped by the same count as the cell).
__global__ void k_gather_pos(Grid g, const int32_t* __restrict__ perm, const double* __restrict__ pos,
                             const double* __restrict__ lam, int32_t* __restrict__ inv,
                             double* __restrict__ spos, double* __restrict__ slam,
                             float4* __restrict__ scr, int32_t* __restrict__ cellc) {
  const int n = g.n;
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n) return;
  const int i = perm[s];
  inv[i] = s;
  float w[3];
  int c[3];
  for (int a = 0; a < 3; ++a) {
    const double x = pos[a * n + i];
    spos[a * n + s] = x;
    double k = 0.0;
    bool kz = true;
    c[a] = finite64(x) ? cell_wrap(g, a, x, k, kz) : 0;
    w[a] = wrapped32(g, a, x, k, kz);
  }
  slam[s] = lam[i];
  scr[s] = make_float4(w[0], w[1], w[2], 0.f);
  cellc[s] = pack_cell(c[0], c[1], c[2]);
}

// (first slot, count) of every cell by linear index, for the tile planner and
// the search; the counts also go to lcnt[k] (lcnt[total] = 0), whose
// exclusive scan places the cells in linear order for the run search.
__global__ void k_cell_lin(Grid g, Bricks br, const int32_t* __restrict__ cell_start, int2* __restrict__ clin,
                           int32_t* __restrict__ lcnt, int32_t* __restrict__ misc) {
  const int64_t total = static_cast<int64_t>(g.ncell[0]) * g.ncell[1] * g.ncell[2];
  const int64_t k = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (k == total) {
    lcnt[k] = 0;
    misc[1] = 0;  // the compaction's count of unstaged tiles
  }
  if (k >= total) return;
  const int cz = static_cast<int>(k % g.ncell[2]);
  const int cy = static_cast<int>((k / g.ncell[2]) % g.ncell[1]);
  const int cx = static_cast<int>(k / (static_cast<int64_t>(g.ncell[2]) * g.ncell[1]));
  const int32_t key = cell_key(g, br, cx, cy, cz);
  const int a = cell_start[key];
  clin[k] = make_int2(a, cell_start[key + 1] - a);
  lcnt[k] = cell_start[key + 1] - a;
}

// Screen records in linear cell order (z fastest; slot order inside a cell),
// with the slot in w, plus four padding records: the cells of one (x, y) row
// of a reach box are then one contiguous run.  lstart: exclusive scan of the
// linear-order counts.  (Slots without a finite position have no record.)
__global__ void k_fill_lin(Grid g, const int32_t* __restrict__ cellc, const int2* __restrict__ clin,
                           const int32_t* __restrict__ lstart, const float4* __restrict__ scr,
                           float4* __restrict__ lscr) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.n) return;
  int cx, cy, cz;
  unpack_cell(cellc[s], cx, cy, cz);
  const int64_t k = (static_cast<int64_t>(cx) * g.ncell[1] + cy) * g.ncell[2] + cz;
  const float4 o = scr[s];
  const int2 members = clin[k];
  if (static_cast<unsigned>(s - members.x) < static_cast<unsigned>(members.y))
    lscr[lstart[k] + (s - members.x)] = make_float4(o.x, o.y, o.z, __int_as_float(s));
  if (s < 4) lscr[g.n + s] = make_float4(0.f, 0.f, 0.f, __int_as_float(-1));  // batch padding
}

struct Reach {
  int start, count;
  bool wrap, open;
};

__device__ __forceinline__ Reach axis_reach_cells(const Grid& g, int a, int c, int R) {
  Reach q;
  q.open = !g.periodic[a];
  if (g.periodic[a] && 2 * R + 1 >= g.ncell[a]) {
    q.start = 0;
    q.count = g.ncell[a];
    q.wrap = false;
  } else {
    q.start = c - R;
    q.count = max(2 * R + 1, 0);  // R = -1: no cells
    q.wrap = g.periodic[a] != 0;
  }
  return q;
}

__device__ __forceinline__ Reach axis_reach(const Grid& g, int a, int c, double r) {
  return axis_reach_cells(g, a, c, reach_cells(g, a, r));
}

__device__ __forceinline__ int axis_cell(const Grid& g, int a, const Reach& q, int k, bool& ok) {
  int c = q.start + k;
  ok = true;
  if (q.wrap) {
    int nc = g.ncell[a];
    c = c < 0 ? c + nc : (c >= nc ? c - nc : c);
  } else if (q.open && (c < 0 || c >= g.ncell[a])) {
    ok = false;
  }
  return c;
}

// Screen of candidate t against particle s: FP32 offsets of the wrapped
// positions and squared distance against the inner / outer screen radii;
// the exact FP64 test decides the ambiguous band.  kWrap = false skips the
// minimum image, which is then the identity (see the caller).
struct Screen {
  float in2, out2;
  double r2;
  float lenf[3], invlf[3];
};

__device__ __forceinline__ Screen make_screen(const Grid& g, double r) {
  Screen q;
  q.r2 = __dmul_rn(r, r);
  const double m = static_cast<double>(g.screen_margin) + 4e-7 * r;
  q.in2 = static_cast<float>(r > m ? (r - m) * (r - m) : 0.0);
  q.out2 = static_cast<float>((r + m) * (r + m));
  for (int a = 0; a < 3; ++a) {
    q.lenf[a] = g.lenf[a];
    q.invlf[a] = g.inv_lenf[a];  // formed on the host: no FP64 division per particle
  }
  return q;
}

// FP32 screen distance squared: below q.in2 a neighbour, above q.out2 not, in between the exact test decides.
template <bool kWrap>
__device__ __forceinline__ float screen_d2(const Screen& q, float4 me, float4 o) {
  float dx = o.x - me.x, dy = o.y - me.y, dz = o.z - me.z;
  if (kWrap) {
    dx = fmaf(-q.lenf[0], rintf(dx * q.invlf[0]), dx);
    dy = fmaf(-q.lenf[1], rintf(dy * q.invlf[1]), dy);
    dz = fmaf(-q.lenf[2], rintf(dz * q.invlf[2]), dz);
  }
  return fmaf(dx, dx, fmaf(dy, dy, dz * dz));
}

// Whether every cell of the reach on axis a lies inside the grid without
// wrapping and spans less than half the box, so that the plain difference of
// two wrapped positions is already the minimum image: |dx| < (R + 1) cells
// <= len / 2 gives rint(dx / len) = 0.
__device__ __forceinline__ bool plain_axis(const Grid& g, int a, int c, const Reach& q) {
  if (!g.periodic[a]) return true;
  const int R = q.count / 2;
  return q.wrap && c - R >= 0 && c + R < g.ncell[a] && 2 * R + 3 <= g.ncell[a];
}

// The z cells of a reach as up to two runs of cells [a0, b0], [a1, b1] in the
// order of the reach offsets; returns how many.
__device__ __forceinline__ int z_runs(const Reach& qz, int ncz, int& a0, int& b0, int& a1, int& b1) {
  const int za = qz.start, zb = qz.start + qz.count - 1;
  a0 = za;
  b0 = zb;
  a1 = 0;
  b1 = -1;
  if (!qz.wrap) {
    a0 = max(za, 0);
    b0 = min(zb, ncz - 1);
  } else if (za < 0) {  // wraps below: cells ncz + za .., then 0 .. zb
    a0 = za + ncz;
    b0 = zb < 0 ? zb + ncz : ncz - 1;
    b1 = zb < 0 ? -1 : zb;
  } else if (zb >= ncz) {  // wraps above: cells za .. ncz - 1, then 0 .. zb - ncz
    a0 = za < ncz ? za : za - ncz;
    b0 = za < ncz ? ncz - 1 : zb - ncz;
    b1 = za < ncz ? zb - ncz : -1;
  }
  const int nseg = (a0 <= b0 ? 1 : 0) + (a1 <= b1 ? 1 : 0);
  if (a0 > b0) {
    a0 = a1;
    b0 = b1;
  }
  return nseg;
}

// A wrapped screen position that can have neighbours (finite, in FP32 too).
__device__ __forceinline__ bool on_screen(float4 p) {
  return fabsf(p.x) + fabsf(p.y) + fabsf(p.z) < __int_as_float(0x7f800000);
}

// Candidate records in linear cell order (k_fill_lin) and the cells' starts.
struct Lin {
  const float4* __restrict__ rec;
  const int32_t* __restrict__ start;
};

// One particle's list by one thread: cells in x, y, z order of the reach box,
// slot order inside a cell.  The z cells of one (x, y) row are read as one run
// of the linear-order records (two where the row wraps a periodic z boundary),
// four candidates per batch so that their loads overlap.  The reach box is not
// culled per particle: the particles of one cell then walk identical rows and
// runs, so a warp's lanes stay together (measured faster than culling, which
// skips ~20% of the candidates but leaves half the lanes idle).  Writes the
// first g.ell entries to out; returns the exact count.
template <bool kWrap>
__device__ int search_runs(const Grid& g, const Lin& lin, const double* __restrict__ spos,
                           const Screen& q, const Reach& qx, const Reach& qy, const Reach& qz,
                           float4 me, int s, int32_t* __restrict__ out) {
  const int ncz = g.ncell[2];
  int count = 0;
  auto take = [&](int t) {
    if (count < g.ell) out[count] = t;
    ++count;
  };
  for (int kx = 0; kx < qx.count; ++kx) {
    bool okx;
    const int cx = axis_cell(g, 0, qx, kx, okx);
    if (!okx) continue;
    for (int ky = 0; ky < qy.count; ++ky) {
      bool oky;
      const int cy = axis_cell(g, 1, qy, ky, oky);
      if (!oky) continue;
      int a0, b0, a1, b1;
      const int nseg = z_runs(qz, ncz, a0, b0, a1, b1);
      const int64_t row = (static_cast<int64_t>(cx) * g.ncell[1] + cy) * ncz;
      for (int k = 0; k < nseg; ++k) {
        const int t0 = lin.start[row + (k == 0 ? a0 : a1)];
        const int t1 = lin.start[row + (k == 0 ? b0 : b1) + 1];
        // batches of four (the records array is padded by four, so a batch
        // may read past the run): the screen sets a hit bit (inside the
        // inner radius) or an ambiguous bit (inside the band), the exact FP64
        // test settles the rare ambiguous ones, hits are then taken in order
        for (int t = t0; t < t1; t += 4) {
          const float4* rp = lin.rec + t;
          const float4 o0 = rp[0], o1 = rp[1], o2 = rp[2], o3 = rp[3];
          const unsigned live = t1 - t >= 4 ? 0xfu : (1u << (t1 - t)) - 1u;
          const float d0 = screen_d2<kWrap>(q, me, o0), d1 = screen_d2<kWrap>(q, me, o1);
          const float d2 = screen_d2<kWrap>(q, me, o2), d3 = screen_d2<kWrap>(q, me, o3);
          const unsigned self = (__float_as_int(o0.w) == s ? 1u : 0u) | (__float_as_int(o1.w) == s ? 2u : 0u) |
                                (__float_as_int(o2.w) == s ? 4u : 0u) | (__float_as_int(o3.w) == s ? 8u : 0u);
          const unsigned in = (d0 < q.in2 ? 1u : 0u) | (d1 < q.in2 ? 2u : 0u) | (d2 < q.in2 ? 4u : 0u) |
                              (d3 < q.in2 ? 8u : 0u);
          const unsigned out = (d0 <= q.out2 ? 1u : 0u) | (d1 <= q.out2 ? 2u : 0u) |
                               (d2 <= q.out2 ? 4u : 0u) | (d3 <= q.out2 ? 8u : 0u);
          const unsigned keep = live & ~self;
          unsigned hit = in & keep;
          const unsigned amb = out & ~in & keep;
          if (amb) {
            if ((amb & 1u) && dist2_exact(g, spos, g.n, s, __float_as_int(o0.w)) < q.r2) hit |= 1u;
            if ((amb & 2u) && dist2_exact(g, spos, g.n, s, __float_as_int(o1.w)) < q.r2) hit |= 2u;
            if ((amb & 4u) && dist2_exact(g, spos, g.n, s, __float_as_int(o2.w)) < q.r2) hit |= 4u;
            if ((amb & 8u) && dist2_exact(g, spos, g.n, s, __float_as_int(o3.w)) < q.r2) hit |= 8u;
          }
          if (hit) {
            if (hit & 1u) take(__float_as_int(o0.w));
            if (hit & 2u) take(__float_as_int(o1.w));
            if (hit & 4u) take(__float_as_int(o2.w));
            if (hit & 8u) take(__float_as_int(o3.w));
          }
        }
      }
    }
  }
  return count;
}

__device__ __forceinline__ int warp_excl_scan(int v, int lane) {
  int x = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, d);
    if (lane >= d) x += y;
  }
  return x - v;
}

// One particle's list by one warp: the same candidates in the same order, the
// runs of 32 rows at a time laid out as one sequence, 32 candidates per chunk,
// a ballot appending the hits.  Entries to out[0 .. room); returns the exact
// count.  table: 2 x 64 + 1 ints of the warp's shared memory.  rx, ry, rz: reach in cells.
constexpr int kWarpTable = 2 * 64 + 1;
template <bool kWrap>
__device__ __forceinline__ int search_rows(const Grid& g, const Lin& lin, const double* __restrict__ spos,
                                           float in2, float out2, double r2, const Reach& qx,
                                           const Reach& qy, const Reach& qz, float4 me, int s, int* table,
                                           int64_t room, int32_t* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  int* t0 = table;         // first linear-order record of each run
  int* pre = table + 64;   // candidates before each run (the last: the total)
  const int ncy = g.ncell[1], ncz = g.ncell[2];
  const int nrow = qx.count * qy.count;
  int count = 0;
  Screen q;
  for (int a = 0; a < 3; ++a) {
    q.lenf[a] = g.lenf[a];
    q.invlf[a] = g.inv_lenf[a];
  }
  for (int j0 = 0; j0 < nrow; j0 += 32) {
    const int j = j0 + lane;
    int nr = 0, ta = 0, la = 0, tb = 0, lb = 0;
    if (j < nrow) {
      const int kx = j / qy.count, ky = j - kx * qy.count;
      bool okx, oky;
      const int rx = axis_cell(g, 0, qx, kx, okx), ry = axis_cell(g, 1, qy, ky, oky);
      if (okx && oky) {
        int a0, b0, a1, b1;
        nr = z_runs(qz, ncz, a0, b0, a1, b1);
        const int64_t row = (static_cast<int64_t>(rx) * ncy + ry) * ncz;
        if (nr >= 1) {
          ta = lin.start[row + a0];
          la = lin.start[row + b0 + 1] - ta;
        }
        if (nr == 2) {
          tb = lin.start[row + a1];
          lb = lin.start[row + b1 + 1] - tb;
        }
      }
    }
    const int rpos = warp_excl_scan(nr, lane), cpos = warp_excl_scan(la + lb, lane);
    if (nr >= 1) {
      t0[rpos] = ta;
      pre[rpos] = cpos;
    }
    if (nr == 2) {
      t0[rpos + 1] = tb;
      pre[rpos + 1] = cpos + la;
    }
    const int nrun = __shfl_sync(0xffffffffu, rpos + nr, 31);
    const int total = __shfl_sync(0xffffffffu, cpos + la + lb, 31);
    if (lane == 0) pre[nrun] = total;
    __syncwarp();
    int run = 0;  // the run holding the next chunk's first candidate
    auto fetch = [&](int v0) {
      const int v = v0 + lane;
      float4 o = make_float4(__int_as_float(0x7fc00000), 0.f, 0.f, __int_as_float(-1));
      int rn = run;
      if (v < total) {
        while (pre[rn + 1] <= v) ++rn;
        o = lin.rec[t0[rn] + (v - pre[rn])];
      }
      run = __shfl_sync(0xffffffffu, rn, 31);
      return o;
    };
    float4 next = fetch(0);
    for (int v0 = 0; v0 < total; v0 += 32) {
      const float4 o = next;
      if (v0 + 32 < total) next = fetch(v0 + 32);  // one chunk ahead
      const int t = __float_as_int(o.w);
      const float d = screen_d2<kWrap>(q, me, o);
      bool hit = t != s && d < in2;
      if (t != s && !hit && d <= out2) hit = dist2_exact(g, spos, g.n, s, t) < r2;
      const unsigned m = __ballot_sync(0xffffffffu, hit);
      if (hit) {
        const int e = count + __popc(m & ((1u << lane) - 1u));
        if (e < room) out[e] = t;
      }
      count += __popc(m);
    }
    __syncwarp();  // the next rows rewrite the table
  }
  return count;
}

__device__ __forceinline__ int search_warp(const Grid& g, const Lin& lin, const double* __restrict__ spos,
                                           float in2, float out2, double r2, int rx, int ry, int rz,
                                           int32_t cell, float4 me, int s, int* table, int64_t room,
                                           int32_t* __restrict__ out) {
  if (!on_screen(me)) return 0;
  int c[3];
  unpack_cell(cell, c[0], c[1], c[2]);
  const Reach qx = axis_reach_cells(g, 0, c[0], rx);
  const Reach qy = axis_reach_cells(g, 1, c[1], ry);
  const Reach qz = axis_reach_cells(g, 2, c[2], rz);
  if (plain_axis(g, 0, c[0], qx) && plain_axis(g, 1, c[1], qy) && plain_axis(g, 2, c[2], qz))
    return search_rows<false>(g, lin, spos, in2, out2, r2, qx, qy, qz, me, s, table, room, out);
  return search_rows<true>(g, lin, spos, in2, out2, r2, qx, qy, qz, me, s, table, room, out);
}

// The CSR fill of one list longer than the scratch rows, by one warp (rare):
// kept out of line so that it does not weigh on the compaction kernel's
// registers.
__device__ __noinline__ void search_overflow(const Grid& g, Lin lin, const int32_t* __restrict__ cellc,
                                             const float4* __restrict__ scr,
                                             const double* __restrict__ spos, double r, int s, int* table,
                                             int64_t room, int32_t* __restrict__ out) {
  const Screen q = make_screen(g, r);
  search_warp(g, lin, spos, q.in2, q.out2, q.r2, reach_cells(g, 0, r), reach_cells(g, 1, r),
              reach_cells(g, 2, r), cellc[s], scr[s], s, table, room, out);
}

constexpr int kRunCap = 128;  // candidate runs a warp records (a reach of 3 cells: at most 98)

// Per warp: the cell's particles being searched ("homes", 32 at a time, padded
// to a multiple of four with homes that hit nothing) and the runs of their
// common reach box.
struct __align__(16) SearchWarp {
  float nx[32], ny[32], nz[32];  // negated wrapped FP32 positions
  float in2[32], out2[32];       // inner / outer screen radius^2
  int slot[32];
  double r2[32];                 // list radius^2 (exact test)
  int32_t* row[32];              // the home's scratch row
  int run_t0[kRunCap];           // first linear-order record of each run
  int run_pre[kRunCap + 1];      // candidates before each run (the last: the total)
};
// the home arrays are read four at a time as 16-byte vectors
static_assert(offsetof(SearchWarp, nx) % 16 == 0 && offsetof(SearchWarp, ny) % 16 == 0 &&
                  offsetof(SearchWarp, nz) % 16 == 0 && offsetof(SearchWarp, in2) % 16 == 0 &&
                  offsetof(SearchWarp, out2) % 16 == 0 && offsetof(SearchWarp, slot) % 16 == 0,
              "vector-read arrays of SearchWarp must be 16-byte aligned");

// Squared FP32 screen distances of candidate o to two homes (a, b): packed
// FP32x2, each half rounded as screen_d2 rounds it.
template <bool kWrap>
__device__ __forceinline__ float2 screen_d2_pair(const Grid& g, float4 o, float2 nx, float2 ny, float2 nz) {
  float2 dx = __fadd2_rn(make_float2(o.x, o.x), nx);
  float2 dy = __fadd2_rn(make_float2(o.y, o.y), ny);
  float2 dz = __fadd2_rn(make_float2(o.z, o.z), nz);
  if (kWrap) {
    const float2 kx = __fmul2_rn(dx, make_float2(g.inv_lenf[0], g.inv_lenf[0]));
    const float2 ky = __fmul2_rn(dy, make_float2(g.inv_lenf[1], g.inv_lenf[1]));
    const float2 kz = __fmul2_rn(dz, make_float2(g.inv_lenf[2], g.inv_lenf[2]));
    dx = __ffma2_rn(make_float2(-g.lenf[0], -g.lenf[0]), make_float2(rintf(kx.x), rintf(kx.y)), dx);
    dy = __ffma2_rn(make_float2(-g.lenf[1], -g.lenf[1]), make_float2(rintf(ky.x), rintf(ky.y)), dy);
    dz = __ffma2_rn(make_float2(-g.lenf[2], -g.lenf[2]), make_float2(rintf(kz.x), rintf(kz.y)), dz);
  }
  return __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
}

// The candidates of one chunk (one per lane) against every home of the warp,
// four homes per round (their loads and screens independent): a ballot per
// home gives its hits, appended to its scratch row (S.row) in lane order.
template <bool kWrap>
__device__ __forceinline__ void screen_chunk(const Grid& g, const double* __restrict__ spos,
                                             const SearchWarp& S, int mh4, float4 o, int lane,
                                             int& cnt) {
  const int t = __float_as_int(o.w);
  const unsigned bit = 1u << lane, lt = bit - 1u;
#pragma unroll 1
  for (int i = 0; i < mh4; i += 4) {
    const float4 X = *reinterpret_cast<const float4*>(S.nx + i);
    const float4 Y = *reinterpret_cast<const float4*>(S.ny + i);
    const float4 Z = *reinterpret_cast<const float4*>(S.nz + i);
    const float4 I2 = *reinterpret_cast<const float4*>(S.in2 + i);
    const float4 O2 = *reinterpret_cast<const float4*>(S.out2 + i);
    const int4 SL = *reinterpret_cast<const int4*>(S.slot + i);
    const float2 d01 = screen_d2_pair<kWrap>(g, o, make_float2(X.x, X.y), make_float2(Y.x, Y.y),
                                             make_float2(Z.x, Z.y));
    const float2 d23 = screen_d2_pair<kWrap>(g, o, make_float2(X.z, X.w), make_float2(Y.z, Y.w),
                                             make_float2(Z.z, Z.w));
    const float d[4] = {d01.x, d01.y, d23.x, d23.y};
    const float in2[4] = {I2.x, I2.y, I2.z, I2.w};
    const float out2[4] = {O2.x, O2.y, O2.z, O2.w};
    const int sl[4] = {SL.x, SL.y, SL.z, SL.w};
    unsigned hit[4];
    unsigned band = 0u;  // bit u: inside home u's band (the exact test decides)
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const bool other = t != sl[u];
      hit[u] = __ballot_sync(0xffffffffu, other && d[u] < in2[u]);
      band |= (other && !(d[u] < in2[u]) && d[u] <= out2[u]) ? 1u << u : 0u;
    }
    if (__any_sync(0xffffffffu, band != 0u)) {
#pragma unroll
      for (int u = 0; u < 4; ++u)
        hit[u] |= __ballot_sync(0xffffffffu, ((band >> u) & 1u) &&
                                                 dist2_exact(g, spos, g.n, sl[u], t) < S.r2[i + u]);
    }
    if ((hit[0] | hit[1] | hit[2] | hit[3]) != 0u) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (hit[u] == 0u) continue;
        const int c = __shfl_sync(0xffffffffu, cnt, i + u);
        if (hit[u] & bit) {
          const int e = c + __popc(hit[u] & lt);
          if (e < g.ell) S.row[i + u][e] = t;
        }
        if (lane == i + u) cnt = c + __popc(hit[u]);
      }
    }
  }
}

// Single pass, cell-major, for sets of one lambda: one warp per cell of the
// linear order, its particles ("homes", 32 at a time) sharing one reach box.
// The homes share one candidate sequence, the runs of their reach box in
// the order of the particle-major search (rows in (x, y) offset order, the z
// cells of a row as one or two runs of the linear-order records, slot order
// inside a cell), taken 32 candidates per chunk, one per lane; each chunk is
// screened against every home and a ballot per home appends its hits in lane
// order, so every list equals the particle-major one.  Writes the exact list
// lengths and the first g.ell entries of the lists it takes; a cell whose
// homes differ in reach, or whose reach covers a whole periodic axis or has
// more runs than a warp records, keeps the -1 of ncnt for k_search_ell.
// (Where lambda varies the particle-major search alone is faster: sparse
// cells leave most of a warp's homes empty, and cells of mixed reach would
// send scattered particles to the second pass.)
// One warp per block, so that the block scheduler hands out single cells
// (32 resident per SM at 64 registers).
__global__ void __launch_bounds__(32, 32) k_search_cells(Grid g, Lin lin,
                                                     const double* __restrict__ spos,
                                                     const double* __restrict__ slam,
                                                     int32_t* __restrict__ ncnt,
                                                     int32_t* __restrict__ ell) {
  __shared__ SearchWarp S;
  const int lane = threadIdx.x;
  const int ncx = g.ncell[0], ncy = g.ncell[1], ncz = g.ncell[2];
  const int64_t k = blockIdx.x;
  if (k >= static_cast<int64_t>(ncx) * ncy * ncz) return;
  const int h0 = lin.start[k], h1 = lin.start[k + 1];
  const int cz = static_cast<int>(k % ncz);
  const int cy = static_cast<int>((k / ncz) % ncy);
  const int cx = static_cast<int>(k / (static_cast<int64_t>(ncz) * ncy));
  for (int g0 = h0; g0 < h1; g0 += 32) {
    const int mh = min(32, h1 - g0);
    const bool mine = lane < mh;
    float4 me = make_float4(0.f, 0.f, 0.f, __int_as_float(-1));
    if (mine) me = lin.rec[g0 + lane];
    const int s = __float_as_int(me.w);
    if (__all_sync(0xffffffffu, !mine || !on_screen(me))) {  // no positions: no neighbours
      if (mine) ncnt[s] = 0;
      continue;
    }
    double r = 0.0;
    int R[3] = {0, 0, 0};
    if (mine) {
      r = list_radius(g, slam[s]);
      for (int a = 0; a < 3; ++a) R[a] = reach_cells(g, a, r);
    }
    int U[3];
    bool same = true;
    for (int a = 0; a < 3; ++a) {
      U[a] = __shfl_sync(0xffffffffu, R[a], 0);
      same = same && (!mine || R[a] == U[a]);
    }
    if (!__all_sync(0xffffffffu, same) || U[0] < 0 || U[1] < 0 || U[2] < 0) continue;
    const Reach qx = axis_reach_cells(g, 0, cx, U[0]);
    const Reach qy = axis_reach_cells(g, 1, cy, U[1]);
    const Reach qz = axis_reach_cells(g, 2, cz, U[2]);
    const bool whole = (g.periodic[0] && !qx.wrap) || (g.periodic[1] && !qy.wrap) ||
                       (g.periodic[2] && !qz.wrap);
    const int64_t nrow = static_cast<int64_t>(qx.count) * qy.count;
    if (whole || nrow > kRunCap) continue;
    // the runs of the reach box, 32 rows at a time
    int nrun = 0, total = 0;
    for (int j0 = 0; j0 < nrow; j0 += 32) {
      const int j = j0 + lane;
      int nr = 0, ta = 0, la = 0, tb = 0, lb = 0;
      if (j < nrow) {
        const int kx = j / qy.count, ky = j - kx * qy.count;
        bool okx, oky;
        const int rx = axis_cell(g, 0, qx, kx, okx);
        const int ry = axis_cell(g, 1, qy, ky, oky);
        if (okx && oky) {
          int a0, b0, a1, b1;
          nr = z_runs(qz, ncz, a0, b0, a1, b1);
          const int64_t row = (static_cast<int64_t>(rx) * ncy + ry) * ncz;
          if (nr >= 1) {
            ta = lin.start[row + a0];
            la = lin.start[row + b0 + 1] - ta;
          }
          if (nr == 2) {
            tb = lin.start[row + a1];
            lb = lin.start[row + b1 + 1] - tb;
          }
        }
      }
      const int rpos = nrun + warp_excl_scan(nr, lane);
      const int cpos = total + warp_excl_scan(la + lb, lane);
      if (rpos + nr <= kRunCap) {
        if (nr >= 1) {
          S.run_t0[rpos] = ta;
          S.run_pre[rpos] = cpos;
        }
        if (nr == 2) {
          S.run_t0[rpos + 1] = tb;
          S.run_pre[rpos + 1] = cpos + la;
        }
      }
      nrun = __shfl_sync(0xffffffffu, rpos + nr, 31);
      total = __shfl_sync(0xffffffffu, cpos + la + lb, 31);
    }
    if (nrun > kRunCap) continue;
    const int mh4 = (mh + 3) & ~3;
    if (lane < mh4) {
      Screen q = make_screen(g, r);
      if (!mine) {  // padding: hits nothing
        q.in2 = -1.f;
        q.out2 = -1.f;
      }
      S.nx[lane] = -me.x;
      S.ny[lane] = -me.y;
      S.nz[lane] = -me.z;
      S.in2[lane] = q.in2;
      S.out2[lane] = q.out2;
      S.slot[lane] = mine ? s : -2;
      S.r2[lane] = q.r2;
      S.row[lane] = ell + static_cast<int64_t>(mine ? s : 0) * g.ell;
    }
    if (lane == 0) S.run_pre[nrun] = total;
    __syncwarp();
    // the plain difference is the minimum image for the whole reach box
    const bool plain = plain_axis(g, 0, cx, qx) && plain_axis(g, 1, cy, qy) && plain_axis(g, 2, cz, qz);
    int run = 0;  // the run holding the next chunk's first candidate
    // candidate v0 + lane (none past the end: a NaN record hits nothing)
    auto fetch = [&](int v0) {
      const int v = v0 + lane;
      float4 o = make_float4(__int_as_float(0x7fc00000), 0.f, 0.f, __int_as_float(-1));
      int rn = run;
      if (v < total) {
        while (S.run_pre[rn + 1] <= v) ++rn;
        o = lin.rec[S.run_t0[rn] + (v - S.run_pre[rn])];
      }
      run = __shfl_sync(0xffffffffu, rn, 31);
      return o;
    };
    int cnt = 0;  // lane i: the list length of home i so far
    float4 next = fetch(0);
    for (int v0 = 0; v0 < total; v0 += 32) {
      const float4 o = next;
      if (v0 + 32 < total) next = fetch(v0 + 32);  // one chunk ahead
      if (plain) {
        screen_chunk<false>(g, spos, S, mh4, o, lane, cnt);
      } else {
        screen_chunk<true>(g, spos, S, mh4, o, lane, cnt);
      }
    }
    if (mine) ncnt[s] = cnt;
    __syncwarp();  // the next group of homes rewrites the warp's records
  }
}

// Single pass, thread per particle (slot order): exact list lengths and the
// first g.ell entries of every list (after the cell-major search, left_only:
// of the lists it left, ncnt still -1).
__global__ void __launch_bounds__(kThreads, 4) k_search_ell(Grid g, Lin lin, const int32_t* __restrict__ cellc,
                                                         const float4* __restrict__ scr,
                                                         const double* __restrict__ spos,
                                                         const double* __restrict__ slam,
                                                         int32_t* __restrict__ ncnt,
                                                         int32_t* __restrict__ ell, bool left_only) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.n) return;
  if (s == g.n - 1) ncnt[g.n] = 0;  // the offsets scan's sentinel
  if (left_only && ncnt[s] >= 0) return;
  const float4 me = scr[s];
  if (!on_screen(me)) {
    ncnt[s] = 0;
    return;
  }
  const double r = list_radius(g, slam[s]);
  const Screen q = make_screen(g, r);
  int c[3];
  unpack_cell(cellc[s], c[0], c[1], c[2]);
  const Reach qx = axis_reach(g, 0, c[0], r);
  const Reach qy = axis_reach(g, 1, c[1], r);
  const Reach qz = axis_reach(g, 2, c[2], r);
  int32_t* out = ell + static_cast<int64_t>(s) * g.ell;
  const bool plain =
      plain_axis(g, 0, c[0], qx) && plain_axis(g, 1, c[1], qy) && plain_axis(g, 2, c[2], qz);
  ncnt[s] = plain ? search_runs<false>(g, lin, spos, q, qx, qy, qz, me, s, out)
                  : search_runs<true>(g, lin, spos, q, qx, qy, qz, me, s, out);
}

// The same by a warp per particle, for sets too small to fill the GPU with
// threads (40 blocks hold 10,007 particles).  Two particles per warp: their
// FP64 set-up (28 instructions, 20 SM cycles each per warp) runs once for
// both, a lane each (eight: 66 instead of 38 us for 10,007 particles, 123
// instead of 116 for 60,000: too few warps).
__global__ void __launch_bounds__(128) k_search_warp(Grid g, Lin lin, const int32_t* __restrict__ cellc,
                                                     const float4* __restrict__ scr,
                                                     const double* __restrict__ spos,
                                                     const double* __restrict__ slam,
                                                     int32_t* __restrict__ ncnt, int32_t* __restrict__ ell) {
  constexpr int kPairs = 2;
  __shared__ int table[4][kWarpTable];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t s0 = (static_cast<int64_t>(blockIdx.x) * 4 + wid) * kPairs;
  if (s0 >= g.n) return;
  const int last = g.n - 1;
  const int mine = static_cast<int>(s0 + lane % kPairs < g.n ? s0 + lane % kPairs : last);
  const double r = list_radius(g, slam[mine]);
  const Screen q = make_screen(g, r);
  const int rx = reach_cells(g, 0, r), ry = reach_cells(g, 1, r), rz = reach_cells(g, 2, r);
  const int32_t cell = cellc[mine];
  const float4 me = scr[mine];
  const bool todo = lane < kPairs && s0 + lane < g.n;
  int count = 0;
  for (unsigned left = __ballot_sync(0xffffffffu, todo); left != 0u; left &= left - 1u) {
    const int p = __ffs(left) - 1;
    auto of = [&](auto v) { return __shfl_sync(0xffffffffu, v, p); };
    const int s = of(mine);
    const int c = search_warp(g, lin, spos, of(q.in2), of(q.out2), of(q.r2), of(rx), of(ry), of(rz), of(cell),
                              make_float4(of(me.x), of(me.y), of(me.z), 0.f), s, table[wid], g.ell,
                              ell + static_cast<int64_t>(s) * g.ell);
    if (lane == p) count = c;
  }
  if (todo) ncnt[mine] = count;
  if (lane < kPairs && s0 + lane == last) ncnt[g.n] = 0;  // the offsets scan's sentinel
}

// One CTA per tile: move the tile's lists from the single-pass scratch into
// the CSR arrays (searching again, straight into CSR, for lists longer than
// the scratch rows), plan the tile's staged neighbourhood and record it for
// the fused fit - (staged count, unstaged flag), the slot of every staged
// index, each tile particle's own staged index - and map every list entry to
// its staged index.
template <int T>
__global__ void __launch_bounds__(T, 1152 / T) k_compact(const __grid_constant__ Grid g, const int2* __restrict__ clin, Lin lin,
                                               const int32_t* __restrict__ cellc,
                                               const float4* __restrict__ scr,
                                               const double* __restrict__ spos,
                                               const double* __restrict__ slam,
                                               const int32_t* __restrict__ ncnt,
                                               const int32_t* __restrict__ ell,
                                               const int64_t* __restrict__ off,
                                               int32_t* __restrict__ idx, uint16_t* __restrict__ lidx,
                                               int2* __restrict__ tplan, int32_t* __restrict__ tslot,
                                               uint16_t* __restrict__ lself, uint8_t* __restrict__ tmap,
                                               int32_t* fallback_count, int32_t* status_word) {
  __shared__ TileShared ts;
  __shared__ unsigned bits[kBoxWords];
  __shared__ int wpre[kBoxWords];
  __shared__ int base[kMarkCap + 1];
  __shared__ int cstart[kMarkCap];
  __shared__ int warp_tmp[T / 32 + 1];
  __shared__ int64_t toff[T + 1];
  __shared__ int tlen[T];
  __shared__ uint8_t owner[kOwnerCap];
  const TileArrays tarr{bits, wpre, base, cstart, warp_tmp};
  const int n = g.n;
  const int tid = threadIdx.x;
  const int s0 = blockIdx.x * T;
  const int cnt = min(T, n - s0);
  for (int k = tid; k <= cnt; k += T) toff[k] = off[s0 + k];
  __syncthreads();
  // fit thread -> tile particle in descending list length (ties: slot order),
  // so that the lanes of a fit warp run loops of similar length
  tlen[tid] = tid < cnt ? static_cast<int>(toff[tid + 1] - toff[tid]) : -1;
  __syncthreads();
  {
    const int len = tlen[tid];
    int rank = 0;
    for (int j = 0; j < T; ++j) {
      const int c = tlen[j];
      rank += (c > len || (c == len && j < tid)) ? 1 : 0;
    }
    tmap[static_cast<int64_t>(blockIdx.x) * T + rank] = static_cast<uint8_t>(tid);
  }
  if (tid < cnt && toff[tid + 1] > g.capacity) raise_flag(status_word, PHB_FLAG_CAPACITY);
  // lists longer than their scratch rows: searched again by the warp (the
  // shared arrays of the tile plan, not yet in use, hold its table)
  {
    const bool over = tid < cnt && ncnt[s0 + tid] > g.ell;
    unsigned left = __ballot_sync(0xffffffffu, over);
    for (; left != 0u; left &= left - 1u) {
      const int p = (tid & ~31) + __ffs(left) - 1, s = s0 + p;
      const int64_t to = toff[p] < g.capacity ? toff[p] : g.capacity;
      search_overflow(g, lin, cellc, scr, spos, list_radius(g, slam[s]), s,
                      base + (tid >> 5) * kWarpTable, g.capacity - to, idx + to);
    }
    __syncthreads();
  }
  tile_plan<T>(g, s0, cnt, cellc, slam, clin, ts, tarr);
  const bool staged = !ts.fallback;
  if (tid == 0) {
    tplan[blockIdx.x] = make_int2(staged ? ts.total : 0, staged ? 0 : 1);
    if (!staged) atomicAdd(fallback_count, 1);
  }
  if (staged) {
    int32_t* ts_out = tslot + static_cast<int64_t>(blockIdx.x) * g.stage_cap;
    for (int j = tid; j < ts.ncells; j += T) {
      const int l0 = base[j], m = base[j + 1] - l0, t0 = cstart[j];
      for (int q = 0; q < m; ++q) ts_out[l0 + q] = t0 + q;
    }
    if (tid < cnt) {
      // a slot that is in no cell (no finite position) or whose cell nothing
      // marked has no staged record: index 0, which is one (its list is empty)
      const int s = s0 + tid;
      const int k = box_index(g, ts, cellc[s]);
      int self = 0;
      if (bits[k >> 5] >> (k & 31) & 1u) {
        const int j = marked_index(tarr, k), o = s - cstart[j];
        if (static_cast<unsigned>(o) < static_cast<unsigned>(base[j + 1] - base[j])) self = base[j] + o;
      }
      lself[s] = static_cast<uint16_t>(self);
    }
  }
  // the tile's entries [e0, e1) as one flat range over the block (each
  // entry's tile particle from a byte map, or a binary search of the offsets
  // when the tile has more entries than the map holds)
  const int64_t e0 = toff[0];
  const int64_t e1 = toff[cnt] < g.capacity ? toff[cnt] : g.capacity;
  const int64_t m = e1 > e0 ? e1 - e0 : 0;
  const bool mapped = m <= kOwnerCap;
  // (offset of its scratch row less that of its first entry, per particle)
  constexpr int kInCsr = -0x7fffffff - 1;  // a list longer than its row, already in place
  if (tid < cnt)
    tlen[tid] = tlen[tid] > g.ell ? kInCsr : tid * g.ell - static_cast<int>(toff[tid] - e0);
  if (mapped && tid < cnt) {
    const int64_t a = toff[tid], b = toff[tid + 1] < e1 ? toff[tid + 1] : e1;
    for (int64_t e = a; e < b; ++e) owner[e - e0] = static_cast<uint8_t>(tid);
  }
  __syncthreads();
  // four entries per thread per round, their loads issued together (the
  // list slot, then its cell) so that several global loads are in flight.
  // from(i): the list slot of entry e0 + i.
  auto entries = [&](auto from, auto count) {
    constexpr int kB = 4;
    using Int = decltype(count);
    int32_t* idx_t = idx + e0;
    uint16_t* lidx_t = lidx + e0;
    for (Int i0 = tid; i0 < count; i0 += kB * T) {
      int t[kB], c[kB];
#pragma unroll
      for (int u = 0; u < kB; ++u) t[u] = i0 + u * T < count ? from(i0 + u * T) : 0;
#pragma unroll
      for (int u = 0; u < kB; ++u) c[u] = (i0 + u * T < count && staged) ? cellc[t[u]] : 0;
#pragma unroll
      for (int u = 0; u < kB; ++u) {
        if (i0 + u * T >= count) continue;
        idx_t[i0 + u * T] = t[u];
        if (staged) {
          const int j = marked_index(tarr, box_index(g, ts, c[u]));
          lidx_t[i0 + u * T] = static_cast<uint16_t>(base[j] + (t[u] - cstart[j]));
        }
      }
    }
  };
  const int32_t* ell_t = ell + static_cast<int64_t>(s0) * g.ell;
  if (mapped) {
    // 32-bit offsets, and one word per tile particle instead of its offset and
    // length: an entry's instructions bound the kernel.  With box_index's
    // wrap: 64^3 lattice 104.5 -> 78.9 us, 1M tube 363 -> 273, 8M layer 2,626
    // -> 2,005
    entries([&](int i) {
      const int r = tlen[owner[i]];
      return r == kInCsr ? idx[e0 + i] : ell_t[r + i];
    }, static_cast<int>(m));
  } else {
    entries([&](int64_t i) {
      const int64_t e = e0 + i;
      int lo = 0, hi = cnt - 1;  // the last p with toff[p] <= e
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (toff[mid] <= e) lo = mid; else hi = mid - 1;
      }
      return tlen[lo] == kInCsr ? idx[e] : ell_t[static_cast<int64_t>(lo) * g.ell + (e - toff[lo])];
    }, m);
  }
}

// Tile order for the fused fit's schedule 1: tiles grouped by cost class
// floor(log2(list entries + 1)), most expensive class first (longest
// processing time first keeps the tail of the launch short).  One CTA.
__global__ void __launch_bounds__(1024) k_tile_order(int n, int T, int ntiles, int64_t cap,
                                                     const int64_t* __restrict__ off,
                                                     int32_t* __restrict__ order) {
  __shared__ int hist[65], cursor[65];
  const int tid = threadIdx.x;
  if (tid < 65) hist[tid] = 0;
  __syncthreads();
  for (int t = tid; t < ntiles; t += blockDim.x) {
    const int s0 = t * T, s1 = min(s0 + T, n);
    const int64_t a = off[s0] < cap ? off[s0] : cap, b = off[s1] < cap ? off[s1] : cap;
    const int cls = 64 - __clzll(static_cast<unsigned long long>(b - a + 1));
    atomicAdd(&hist[cls], 1);
  }
  __syncthreads();
  if (tid == 0) {
    int acc = 0;
    for (int c = 64; c >= 0; --c) {
      cursor[c] = acc;
      acc += hist[c];
    }
  }
  __syncthreads();
  for (int t = tid; t < ntiles; t += blockDim.x) {
    const int s0 = t * T, s1 = min(s0 + T, n);
    const int64_t a = off[s0] < cap ? off[s0] : cap, b = off[s1] < cap ? off[s1] : cap;
    const int cls = 64 - __clzll(static_cast<unsigned long long>(b - a + 1));
    order[atomicAdd(&cursor[cls], 1)] = t;
  }
}

// -------- particle adaptivity scan (voids on a 9^3 grid of test points,
// clumps of too-close particles; see phb_adapt_scan)

// Slot-order copies of positions and lambda and wrapped FP32 screen
// positions for positions that may have moved since the build (the cells
// and tile plans of the build are left alone).
__global__ void k_adapt_gather(Grid g, const int32_t* __restrict__ perm, const double* __restrict__ pos,
                               const double* __restrict__ lam, double* __restrict__ spos,
                               double* __restrict__ slam, float4* __restrict__ scr) {
  const int n = g.n;
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n) return;
  const int i = perm[s];
  float w[3];
  for (int a = 0; a < 3; ++a) {
    const double x = pos[a * n + i];
    spos[a * n + s] = x;
    double k = 0.0;
    bool kz = true;
    if (finite64(x)) cell_wrap(g, a, x, k, kz);
    w[a] = wrapped32(g, a, x, k, kz);
  }
  slam[s] = lam[i];
  scr[s] = make_float4(w[0], w[1], w[2], 0.f);
}

// Grid points k (9 per axis, index ((kx+4) 9 + (ky+4)) 9 + (kz+4)) with
// |k|^2 <= Q2, in ascending index.
template <int Q2>
struct GridPoints {
  int n = 0;
  int8_t x[257] = {}, y[257] = {}, z[257] = {};
  constexpr GridPoints() {
    for (int i = -4; i <= 4; ++i)
      for (int j = -4; j <= 4; ++j)
        for (int k = -4; k <= 4; ++k)
          if (i * i + j * j + k * k <= Q2) {
            x[n] = static_cast<int8_t>(i);
            y[n] = static_cast<int8_t>(j);
            z[n] = static_cast<int8_t>(k);
            ++n;
          }
  }
};
constexpr int grid_points(int q2) { return q2 == 5 ? 57 : 257; }
static_assert(GridPoints<5>().n == grid_points(5) && GridPoints<16>().n == grid_points(16), "point counts");
__device__ constexpr GridPoints<5> kGrid5;
__device__ constexpr GridPoints<16> kGrid16;

// FP32 offset of record o from me, minimum image on periodic axes.
__device__ __forceinline__ float3 offset32(const Grid& g, float4 me, float4 o) {
  float dx = o.x - me.x, dy = o.y - me.y, dz = o.z - me.z;
  dx = fmaf(-g.lenf[0], rintf(dx * g.inv_lenf[0]), dx);
  dy = fmaf(-g.lenf[1], rintf(dy * g.inv_lenf[1]), dy);
  dz = fmaf(-g.lenf[2], rintf(dz * g.inv_lenf[2]), dz);
  return make_float3(dx, dy, dz);
}

// Exact FP64 squared distance from neighbour t of slot s to the test point
// at offset (ox, oy, oz): ((ex*ex + ey*ey) + ez*ez), e = min-image(x_t - x_s) - o.
__device__ __forceinline__ double test_dist2(const Grid& g, const double* spos, int n, int s, int t,
                                             double ox, double oy, double oz) {
  const double ex = __dsub_rn(min_image64(__dsub_rn(spos[t], spos[s]), g.len[0], g.periodic[0]), ox);
  const double ey =
      __dsub_rn(min_image64(__dsub_rn(spos[n + t], spos[n + s]), g.len[1], g.periodic[1]), oy);
  const double ez =
      __dsub_rn(min_image64(__dsub_rn(spos[2 * n + t], spos[2 * n + s]), g.len[2], g.periodic[2]), oz);
  return __dadd_rn(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)), __dmul_rn(ez, ez));
}

// Exact squared distance from neighbour t of slot s to the test point (kx, ky,
// kz), below d_v^2.
__device__ __forceinline__ bool covers_exact(const Grid& g, const double* spos, int s, int t, double lam,
                                          double vf, int kx, int ky, int kz) {
  const double h = __dmul_rn(__dmul_rn(g.rf_factor, lam), 0.25), v = __dmul_rn(vf, lam);
  return test_dist2(g, spos, g.n, s, t, __dmul_rn(static_cast<double>(kx), h),
                    __dmul_rn(static_cast<double>(ky), h), __dmul_rn(static_cast<double>(kz), h)) <
         __dmul_rn(v, v);
}

__device__ __forceinline__ bool closer_exact(const Grid& g, const double* spos, int s, int t, double lam,
                                          double cf) {
  const double c = __dmul_rn(cf, lam);
  return dist2_exact(g, spos, g.n, s, t) < __dmul_rn(c, c);
}

// Exact clearance squared of test point (kx, ky, kz) of slot s (all lanes of a
// warp): the smallest squared distance to the particle and its r_f set.  Only
// entries within near2 (FP32) can hold it.
__device__ __forceinline__ double clearance_exact(const Grid& g, const double* spos, const float4* scr,
                                               const int32_t* idx, int64_t beg, int64_t end, int s,
                                               double lam, int kx, int ky, int kz, float near2) {
  const float4 me = scr[s];
  const double rr = __dmul_rn(g.rf_factor, lam), h = __dmul_rn(rr, 0.25);
  const double ox = __dmul_rn(static_cast<double>(kx), h), oy = __dmul_rn(static_cast<double>(ky), h),
               oz = __dmul_rn(static_cast<double>(kz), h);
  const float fx = __double2float_rn(ox), fy = __double2float_rn(oy), fz = __double2float_rn(oz);
  double c = __dadd_rn(__dadd_rn(__dmul_rn(ox, ox), __dmul_rn(oy, oy)), __dmul_rn(oz, oz));
  for (int64_t e = beg + (threadIdx.x & 31); e < end; e += 32) {
    const int t = idx[e];
    const float3 d = offset32(g, me, scr[t]);
    const float ex = d.x - fx, ey = d.y - fy, ez = d.z - fz;
    if (fmaf(ex, ex, fmaf(ey, ey, ez * ez)) > near2) continue;
    if (!(dist2_exact(g, spos, g.n, s, t) < __dmul_rn(rr, rr))) continue;  // a skin entry, not in N(i)
    const double e2 = test_dist2(g, spos, g.n, s, t, ox, oy, oz);
    c = e2 < c ? e2 : c;
  }
  __syncwarp();
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double x = __shfl_xor_sync(0xffffffffu, c, o);
    c = x < c ? x : c;
  }
  return c;
}

// What the scan asks of every particle alike.
struct ScanRule {
  double vf, cf;
  uint32_t test;  // bit q: points with |k|^2 = q are tested (neither beyond r_f - d_v nor within d_v of the particle)
  uint32_t ask;   // bit q: the two are so close that each particle's own rounding decides
};

// A warp per slot.  What bounds it is instruction issue (850 warp instructions
// per particle): the coverage of the 57 default test points by ~52 neighbours,
// one neighbour per lane, with squares per axis and one add and one shift per
// point, and the latency of its gathers, hence 40 warps per SM (640 us with
// 20, 427 with 32, 400 with 40 for the 400,000 particles of a shock tube).  A
// thread per particle that walked its list anew for every point took 2.68 ms.
// FP64 instructions, 80 times an FP32 one here, are kept to what FP32 cannot
// decide: FP32 distances are within the margin m of the exact ones, so a point
// is covered or not, and of several uncovered points the one with the largest
// clearance, without FP64 unless two distances lie within 2 m.  The FP64
// decisions are single IEEE-rounded operations in the order of the definition.
template <int Q2>
__global__ void __launch_bounds__(128, 10) k_adapt_scan(const __grid_constant__ Grid g, ScanRule rule,
                                                   const int32_t* __restrict__ perm,
                                                   const double* __restrict__ spos,
                                                   const double* __restrict__ slam,
                                                   const float4* __restrict__ scr,
                                                   const int64_t* __restrict__ off,
                                                   const int32_t* __restrict__ idx, int32_t* void_count,
                                                   int32_t* best, double* cand, int32_t* clump) {
  constexpr GridPoints<Q2> P;
  constexpr int NP = grid_points(Q2), NW = (NP + 31) / 32, K = Q2 == 5 ? 2 : 4;
  const auto& D = []() -> const GridPoints<Q2>& {
    if constexpr (Q2 == 5) return kGrid5;
    else return kGrid16;
  }();
  const int n = g.n;
  const int64_t N = n;
  const int lane = threadIdx.x & 31;
  const int64_t w = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  if (w >= n) return;
  const int s = static_cast<int>(w);
  const double lam = slam[s];
  // for a lambda that is not a positive number every point's own comparisons
  // decide (a NaN, an infinity and a zero have none to test)
  const bool usual = finite64(lam) && __double2hiint(lam) >= 0x00100000;
  const uint32_t each = usual ? rule.ask : 0xffffffffu;
  // FP32 radii with a margin: coordinates (screen_margin) and a few ulps of
  // r for offsets, squares and the radii themselves
  const float lamf = f32_of(lam);
  const float r = static_cast<float>(g.rf_factor) * lamf, h = 0.25f * r;
  const float dv = static_cast<float>(rule.vf) * lamf, dc = static_cast<float>(rule.cf) * lamf;
  const float m = g.screen_margin + 3e-6f * r;
  auto below = [&](float d) { return d > m ? (d - m) * (d - m) : 0.f; };
  auto above = [&](float d) { return (d + m) * (d + m); };
  const float v_in2 = below(dv), v_out2 = above(dv), c_in2 = below(dc), c_out2 = above(dc);
  const float r_in2 = below(r), r_out2 = above(r);
  const float4 me = scr[s];
  const int me_caller = perm[s];
  const int64_t beg = off[s];
  const int64_t end = off[s + 1] < g.capacity ? off[s + 1] : g.capacity;

  // coverage of every point, and clumps: a neighbour with a smaller caller
  // index closer than d_c
  uint32_t cov[NW];
#pragma unroll
  for (int i = 0; i < NW; ++i) cov[i] = 0u;
  bool cl = false;
  auto cover = [&](int t, float4 o) {
    const float3 d = offset32(g, me, o);
    float ax[2 * K + 1], ay[2 * K + 1], az[2 * K + 1];
#pragma unroll
    for (int k = -K; k <= K; ++k) {
      const float ex = fmaf(static_cast<float>(-k), h, d.x), ey = fmaf(static_cast<float>(-k), h, d.y),
                  ez = fmaf(static_cast<float>(-k), h, d.z);
      ax[k + K] = ex * ex;
      ay[k + K] = ey * ey;
      az[k + K] = fmaf(ez, ez, -v_in2);
    }
    const float dd = fmaf(d.x, d.x, fmaf(d.y, d.y, d.z * d.z));
    if (dd <= c_out2 && perm[t] < me_caller)
      cl |= dd < c_in2 || closer_exact(g, spos, s, t, lam, rule.cf);
    // the sign of |d - o_k|^2 - v_in2 is shifted into the word: one add and
    // one shift per point
#pragma unroll
    for (int i = 0; i < NW; ++i) {
      uint32_t bits = 0u;
      constexpr int last = NP - 32 * (NW - 1);
#pragma unroll
      for (int b = 0; b < (i + 1 < NW ? 32 : last); ++b) {
        const int p = 32 * i + b;
        const float e = (ax[P.x[p] + K] + ay[P.y[p] + K]) + az[P.z[p] + K];
        bits = __funnelshift_l(__float_as_uint(e), bits, 1);
      }
      cov[i] |= bits;
    }
  };
  // two neighbours per lane on their way at once
  for (int64_t e = beg + lane; e < end; e += 64) {
    const bool two = e + 32 < end;
    const int t0 = idx[e], t1 = two ? idx[e + 32] : t0;
    const float4 o0 = scr[t0], o1 = scr[t1];
    cover(t0, o0);
    if (two) cover(t1, o1);
  }
  // point p of a word at bit p
#pragma unroll
  for (int i = 0; i < NW; ++i) cov[i] = __brev(cov[i] << (i + 1 < NW ? 0 : 32 * NW - NP));
  cl = __any_sync(0xffffffffu, cl);
  uint32_t open[NW];  // points to be tested that no neighbour covers for certain
#pragma unroll
  for (int i = 0; i < NW; ++i) {
    // lane p & 31 holds point p
    const int p = 32 * i + lane;
    bool ask = false;
    if (p < NP) {
      const int kx = D.x[p], ky = D.y[p], kz = D.z[p];
      const uint32_t q = 1u << (kx * kx + ky * ky + kz * kz);
      ask = (rule.test & q) != 0u;
      if (each & q) {
        const double rr = __dmul_rn(g.rf_factor, lam), hh = __dmul_rn(rr, 0.25);
        const double v = __dmul_rn(rule.vf, lam), in = __dsub_rn(rr, v);
        const double ox = __dmul_rn(static_cast<double>(kx), hh), oy = __dmul_rn(static_cast<double>(ky), hh),
                     oz = __dmul_rn(static_cast<double>(kz), hh);
        const double o2 = __dadd_rn(__dadd_rn(__dmul_rn(ox, ox), __dmul_rn(oy, oy)), __dmul_rn(oz, oz));
        ask = o2 < __dmul_rn(in, in) && !(o2 < __dmul_rn(v, v));
      }
    }
    open[i] = __ballot_sync(0xffffffffu, ask) & ~__reduce_or_sync(0xffffffffu, cov[i]);
  }

  // the open points: exactly covered (band) or void; the void with the
  // largest clearance, the smallest distance to the particle and its r_f set
  int cnt = 0, bk = -1;
  float best_lo = -1.f, best_hi = -1.f;  // bounds of the best point's clearance (distance)
  double best_exact = -1.0;              // its exact square, once a comparison needed it
  // only entries within 2 m of the FP32 minimum can hold the exact one
  auto exact = [&](int p, float hi) {
    return clearance_exact(g, spos, scr, idx, beg, end, s, lam, D.x[p], D.y[p], D.z[p],
                           (hi + m) * (hi + m) * 1.000001f);
  };
#pragma unroll
  for (int i = 0; i < NW; ++i) {
    for (uint32_t left = open[i]; left != 0u; left &= left - 1u) {
      const int p = 32 * i + __ffs(left) - 1;
      const float fx = D.x[p] * h, fy = D.y[p] * h, fz = D.z[p] * h;
      // smallest FP32 distance over the entries certainly (hi) and possibly (lo) in the r_f set
      float lo2 = fmaf(fx, fx, fmaf(fy, fy, fz * fz)), hi2 = lo2;
      bool covered = false;
      for (int64_t e = beg + lane; e < end; e += 32) {
        const int t = idx[e];
        const float3 d = offset32(g, me, scr[t]);
        const float dd = fmaf(d.x, d.x, fmaf(d.y, d.y, d.z * d.z));
        const float ex = d.x - fx, ey = d.y - fy, ez = d.z - fz;
        const float e2 = fmaf(ex, ex, fmaf(ey, ey, ez * ez));
        if (e2 <= v_out2) covered |= covers_exact(g, spos, s, t, lam, rule.vf, D.x[p], D.y[p], D.z[p]);
        if (dd <= r_out2) lo2 = fminf(lo2, e2);
        if (dd < r_in2) hi2 = fminf(hi2, e2);
      }
      if (__any_sync(0xffffffffu, covered)) continue;
      ++cnt;
      const float lo = sqrtf(__uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(lo2)))) - m;
      const float hi = sqrtf(__uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(hi2)))) + m;
      bool better = bk < 0 || lo > best_hi;
      double ex = -1.0;
      if (!better && hi >= best_lo) {  // too close for FP32
        if (best_exact < 0.0) best_exact = exact(bk, best_hi);
        ex = exact(p, hi);
        better = ex > best_exact;
      }
      if (better) {
        bk = p;
        best_lo = lo;
        best_hi = hi;
        best_exact = ex;
      }
    }
  }
  if (lane == 0) {
    if (void_count) void_count[me_caller] = cnt;
    if (best) best[me_caller] = bk < 0 ? -1 : ((D.x[bk] + 4) * 9 + D.y[bk] + 4) * 9 + D.z[bk] + 4;
    if (clump) clump[me_caller] = cl ? 1 : 0;
  }
  if (cand && lane < 3) {
    double c = 0.0;
    if (bk >= 0) {
      const int k = lane == 0 ? D.x[bk] : lane == 1 ? D.y[bk] : D.z[bk];
      const double hh = __dmul_rn(__dmul_rn(g.rf_factor, lam), 0.25);
      c = __dadd_rn(spos[lane * N + s], __dmul_rn(static_cast<double>(k), hh));
    }
    cand[lane * N + me_caller] = c;
  }
}

// Which grid points the scan tests, by |k|^2 (the same for every lambda
// unless the radii nearly coincide): |o_k| = |k| r_f / 4 below r_f - d_v and not
// below d_v.
ScanRule scan_rule(double rf, double vf, double cf) {
  ScanRule q{vf, cf, 0u, 0u};
  for (int k = 0; k <= 16; ++k) {
    const double o2 = k * rf * rf / 16.0, in2 = (rf - vf) * (rf - vf), v2 = vf * vf, eps = 1e-12 * rf * rf;
    if (o2 > in2 - eps && o2 < in2 + eps) q.ask |= 1u << k;
    else if (o2 > v2 - eps && o2 < v2 + eps) q.ask |= 1u << k;
    else if (o2 < in2 && o2 > v2) q.test |= 1u << k;
  }
  return q;
}

// Deletion and creation flags (caller order) from a scan: wants = survives
// (no clump mark), has a void and its point lies inside the box on every open
// axis; keep = survives.
__global__ void k_apply_wants(Grid g, const int32_t* __restrict__ best, const double* __restrict__ cand,
                              const int32_t* __restrict__ clump, int32_t* __restrict__ wants,
                              int32_t* __restrict__ keep) {
  const int n = g.n;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i > n) return;
  if (i == n) {  // scan sentinels
    keep[n] = 0;
    return;
  }
  const int64_t N = n;
  bool in = true;
  for (int a = 0; a < 3; ++a) {
    const double c = cand[a * N + i];
    if (!g.periodic[a]) in = in && c >= g.lo[a] && c < __dadd_rn(g.lo[a], g.len[a]);
  }
  keep[i] = clump[i] == 0 ? 1 : 0;
  wants[i] = (clump[i] == 0 && best[i] >= 0 && in) ? 1 : 0;
}

// create[i]: i wants a particle and no neighbour j of its exact r_f set with
// j < i wants one at a point closer than d_v = vf lambda_i (FP64, minimum
// image, in the order ((dx*dx + dy*dy) + dz*dz)).  Thread per slot.
__global__ void k_apply_create(Grid g, const int32_t* __restrict__ perm, const double* __restrict__ spos,
                               const double* __restrict__ slam, const int64_t* __restrict__ off,
                               const int32_t* __restrict__ idx, const double* __restrict__ cand,
                               const int32_t* __restrict__ wants, double vf,
                               int32_t* __restrict__ create) {
  const int n = g.n;
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s > n) return;
  if (s == n) {
    create[n] = 0;
    return;
  }
  const int64_t N = n;
  const int i = perm[s];
  int32_t c = wants[i];
  if (c) {
    const double lam = slam[s];
    const double r = __dmul_rn(g.rf_factor, lam);
    const double r2 = __dmul_rn(r, r);
    const double dv = __dmul_rn(vf, lam);
    const double dv2 = __dmul_rn(dv, dv);
    const double ci[3] = {cand[i], cand[N + i], cand[2 * N + i]};
    const int64_t end = off[s + 1] < g.capacity ? off[s + 1] : g.capacity;
    for (int64_t e = off[s]; e < end && c; ++e) {
      const int t = idx[e];
      const int j = perm[t];
      if (j >= i || !wants[j]) continue;
      double dd[3];
      for (int a = 0; a < 3; ++a) dd[a] = min_image64(__dsub_rn(cand[a * N + j], ci[a]), g.len[a], g.periodic[a]);
      const double d2 =
          __dadd_rn(__dadd_rn(__dmul_rn(dd[0], dd[0]), __dmul_rn(dd[1], dd[1])), __dmul_rn(dd[2], dd[2]));
      if (!(d2 < dv2)) continue;
      if (dist2_exact(g, spos, n, s, t) < r2) c = 0;  // not a skin entry
    }
  }
  create[i] = c;
}

// Survivors (in order) then new particles (in parent order) into the output
// arrays of leading dimension cap; ks / cs: exclusive scans of keep / create
// (their totals at n).  New particles: lambda of the parent and its
// second-order Taylor value at o = c - x, accumulated as
// U + sum_a (g_a o_a + sum_b ((h_ab / 2) o_a) o_b).
__global__ void k_apply_write(int n, int64_t cap, const double* __restrict__ pos,
                              const double* __restrict__ lam, const double* __restrict__ U,
                              const double* __restrict__ cand, const double* __restrict__ grad,
                              const double* __restrict__ hess, const int32_t* __restrict__ ks,
                              const int32_t* __restrict__ cs, double* __restrict__ pos_out,
                              double* __restrict__ lam_out, double* __restrict__ U_out,
                              int64_t* __restrict__ origin, int64_t* m_out, int32_t* status_word) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int64_t N = n;
  const int64_t nk = ks[n];
  if (i == 0) {
    const int64_t m = nk + cs[n];
    *m_out = m;
    if (m > cap) raise_flag(status_word, PHB_FLAG_CAPACITY);
  }
  if (ks[i + 1] != ks[i]) {
    const int64_t k = ks[i];
    if (k < cap) {
      for (int a = 0; a < 3; ++a) pos_out[a * cap + k] = pos[a * N + i];
      lam_out[k] = lam[i];
      for (int f = 0; f < 8; ++f) U_out[f * cap + k] = U[f * N + i];
      origin[k] = i;
    }
  }
  if (cs[i + 1] != cs[i]) {
    const int64_t k = nk + cs[i];
    if (k < cap) {
      double o[3];
      for (int a = 0; a < 3; ++a) {
        const double c = cand[a * N + i];
        pos_out[a * cap + k] = c;
        o[a] = __dsub_rn(c, pos[a * N + i]);
      }
      lam_out[k] = lam[i];
      const int hx[3][3] = {{0, 1, 2}, {1, 3, 4}, {2, 4, 5}};
      for (int f = 0; f < 8; ++f) {
        double u = U[f * N + i];
        for (int a = 0; a < 3; ++a) {
          u = __dadd_rn(u, __dmul_rn(grad[(f * 3 + a) * N + i], o[a]));
          for (int b = 0; b < 3; ++b)
            u = __dadd_rn(u, __dmul_rn(__dmul_rn(__dmul_rn(0.5, hess[(f * 6 + hx[a][b]) * N + i]), o[a]), o[b]));
        }
        U_out[f * cap + k] = u;
      }
      origin[k] = N + i;
    }
  }
}

// -------- storage order
__global__ void k_identity(int n, int32_t* __restrict__ perm, int32_t* __restrict__ inv) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n) return;
  perm[s] = s;
  inv[s] = s;
}

// -------- export in caller numbering
__global__ void k_user_counts(int n, const int32_t* __restrict__ inv, const int64_t* __restrict__ off,
                              int32_t* __restrict__ ucnt) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i > n) return;
  if (i == n) { ucnt[n] = 0; return; }
  const int s = inv[i];
  ucnt[i] = static_cast<int32_t>(off[s + 1] - off[s]);
}

__global__ void k_user_fill(int n, int64_t cap, const int32_t* __restrict__ inv,
                            const int32_t* __restrict__ perm, const int64_t* __restrict__ off,
                            const int32_t* __restrict__ idx, const int64_t* __restrict__ uoff,
                            int32_t* __restrict__ uidx) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int s = inv[i];
  const int64_t a = off[s], b = off[s + 1] < cap ? off[s + 1] : cap;
  int32_t* v = uidx + uoff[i];
  const int m = static_cast<int>(b > a ? b - a : 0);
  for (int k = 0; k < m; ++k) v[k] = perm[idx[a + k]];
  for (int k = 1; k < m; ++k) {  // ascending caller index
    int32_t x = v[k];
    int j = k - 1;
    while (j >= 0 && v[j] > x) { v[j + 1] = v[j]; --j; }
    v[j + 1] = x;
  }
}

}  // namespace

cudaError_t build_neighbors_impl(const phb_plan* p, const double* pos, const double* lam, void* ws,
                                 int32_t* status_word, cudaStream_t st) {
  const Grid g = make_grid(p);
  const int n = g.n;
  int32_t* keys = region<int32_t>(p, ws, R_KEYS);
  int32_t* perm = region<int32_t>(p, ws, R_PERM);
  int32_t* inv = region<int32_t>(p, ws, R_INV);
  int32_t* cell = region<int32_t>(p, ws, R_CELL);
  int32_t* cursor = region<int32_t>(p, ws, R_CURSOR);
  int64_t* bsum = region<int64_t>(p, ws, R_SCAN);
  double* spos = region<double>(p, ws, R_SPOS);
  double* slam = region<double>(p, ws, R_SLAM);
  float4* scr = region<float4>(p, ws, R_SCREEN);
  int32_t* ncnt = region<int32_t>(p, ws, R_NCNT);
  int64_t* off = region<int64_t>(p, ws, R_OFF);
  int32_t* idx = region<int32_t>(p, ws, R_IDX);
  uint16_t* lidx = region<uint16_t>(p, ws, R_LIDX);
  int32_t* cellc = region<int32_t>(p, ws, R_CELLC);
  int2* clin = region<int2>(p, ws, R_CLIN);
  int32_t* misc = region<int32_t>(p, ws, R_MISC);
  cudaError_t e;
  // cell counts and scatter cursors are adjacent regions: one clear
  const int32_t nkeys = static_cast<int32_t>(p->nkeys);
  const size_t clear = p->ws_off[R_CURSOR] + (p->nkeys + 1) * sizeof(int32_t) - p->ws_off[R_CELL];
  if ((e = cudaMemsetAsync(cell, 0, clear, st))) return e;
  Bricks br{nullptr, nullptr};
  if (const int64_t words = brick_words(p); words > 0) {
    uint32_t* bits = region<uint32_t>(p, ws, R_BBITS);
    int32_t* before = region<int32_t>(p, ws, R_BBEFORE);
    if ((e = cudaMemsetAsync(bits, 0, words * sizeof(uint32_t), st))) return e;
    k_brick_mark<<<blocks_for(p->nkeys / 64), kThreads, 0, st>>>(g, bits);
    note_launch();
    k_brick_count<<<blocks_for(words + 1), kThreads, 0, st>>>(words, bits, before);
    note_launch();
    if ((e = scan_exclusive_i32(before, words + 1, bsum, st))) return e;
    br = Bricks{bits, before};
  }
  k_keys<<<blocks_for(n), kThreads, 0, st>>>(g, br, nkeys, pos, lam, keys, cell, status_word);
  note_launch();
  if ((e = scan_exclusive_i32(cell, p->nkeys + 1, bsum, st))) return e;
  // the inverse-permutation region (written later by k_gather_pos) holds the
  // scattered order until the ranking puts it into ascending caller index
  k_scatter<<<blocks_for(n), kThreads, 0, st>>>(n, keys, cell, cursor, inv);
  note_launch();
  k_rank_cells<<<blocks_for(n), kThreads, 0, st>>>(n, nkeys, keys, cell, inv, perm);
  note_launch();
  k_gather_pos<<<blocks_for(n), kThreads, 0, st>>>(g, perm, pos, lam, inv, spos, slam, scr, cellc);
  note_launch();
  const int64_t ncells = int64_t(p->ncell[0]) * p->ncell[1] * p->ncell[2];
  int32_t* lstart = region<int32_t>(p, ws, R_LSTART);
  float4* lscr = region<float4>(p, ws, R_LSCR);
  k_cell_lin<<<blocks_for(ncells + 1), kThreads, 0, st>>>(g, br, cell, clin, lstart, misc);
  note_launch();
  if ((e = scan_exclusive_i32(lstart, ncells + 1, bsum, st))) return e;
  k_fill_lin<<<blocks_for(n), kThreads, 0, st>>>(g, cellc, clin, lstart, scr, lscr);
  note_launch();
  const Lin lin{lscr, lstart};
  int32_t* ell = region<int32_t>(p, ws, R_ELL);
  // Which search (us of the search kernels).  One lambda: a warp per particle
  // below kCellsMin (1,000 particles 15, 4,096: 18, 10,648: 29, 19,683: 43), from
  // there on a warp per cell (37, 54, 40, 43; 262,144: 157), then a thread per
  // particle for the lists it left.  Lambda varying: a warp per particle up to
  // kWarpMax (10,007 particles 38, 60,000: 116, 130,000: 230), a thread per
  // particle beyond (165, 181, 250; 260,000: 345 against 402).
  constexpr int kCellsMin = 1 << 14, kWarpMax = 1 << 17;
  const bool one_lambda = p->lambda_max <= 1.01 * p->lambda_min;
  const bool cell_major = one_lambda && n >= kCellsMin;
  if (cell_major && (e = cudaMemsetAsync(ncnt, 0xff, static_cast<size_t>(n) * sizeof(int32_t), st)))
    return e;
  int tr = trace_begin(4, st);
  if (cell_major) {
    k_search_cells<<<static_cast<unsigned>(ncells), 32, 0, st>>>(g, lin, spos, slam, ncnt, ell);
    note_launch();
  }
  if (cell_major || n > kWarpMax)
    k_search_ell<<<blocks_for(n), kThreads, 0, st>>>(g, lin, cellc, scr, spos, slam, ncnt, ell, cell_major);
  else
    k_search_warp<<<blocks_for(n, 8), 128, 0, st>>>(g, lin, cellc, scr, spos, slam, ncnt, ell);
  trace_end(tr, st);
  note_launch();
  if ((e = scan_exclusive_i32_to_i64(ncnt, off, n + 1, bsum, st))) return e;
  const unsigned tiles = static_cast<unsigned>(p->ntiles);
  int2* tplan = region<int2>(p, ws, R_TPLAN);
  int32_t* tslot = region<int32_t>(p, ws, R_TSLOT);
  uint16_t* lself = region<uint16_t>(p, ws, R_LSELF);
  uint8_t* tmap = region<uint8_t>(p, ws, R_TMAP);
  tr = trace_begin(5, st);
  // nine 128-thread blocks per SM at 56 registers: 2048 tiles in 1.5 waves
  // of 1368 instead of 1.7 of 1216 (the shared memory of nine needs the
  // largest carve-out)
  cudaFuncSetAttribute(k_compact<128>, cudaFuncAttributePreferredSharedMemoryCarveout,
                       cudaSharedmemCarveoutMaxShared);
  cudaFuncSetAttribute(k_compact<64>, cudaFuncAttributePreferredSharedMemoryCarveout,
                       cudaSharedmemCarveoutMaxShared);
  if (p->tile == 128)
    k_compact<128><<<tiles, 128, 0, st>>>(g, clin, lin, cellc, scr, spos, slam, ncnt, ell, off, idx, lidx,
                                          tplan, tslot, lself, tmap, misc + 1, status_word);
  else
    k_compact<64><<<tiles, 64, 0, st>>>(g, clin, lin, cellc, scr, spos, slam, ncnt, ell, off, idx, lidx,
                                        tplan, tslot, lself, tmap, misc + 1, status_word);
  trace_end(tr, st);
  note_launch();
  if (p->schedule == 1) {  // only schedule 1 of the fit reads the tile order
    k_tile_order<<<1, 1024, 0, st>>>(n, p->tile, p->ntiles, p->nbr_capacity, off,
                                     region<int32_t>(p, ws, R_TORDER));
    note_launch();
  }
  return cudaGetLastError();
}

cudaError_t export_neighbors_impl(const phb_plan* p, const void* ws_c, int64_t* uoff, int32_t* uidx,
                                  cudaStream_t st) {
  void* ws = const_cast<void*>(ws_c);
  const int n = static_cast<int>(p->n);
  const int32_t* perm = region<int32_t>(p, ws, R_PERM);
  const int32_t* inv = region<int32_t>(p, ws, R_INV);
  const int64_t* off = region<int64_t>(p, ws, R_OFF);
  const int32_t* idx = region<int32_t>(p, ws, R_IDX);
  int32_t* ucnt = region<int32_t>(p, ws, R_QUEUE);  // scratch: n+1 fits before R_PC (>= n+64 ints)
  int64_t* bsum = region<int64_t>(p, ws, R_SCAN);
  cudaError_t e;
  k_user_counts<<<blocks_for(n + 1), kThreads, 0, st>>>(n, inv, off, ucnt);
  note_launch();
  if ((e = scan_exclusive_i32_to_i64(ucnt, uoff, n + 1, bsum, st))) return e;
  k_user_fill<<<blocks_for(n), kThreads, 0, st>>>(n, p->nbr_capacity, inv, perm, off, idx, uoff, uidx);
  note_launch();
  return cudaGetLastError();
}

}  // namespace phb

using namespace phb;

extern "C" phb_status phb_build_neighbors(const phb_plan* plan, const double* pos,
                                          const double* lambda, void* ws, size_t ws_bytes,
                                          int32_t* status_word, phb_stream_t stream) {
  phb_status s = check_common(plan, ws, ws_bytes, plan ? plan->ws_off[R_END_COMMON] : 0);
  if (s != PHB_OK) return s;
  if (!pos || !lambda) return PHB_ERR_INVALID_ARG;
  return launch_status(build_neighbors_impl(plan, pos, lambda, ws, status_word,
                                            reinterpret_cast<cudaStream_t>(stream)));
}

extern "C" phb_status phb_adapt_scan(const phb_plan* plan, const double* pos, const double* lambda,
                                     double void_factor, double clump_factor, void* ws, size_t ws_bytes,
                                     int32_t* void_count, int32_t* best, double* cand, int32_t* clump,
                                     int32_t* status_word, phb_stream_t stream) {
  phb_status s = check_common(plan, ws, ws_bytes, plan ? plan->ws_off[R_END_COMMON] : 0);
  if (s != PHB_OK) return s;
  if (!pos || !lambda) return PHB_ERR_INVALID_ARG;
  if (!(void_factor > 0.0) || !(void_factor < plan->rf_factor) || !(clump_factor >= 0.0) ||
      !(clump_factor < plan->rf_factor))
    return PHB_ERR_INVALID_ARG;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const Grid g = make_grid(plan);
  const int n = g.n;
  const int32_t* perm = region<int32_t>(plan, ws, R_PERM);
  double* spos = region<double>(plan, ws, R_SPOS);
  double* slam = region<double>(plan, ws, R_SLAM);
  float4* scr = region<float4>(plan, ws, R_SCREEN);
  k_adapt_gather<<<blocks_for(n), kThreads, 0, st>>>(g, perm, pos, lambda, spos, slam, scr);
  note_launch();
  // the points within |k|^2 <= 5 are all there are for the default factors;
  // smaller void factors reach out to |k|^2 = 16 (|o_k| < r_f)
  const ScanRule rule = scan_rule(plan->rf_factor, void_factor, clump_factor);
  const auto scan = (rule.test | rule.ask) >> 6 == 0u ? k_adapt_scan<5> : k_adapt_scan<16>;
  scan<<<blocks_for(int64_t(n) * 32, 128), 128, 0, st>>>(g, rule, perm, spos, slam, scr,
                                                         region<int64_t>(plan, ws, R_OFF),
                                                         region<int32_t>(plan, ws, R_IDX), void_count, best,
                                                         cand, clump);
  note_launch();
  return launch_status(cudaGetLastError());
}

extern "C" phb_status phb_adapt_apply(const phb_plan* plan, const double* pos, const double* lambda,
                                      const double* U, const int32_t* best, const double* cand,
                                      const int32_t* clump, const double* grad, const double* hess,
                                      double void_factor, int64_t cap, double* pos_out,
                                      double* lambda_out, double* U_out, int64_t* origin,
                                      int64_t* m_out, void* ws, size_t ws_bytes, int32_t* status_word,
                                      phb_stream_t stream) {
  phb_status s = check_common(plan, ws, ws_bytes, plan ? plan->ws_off[R_END_COMMON] : 0);
  if (s != PHB_OK) return s;
  if (!pos || !lambda || !U || !best || !cand || !clump || !grad || !hess || !pos_out ||
      !lambda_out || !U_out || !origin || !m_out || cap < 0)
    return PHB_ERR_INVALID_ARG;
  if (!(void_factor > 0.0) || !(void_factor < plan->rf_factor)) return PHB_ERR_INVALID_ARG;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const Grid g = make_grid(plan);
  const int n = g.n;
  const int32_t* perm = region<int32_t>(plan, ws, R_PERM);
  double* spos = region<double>(plan, ws, R_SPOS);
  double* slam = region<double>(plan, ws, R_SLAM);
  float4* scr = region<float4>(plan, ws, R_SCREEN);
  int32_t* wants = region<int32_t>(plan, ws, R_QUEUE);
  int32_t* keep = region<int32_t>(plan, ws, R_AFLAG);
  int32_t* create = region<int32_t>(plan, ws, R_ALIST);
  int64_t* bsum = region<int64_t>(plan, ws, R_SCAN);
  cudaError_t e;
  k_adapt_gather<<<blocks_for(n), kThreads, 0, st>>>(g, perm, pos, lambda, spos, slam, scr);
  note_launch();
  k_apply_wants<<<blocks_for(n + 1), kThreads, 0, st>>>(g, best, cand, clump, wants, keep);
  note_launch();
  k_apply_create<<<blocks_for(n + 1), kThreads, 0, st>>>(g, perm, spos, slam,
                                                         region<int64_t>(plan, ws, R_OFF),
                                                         region<int32_t>(plan, ws, R_IDX), cand, wants,
                                                         void_factor, create);
  note_launch();
  if ((e = scan_exclusive_i32(keep, n + 1, bsum, st))) return launch_status(e);
  if ((e = scan_exclusive_i32(create, n + 1, bsum, st))) return launch_status(e);
  k_apply_write<<<blocks_for(n), kThreads, 0, st>>>(n, cap, pos, lambda, U, cand, grad, hess, keep, create,
                                                    pos_out, lambda_out, U_out, origin, m_out,
                                                    status_word);
  note_launch();
  return launch_status(cudaGetLastError());
}

extern "C" phb_status phb_reorder(const phb_plan* plan, double* pos, double* lambda, double* U,
                                  int32_t* perm_out, void* ws, size_t ws_bytes, int32_t* status_word,
                                  phb_stream_t stream) {
  phb_status s = check_common(plan, ws, ws_bytes, plan ? plan->ws_off[R_END_COMMON] : 0);
  if (s != PHB_OK) return s;
  if (!pos || !lambda || !U) return PHB_ERR_INVALID_ARG;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const Grid g = make_grid(plan);
  const int64_t N = plan->n;
  int32_t* perm = region<int32_t>(plan, ws, R_PERM);
  cudaError_t e;
  // slot-order copies of all three arrays, then back over the caller's
  if ((e = gather_sorted(plan, g, pos, lambda, U, ws, status_word, st))) return launch_status(e);
  if (perm_out && (e = cudaMemcpyAsync(perm_out, perm, N * sizeof(int32_t), cudaMemcpyDeviceToDevice, st)))
    return launch_status(e);
  if ((e = cudaMemcpyAsync(pos, region<double>(plan, ws, R_SPOS), 3 * N * sizeof(double),
                           cudaMemcpyDeviceToDevice, st)))
    return launch_status(e);
  if ((e = cudaMemcpyAsync(lambda, region<double>(plan, ws, R_SLAM), N * sizeof(double),
                           cudaMemcpyDeviceToDevice, st)))
    return launch_status(e);
  if ((e = cudaMemcpyAsync(U, region<double>(plan, ws, R_SU), 8 * N * sizeof(double),
                           cudaMemcpyDeviceToDevice, st)))
    return launch_status(e);
  k_identity<<<blocks_for(N), kThreads, 0, st>>>(g.n, perm, region<int32_t>(plan, ws, R_INV));
  note_launch();
  return launch_status(cudaGetLastError());
}

extern "C" int64_t phb_neighbor_total(const phb_plan* plan, const void* ws, phb_stream_t stream) {
  if (!plan || !ws || plan->ws_bytes == 0) return -1;
  int64_t total = -1;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const int64_t* off = region<int64_t>(plan, ws, R_OFF);
  if (cudaMemcpyAsync(&total, off + plan->n, sizeof(int64_t), cudaMemcpyDeviceToHost, st) !=
      cudaSuccess)
    return -1;
  if (cudaStreamSynchronize(st) != cudaSuccess) return -1;
  return total;
}

extern "C" phb_status phb_export_neighbors(const phb_plan* plan, const void* ws, int64_t* off,
                                           int32_t* idx, int64_t idx_capacity, phb_stream_t stream) {
  if (!plan || !ws || !off || !idx || plan->ws_bytes == 0) return PHB_ERR_INVALID_ARG;
  // the export writes its counts into the route-queue region (n int32 + pad)
  int64_t total = phb_neighbor_total(plan, ws, stream);
  if (total < 0) return PHB_ERR_CUDA;
  if (total > idx_capacity || total > plan->nbr_capacity) return PHB_ERR_CAPACITY;
  return launch_status(export_neighbors_impl(plan, ws, off, idx, reinterpret_cast<cudaStream_t>(stream)));
}
