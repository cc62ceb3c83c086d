// One-sided (row) Jacobi SVD of small matrices on a cluster of CTAs (K3: the
// truncated splits of Sec. 1.1.3 and the reduced factors of the randomised
// truncation).
//
// The M rows of G (length N) are rotated pairwise until they are orthogonal,
// the same rotations accumulating in WH (M x M, from the identity): WH G_0 =
// G.  A row of G and its row of WH are one vector of N + M entries.
//
// Order and arithmetic are part of the results.  The phases of the singular
// vectors follow from the order of the rotations and from every rounding, and
// the randomised truncations sketch in the basis that these phases give: where
// a spectrum is flat, another order moves a network's messages by 1e-5 in full
// precision.  So the pairs go round a circle tournament (round r: row M' - 1
// against row r, row r + q against row r - q, mod M' - 1, M' = M rounded up to
// even), the four sums of a pair are taken lane by lane (32 or 16 lanes) with
// one addition tree, and every product and sum is rounded as written here (fma
// calls, and products that no addition can take up).  JacOrder names the three
// forms that results so far were computed in; k_jacobi (device memory) rotates
// as kJacPlain32.
//
// Distribution: the P = M' / 2 pairs of a round lie on C CTAs, pp places each,
// a warp a place, both rows in shared memory.  From round to round the first
// rows of the places move one place left and the second rows one place right
// (turning at the ends; row M' - 1 stays): inside a CTA the rows stay where
// they are and the places' slots move round two rings of pp + 2 slots; at its
// ends a warp pushes the row that leaves into the neighbour's next slot,
// completing on that CTA's mbarrier, and waits for the one that comes.  A
// neighbour pushes at the end of round r into the slot whose row left at the
// end of round r - 2: it has had this CTA's push of round r - 1, which came
// after the block barrier of round r - 2.  One barrier a direction and round
// parity: a push of round r + 2 needs this CTA's push of round r + 1, made by
// the same warp after its wait for round r.
//
// What bounds it.  complex128: the FP64 unit (a warp-wide instruction 64
// clocks, one every 19 clocks an SM), so the square roots and the quotients of
// a pair are taken side by side in lanes of one instruction and the sums share
// their addition tree (6 additions for 20), two pairs a CTA: 128 instructions
// a pair, half of them scalars.  complex64: the chain of one reduction and
// five roots and quotients a round.  Measured, us, one CTA with all rows (a warp
// or half a warp a pair, every lane its own scalars) and here: complex128 8 x 8
// 261 and 178, 31 x 40 6170 and 1430, 64 x 64 28400 and 3470 (graded rows 62600
// and 8090); complex64 31 x 40 315 and 278, 64 x 64 1030 and 717, 96 x 90 1737 and
// 1167 (long rows of few pairs are no faster: 20 x 900 323 and 354); from device
// memory and here: complex128 128 x 128 45600 and 11250.
#include <cooperative_groups.h>

#include <algorithm>
#include <atomic>
#include <cstdint>

#include "kernels.h"
#include "push.h"

namespace cg = cooperative_groups;

namespace bbp {

namespace {

constexpr int kJacMaxCluster = 16;
constexpr int kJacWarps = 20;
constexpr size_t kJacSmemMax = 227 * 1024;
constexpr size_t kJacStaged = 211 * 1024;   // rows that one CTA's shared memory held: the staged orders

template <typename C> struct RealJ;
template <> struct RealJ<double2> { using T = double; };
template <> struct RealJ<float2> { using T = float; };
template <typename C> __device__ __forceinline__ C mkj(typename RealJ<C>::T re, typename RealJ<C>::T im) {
  C r;
  r.x = re;
  r.y = im;
  return r;
}

template <typename R>
__device__ __forceinline__ R sum1(R v) {
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Lanes of a pair's sums, and which product of e y is rounded by itself.
enum JacOrder { kJacPlain32 = 0, kJacStaged32 = 1, kJacStaged16 = 2 };

// Rotates rows x and y (N entries of G, len = N + M with those of WH) so that
// their G parts become orthogonal; returns 1 when a rotation was applied.  A
// warp; every lane takes the same decision.
template <typename C, int ORD>
__device__ __forceinline__ int rotate_rows(C* __restrict__ xr, C* __restrict__ yr, int N, int len, int lane,
                                           typename RealJ<C>::T tol, typename RealJ<C>::T floor) {
  using R = typename RealJ<C>::T;
  const unsigned all = 0xffffffffu;
  const bool up = lane & 16, odd = lane & 8;
  R p0 = 0, p1 = 0;                      // lower lanes: |x|^2, Re x conj(y); upper: |y|^2, Im x conj(y)
  if constexpr (ORD == kJacStaged16) {
#pragma unroll 4
    for (int c = lane & 15; c < N; c += 16) {
      const C x = xr[c], y = yr[c];
      const C u = up ? y : x;
      const R a = up ? x.y : x.x, b = up ? -x.x : x.y;
      p0 += fma(u.x, u.x, u.y * u.y);
      p1 += fma(a, y.x, b * y.y);
    }
  } else {
    R al = 0, be = 0, gx = 0, gy = 0;
#pragma unroll 4
    for (int c = lane; c < N; c += 32) {
      const C x = xr[c], y = yr[c];
      al += fma(x.x, x.x, x.y * x.y);
      be += fma(y.x, y.x, y.y * y.y);
      gx += fma(x.x, y.x, x.y * y.y);
      gy += fma(x.y, y.x, -(x.x * y.y));
    }
    p0 = (up ? be : al) + __shfl_xor_sync(all, up ? al : be, 16);
    p1 = (up ? gy : gx) + __shfl_xor_sync(all, up ? gx : gy, 16);
  }
  R v = (odd ? p1 : p0) + __shfl_xor_sync(all, odd ? p0 : p1, 8);
  v += __shfl_xor_sync(all, v, 4);
  v += __shfl_xor_sync(all, v, 2);
  v += __shfl_xor_sync(all, v, 1);
  const R al = __shfl_sync(all, v, 0), gx = __shfl_sync(all, v, 8);
  const R be = __shfl_sync(all, v, 16), gy = __shfl_sync(all, v, 24);
  const R rt = sqrt(odd ? fma(gx, gx, gy * gy) : v);     // |g| beside the two norms
  const R g = __shfl_sync(all, rt, 8);
  if (g == 0 || g <= tol * __shfl_sync(all, rt, 0) * __shfl_sync(all, rt, 16)) return 0;
  // a row below eps ||Z|| carries nothing at working precision; orthogonalising
  // it (in subnormal arithmetic, at worst) would never meet the test above
  const R lo = fmin(al, be);
  if (lo <= floor) return 0;
  // rows whose norms differ by more than 1e30 (1e15 in complex64) do not
  // affect each other at working precision; rotating them only churns
  // rounding noise (and never meets the relative test once a norm is subnormal)
  const R far = sizeof(R) == 8 ? (R)1e-60 : (R)1e-30;
  if (lo <= far * fmax(al, be)) return 0;
  const R num = up ? be - al : (odd ? gy : gx), den = up ? 2 * g : g;
  const R quo = num / den;
  const R ex = __shfl_sync(all, quo, 0), ey = __shfl_sync(all, quo, 8), zeta = __shfl_sync(all, quo, 16);
  const R t = (zeta >= 0 ? (R)1 : (R)-1) / (fabs(zeta) + sqrt(fma(zeta, zeta, (R)1)));
  const R cs = (R)1 / sqrt(fma(t, t, (R)1)), sn = cs * t;
#pragma unroll 4
  for (int c = lane; c < len; c += 32) {
    const C x = xr[c], y = yr[c];
    const R wx = fma(ex, y.x, -(ey * y.y));
    const R wy = ORD == kJacPlain32 ? fma(ex, y.y, ey * y.x) : fma(ey, y.x, ex * y.y);
    xr[c] = mkj<C>(fma(x.x, cs, -(wx * sn)), fma(x.y, cs, -(wy * sn)));
    yr[c] = mkj<C>(fma(x.x, sn, wx * cs), fma(x.y, sn, wy * cs));
  }
  return 1;
}

struct JacArgs {
  int M, N, pp;                          // rows, row length, places a CTA
  int ldz, conj_t;                       // G_0[a][c] = Z[a ldz + c], or conj(Z[c ldz + a])
  int m, n, k;                           // exact SVD outputs (U, Rem not null): U m x k, Rem k x n
  double tol, floor_rel;
  int max_sweeps;
};

// ||Z||^2 between 2^-kJacUnscaled and 2^kJacUnscaled: the rows are taken as they are;
// beyond, scaled by a power of two to a norm near one (every rounding stays the
// same, and no square of an entry that matters leaves the range).
template <typename C> constexpr int kJacUnscaled = sizeof(C) == sizeof(float2) ? 40 : 400;

__host__ __device__ inline size_t jac_header(int M) {
  const size_t Mp = M + (M & 1);
  return 64 + 176 + 512 + ((2 * sizeof(double) + sizeof(int)) * Mp + 15) / 16 * 16;
}

template <typename C, int ORD, bool CL>
__global__ void __launch_bounds__(32 * kJacWarps, 1) k_jac(JacArgs p, const C* __restrict__ Z, C* __restrict__ Gout,
                                                C* __restrict__ WHout, double* __restrict__ sigma,
                                                int* __restrict__ idx, double* __restrict__ zn2_out, int* counters,
                                                C* __restrict__ U, C* __restrict__ Rem, int* status, double* flops) {
  using R = typename RealJ<C>::T;
  cg::cluster_group cl = cg::this_cluster();
  const int cs = CL ? (int)cl.num_blocks() : 1, cr = CL ? (int)cl.block_rank() : 0;
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  const int M = p.M, N = p.N, pp = p.pp, len = N + M;
  const int ld = (len + 1) & ~1;         // entries of a row in shared memory (16-byte rows)
  const int Mp = M + (M & 1), P = Mp / 2, rounds = Mp - 1;
  const int q0 = cr * pp, pl = min(pp, P - q0);     // first place and number of places of this CTA
  const int S = pp + 2;                  // slots of a ring
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const uint32_t bars = saddr(smem_raw);            // first rows in (by parity), second rows in, counts
  volatile int* failed = (volatile int*)(smem_raw + 48);
  int* s_rot = (int*)(smem_raw + 52);
  double* s_sum = (double*)(smem_raw + 64);         // [0] this CTA's sum, [1 ..] warps' sums
  int* s_cnt = (int*)(smem_raw + 64 + 176);         // [2][16][4] rotations of a sweep, by CTA
  double* s_sig = (double*)(smem_raw + 64 + 176 + 512);   // [Mp] singular values
  double* s_inv = s_sig + Mp;            // [Mp] their inverses, zero below the floor
  int* s_rank = (int*)(s_inv + Mp);      // [Mp], and a pad to sixteen bytes
  C* rows = (C*)(smem_raw + jac_header(M));
  // first rows: slot (j + R) mod S of place j in round R (all sweeps counted
  // through), row M' - 1 in a slot of its own; second rows: slot (j - R) mod S
  // (one CTA alone: row a at rows + a ld)
  auto ring_a = [&](int j, int r) { return rows + (size_t)((j + r) % S) * ld; };
  auto ring_b = [&](int j, int r) { return rows + (size_t)(S + (j + r * (S - 1)) % S) * ld; };
  C* const fixed = rows + (size_t)(2 * S) * ld;
  auto first = [&](int j, int r) {       // rows of place j
    if constexpr (CL) return q0 + j == 0 ? fixed : ring_a(j, r);
    else return rows + (size_t)(j == 0 ? Mp - 1 : (r + j) % rounds) * ld;
  };
  auto second = [&](int j, int r) {
    if constexpr (CL) return ring_b(j, r);
    else return rows + (size_t)((r - j % rounds + rounds) % rounds) * ld;
  };
  auto id_a = [&](int j) { return q0 + j == 0 ? Mp - 1 : q0 + j; };             // rows of the places
  auto id_b = [&](int j) { return q0 + j == 0 ? 0 : Mp - 1 - (q0 + j); };       // when a sweep begins
  const C zero = mkj<C>(0, 0);
  if (tid == 0) {
    for (int q = 0; q < 6; ++q) bar_init(bars + 8 * q);
    *failed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }

  // ---- load
  double part = 0.0;
#pragma unroll 4
  for (int e = tid; e < 2 * pl * ld; e += nt) {
    // neighbouring threads along the contiguous index of Z
    const int rr = p.conj_t ? e % (2 * pl) : e / ld, c = p.conj_t ? e / (2 * pl) : e - rr * ld;
    const int j = rr >> 1, a = rr & 1 ? id_b(j) : id_a(j);
    if (!CL && a >= M) continue;         // (no slot for the row that rounds M up)
    C v = zero;
    if (a < M) {
      if (c < N) {
        v = p.conj_t ? Z[(size_t)c * p.ldz + a] : Z[(size_t)a * p.ldz + c];
        if (p.conj_t) v.y = -v.y;
        part += (double)v.x * v.x + (double)v.y * v.y;
      } else if (c - N == a) {
        v = mkj<C>(1, 0);
      }
    }
    (rr & 1 ? second(j, 0) : first(j, 0))[c] = v;
  }
  part = sum1(part);
  if (lane == 0) s_sum[1 + warp] = part;
  __syncthreads();
  if (tid == 0) {
    double s = 0.0;
    for (int w = 0; w < nw; ++w) s += s_sum[1 + w];
    s_sum[0] = s;
  }
  double zn2 = 0.0;
  if constexpr (CL) {
    cl.sync();                           // (also: the barriers are ready before the first push)
    for (int q = 0; q < cs; ++q) zn2 += cl.map_shared_rank(s_sum, q)[0];
    cl.sync();
  } else {
    __syncthreads();
    zn2 = s_sum[0];
  }
  if (cr == 0 && tid == 0 && zn2_out) *zn2_out = zn2;
  int ex2 = 0;
  if (zn2 > 0.0 && isfinite(zn2)) {
    int e;
    frexp(zn2, &e);
    if (abs(e) > kJacUnscaled<C>) ex2 = e / 2;
    if (sizeof(R) == 4) ex2 = min(max(ex2, -120), 120);
  }
  const R up = (R)ldexp(1.0, -ex2), down = (R)ldexp(1.0, ex2);
  const R floor = (R)(p.floor_rel * (zn2 * ldexp(1.0, -2 * ex2)));
  if (ex2 != 0)
    for (int rr = warp; rr < 2 * pl; rr += nw) {
      C* row = rr & 1 ? second(rr >> 1, 0) : first(rr >> 1, 0);
      if ((rr & 1 ? id_b(rr >> 1) : id_a(rr >> 1)) >= M) continue;
      for (int c = lane; c < N; c += 32) row[c] = mkj<C>(row[c].x * up, row[c].y * up);
    }
  __syncthreads();

  // ---- sweeps
  const uint32_t row_bytes = (uint32_t)(sizeof(C) * (size_t)ld);
  // the warps at the CTA's ends wait for the rows of round r
  auto arrive = [&](int r) {
    if constexpr (CL) {
      if (warp == (pl - 1) % nw && cr < cs - 1) {
        if (lane == 0) bar_expect(bars + 8 * (r & 1), row_bytes);
        __syncwarp();
        bar_wait(bars + 8 * (r & 1), (r - 1) >> 1 & 1, failed);
      }
      if (warp == 0 && cr > 0) {
        if (lane == 0) bar_expect(bars + 16 + 8 * (r & 1), row_bytes);
        __syncwarp();
        bar_wait(bars + 16 + 8 * (r & 1), (r - 1) >> 1 & 1, failed);
      }
    }
  };
  auto send = [&](const C* row, C* to, uint32_t bar, int rank) {
    const uint32_t src = saddr(row), dst = CL ? remote(saddr(to), rank) : 0u, b = CL ? remote(bar, rank) : 0u;
    for (uint32_t o = 16 * lane; o < row_bytes; o += 512) push128(dst + o, b, lds128(src + o));
  };
  auto copy = [&](const C* row, C* to) {
    const uint32_t src = saddr(row), dst = saddr(to);
    for (uint32_t o = 16 * lane; o < row_bytes; o += 512) sts128(dst + o, lds128(src + o));
  };
  const R tol = (R)p.tol;
  int sweeps = 0, rot_total = 0, R0 = 0;
  uint32_t ph_cnt = 0;                   // phases of the counts' barriers
  bool converged = false;
  while (sweeps < p.max_sweeps) {
    int rot = 0;
    for (int r = 0; r < rounds; ++r, ++R0) {
      if (R0 > 0) arrive(R0);
      for (int j = warp; j < pl; j += nw) {
        C* x = first(j, CL ? R0 : r);
        C* y = second(j, CL ? R0 : r);
        if (q0 + j > 0 || Mp == M) rot += rotate_rows<C, ORD>(x, y, N, len, lane, tol, floor);
        if constexpr (CL) {
          __syncwarp();
          // first rows go left: out of the CTA, or from place 1 to place 0 as its second row
          if (j == 0 && cr > 0) send(x, ring_a(pp - 1, R0 + 1), bars + 8 * ((R0 + 1) & 1), cr - 1);
          else if (q0 + j == 1) copy(x, ring_b(0, R0 + 1));
          // second rows go right: out of the CTA, or at the last place become its first row
          if (j == pl - 1) {
            if (cr < cs - 1) send(y, ring_b(0, R0 + 1), bars + 16 + 8 * ((R0 + 1) & 1), cr + 1);
            else copy(y, ring_a(j, R0 + 1));
          }
        }
      }
      __syncthreads();
    }
    // rotations of the sweep over the cluster
    if (tid == 0) *s_rot = 0;
    __syncthreads();
    if (lane == 0 && rot) atomicAdd(s_rot, rot);
    __syncthreads();
    int total = *s_rot;
    if constexpr (CL) {
      const int par = sweeps & 1;
      if (tid == 0) bar_expect(bars + 32 + 8 * par, 16u * cs);
      if (tid < cs)
        push128(remote(saddr(s_cnt + (par * kJacMaxCluster + cr) * 4), tid), remote(bars + 32 + 8 * par, tid),
                make_float4(__int_as_float(total), 0.f, 0.f, 0.f));
      bar_wait(bars + 32 + 8 * par, (ph_cnt >> par) & 1u, failed);
      ph_cnt ^= 1u << par;
      total = 0;
      for (int q = 0; q < cs; ++q) total += s_cnt[(par * kJacMaxCluster + q) * 4];
    }
    __syncthreads();
    const bool bad = *failed != 0;       // an exchange that ran out: no result
    __syncthreads();
    ++sweeps;
    rot_total += total;
    if (total == 0 || bad) { converged = total == 0 && !bad; break; }
  }
  if (R0 > 0) arrive(R0);                // the rows are back at their places
  __syncthreads();
  if (*failed) converged = false;

  // ---- row norms in double, ranks by size, outputs
  for (int rr = warp; rr < 2 * pl; rr += nw) {
    const int j = rr >> 1, id = rr & 1 ? id_b(j) : id_a(j);
    if (id >= M) continue;
    const C* row = rr & 1 ? second(j, CL ? R0 : 0) : first(j, CL ? R0 : 0);
    double a = 0.0;
    for (int c = lane; c < N; c += 32) {
      const double x = row[c].x, y = row[c].y;
      a += fma(x, x, y * y);
    }
    a = sum1(a);
    if (lane == 0) s_sig[id] = sqrt(a) * ldexp(1.0, ex2);
  }
  __syncthreads();
  if constexpr (CL) {
    cl.sync();
    for (int e = tid; e < M; e += nt) {
      const int q = (e == Mp - 1 ? 0 : (e < P ? e : Mp - 1 - e)) / pp;   // the CTA of the row's place
      if (q != cr) s_sig[e] = cl.map_shared_rank(s_sig, q)[e];
    }
    cl.sync();                           // (no remote access after this)
  }
  const double smin = sqrt(p.floor_rel * zn2);
  for (int rr = warp; rr < 2 * pl; rr += nw) {
    const int j = rr >> 1, a = rr & 1 ? id_b(j) : id_a(j);
    if (a >= M) continue;
    // a total order (non-finite norms last), so the ranks are a permutation
    const double sg = s_sig[a];
    const double sa = sg >= 0.0 && isfinite(sg) ? sg : -1.0;
    int rank = 0;
    for (int b = lane; b < M; b += 32) {
      const double t = s_sig[b], sb = t >= 0.0 && isfinite(t) ? t : -1.0;
      rank += sb > sa || (sb == sa && b < a);
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
    if (lane == 0) {
      s_rank[a] = rank;
      s_inv[a] = sg > smin && sg > 0.0 ? 1.0 / sg : 0.0;
      if (sigma) sigma[a] = sg;
      if (idx && rank < p.k) idx[rank] = a;
    }
  }
  __syncthreads();
#pragma unroll 2
  for (int e = tid; e < 2 * pl * len; e += nt) {
    const int rr = p.conj_t ? e % (2 * pl) : e / len, c = p.conj_t ? e / (2 * pl) : e - rr * len;
    const int j = rr >> 1, a = rr & 1 ? id_b(j) : id_a(j);
    if (a >= M) continue;
    const C x = (rr & 1 ? second(j, CL ? R0 : 0) : first(j, CL ? R0 : 0))[c];
    const int rank = s_rank[a];
    const bool top = U && rank < p.k;
    const double sg = s_sig[a];
    if (c < N) {
      const C g = mkj<C>(x.x * down, x.y * down);
      if (Gout) Gout[(size_t)a * N + c] = g;
      if (top && p.m <= p.n) Rem[(size_t)rank * p.n + c] = g;       // U = WH^H, Rem = G
      if (top && p.m > p.n) {            // rows of Z^H: U = G^H / sigma, Rem = sigma WH
        const R is = (R)s_inv[a];
        U[(size_t)c * p.k + rank] = mkj<C>(g.x * is, -g.y * is);
      }
    } else {
      const int w = c - N;
      if (WHout) WHout[(size_t)a * M + w] = x;
      if (top && p.m <= p.n) U[(size_t)w * p.k + rank] = mkj<C>(x.x, -x.y);
      if (top && p.m > p.n) Rem[(size_t)rank * p.n + w] = mkj<C>(x.x * (R)sg, x.y * (R)sg);
    }
  }
  if (tid == 0 && !converged) *status = 1;   // the sweep limit, or an exchange that ran out
  if (cr == 0 && tid == 0) {
    if (counters) {
      counters[0] = counters[1] = 0;
      counters[2] = sweeps;
      counters[3] = rot_total;
    }
    if (flops)
      atomicAdd(flops, (double)sweeps * 0.5 * M * (M - 1) * 16.0 * N + (double)rot_total * 18.0 * (N + M));
  }
}

struct JacPlan {
  int cs = 0, pp = 0, order = 0;
  size_t bytes = 0;
};

// Places a CTA.  complex128: two (four pairs an SM wait for its FP64 unit:
// 64 clocks a warp-wide instruction; 64 rows 7.26 ms, on four places 7.62).
// complex64: one CTA up to twenty places, nine of long rows (pushing rows costs
// more than several CTAs save: 40 x 40 692 us, on a cluster of five 749; 40 x 200
// 1003 and 907), else four a CTA (96 x 96 2450 us, eight 2585, sixteen 3104).  More when sixteen CTAs need it, and one
// CTA alone where a cluster's rings (pp + 2 slots each) do not fit.
template <typename C>
bool jac_plan(int M, int N, JacPlan& p) {
  const bool c64 = sizeof(C) == sizeof(float2);
  const int P = (M + 1) / 2, pref = c64 ? 4 : 2;
  const size_t row = sizeof(C) * (size_t)((N + M + 1) & ~1);
  const bool staged = sizeof(C) * ((size_t)M * N + (size_t)M * M) <= kJacStaged;
  p.order = !staged ? kJacPlain32 : (M > 64 ? kJacStaged16 : kJacStaged32);
  if (P > (c64 ? (N + M <= 160 ? 20 : 9) : pref)) {
    p.pp = std::max(pref, (P + kJacMaxCluster - 1) / kJacMaxCluster);
    p.cs = (P + p.pp - 1) / p.pp;
    p.bytes = jac_header(M) + row * (2 * (p.pp + 2) + 1);
    if (p.bytes <= kJacSmemMax) return true;
  }
  p.pp = P;
  p.cs = 1;
  p.bytes = jac_header(M) + row * M;
  return p.bytes <= kJacSmemMax;
}

template <typename C, int ORD, bool CL>
cudaError_t jac_run(const JacPlan& p, const JacArgs& a, const C* Z, C* G, C* WH, double* sigma, int* idx, double* zn2,
                    int* counters, C* U, C* Rem, int* status, double* flops, cudaStream_t s) {
  auto kern = k_jac<C, ORD, CL>;
  static std::atomic<unsigned long long> done{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = 1ull << (dev & 63);
  if (!(done.load(std::memory_order_relaxed) & bit)) {
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kJacSmemMax)) != cudaSuccess)
      return e;
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) != cudaSuccess) return e;
    done.fetch_or(bit);
  }
  if (p.cs == 0) return cudaSuccess;     // (the attributes only)
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.cs, 1, 1);
  // (eight warps load and store short rows, all long ones)
  const int least = (a.M * (a.N + a.M)) / p.cs >= 8192 ? kJacWarps : 8;
  cfg.blockDim = dim3(32 * std::min(std::max(p.pp, least), kJacWarps), 1, 1);
  cfg.dynamicSmemBytes = p.bytes;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = p.cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = CL ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, a, Z, G, WH, sigma, idx, zn2, counters, U, Rem, status, flops);
}

template <typename C, int ORD>
cudaError_t jac_order(const JacPlan& p, bool cl, const JacArgs& a, const C* Z, C* G, C* WH, double* sigma, int* idx,
                      double* zn2, int* counters, C* U, C* Rem, int* status, double* flops, cudaStream_t s) {
  return cl ? jac_run<C, ORD, true>(p, a, Z, G, WH, sigma, idx, zn2, counters, U, Rem, status, flops, s)
            : jac_run<C, ORD, false>(p, a, Z, G, WH, sigma, idx, zn2, counters, U, Rem, status, flops, s);
}
template <typename C>
cudaError_t jac_pick(const JacPlan& p, bool cl, const JacArgs& a, const C* Z, C* G, C* WH, double* sigma, int* idx,
                     double* zn2, int* counters, C* U, C* Rem, int* status, double* flops, cudaStream_t s) {
  if (p.order == kJacStaged16)
    return jac_order<C, kJacStaged16>(p, cl, a, Z, G, WH, sigma, idx, zn2, counters, U, Rem, status, flops, s);
  if (p.order == kJacStaged32)
    return jac_order<C, kJacStaged32>(p, cl, a, Z, G, WH, sigma, idx, zn2, counters, U, Rem, status, flops, s);
  return jac_order<C, kJacPlain32>(p, cl, a, Z, G, WH, sigma, idx, zn2, counters, U, Rem, status, flops, s);
}

template <typename C>
cudaError_t jac_t(const C* Z, int ldz, bool conj_t, int M, int N, int k, C* G, C* WH, double* sigma, int* idx,
                  double* zn2, int* counters, int m, int n, C* U, C* Rem, double tol, double floor_rel,
                  int max_sweeps, int* status, cudaStream_t s) {
  JacPlan p;
  if (!jac_plan<C>(M, N, p)) return cudaErrorInvalidValue;
  KTimerScope timer(KC_JACOBI, s, 0.0);
  JacArgs a;
  a.M = M;
  a.N = N;
  a.pp = p.pp;
  a.ldz = ldz;
  a.conj_t = conj_t ? 1 : 0;
  a.m = m;
  a.n = n;
  a.k = k;
  a.tol = tol;
  a.floor_rel = floor_rel;
  a.max_sweeps = max_sweeps;
  return jac_pick<C>(p, p.cs > 1, a, Z, G, WH, sigma, idx, zn2, counters, U, Rem, status,
                     ktimer_device_flops(KC_JACOBI), s);
}

template <typename C>
cudaError_t jac_optin() {
  JacPlan p;
  JacArgs a = {};
  for (int order : {kJacPlain32, kJacStaged32, kJacStaged16})
    for (bool cl : {false, true}) {
      p.order = order;
      cudaError_t r = jac_pick<C>(p, cl, a, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr,
                                  nullptr, nullptr, nullptr, 0);
      if (r != cudaSuccess) return r;
    }
  return cudaSuccess;
}

}  // namespace

cudaError_t init_jac_attributes() {
  cudaError_t e = jac_optin<float2>();
  return e != cudaSuccess ? e : jac_optin<double2>();
}

bool jac_fits(int M, int N, size_t elem) {
  JacPlan p;
  return elem == sizeof(double2) ? jac_plan<double2>(M, N, p) : jac_plan<float2>(M, N, p);
}

cudaError_t launch_jac(const float2* Z, int ldz, bool conj_t, int M, int N, int k, float2* G, float2* WH,
                       double* sigma, int* idx, double* zn2, int* counters, int m, int n, float2* U, float2* Rem,
                       double tol, double floor_rel, int max_sweeps, int* status, cudaStream_t s) {
  return jac_t(Z, ldz, conj_t, M, N, k, G, WH, sigma, idx, zn2, counters, m, n, U, Rem, tol, floor_rel, max_sweeps,
               status, s);
}
cudaError_t launch_jac(const double2* Z, int ldz, bool conj_t, int M, int N, int k, double2* G, double2* WH,
                       double* sigma, int* idx, double* zn2, int* counters, int m, int n, double2* U, double2* Rem,
                       double tol, double floor_rel, int max_sweeps, int* status, cudaStream_t s) {
  return jac_t(Z, ldz, conj_t, M, N, k, G, WH, sigma, idx, zn2, counters, m, n, U, Rem, tol, floor_rel, max_sweeps,
               status, s);
}

}  // namespace bbp
