// One-sided (row) Jacobi SVD of small matrices on a cluster of CTAs (K3: the
// truncated splits of Sec. 1.1.3 and the reduced factors of the randomised
// truncation).
//
// The M rows of G (length N) are rotated pairwise until they are orthogonal,
// the same rotations accumulating in WH (M x M, from the identity): WH G_0 =
// G.  A row of G and its row of WH are one vector of N + M entries.
//
// Distribution: 2 C blocks of bs rows on C CTAs, two a CTA ("top", "bottom").
// A step rotates every pair (top i, bottom j): bs rounds of bs disjoint pairs,
// a warp a pair, top row i staying in warp i's registers over the rounds.
// Then the blocks move one place round the tournament (Brent and Luk's
// ordering of blocks), pushed into the neighbours' shared memory; after 2 C -
// 1 steps every two blocks have met and each is back home.  The pairs within
// a block are rotated when a sweep begins.  A block is pushed into one of
// three buffers in turn, completing on the receiver's mbarrier: a neighbour
// pushes at the end of step s into the buffer whose last contents left at the
// end of step s - 2, which its own push at the end of step s - 1 proves, so
// no other handshake is needed.
//
// A rotation is given by tau = t e^{i phi} (t = tan theta), x' = c (x - tau
// y), y' = c (y + conj(tau) x).  Any tau gives a unitary step once c = 1 /
// sqrt(1 + |tau|^2) holds to working precision, so tau itself is formed in
// float from the float images of the sums in both types (an error d of the
// angle leaves d times the pair's inner product, which the next sweep takes);
// c, sigma = c tau and the squared norms (al' = al - t |g|, be' = be + t |g|,
// taken anew when they cancel and in every sweep) are in the element's type.
//
// What bounds it: complex128, the FP64 pipe (a warp-wide multiply-add takes
// 64 clocks of its sub-partition): 4 for the inner product and 12 for the
// rotation per 32 entries, about 20 a pair besides, so four pairs a CTA, one
// per sub-partition, and as many CTAs as that gives; complex64, the chain of
// one reduction and the scalars per round (about 600 clocks).
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
constexpr size_t kJacSmemMax = 227 * 1024;

template <typename C> struct RealJ;
template <> struct RealJ<double2> { using T = double; };
template <> struct RealJ<float2> { using T = float; };
template <typename C> __device__ __forceinline__ C mkj(typename RealJ<C>::T re, typename RealJ<C>::T im) {
  C r;
  r.x = re;
  r.y = im;
  return r;
}

// float image of x (about six digits in double, by its high word: no FP64
// conversion), and the exact double of a float
__device__ __forceinline__ float image(float x) { return x; }
__device__ __forceinline__ float image(double x) {
  const int hi = __double2hiint(x);
  const int e = ((hi >> 20) & 0x7ff) - 1023 + 127;
  if (e <= 0) return 0.f;
  if (e >= 255) return __int_as_float((hi & 0x80000000) | 0x7f800000);
  return __int_as_float((hi & 0x80000000) | (e << 23) | ((hi & 0xfffff) << 3));
}
__device__ __forceinline__ void widen(float x, float& r) { r = x; }
__device__ __forceinline__ void widen(float x, double& r) {
  const int b = __float_as_int(x);
  const int e = (b >> 23) & 0xff;
  r = e == 0 ? 0.0
             : __hiloint2double((b & 0x80000000) | ((e - 127 + 1023) << 20) | ((b & 0x7fffff) >> 3), (b & 7) << 29);
}
// x 2^-e and the exponent e of the larger of two magnitudes (double: so that
// the images are in float's range)
__device__ __forceinline__ int top_exponent(double a, double b) {
  return max((__double2hiint(a) >> 20) & 0x7ff, (__double2hiint(b) >> 20) & 0x7ff) - 1023;
}
__device__ __forceinline__ float image_scaled(double x, int e) {   // image of x 2^-e
  const int hi = __double2hiint(x), ex = ((hi >> 20) & 0x7ff) - 1023 + 127 - e;
  if (((hi >> 20) & 0x7ff) == 0 || ex <= 0) return 0.f;
  if (ex >= 255) return __int_as_float((hi & 0x80000000) | 0x7f7fffff);
  return __int_as_float((hi & 0x80000000) | (ex << 23) | ((hi & 0xfffff) << 3));
}
__device__ __forceinline__ int top_exponent(float, float) { return 0; }
__device__ __forceinline__ float image_scaled(float x, int) { return x; }

// 1 / sqrt(q), q in [1, 2]: a float seed and Newton (float) or one cubically
// convergent Householder step (double)
__device__ __forceinline__ float inv_root(float q) {
  const float y = rsqrtf(q);
  return fmaf(0.5f * y, fmaf(-q * y, y, 1.f), y);
}
__device__ __forceinline__ double inv_root(double q) {
  double y;
  widen(rsqrtf(image(q)), y);
  const double e = fma(-q * y, y, 1.0);          // (six digits in: one step leaves 1e-18)
  return fma(y * e, fma(0.375, e, 0.5), y);
}

// two sums over the warp, both in every lane
template <typename R>
__device__ __forceinline__ void sum2(R& a, R& b, int lane) {
  const bool up = lane & 16;
  R v = (up ? b : a) + __shfl_xor_sync(0xffffffffu, up ? a : b, 16);
#pragma unroll
  for (int o = 8; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  a = __shfl_sync(0xffffffffu, v, 0);
  b = __shfl_sync(0xffffffffu, v, 16);
}
template <typename R>
__device__ __forceinline__ R sum1(R v) {
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

struct JacArgs {
  int M, N, bs, nb;                      // rows, row length, rows a block, buffers (1 or 3)
  int ldz, conj_t;                       // G_0[a][c] = Z[a ldz + c], or conj(Z[c ldz + a])
  int m, n, k;                           // exact SVD outputs (U, Rem not null): U m x k, Rem k x n
  double tol, floor_rel;
  int max_sweeps;
};

// E: entries of a row (N + M) a lane holds (0: rows stay in shared memory).
template <typename C, int E, bool CL>
__global__ void __launch_bounds__(512, 1) k_jac(JacArgs p, const C* __restrict__ Z, C* __restrict__ Gout,
                                                C* __restrict__ WHout, double* __restrict__ sigma,
                                                int* __restrict__ idx, double* __restrict__ zn2_out, int* counters,
                                                C* __restrict__ U, C* __restrict__ Rem, int* status, double* flops) {
  using R = typename RealJ<C>::T;
  cg::cluster_group cl = cg::this_cluster();
  const int cs = CL ? (int)cl.num_blocks() : 1, cr = CL ? (int)cl.block_rank() : 0;
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5;
  const int M = p.M, N = p.N, bs = p.bs, len = N + M;
  const int ld = (len + 1) & ~1;         // entries of a row in shared memory (16-byte rows)
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const uint32_t bars = saddr(smem_raw);            // blocks (three), counts (two)
  volatile int* failed = (volatile int*)(smem_raw + 48);
  int* s_rot = (int*)(smem_raw + 52);
  double* s_sum = (double*)(smem_raw + 64);         // [2 cs] sums and sweep counts of the CTAs
  int* s_cnt = (int*)(s_sum + kJacMaxCluster);      // [2][cs][4]
  double* s_sig = (double*)(smem_raw + 64 + 128 + 512);   // [2 cs bs] singular values (in home order)
  const size_t hdr = 64 + 128 + 512 + sizeof(double) * (size_t)(2 * cs * bs);
  // buffer b: two blocks of bs rows, then their squared norms
  const uint32_t blk = (uint32_t)(sizeof(C) * (size_t)ld * bs), nrm = (uint32_t)((sizeof(R) * bs + 15) & ~15u);
  const uint32_t half = blk + nrm, buf = 2 * half;
  unsigned char* base = smem_raw + ((hdr + 15) & ~size_t(15));
  auto rows = [&](int b, int h) { return (C*)(base + (size_t)b * buf + (size_t)h * half); };
  auto norms = [&](int b, int h) { return (R*)(base + (size_t)b * buf + (size_t)h * half + blk); };
  const C zero = mkj<C>(0, 0);
  if (tid == 0) {
    for (int q = 0; q < 5; ++q) bar_init(bars + 8 * q);
    *failed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }

  // ---- load: block 2 cr at the top, 2 cr + 1 at the bottom
  double part = 0.0;
  for (int rr = warp; rr < 2 * bs; rr += nt >> 5) {
    const int a = 2 * cr * bs + rr;
    C* row = rows(0, rr / bs) + (size_t)(rr % bs) * ld;
    for (int c = lane; c < ld; c += 32) {
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
      row[c] = v;
    }
  }
  part = sum1(part);
  __syncthreads();
  if (lane == 0) s_sig[warp] = part;     // (at most 2 bs warps: bs of them)
  __syncthreads();
  if (tid == 0) {
    double s = 0.0;
    for (int w = 0; w < nt >> 5; ++w) s += s_sig[w];
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
  // the rows are scaled by a power of two so that ||G|| is near one
  int ex2 = 0;
  if (zn2 > 0.0 && isfinite(zn2)) {
    int e;
    frexp(zn2, &e);
    ex2 = e / 2;
    if (sizeof(R) == 4) ex2 = min(max(ex2, -120), 120);
  }
  const R up = (R)ldexp(1.0, -ex2), down = (R)ldexp(1.0, ex2);
  const R floor = (R)(p.floor_rel * (zn2 * ldexp(1.0, -2 * ex2)));
  for (int e = tid; e < 2 * bs * N; e += nt) {
    const int rr = e / N, c = e - rr * N;
    C* x = rows(0, rr / bs) + (size_t)(rr % bs) * ld + c;
    *x = mkj<C>(x->x * up, x->y * up);
  }
  __syncthreads();

  const R far = sizeof(R) == 8 ? (R)1e-60 : (R)1e-30;
  const float ftol = (float)p.tol;
  int rot = 0;
  // one pair: x (squared norm al) in registers, or at xr when rows are too
  // long for that (E = 0), and y at row (squared norm at nb)
  constexpr int EX = E > 0 ? E : 1;
  auto pair = [&](C (&x)[EX], C* xr, R& al, C* row, R* nb) {
    C y[EX];
    R gx = 0, gy = 0;
    if constexpr (E > 0) {
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int c = lane + 32 * e;
        y[e] = c < len ? row[c] : zero;
        if (c < N) {                     // x conj(y)
          gx = fma(x[e].y, y[e].y, fma(x[e].x, y[e].x, gx));
          gy = fma(-x[e].x, y[e].y, fma(x[e].y, y[e].x, gy));
        }
      }
    } else {
      for (int c = lane; c < N; c += 32) {
        const C u = xr[c], v = row[c];
        gx = fma(u.y, v.y, fma(u.x, v.x, gx));
        gy = fma(-u.x, v.y, fma(u.y, v.x, gy));
      }
    }
    const R be = *nb;
    sum2(gx, gy, lane);
    // negligible against the rows' norms, a row below eps ||Z|| (it carries
    // nothing at working precision, and would never meet the first test), or
    // norms too far apart to affect each other
    const int ge = top_exponent(gx, gy);
    const float fx = image_scaled(gx, ge), fy = image_scaled(gy, ge);
    const float g2 = fx * fx + fy * fy;
    if (g2 == 0.f) return;
    const float ig = rsqrtf(g2), g = g2 * ig;
    float gs = g;                        // g on the scale of the norms
    if (sizeof(R) == 8) gs = ldexpf(g, max(ge, -200));
    if (gs * rsqrtf(image(al)) * rsqrtf(image(be)) <= ftol) return;
    const R lo = al < be ? al : be, hi = al < be ? be : al;
    if (lo <= floor || lo <= far * hi) return;
    const float zeta = 0.5f * image_scaled(be - al, ge) * ig;
    const float az = fabsf(zeta);
    const float t = az > 1e15f ? __fdividef(0.5f, az) : __fdividef(1.f, az + sqrtf(fmaf(az, az, 1.f)));
    const float ft = copysignf(t, zeta) * ig;
    R tx, ty;
    widen(ft * fx, tx);
    widen(ft * fy, ty);
    const R c = inv_root(fma(tx, tx, fma(ty, ty, (R)1)));
    const R sx = c * tx, sy = c * ty;
    const R d = fma(tx, gx, ty * gy);    // t |g|
    auto turn = [&](C& u, C& v) {        // c u - sigma v, c v + conj(sigma) u
      const C a = u, b = v;
      u.x = fma(sy, b.y, fma(-sx, b.x, c * a.x));
      u.y = fma(-sy, b.x, fma(-sx, b.y, c * a.y));
      v.x = fma(sy, a.y, fma(sx, a.x, c * b.x));
      v.y = fma(-sy, a.x, fma(sx, a.y, c * b.y));
    };
    if constexpr (E > 0) {
#pragma unroll
      for (int e = 0; e < E; ++e) {
        turn(x[e], y[e]);
        const int q = lane + 32 * e;
        if (q < len) row[q] = y[e];
      }
    } else {
      for (int q = lane; q < len; q += 32) {
        C u = xr[q], v = row[q];
        turn(u, v);
        xr[q] = u;
        row[q] = v;
      }
    }
    R na = al - d, nbe = be + d;
    if (na < (R)0.25 * al || nbe < (R)0.25 * be) {   // cancelled: take both anew
      R a = 0, b = 0;
      if constexpr (E > 0) {
#pragma unroll
        for (int e = 0; e < E; ++e)
          if (lane + 32 * e < N) {
            a = fma(x[e].y, x[e].y, fma(x[e].x, x[e].x, a));
            b = fma(y[e].y, y[e].y, fma(y[e].x, y[e].x, b));
          }
      } else {
        for (int q = lane; q < N; q += 32) {
          const C u = xr[q], v = row[q];
          a = fma(u.y, u.y, fma(u.x, u.x, a));
          b = fma(v.y, v.y, fma(v.x, v.x, b));
        }
      }
      sum2(a, b, lane);
      na = a;
      nbe = b;
    }
    al = na;
    __syncwarp();
    if (lane == 0) *nb = nbe;
    ++rot;
  };
  auto load_row = [&](C (&x)[EX], const C* r) {
    if constexpr (E > 0) {
#pragma unroll
      for (int e = 0; e < E; ++e) x[e] = lane + 32 * e < len ? r[lane + 32 * e] : zero;
    }
  };
  auto store_row = [&](const C (&x)[EX], C* r) {
    if constexpr (E > 0) {
#pragma unroll
      for (int e = 0; e < E; ++e)
        if (lane + 32 * e < len) r[lane + 32 * e] = x[e];
    }
  };

  int sweeps = 0, rot_total = 0, cur = 0;
  uint32_t ph = 0, ph_cnt = 0;           // phases of the block barriers and of the counts
  bool converged = false;
  C x[EX];
  const int steps = 2 * cs - 1;
  while (sweeps < p.max_sweeps) {
    rot = 0;
    // squared norms, and the pairs within each block: warp w < bs / 2 works
    // on the top block, the others on the bottom one
    for (int rr = warp; rr < 2 * bs; rr += nt >> 5) {
      const C* row = rows(cur, rr / bs) + (size_t)(rr % bs) * ld;
      R a = 0;
      for (int c = lane; c < N; c += 32) a = fma(row[c].y, row[c].y, fma(row[c].x, row[c].x, a));
      a = sum1(a);
      if (lane == 0) norms(cur, rr / bs)[rr % bs] = a;
    }
    __syncthreads();
    const int bp = bs + (bs & 1), hp = bp / 2;       // rounds of a block's own tournament
    for (int r = 0; r < bp - 1; ++r) {
      for (int w = warp; w < 2 * hp; w += nt >> 5) {
        const int h = w / hp, q = w % hp;
        const int i = q == 0 ? bp - 1 : (r + q) % (bp - 1), j = q == 0 ? r : (r - q + bp - 1) % (bp - 1);
        if (i < bs && j < bs) {
          C* rx = rows(cur, h) + (size_t)i * ld;
          R al = norms(cur, h)[i];
          load_row(x, rx);
          const int was = rot;
          pair(x, rx, al, rows(cur, h) + (size_t)j * ld, norms(cur, h) + j);
          if (rot != was) {
            store_row(x, rx);
            if (lane == 0) norms(cur, h)[i] = al;
          }
        }
      }
      __syncthreads();
    }
    // the blocks' tournament
    for (int s = 0; s < steps; ++s) {
      R al = 0;
      C* rx = rows(cur, 0) + (size_t)min(warp, bs - 1) * ld;
      if (warp < bs) {
        al = norms(cur, 0)[warp];
        load_row(x, rx);
      }
      for (int r = 0; r < bs; ++r) {
        if (warp < bs) {
          int j = warp + r;
          if (j >= bs) j -= bs;
          pair(x, rx, al, rows(cur, 1) + (size_t)j * ld, norms(cur, 1) + j);
        }
        __syncthreads();
      }
      if (warp < bs) {
        store_row(x, rx);
        if (lane == 0) norms(cur, 0)[warp] = al;
      }
      if constexpr (CL) {
        __syncthreads();
        // top blocks move right (the first stays, the last turns), bottom
        // blocks left (the first turns)
        const int nxt = cur == 2 ? 0 : cur + 1;
        const bool keep_top = cr == 0, turn = cr == cs - 1;
        if (tid == 0) bar_expect(bars + 8 * nxt, half * (uint32_t)((cr > 0) + (cr < cs - 1)));
        const uint32_t src = saddr(base) + cur * buf, dst = saddr(base) + nxt * buf;
        const uint32_t bt = remote(bars + 8 * nxt, min(cr + 1, cs - 1)), bb = remote(bars + 8 * nxt, cr == 0 ? 1 : cr - 1);
        const uint32_t dt = remote(dst, min(cr + 1, cs - 1));                  // neighbour's top
        const uint32_t db = remote(cr == 0 ? dst : dst + half, cr == 0 ? 1 : cr - 1);   // its bottom (its top from CTA 0)
        for (uint32_t o = 16 * tid; o < half; o += 16 * nt) {
          float4 v = lds128(src + o);
          if (keep_top) sts128(dst + o, v);
          else if (turn) sts128(dst + half + o, v);
          else push128(dt + o, bt, v);
          v = lds128(src + half + o);
          push128(db + o, bb, v);
        }
        cur = nxt;
        bar_wait(bars + 8 * cur, (ph >> cur) & 1u, failed);
        ph ^= 1u << cur;
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
      if (tid == 0) bar_expect(bars + 8 * (3 + par), 16u * cs);
      if (tid < cs)
        push128(remote(saddr(s_cnt + (par * kJacMaxCluster + cr) * 4), tid), remote(bars + 8 * (3 + par), tid),
                make_float4(__int_as_float(total), 0.f, 0.f, 0.f));
      bar_wait(bars + 8 * (3 + par), (ph_cnt >> par) & 1u, failed);
      ph_cnt ^= 1u << par;
      total = 0;
      for (int q = 0; q < cs; ++q) total += s_cnt[(par * kJacMaxCluster + q) * 4];
    }
    __syncthreads();
    ++sweeps;
    rot_total += total;
    if (total == 0 || *failed) { converged = total == 0; break; }
  }

  // ---- row norms in double, ranks by size, outputs
  for (int rr = warp; rr < 2 * bs; rr += nt >> 5) {
    const C* row = rows(cur, rr / bs) + (size_t)(rr % bs) * ld;
    double a = 0.0;
    for (int c = lane; c < N; c += 32) a += (double)row[c].x * row[c].x + (double)row[c].y * row[c].y;
    a = sum1(a);
    if (lane == 0) s_sig[2 * cr * bs + rr] = sqrt(a) * ldexp(1.0, ex2);
  }
  __syncthreads();
  if constexpr (CL) {
    cl.sync();
    for (int e = tid; e < 2 * cs * bs; e += nt) {
      const int q = e / (2 * bs);
      if (q != cr) s_sig[e] = cl.map_shared_rank(s_sig, q)[e];
    }
    cl.sync();                           // (no remote access after this)
  }
  const double smin = sqrt(p.floor_rel * zn2);
  for (int rr = warp; rr < 2 * bs; rr += nt >> 5) {
    const int a = 2 * cr * bs + rr;
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
    const C* g = rows(cur, rr / bs) + (size_t)(rr % bs) * ld;
    const C* w = g + N;
    if (sigma && lane == 0) sigma[a] = sg;
    if (idx && lane == 0 && rank < p.k) idx[rank] = a;
    if (Gout)
      for (int c = lane; c < N; c += 32) Gout[(size_t)a * N + c] = mkj<C>(g[c].x * down, g[c].y * down);
    if (WHout)
      for (int c = lane; c < M; c += 32) WHout[(size_t)a * M + c] = w[c];
    if (U && rank < p.k) {
      if (p.m <= p.n) {                  // U = WH^H, Rem = G
        for (int c = lane; c < M; c += 32) U[(size_t)c * p.k + rank] = mkj<C>(w[c].x, -w[c].y);
        for (int c = lane; c < N; c += 32) Rem[(size_t)rank * p.n + c] = mkj<C>(g[c].x * down, g[c].y * down);
      } else {                           // rows of Z^H: U = G^H / sigma, Rem = sigma WH
        const R is = sg > smin && sg > 0.0 ? (R)(1.0 / sg) : (R)0, s1 = (R)sg;
        for (int c = lane; c < N; c += 32)
          U[(size_t)c * p.k + rank] = mkj<C>(g[c].x * down * is, -(g[c].y * down) * is);
        for (int c = lane; c < M; c += 32) Rem[(size_t)rank * p.n + c] = mkj<C>(w[c].x * s1, w[c].y * s1);
      }
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
  int cs = 0, bs = 0, nb = 0, e = 0;
  size_t bytes = 0;
};

template <typename C>
bool jac_fit(int M, int N, int cs, JacPlan& p) {
  static const int kE[] = {2, 4, 6, 8, 12};
  const size_t R = sizeof(C) / 2;
  p.cs = cs;
  p.bs = (M + 2 * cs - 1) / (2 * cs);
  p.nb = cs > 1 ? 3 : 1;
  const int per = (N + M + 31) / 32;
  p.e = 0;
  for (int e : kE)
    if (e >= per && (sizeof(C) == sizeof(float2) || e <= 8)) { p.e = e; break; }
  if (p.bs > 16) return false;
  const size_t ld = (size_t)((N + M + 1) & ~1);
  const size_t half = sizeof(C) * ld * p.bs + ((R * p.bs + 15) & ~size_t(15));
  const size_t hdr = 64 + 128 + 512 + sizeof(double) * (size_t)std::max(2 * cs * p.bs, 16);
  p.bytes = ((hdr + 15) & ~size_t(15)) + 2 * half * p.nb;
  return p.bytes <= kJacSmemMax;
}

// CTAs of an M-row problem: complex128 four pairs a CTA (one per FP64
// sub-partition), complex64 eight.
template <typename C>
bool jac_plan(int M, int N, JacPlan& p) {
  const int pairs = sizeof(C) == sizeof(float2) ? 8 : 4;
  const int want = std::min(kJacMaxCluster, std::max(1, (M + 2 * pairs - 1) / (2 * pairs)));
  for (int cs = want; cs <= kJacMaxCluster; ++cs)
    if (jac_fit<C>(M, N, cs, p)) return true;
  for (int cs = want - 1; cs >= 1; --cs)
    if (jac_fit<C>(M, N, cs, p)) return true;
  return false;
}

template <typename C, int E, bool CL>
cudaError_t jac_run(const JacPlan& p, const JacArgs& a, const C* Z, C* G, C* WH, double* sigma, int* idx, double* zn2,
                    int* counters, C* U, C* Rem, int* status, double* flops, cudaStream_t s) {
  auto kern = k_jac<C, E, CL>;
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
  cfg.blockDim = dim3(32 * std::max(p.bs + (p.bs & 1), 1), 1, 1);
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

template <typename C>
cudaError_t jac_pick(const JacPlan& p, bool cl, const JacArgs& a, const C* Z, C* G, C* WH, double* sigma, int* idx,
                     double* zn2, int* counters, C* U, C* Rem, int* status, double* flops, cudaStream_t s) {
#define BBP_JAC(E)                                                                                       \
  case E:                                                                                                \
    return cl ? jac_run<C, E, true>(p, a, Z, G, WH, sigma, idx, zn2, counters, U, Rem, status, flops, s)  \
              : jac_run<C, E, false>(p, a, Z, G, WH, sigma, idx, zn2, counters, U, Rem, status, flops, s)
  switch (p.e) {
    BBP_JAC(0);
    BBP_JAC(2);
    BBP_JAC(4);
    BBP_JAC(6);
    BBP_JAC(8);
    default: break;
  }
  if constexpr (sizeof(C) == sizeof(float2)) {
    switch (p.e) {
      BBP_JAC(12);
      default: break;
    }
  }
#undef BBP_JAC
  return cudaErrorInvalidValue;
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
  a.bs = p.bs;
  a.nb = p.nb;
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
  for (int e : {0, 2, 4, 6, 8, 12})
    for (bool cl : {false, true}) {
      if (e > 8 && sizeof(C) != sizeof(float2)) continue;
      p.e = e;
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
