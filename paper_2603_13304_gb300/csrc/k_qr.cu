// Blocked Householder QR (Sec. 2.3.3: the canonical moves, the message
// distances and the orthonormalisations of the truncation), one CTA or a
// thread-block cluster per panel.
//
// A panel A (m x n, row-major) is cut into row slices, one per CTA of a
// cluster of cs <= 16 CTAs; each slice stays in that CTA's shared memory
// (column-major, odd column stride) for the whole factorisation.  The columns
// go in blocks of kNB = 8:
//  steps   the block's eight columns are held in registers (complex64: a
//          thread per row; complex128: four warps per 32 rows, two columns
//          each, so that a step's FP64 work spreads over the SM's four
//          sub-partitions).  Householder step J needs the norm of x (column J
//          below row J) and x^H a_c for the block's other columns only:
//          sixteen real sums, one reduction tree over the warp, one exchange
//          over the CTA's warps and, in a cluster, one push of the CTA's sums
//          (and of row J, from its owner) into every CTA's receive buffer,
//          completing on that CTA's mbarrier.  One warp of each CTA then
//          forms the reflector (from the same values in every CTA); the sums
//          against the block's earlier reflectors give V^H V, from which
//          another warp builds T of the compact WY form (T_jj = tau_j,
//          T_0:j,j = -tau_j T_0:j,0:j (V^H V)_0:j,j) beside the next steps.
//  update  the columns right of the block take I - V T^H V^H as two passes
//          over shared memory, W = V^H A and A -= V F with F = T^H W.  In a
//          cluster the partial W of column c go to CTA c mod cs, which sums
//          them in rank order, multiplies and pushes F to every CTA.
// Q = H_0 ... H_{k-1} [I; 0] is formed backwards in place by the same two
// passes with T in place of T^H.
//
// Convention: H = I - tau v v^H, v_j = 1, R has a real diagonal beta_j, the
// factorisation applies H_j^H.  complex64 columns are scaled by a power of
// two near their largest magnitude when they are loaded and R is scaled back
// when it is stored (both exact), so that their squares neither overflow nor
// underflow and the complex64 kernel does no FP64 arithmetic.
//
// What bounds it: a step is a chain of one reduction tree, the exchange, a
// square root and two reciprocals (about 2000 clocks in complex64 on a
// cluster, 6000 in complex128); the O(m n^2) work runs in the two passes,
// bound by FMA issue and shared-memory bandwidth, or, in complex128, by the
// FP64 rate of the CTA's SM (two multiply-adds a clock).  The column-by-column
// form (every trailing column dotted and updated once per step, a cluster
// barrier per step) spent 4.2 us a step on instruction issue and barriers.
// Measured with Q, us, column by column and blocked: complex64 2304 x 96 on
// nine CTAs 648 and 326, 2304 x 64 358 and 187, 432 x 40 182 (one CTA) and 86;
// complex128 512 x 64 on sixteen CTAs 1530 and 615, 32 x 8 66 and 33.
#include <cooperative_groups.h>

#include <algorithm>
#include <atomic>
#include <cstdint>
#include <type_traits>

#include "kernels.h"
#include "push.h"

namespace cg = cooperative_groups;

namespace bbp {

namespace {

template <typename C> struct RealT;
template <> struct RealT<double2> { using T = double; };
template <> struct RealT<float2> { using T = float; };

template <typename C> __device__ __forceinline__ C mk(typename RealT<C>::T re, typename RealT<C>::T im) {
  C r;
  r.x = re;
  r.y = im;
  return r;
}
template <typename C> __device__ __forceinline__ C mul(C a, C b) {
  return mk<C>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
template <typename C> __device__ __forceinline__ C mulc(C a, C b) {   // conj(a) b
  return mk<C>(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x);
}
template <typename C> __device__ __forceinline__ C add(C a, C b) { return mk<C>(a.x + b.x, a.y + b.y); }
// s += conj(a) b, s -= a b, s += a b, as chains of fused multiply-adds (a sum
// of products added at the end would take half as many instructions again)
template <typename C> __device__ __forceinline__ void fmac(C& s, C a, C b) {
  s.x = fma(a.y, b.y, fma(a.x, b.x, s.x));
  s.y = fma(-a.y, b.x, fma(a.x, b.y, s.y));
}
template <typename C> __device__ __forceinline__ void fnma(C& s, C a, C b) {
  s.x = fma(a.y, b.y, fma(-a.x, b.x, s.x));
  s.y = fma(-a.y, b.x, fma(-a.x, b.y, s.y));
}
template <typename C> __device__ __forceinline__ void fma2(C& s, C a, C b) {
  s.x = fma(-a.y, b.y, fma(a.x, b.x, s.x));
  s.y = fma(a.y, b.x, fma(a.x, b.y, s.y));
}

constexpr int kNB = 8;                   // reflectors a block
constexpr int kQrThreads = 512;
constexpr size_t kQrSmemMax = 227 * 1024;

// Sixteen sums over the warp, halving the set at every level (16 shuffles in
// all); lane L returns sum L >> 1.
template <typename R>
__device__ __forceinline__ R reduce16(R (&v)[16], int lane) {
#pragma unroll
  for (int w = 8; w >= 1; w >>= 1) {
    const bool up = (lane & (2 * w)) != 0;
#pragma unroll
    for (int q = 0; q < w; ++q) {
      const R send = up ? v[q] : v[q + w];
      const R keep = up ? v[q + w] : v[q];
      v[q] = keep + __shfl_xor_sync(0xffffffffu, send, 2 * w);
    }
  }
  return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// Pushes sixteen values, value i in lane src0 + i, as sixteen-byte chunks to
// the same offset of CTAs q0, q0 + dq, ... < cs: the calling lanes take chunk
// `chunk` of four (complex64) or eight (complex128).  Every lane of the warp
// takes part in the shuffles.
__device__ __forceinline__ void push16(float my, int src0, int chunk, uint32_t at, uint32_t bar, bool on, int q0,
                                       int dq, int cs) {
  const float v0 = __shfl_sync(0xffffffffu, my, src0 + 4 * chunk), v1 = __shfl_sync(0xffffffffu, my, src0 + 4 * chunk + 1);
  const float v2 = __shfl_sync(0xffffffffu, my, src0 + 4 * chunk + 2), v3 = __shfl_sync(0xffffffffu, my, src0 + 4 * chunk + 3);
  if (on)
    for (int q = q0; q < cs; q += dq) push(remote(at + 16 * chunk, q), remote(bar, q), v0, v1, v2, v3);
}
__device__ __forceinline__ void push16(double my, int src0, int chunk, uint32_t at, uint32_t bar, bool on, int q0,
                                       int dq, int cs) {
  const double v0 = __shfl_sync(0xffffffffu, my, src0 + 2 * chunk), v1 = __shfl_sync(0xffffffffu, my, src0 + 2 * chunk + 1);
  if (on)
    for (int q = q0; q < cs; q += dq) push(remote(at + 16 * chunk, q), remote(bar, q), v0, v1);
}

// Shared memory of one CTA: byte offsets after the slice (n columns of ld).
struct QrLayout {
  size_t bars, part, rowl, recv, rowb, step, svec, xcol, wbuf, fbuf, fown, sv, tau, scale, dbuf, bytes;
};
constexpr int kDotGroups = 2;            // complex128: 32-column groups in one trip of the W pass
template <typename C>
__host__ __device__ inline QrLayout qr_layout(int rows, int n, int k, int cs, bool want_q, bool dots_by_column) {
  const size_t R = sizeof(C) / 2;
  const bool c64 = sizeof(C) == 8;
  QrLayout L;
  size_t o = sizeof(C) * (size_t)(rows | 1) * n;
  o = (o + 15) & ~size_t(15);
  L.bars = o; o += 48;                     // four mbarriers (steps by parity, W, F), the failure mark
  L.part = o; o += R * (kQrThreads / 32) * 16;   // partial sums of a step
  L.rowl = o; o += R * 16;                 // row J, in its owner
  L.recv = o; o += cs > 1 ? R * 2 * cs * 16 : 0;   // [parity][source][16]
  L.rowb = o; o += cs > 1 ? R * 2 * 16 : 0;
  L.step = o; o += R * 32;                 // sc, the new diagonal, the block's factors or tau
  L.svec = o; o += R * 2 * 16;             // [parity] V^H V of the step's column
  L.xcol = o; o += c64 ? 0 : sizeof(C) * 2 * rows;   // [parity] x of the step
  L.wbuf = o; o += cs > 1 ? R * 16 * (size_t)cs * ((n + cs - 1) / cs) : 0;   // [source][own column][16]
  L.fbuf = o; o += R * 16 * (size_t)n;     // W, then F, by column
  L.fown = o; o += R * 16 * kNB;
  const size_t ks = want_q ? (k + kNB - 1) / kNB * kNB : kNB;   // every block's when Q is formed, else one
  L.sv = o; o += sizeof(C) * ks * kNB;   // per block: T above the diagonal, the top rows of V below it
  L.tau = o; o += sizeof(C) * ks;
  L.scale = o; o += c64 ? sizeof(float) * (size_t)((n + 3) & ~3) : 0;   // powers of two of the columns
  L.dbuf = o; o += dots_by_column ? R * kDotGroups * 4 * 16 * 32 : 0;
  L.bytes = o;
  return L;
}

// r = sqrt(q) and ir = 1 / sqrt(q); 1 / d.  A float seed and one Newton step
// (float) or one cubically convergent Householder step (double, with the
// exponent taken out so that the seed is in float's range), r with one more
// Newton correction.  The IEEE square root and divisions are longer dependent
// chains, which every step would wait for.
__device__ __forceinline__ void root(float q, float& r, float& ir) {
  float y = rsqrtf(q);
  y = fmaf(0.5f * y, fmaf(-q * y, y, 1.f), y);
  r = q * y;
  r = fmaf(fmaf(-r, r, q), 0.5f * y, r);
  ir = fmaf(y, fmaf(-r, y, 1.f), y);
}
__device__ __forceinline__ double exp_add(double x, int e) {   // x 2^e, all normal
  return __hiloint2double(__double2hiint(x) + (e << 20), __double2loint(x));
}
__device__ __forceinline__ void root(double q, double& r, double& ir) {
  const int h = ((((__double2hiint(q) >> 20) & 0x7ff) - 1023) & ~1) / 2;
  q = exp_add(q, -2 * h);                // in [1, 4)
  double y = (double)rsqrtf((float)q);
  const double e = fma(-q * y, y, 1.0);
  y = fma(y * e, fma(0.375, e, 0.5), y);
  r = q * y;
  r = fma(fma(-r, r, q), exp_add(y, -1), r);
  ir = exp_add(y, -h);
  r = exp_add(r, h);
}
__device__ __forceinline__ float recip(float d) {
  const float y = __fdividef(1.f, d);
  return fmaf(y, fmaf(-d, y, 1.f), y);
}
__device__ __forceinline__ double recip(double d) {
  const int h = ((__double2hiint(d) >> 20) & 0x7ff) - 1023;
  d = exp_add(d, -h);
  const double y = (double)__fdividef(1.f, (float)d);
  const double e = fma(-d, y, 1.0);
  return exp_add(fma(y, fma(e, e, e), y), -h);
}
// largest sum of squares the reflector is formed from, and the smallest
template <typename R> __device__ __forceinline__ bool in_range(R q);
template <> __device__ __forceinline__ bool in_range<float>(float q) { return q > 1e-36f && q < 1e37f; }
template <> __device__ __forceinline__ bool in_range<double>(double q) {   // 2^-960 .. 2^960, by the exponent
  const int h = (__double2hiint(q) >> 20) & 0xfff;
  return h > 63 && h < 1983;
}

// The reflector of x (norm^2 S) below alpha = (ar, ai): tau, sc = 1 / (alpha -
// beta) and the new diagonal; beta = -sign(ar) |(alpha, x)|.  Columns out of
// range (not finite, or negligible) are left as they are: tau = sc = 0.
template <typename C, typename R>
__device__ __forceinline__ void reflector(R S, R ar, R ai, C& tau, C& sc, C& diag) {
  tau = sc = mk<C>(0, 0);
  diag = mk<C>(ar, ai);
  const R b2 = ai * ai, q = fma(ar, ar, b2 + S);
  if ((S == 0 && ai == 0) || !in_range(q)) return;
  R nb, inb;
  root(q, nb, inb);
  const R bs = -copysign(nb, ar), ibs = -copysign(inb, ar);
  const R dx = ar - bs, idd = recip(fma(dx, dx, b2));   // 1 / (alpha - beta) = conj(d) / |d|^2
  tau = mk<C>(-dx * ibs, -ai * ibs);
  sc = mk<C>(dx * idd, -ai * idd);
  diag = mk<C>(bs, 0);
}

// Sum over cnt <= 16 sources of value lane & 15 (sources of 16 values at p).
template <typename R>
__device__ __forceinline__ R combine(const R* p, int cnt, int lane) {
  R v[8];
  const R* s = p + (lane >> 4) * 16 + (lane & 15);
#pragma unroll
  for (int q = 0; q < 8; ++q) v[q] = 2 * q + (lane >> 4) < cnt ? s[32 * q] : (R)0;
#pragma unroll
  for (int w = 4; w >= 1; w >>= 1)
#pragma unroll
    for (int q = 0; q < w; ++q) v[q] += v[q + w];
  return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 16);
}

// Four sums over the warp; lane L returns sum L >> 3.
template <typename R>
__device__ __forceinline__ R reduce4(R a, R b, R c, R d, int lane) {
  const bool h4 = lane & 16, h3 = lane & 8;
  const R s0 = h4 ? a : c, s1 = h4 ? b : d;
  a = (h4 ? c : a) + __shfl_xor_sync(0xffffffffu, s0, 16);
  b = (h4 ? d : b) + __shfl_xor_sync(0xffffffffu, s1, 16);
  const R s2 = h3 ? a : b;
  R v = (h3 ? b : a) + __shfl_xor_sync(0xffffffffu, s2, 8);
  v += __shfl_xor_sync(0xffffffffu, v, 4);
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  return v + __shfl_xor_sync(0xffffffffu, v, 1);
}

struct QrPlan {
  int cs = 0, rows = 0, nt = 0, rpt = 0;
  bool dots_by_column = false;
  size_t bytes = 0;
};

// a layout of m x n rows on cs CTAs; false when it does not fit
template <typename C>
bool qr_fit(int m, int n, bool want_q, int cs, QrPlan& p) {
  const bool c64 = sizeof(C) == sizeof(float2);
  if (n > 4095) return false;
  p.cs = cs;
  p.rows = (m + cs - 1) / cs;
  // complex64: a thread per row, and enough warps for the columns of the
  // passes; complex128: four warps per 32 rows in the steps
  const int need = c64 ? (p.rows + 31) / 32 * 32 : (p.rows + 31) / 32 * 128;
  p.nt = std::min(kQrThreads, std::max({128, need, c64 ? (n + 1) / 2 * 32 : 256}));
  const int per = c64 ? p.nt : p.nt / 4;
  const int rpt = (p.rows + per - 1) / per;
  p.rpt = rpt <= 1 ? 1 : (rpt <= 2 ? 2 : 4);
  if (rpt > 4) return false;
  for (int v = c64 ? 0 : 1; v >= 0; --v) {
    p.dots_by_column = v != 0;
    p.bytes = qr_layout<C>(p.rows, n, std::min(m, n), cs, want_q, v != 0).bytes;
    if (p.bytes <= kQrSmemMax) return true;
  }
  return false;
}

// CTAs of a panel.  complex64: about 128 rows a CTA and at most nine CTAs (two
// such clusters share one GPC's SMs, so that the panels of concurrent streams
// still place); measured with Q, us: 432 x 40 100 on 2 CTAs, 86 on 4, 78 on 8;
// 1296 x 96 307 on 6, 274 on 9; 2304 x 96 326 on 9, 276 on 16.  complex128
// is bound by the FP64 rate of its SMs: 32 rows a CTA (one row a lane), once
// the panel has the work for it; 512 x 64 1804 us on 4 CTAs, 615 on 16;
// 64 x 16 146 on 1, 102 on 2.
template <typename C>
bool qr_plan(int m, int n, bool want_q, int cluster, QrPlan& p) {
  if (m < 1 || n < 1) return false;
  if (cluster > 0) return cluster <= kPanelMaxCluster && qr_fit<C>(m, n, want_q, cluster, p);
  const double work = (double)std::max(m, n) * std::min(m, n) * std::min(m, n);
  int want = 1;
  if (m >= n) {
    if (sizeof(C) == sizeof(float2)) want = (int)std::min(9.0, std::ceil(m / 128.0));
    else want = (int)std::min<double>(kPanelMaxCluster, std::min(std::ceil(m / 32.0), work / 8192));
  }
  for (int cs = std::max(1, want); cs <= kPanelMaxCluster; ++cs)
    if (qr_fit<C>(m, n, want_q, cs, p)) return true;
  return false;
}

// Columns a warp takes at a time in the passes (one to three): the fewest
// issue slots over all rounds of the nw warps, 32 multiply-adds a column and
// about 14 for the reflectors' loads a row chunk.
__device__ __forceinline__ int columns_per_warp(int width, int nw) {
  int best = 1, cost = 1 << 30;
  for (int c = 1; c <= 3; ++c) {
    const int k = (width + c * nw - 1) / (c * nw) * (32 * c + 14);
    if (k < cost) { cost = k; best = c; }
  }
  return best;
}

// RPT: rows a thread holds in the steps; CL: a cluster of more than one CTA.
template <typename C, int RPT, bool CL>
__global__ void __launch_bounds__(kQrThreads, 1) k_bqr(const C* Ag, int m_all, int n, int rb,
                                                       long long stride, int rows, int dots_by_column, int conj_t,
                                                       C* Qg, C* __restrict__ Rg) {
  using R = typename RealT<C>::T;
  constexpr bool c64 = sizeof(R) == 4;
  cg::cluster_group cl = cg::this_cluster();
  const int cs = CL ? (int)cl.num_blocks() : 1, cr = CL ? (int)cl.block_rank() : 0;
  const int panel = blockIdx.x / cs, npanel = gridDim.x / cs;
  const int m = min(rb, m_all - panel * rb);
  const int k = min(m, n);
  Ag += panel * stride;
  if (Qg) Qg += panel * stride;
  if (Rg) Rg += (long long)panel * n * n;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  const QrLayout L = qr_layout<C>(rows, n, min(rb, n), cs, Qg != nullptr, dots_by_column != 0);
  C* A = (C*)smem_raw;                   // local row t of column c at A[c * ld + t]
  const uint32_t bars = saddr(smem_raw + L.bars);   // steps (parity 0, 1), W, F
  volatile int* failed = (volatile int*)(smem_raw + L.bars + 32);
  R* part = (R*)(smem_raw + L.part);
  R* rowl = (R*)(smem_raw + L.rowl);
  R* recv = (R*)(smem_raw + L.recv);
  R* rowb = (R*)(smem_raw + L.rowb);
  R* step = (R*)(smem_raw + L.step);
  C* svec = (C*)(smem_raw + L.svec);
  C* xcol = (C*)(smem_raw + L.xcol);
  R* wbuf = (R*)(smem_raw + L.wbuf);
  R* fbuf = (R*)(smem_raw + L.fbuf);
  R* fown = (R*)(smem_raw + L.fown);
  C* sv = (C*)(smem_raw + L.sv);
  C* s_tau = (C*)(smem_raw + L.tau);
  float* s_scale = (float*)(smem_raw + L.scale);
  R* dbuf = (R*)(smem_raw + L.dbuf);
  const int ld = rows | 1;
  const int ncl = (n + cs - 1) / cs;
  const int r0 = cr * rows;
  const int mr = max(0, min(rows, m - r0));
  const C zero = mk<C>(0, 0), one = mk<C>(1, 0);
  constexpr int kChunks = c64 ? 4 : 8;   // sixteen-byte chunks of sixteen values
  constexpr uint32_t k16 = 16 * sizeof(R);
  const uint32_t csinv = (65536u + cs - 1) / cs;     // c / cs = c csinv >> 16 (c < 4096, cs <= 16)
  uint32_t ph_step = 0, ph_w = 0, ph_f = 0;          // phases of the barriers (steps: a bit per parity)
  if (CL && tid == 0) {
    for (int q = 0; q < 4; ++q) bar_init(bars + 8 * q);
    *failed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }

  if (conj_t) {                          // the panel is the conjugate transpose of an n x m matrix
    for (int c = warp; c < n; c += nw) {
      const C* src = Ag + (long long)c * m + r0;
#pragma unroll 4
      for (int t = lane; t < mr; t += 32) {
        const C x = src[t];
        A[c * ld + t] = mk<C>(x.x, -x.y);
      }
    }
  } else {
    for (int t = warp; t < mr; t += nw) {
      const C* src = Ag + (long long)(r0 + t) * n;
#pragma unroll 4
      for (int c = lane; c < n; c += 32) A[c * ld + t] = src[c];
    }
  }
  const int ks = Qg ? (k + kNB - 1) / kNB * kNB : kNB;
  for (int e = tid; e < ks * kNB; e += nt) sv[e] = zero;   // (a last block of fewer columns reads all of T)
  for (int e = tid; e < ks; e += nt) s_tau[e] = zero;
  if constexpr (c64) {
    // the power of two near each column's largest magnitude over the cluster
    __syncthreads();
    unsigned* smax = (unsigned*)s_scale;
    for (int c = warp; c < n; c += nw) {
      float a = 0.f;
      for (int t = lane; t < mr; t += 32) {
        const C x = A[c * ld + t];
        a = fmaxf(a, fmaxf(fabsf(x.x), fabsf(x.y)));
      }
      const unsigned b = __reduce_max_sync(0xffffffffu, __float_as_uint(a));
      if (lane == 0) smax[c] = b;
    }
    unsigned mx = 0;
    if constexpr (CL) {
      cl.sync();                         // (also: every CTA's barriers are ready before the first push)
      if (tid < n)
        for (int q = 0; q < cs; ++q) mx = max(mx, cl.map_shared_rank(smax, q)[tid]);
      cl.sync();
    } else {
      __syncthreads();
      if (tid < n) mx = smax[tid];
      __syncthreads();
    }
    // (columns past the CTA's threads, and columns that are zero or not
    // finite, stay as they are)
    if (tid < n) s_scale[tid] = mx == 0 || mx >= 0x7f800000u ? 1.f : __uint_as_float(min(max(mx >> 23, 1u), 253u) << 23);
    for (int c = nt + tid; c < n; c += nt) s_scale[c] = 1.f;
    __syncthreads();
    for (int c = warp; c < n; c += nw) {
      const float is = __uint_as_float((254u << 23) - __float_as_uint(s_scale[c]));
      for (int t = lane; t < mr; t += 32) {
        const C x = A[c * ld + t];
        A[c * ld + t] = mk<C>(x.x * is, x.y * is);
      }
    }
    __syncthreads();
  } else {
    if constexpr (CL) cl.sync();         // every CTA's barriers are ready before the first push
    else __syncthreads();
  }

  // reflector u of the block at b0, local row t
  auto vel = [&](int b0, int nbB, int u, int t) {
    if (u >= nbB) return zero;
    const int g = r0 + t;
    return g > b0 + u ? A[(b0 + u) * ld + t] : (g == b0 + u ? one : zero);
  };
  // W = V^H A for columns [c0, c1), CPW columns a warp, lanes over rows
  auto dots_rows = [&](auto cpw, int b0, int nbB, int c0, int c1) {
    constexpr int CPW = decltype(cpw)::value;
    const int t0 = b0 > r0 ? ((b0 - r0) & ~31) : 0;
    for (int c = c0 + warp * CPW; c < c1; c += nw * CPW) {
      C acc[CPW][kNB];
#pragma unroll
      for (int q = 0; q < CPW; ++q)
#pragma unroll
        for (int u = 0; u < kNB; ++u) acc[q][u] = zero;
      int yo[CPW];
#pragma unroll
      for (int q = 0; q < CPW; ++q) yo[q] = min(c + q, c1 - 1) * ld;
      for (int t = t0 + lane; t < mr; t += 32) {
        C y[CPW];
#pragma unroll
        for (int q = 0; q < CPW; ++q) y[q] = A[yo[q] + t];
        if (nbB == kNB && r0 + (t - lane) >= b0 + kNB) {
          const int vo = b0 * ld + t;
#pragma unroll
          for (int u = 0; u < kNB; ++u) {
            const C v = A[vo + u * ld];
#pragma unroll
            for (int q = 0; q < CPW; ++q) fmac(acc[q][u], v, y[q]);
          }
        } else {
#pragma unroll
          for (int u = 0; u < kNB; ++u) {
            const C v = vel(b0, nbB, u, t);
#pragma unroll
            for (int q = 0; q < CPW; ++q) fmac(acc[q][u], v, y[q]);
          }
        }
      }
#pragma unroll
      for (int q = 0; q < CPW; ++q) {
        R v[16];
#pragma unroll
        for (int u = 0; u < kNB; ++u) {
          v[2 * u] = acc[q][u].x;
          v[2 * u + 1] = acc[q][u].y;
        }
        const R w = reduce16(v, lane);   // lane 2 i: value i
        const int cc = c + q;
        if constexpr (CL) {              // to CTA cc mod cs
          const R half = __shfl_sync(0xffffffffu, w, 2 * (lane & 15));
          const int ci = (int)(((uint32_t)cc * csinv) >> 16), own = cc - ci * cs;
          push16(half, 0, lane & (kChunks - 1), saddr(wbuf) + k16 * (uint32_t)(cr * ncl + ci), bars + 16,
                 cc < c1 && lane < kChunks, own, cs, cs);
        } else {
          if (cc < c1 && !(lane & 1)) fbuf[cc * 16 + (lane >> 1)] = w;
        }
      }
    }
  };
  // the same with a lane per column and a quarter of the rows per warp
  // (complex128: a tree over the lanes would cost half as many FP64 additions
  // again as the products of a 32-row slice; here three per value)
  auto dots_columns = [&](int b0, int nbB, int c0, int c1) {
    const int tb = max(0, min(mr, b0 - r0)), quarter = (mr - tb + 3) >> 2;
    const int rs = warp & 3, gw = warp >> 2;
    for (int g0 = c0; g0 < c1; g0 += 32 * kDotGroups) {
      if (gw < kDotGroups) {
        const int c = g0 + 32 * gw + lane;
        C acc[kNB];
#pragma unroll
        for (int u = 0; u < kNB; ++u) acc[u] = zero;
        if (g0 + 32 * gw < c1) {
          const C* yc = A + (size_t)min(c, c1 - 1) * ld;
          const int te = min(mr, tb + (rs + 1) * quarter);
          for (int t = tb + rs * quarter; t < te; ++t) {
            const C y = yc[t];
#pragma unroll
            for (int u = 0; u < kNB; ++u) fmac(acc[u], vel(b0, nbB, u, t), y);
          }
        }
        R* d = dbuf + (size_t)((gw * 4 + rs) * 16) * 32 + lane;
#pragma unroll
        for (int u = 0; u < kNB; ++u) {
          d[(2 * u) * 32] = acc[u].x;
          d[(2 * u + 1) * 32] = acc[u].y;
        }
      }
      __syncthreads();
      for (int e = tid; e < kDotGroups * kNB * 32; e += nt) {
        const int g = e / (kNB * 32), u = (e >> 5) & (kNB - 1), cc = g0 + 32 * g + (e & 31);
        if (cc >= c1) continue;
        const R* d = dbuf + (size_t)(g * 64 + 2 * u) * 32 + (e & 31);
        const R wx = (d[0] + d[16 * 32]) + (d[32 * 32] + d[48 * 32]);
        const R wy = (d[32] + d[17 * 32]) + (d[33 * 32] + d[49 * 32]);
        if constexpr (CL && !c64) {
          const int ci = (int)(((uint32_t)cc * csinv) >> 16), own = cc - ci * cs;
          push(remote(saddr(wbuf) + k16 * (uint32_t)(cr * ncl + ci) + 16 * u, own), remote(bars + 16, own), wx, wy);
        } else {
          fbuf[cc * 16 + 2 * u] = wx;
          fbuf[cc * 16 + 2 * u + 1] = wy;
        }
      }
      __syncthreads();
    }
  };
  auto dots = [&](int b0, int nbB, int c0, int c1) {
    if constexpr (c64) {
      const int cpw = columns_per_warp(c1 - c0, nw);
      if (cpw == 3) dots_rows(std::integral_constant<int, 3>(), b0, nbB, c0, c1);
      else if (cpw == 2) dots_rows(std::integral_constant<int, 2>(), b0, nbB, c0, c1);
      else dots_rows(std::integral_constant<int, 1>(), b0, nbB, c0, c1);
    } else {
      if (dots_by_column) dots_columns(b0, nbB, c0, c1);
      else dots_rows(std::integral_constant<int, 1>(), b0, nbB, c0, c1);
    }
  };
  // entry i of T^H w (fwd) or T w; w is zero from the block's size on
  auto times_t = [&](int b0, bool fwd, const C (&w)[kNB], int i) {
    const C* T = sv + (Qg ? b0 * kNB : 0);
    const C ta = s_tau[(Qg ? b0 : 0) + i];
    C f = zero;
#pragma unroll
    for (int q = 0; q < kNB; ++q) {
      C t = zero;                        // (T^H)_iq or T_iq
      if (fwd) {
        if (q < i) t = T[q * kNB + i];
        else if (q == i) t = ta;
        fmac(f, t, w[q]);
      } else {
        if (q > i) t = T[i * kNB + q];
        else if (q == i) t = ta;
        fma2(f, t, w[q]);
      }
    }
    return f;
  };
  // The phases of the W and F exchange of columns [c0, c1), armed by one thread
  // before the block barrier that precedes the dots.  A CTA that owns none of
  // the columns receives no W and sends no F, so its phase completes as it is
  // armed; what keeps a peer's next W from arriving before that is that the
  // peer needs this CTA's W first, and that is sent after the block barrier.
  auto arm = [&](int c0, int c1) {
    if constexpr (CL) {
      if (tid == 0) {
        const int own = (c1 - cr + cs - 1) / cs - (c0 - cr + cs - 1) / cs;   // own columns in [c0, c1)
        bar_expect(bars + 16, k16 * (uint32_t)(own * cs));
        bar_expect(bars + 24, k16 * (uint32_t)(c1 - c0));
      }
    }
  };
  // W -> F for columns [c0, c1), F to every CTA
  auto factors = [&](int b0, int c0, int c1, bool fwd) {
    if constexpr (CL) {
      bar_wait(bars + 16, ph_w, failed);
      ph_w ^= 1;
      // a half warp per own column, dealt over the warps first
      const int hl = tid & 15, nh = nt >> 4, half = (tid >> 4 & 1) * nw + warp;
      for (int base = c0 / cs; base < ncl; base += nh) {
        const int ci = base + half, c = ci * cs + cr;
        const bool on = ci < ncl && c >= c0 && c < c1;
        R s[4] = {0, 0, 0, 0};
        if (on)
#pragma unroll
          for (int q = 0; q < 16; ++q)
            if (q < cs) s[q & 3] += wbuf[(size_t)(q * ncl + ci) * 16 + hl];
        const R sum = (s[0] + s[1]) + (s[2] + s[3]);
        C w[kNB];
#pragma unroll
        for (int u = 0; u < kNB; ++u) {
          w[u].x = __shfl_sync(0xffffffffu, sum, (lane & 16) + 2 * u);
          w[u].y = __shfl_sync(0xffffffffu, sum, (lane & 16) + 2 * u + 1);
        }
        C f = zero;
        if (__any_sync(0xffffffffu, on)) f = times_t(b0, fwd, w, hl >> 1);
        push16(hl & 1 ? f.y : f.x, lane & 16, hl & (kChunks - 1), saddr(fbuf) + k16 * (uint32_t)c, bars + 24, on,
               hl / kChunks, 16 / kChunks, cs);
      }
      bar_wait(bars + 24, ph_f, failed);
      ph_f ^= 1;
    } else {
      for (int base = c0; base < c1; base += nt >> 3) {   // eight lanes per column
        const int c = base + (tid >> 3), i = tid & 7;
        const bool on = c < c1;
        C* p = (C*)(fbuf + (size_t)(on ? c : c0) * 16);
        C w[kNB];
#pragma unroll
        for (int u = 0; u < kNB; ++u) w[u] = p[u];
        C f = zero;
        if (__any_sync(0xffffffffu, on)) f = times_t(b0, fwd, w, i);
        __syncwarp();                    // the column's W is read before it is overwritten
        if (on) p[i] = f;
      }
    }
  };
  // A -= V F for columns [c0, c1)
  auto update_cpw = [&](auto cpw, int b0, int nbB, int c0, int c1) {
    constexpr int CPW = decltype(cpw)::value;
    const int t0 = b0 > r0 ? ((b0 - r0) & ~31) : 0;
    for (int c = c0 + warp * CPW; c < c1; c += nw * CPW) {
      C f[CPW][kNB];
      int yo[CPW];
#pragma unroll
      for (int q = 0; q < CPW; ++q) {
        const int cc = min(c + q, c1 - 1);
        yo[q] = cc * ld;
        const C* p = (const C*)(fbuf + (size_t)cc * 16);
#pragma unroll
        for (int u = 0; u < kNB; ++u) f[q][u] = p[u];
      }
      for (int t = t0 + lane; t < mr; t += 32) {
        C y[CPW];
#pragma unroll
        for (int q = 0; q < CPW; ++q) y[q] = A[yo[q] + t];
        if (nbB == kNB && r0 + (t - lane) >= b0 + kNB) {
          const int vo = b0 * ld + t;
#pragma unroll
          for (int u = 0; u < kNB; ++u) {
            const C v = A[vo + u * ld];
#pragma unroll
            for (int q = 0; q < CPW; ++q) fnma(y[q], v, f[q][u]);
          }
        } else {
#pragma unroll
          for (int u = 0; u < kNB; ++u) {
            const C v = vel(b0, nbB, u, t);
#pragma unroll
            for (int q = 0; q < CPW; ++q) fnma(y[q], v, f[q][u]);
          }
        }
#pragma unroll
        for (int q = 0; q < CPW; ++q)
          if (c + q < c1) A[yo[q] + t] = y[q];
      }
    }
  };
  auto update = [&](int b0, int nbB, int c0, int c1) {
    if constexpr (c64) {
      const int cpw = columns_per_warp(c1 - c0, nw);
      if (cpw == 3) update_cpw(std::integral_constant<int, 3>(), b0, nbB, c0, c1);
      else if (cpw == 2) update_cpw(std::integral_constant<int, 2>(), b0, nbB, c0, c1);
      else update_cpw(std::integral_constant<int, 1>(), b0, nbB, c0, c1);
    } else {
      update_cpw(std::integral_constant<int, 1>(), b0, nbB, c0, c1);
    }
  };
  // column j of T of the block whose scalars start at sb, a lane per row
  auto t_column = [&](int sb, int j) {
    if (lane >= j) return;
    const C* Tr = sv + (sb + lane) * kNB;
    const C* S = svec + (j & 1) * kNB;
    C acc = mul(s_tau[sb + lane], S[lane]);
#pragma unroll
    for (int q = 1; q < kNB - 1; ++q)
      if (q > lane && q < j) fma2(acc, Tr[q], S[q]);
    const C tj = s_tau[sb + j];
    sv[(sb + lane) * kNB + j] = mul(mk<C>(-tj.x, -tj.y), acc);
  };
  const int qa = lane / kChunks;         // this lane's chunk and its CTAs in a push of a whole warp
  const int chunk = lane & (kChunks - 1);

  // ---- the steps of a block, complex64: a thread per row
  auto steps_rows = [&](int b0, int nbB, int sb) {
    const int naw = min(nw, (rows + 31) >> 5);       // warps that hold rows
    // slot u of x: column (j + u) mod kNB of the block (rotated every step, so
    // that one copy of the step's code serves all of them): slot 0 is the
    // step's column, the columns right of it come next, then the reflectors
    C x[RPT][kNB];
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
      const int t = tid + i * nt;
#pragma unroll
      for (int u = 0; u < kNB; ++u) x[i][u] = (t < mr && u < nbB) ? A[(b0 + u) * ld + t] : zero;
    }
#pragma unroll 1
    for (int j = 0; j < nbB; ++j) {
      const int J = b0 + j, par = j & 1;
      if (warp < naw) {
        C xm[RPT];
#pragma unroll
        for (int i = 0; i < RPT; ++i) xm[i] = r0 + tid + i * nt > J ? x[i][0] : zero;
        R v[16];
#pragma unroll
        for (int u = 1; u < kNB; ++u) {
          C d = zero;
#pragma unroll
          for (int i = 0; i < RPT; ++i) fmac(d, xm[i], x[i][u]);
          v[2 * u] = d.x;
          v[2 * u + 1] = d.y;
        }
        v[0] = v[1] = 0;
#pragma unroll
        for (int i = 0; i < RPT; ++i) v[0] = fmaf(xm[i].y, xm[i].y, fmaf(xm[i].x, xm[i].x, v[0]));
        const R s = reduce16(v, lane);
        if (!(lane & 1)) part[warp * 16 + (lane >> 1)] = s;
#pragma unroll
        for (int i = 0; i < RPT; ++i)    // row J, from the thread that holds it
          if (r0 + tid + i * nt == J) {
#pragma unroll
            for (int u = 0; u < kNB; ++u) ((C*)rowl)[u] = x[i][u];
          }
      }
      if (naw > 1) __syncthreads();
      else __syncwarp();
      if (warp == 0) {
        R my = combine(part, naw, lane), rv = rowl[lane & 15];
        if constexpr (CL) {
          if (lane == 0) bar_expect(bars + 8 * par, k16 * (uint32_t)(cs + 1));
          push16(my, 0, chunk, saddr(recv) + k16 * (uint32_t)(par * cs + cr), bars + 8 * par, true, qa, 32 / kChunks, cs);
          push16(rv, 0, chunk, saddr(rowb) + k16 * (uint32_t)par, bars + 8 * par, J >= r0 && J < r0 + mr, qa,
                 32 / kChunks, cs);
          bar_wait(bars + 8 * par, (ph_step >> par) & 1u, failed);
          my = combine(recv + (size_t)par * cs * 16, cs, lane);
          rv = rowb[par * 16 + (lane & 15)];
        }
        C tau, sc, diag;
        reflector<C, R>(__shfl_sync(0xffffffffu, my, 0), __shfl_sync(0xffffffffu, rv, 0),
                        __shfl_sync(0xffffffffu, rv, 1), tau, sc, diag);
        // lane u: the factor of slot u, or V^H V and the top of V when the
        // slot holds a reflector
        const int u = lane & 7;
        const C s = mk<C>(__shfl_sync(0xffffffffu, my, 2 * u), __shfl_sync(0xffffffffu, my, 2 * u + 1));
        const C row = mk<C>(__shfl_sync(0xffffffffu, rv, 2 * u), __shfl_sync(0xffffffffu, rv, 2 * u + 1));
        if (lane > 0 && lane < kNB) {
          ((C*)step)[2 + lane] = mulc(tau, add(row, mulc(sc, s)));
          const int c = j + lane - kNB;  // the reflector's place in the block
          if (c >= 0) {
            svec[par * kNB + c] = add(mk<C>(row.x, -row.y), mul(sc, mk<C>(s.x, -s.y)));
            sv[(sb + j) * kNB + c] = row;
          }
        }
        if (lane == 0) {
          ((C*)step)[0] = sc;
          ((C*)step)[1] = diag;
          s_tau[sb + j] = tau;
        }
      }
      ph_step ^= 1u << par;
      __syncthreads();
      if (warp == nw - 1) t_column(sb, j);
      if (warp < naw) {
        const C sc = ((const C*)step)[0], diag = ((const C*)step)[1];
        C x0[RPT], v[RPT];
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
          const int g = r0 + tid + i * nt;
          const C y = mul(x[i][0], sc);
          v[i] = g > J ? y : (g == J ? one : zero);
          x0[i] = g > J ? y : (g == J ? diag : x[i][0]);
        }
#pragma unroll
        for (int u = 1; u < kNB; ++u)
          if (j + u < kNB) {
            const C fu = ((const C*)step)[2 + u];
#pragma unroll
            for (int i = 0; i < RPT; ++i) fnma(x[i][u], v[i], fu);
          }
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
#pragma unroll
          for (int u = 1; u < kNB; ++u) x[i][u - 1] = x[i][u];
          x[i][kNB - 1] = x0[i];
        }
      }
    }
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
      const int t = tid + i * nt;
      if (t < mr)
#pragma unroll
        for (int u = 0; u < kNB; ++u) {
          const int c = (nbB + u) & (kNB - 1);
          if (c < nbB) A[(size_t)(b0 + c) * ld + t] = x[i][u];
        }
    }
  };
  // ---- the same in complex128: warp 4 r + p holds columns 2 p, 2 p + 1 of
  // rows 32 (r + i nw / 4) + lane
  auto steps_pairs = [&](int b0, int nbB, int sb) {
    const int p = warp & 3, rc = warp >> 2, nch = nw >> 2, nact = min(nch, (rows + 31) >> 5);
    C x[RPT][2];
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
      const int t = (rc + i * nch) * 32 + lane;
#pragma unroll
      for (int u = 0; u < 2; ++u) x[i][u] = (t < mr && 2 * p + u < nbB) ? A[(size_t)(b0 + 2 * p + u) * ld + t] : zero;
    }
#pragma unroll 1
    for (int j = 0; j < nbB; ++j) {
      const int J = b0 + j, par = j & 1, pj = j >> 1;
      C* xc = xcol + par * rows;
      if (rc < nact) {
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
          const int t = (rc + i * nch) * 32 + lane, g = r0 + t;
          if (p == pj && t < mr) xc[t] = g > J ? (par ? x[i][1] : x[i][0]) : zero;
          if (g == J && t < mr) {
            ((C*)rowl)[2 * p] = x[i][0];
            ((C*)rowl)[2 * p + 1] = x[i][1];
          }
        }
      }
      __syncthreads();
      if (j > 0 && warp == nw - 1) t_column(sb, j - 1);
      R v = 0;                           // lane L: sum L >> 3 of the pair's four
      if (rc < nact) {
        C d0 = zero, d1 = zero;
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
          const int t = (rc + i * nch) * 32 + lane;
          const C xm = t < mr ? xc[t] : zero;
          fmac(d0, xm, x[i][0]);
          fmac(d1, xm, x[i][1]);
        }
        v = reduce4(d0.x, d0.y, d1.x, d1.y, lane);
        if (nact > 1 && !(lane & 7)) part[rc * 16 + 4 * p + (lane >> 3)] = v;
      }
      C row0 = zero, row1 = zero;
      if (nact > 1) {
        __syncthreads();
        if (rc < nact) {
          v = 0;
          for (int r = 0; r < nact; ++r) v += part[r * 16 + 4 * p + (lane >> 3)];
        }
      }
      if (rc < nact) {
        if constexpr (CL && !c64) {
          if (tid == 0) bar_expect(bars + 8 * par, k16 * (uint32_t)(cs + 1));
          if (rc == 0) {
            const int ch = lane & 1, q = lane >> 1;
            const R v0 = __shfl_sync(0xffffffffu, v, 16 * ch), v1 = __shfl_sync(0xffffffffu, v, 16 * ch + 8);
            if (q < cs) {
              const uint32_t off = (uint32_t)sizeof(R) * (4 * p + 2 * ch), bq = remote(bars + 8 * par, q);
              push(remote(saddr(recv) + k16 * (uint32_t)(par * cs + cr) + off, q), bq, v0, v1);
              if (J >= r0 && J < r0 + mr)
                push(remote(saddr(rowb) + k16 * (uint32_t)par + off, q), bq, rowl[4 * p + 2 * ch],
                     rowl[4 * p + 2 * ch + 1]);
            }
          }
          bar_wait(bars + 8 * par, (ph_step >> par) & 1u, failed);
          const R* src = recv + (size_t)par * cs * 16 + 4 * p + (lane >> 3);
          const int q = lane & 7;
          v = (q < cs ? src[q * 16] : (R)0) + (q + 8 < cs ? src[(q + 8) * 16] : (R)0);
          v += __shfl_xor_sync(0xffffffffu, v, 4);
          v += __shfl_xor_sync(0xffffffffu, v, 2);
          v += __shfl_xor_sync(0xffffffffu, v, 1);
          row0 = ((const C*)(rowb + par * 16))[2 * p];
          row1 = ((const C*)(rowb + par * 16))[2 * p + 1];
        } else {
          row0 = ((const C*)rowl)[2 * p];
          row1 = ((const C*)rowl)[2 * p + 1];
        }
      }
      const C s0 = mk<C>(__shfl_sync(0xffffffffu, v, 0), __shfl_sync(0xffffffffu, v, 8));
      const C s1 = mk<C>(__shfl_sync(0xffffffffu, v, 16), __shfl_sync(0xffffffffu, v, 24));
      if (rc == 0 && p == pj) {
        const C al = par ? row1 : row0;
        C tau, sc, diag;
        reflector<C, R>(par ? s1.x : s0.x, al.x, al.y, tau, sc, diag);
        if (lane == 0) {
          ((C*)step)[0] = sc;
          ((C*)step)[1] = diag;
          ((C*)step)[2] = tau;
          s_tau[sb + j] = tau;
        }
      }
      ph_step ^= 1u << par;
      __syncthreads();
      if (rc < nact) {
        const C sc = ((const C*)step)[0], diag = ((const C*)step)[1], tau = ((const C*)step)[2];
        const int c0 = 2 * p, c1 = 2 * p + 1;
        const C sl = lane & 1 ? s1 : s0, rl = lane & 1 ? row1 : row0;   // even lanes: column c0, odd ones: c1
        C f0 = zero, f1 = zero;
        if (c1 > j) {
          C v1 = rl;
          fmac(v1, sc, sl);
          const C f = mulc(tau, v1);
          f0 = mk<C>(__shfl_sync(0xffffffffu, f.x, 0), __shfl_sync(0xffffffffu, f.y, 0));
          f1 = mk<C>(__shfl_sync(0xffffffffu, f.x, 1), __shfl_sync(0xffffffffu, f.y, 1));
        }
        if (rc == 0 && c0 < j && lane < 2 && c0 + lane < j) {
          C v = mk<C>(rl.x, -rl.y);
          fma2(v, sc, mk<C>(sl.x, -sl.y));
          svec[par * kNB + c0 + lane] = v;
          sv[(sb + j) * kNB + c0 + lane] = rl;
        }
        if (c1 >= j) {
#pragma unroll
          for (int i = 0; i < RPT; ++i) {
            const int t = (rc + i * nch) * 32 + lane, g = r0 + t;
            const C y = mul(t < mr ? xc[t] : zero, sc);
            const C v1 = g > J ? y : (g == J ? one : zero);
            if (c0 > j) fnma(x[i][0], v1, f0);
            if (c1 > j) fnma(x[i][1], v1, f1);
            if (c0 == j) x[i][0] = g > J ? y : (g == J ? diag : x[i][0]);
            if (c1 == j) x[i][1] = g > J ? y : (g == J ? diag : x[i][1]);
          }
        }
      }
    }
    __syncthreads();
    if (warp == nw - 1) t_column(sb, nbB - 1);
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
      const int t = (rc + i * nch) * 32 + lane;
#pragma unroll
      for (int u = 0; u < 2; ++u)
        if (t < mr && 2 * p + u < nbB) A[(size_t)(b0 + 2 * p + u) * ld + t] = x[i][u];
    }
  };

  // ---- factorisation
  for (int b0 = 0; b0 < k; b0 += kNB) {
    const int nbB = min(kNB, k - b0), b1 = b0 + nbB, sb = Qg ? b0 : 0;
    if constexpr (c64) steps_rows(b0, nbB, sb);
    else steps_pairs(b0, nbB, sb);
    if (b1 < n) arm(b1, n);              // (the last exchange's waits are over: a block barrier ends every update)
    __syncthreads();
    if (b1 < n) {
      dots(b0, nbB, b1, n);
      if constexpr (!CL) __syncthreads();
      factors(b0, b1, n, true);
      if constexpr (!CL) __syncthreads();
      update(b0, nbB, b1, n);
      __syncthreads();
    }
  }

  // R (k x n, upper triangular; n rows a panel when panels are stacked) from
  // the rows this CTA holds
  if (Rg) {
    const int kr = npanel > 1 ? n : k, hi = cr == cs - 1 ? kr : min(kr, r0 + rows);
    for (int g = r0 + warp; g < hi; g += nw)
      for (int c = lane; c < n; c += 32) {
        C x = zero;
        if (g < k && c >= g) {
          x = A[(size_t)c * ld + g - r0];
          if constexpr (c64) x = mk<C>(x.x * s_scale[c], x.y * s_scale[c]);
        }
        Rg[(long long)g * n + c] = x;
      }
  }
  // no CTA leaves while another may still push to it; an exchange that ran
  // out leaves a NaN
  auto leave = [&](C* out) {
    if constexpr (CL) {
      if (tid == 0 && *failed && out && r0 < m) {
        const R bad = (R)__int_as_float(0x7fffffff);
        out[0] = mk<C>(bad, bad);
      }
      cl.sync();
    }
  };
  __syncthreads();
  if (!Qg) {
    leave(Rg ? Rg + (size_t)(r0 < k ? r0 : 0) * n : nullptr);
    return;
  }

  // ---- Q, the last block first: Q_c -= V (T (V^H Q_c)) right of the block,
  // and for the block's own columns Q_c = e_c - V (T (V^H e_c)), where V^H
  // e_c is a row of the top of V that every CTA holds
  for (int b0 = ((k - 1) / kNB) * kNB; b0 >= 0; b0 -= kNB) {
    const int nbB = min(kNB, k - b0), b1 = b0 + nbB;
    if (b1 < k) {
      dots(b0, nbB, b1, k);
      if constexpr (!CL) __syncthreads();
      factors(b0, b1, k, false);
    }
    for (int e = tid; e < nbB * kNB; e += nt) {   // row i of T (V^H e_a), V^H e_a from the top of V
      const int a = e / kNB, i = e % kNB;
      C f = zero;
      if (i < nbB)
        for (int q = i; q <= a; ++q) {
          const C t = q == i ? s_tau[b0 + i] : sv[(b0 + i) * kNB + q];
          const C v = q == a ? one : sv[(b0 + a) * kNB + q];
          fmac(f, v, t);
        }
      ((C*)fown)[a * kNB + i] = f;
    }
    if (b1 < k) {
      if constexpr (!CL) __syncthreads();
      update(b0, nbB, b1, k);
    }
    __syncthreads();
    if (b0 > 0) arm(b0, k);              // the next block's, ahead of a barrier
    if constexpr (c64) {
      for (int t = tid; t < mr; t += nt) {           // a thread per row
        const int g = r0 + t;
        C v[kNB];
#pragma unroll
        for (int u = 0; u < kNB; ++u) v[u] = vel(b0, nbB, u, t);
#pragma unroll
        for (int a = 0; a < kNB; ++a) {
          if (a >= nbB) break;
          const C* p = (const C*)fown + a * kNB;
          C y = g == b0 + a ? one : zero;
#pragma unroll
          for (int u = 0; u < kNB; ++u) fnma(y, v[u], p[u]);
          A[(size_t)(b0 + a) * ld + t] = y;
        }
      }
      __syncthreads();
    } else {                                         // warp 4 r + p: columns 2 p, 2 p + 1 of 32 rows
      const int p = warp & 3;
      for (int base = 0; base < rows; base += nw * 8) {
        const int t = base + (warp >> 2) * 32 + lane, g = r0 + t;
        C y[2];
#pragma unroll
        for (int a = 0; a < 2; ++a) y[a] = g == b0 + 2 * p + a ? one : zero;
        if (t < mr)
#pragma unroll
          for (int u = 0; u < kNB; ++u) {
            const C v = vel(b0, nbB, u, t);
#pragma unroll
            for (int a = 0; a < 2; ++a)
              if (2 * p + a < nbB) fnma(y[a], v, ((const C*)fown)[(2 * p + a) * kNB + u]);
          }
        __syncthreads();                             // the rows' reflectors are read
        if (t < mr)
#pragma unroll
          for (int a = 0; a < 2; ++a)
            if (2 * p + a < nbB) A[(size_t)(b0 + 2 * p + a) * ld + t] = y[a];
      }
      __syncthreads();
    }
  }
  if (conj_t) {                          // Q^H (k x m)
    for (int c = warp; c < k; c += nw)
      for (int t = lane; t < mr; t += 32) {
        const C x = A[c * ld + t];
        Qg[(long long)c * m + r0 + t] = mk<C>(x.x, -x.y);
      }
  } else {
    for (int t = warp; t < mr; t += nw)
      for (int c = lane; c < k; c += 32) Qg[(long long)(r0 + t) * k + c] = A[c * ld + t];
  }
  __syncthreads();
  leave(conj_t ? Qg + r0 : Qg + (size_t)r0 * k);
}

template <typename C, int RPT, bool CL>
cudaError_t bqr_run(const C* A, int m_all, int n, int rb, long long stride, const QrPlan& p, bool conj_t, C* Q, C* R,
                    cudaStream_t s) {
  auto kern = k_bqr<C, RPT, CL>;
  static std::atomic<unsigned long long> done{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = 1ull << (dev & 63);
  if (!(done.load(std::memory_order_relaxed) & bit)) {
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kQrSmemMax)) != cudaSuccess)
      return e;
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) != cudaSuccess) return e;
    done.fetch_or(bit);
  }
  if (p.nt == 0) return cudaSuccess;     // (the attributes only)
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.cs * ((m_all + rb - 1) / rb), 1, 1);
  cfg.blockDim = dim3(p.nt, 1, 1);
  cfg.dynamicSmemBytes = p.bytes;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = p.cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = CL ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, A, m_all, n, rb, stride, p.rows, p.dots_by_column ? 1 : 0, conj_t ? 1 : 0, Q, R);
}

template <typename C>
cudaError_t bqr_pick(const C* A, int m_all, int n, int rb, long long stride, const QrPlan& p, bool cl, bool conj_t, C* Q,
                     C* R, cudaStream_t s) {
  switch (p.rpt) {
    case 1: return cl ? bqr_run<C, 1, true>(A, m_all, n, rb, stride, p, conj_t, Q, R, s)
                      : bqr_run<C, 1, false>(A, m_all, n, rb, stride, p, conj_t, Q, R, s);
    case 2: return cl ? bqr_run<C, 2, true>(A, m_all, n, rb, stride, p, conj_t, Q, R, s)
                      : bqr_run<C, 2, false>(A, m_all, n, rb, stride, p, conj_t, Q, R, s);
    case 4: return cl ? bqr_run<C, 4, true>(A, m_all, n, rb, stride, p, conj_t, Q, R, s)
                      : bqr_run<C, 4, false>(A, m_all, n, rb, stride, p, conj_t, Q, R, s);
    default: return cudaErrorInvalidValue;
  }
}

template <typename C>
cudaError_t bqr_t(const C* A, int m_all, int n, int rb, long long stride, bool conj_t, C* Q, C* R, int cluster,
                  cudaStream_t s) {
  QrPlan p;
  rb = std::min(rb, m_all);
  if (!qr_plan<C>(rb, n, Q != nullptr, cluster, p)) return cudaErrorInvalidValue;
  return bqr_pick(A, m_all, n, rb, stride, p, p.cs > 1, conj_t, Q, R, s);
}

template <typename C>
cudaError_t bqr_optin() {
  QrPlan p;                              // nt = 0: no launch
  for (int rpt : {1, 2, 4})
    for (bool cl : {false, true}) {
      p.rpt = rpt;
      cudaError_t e = bqr_pick<C>(nullptr, 1, 1, 1, 0, p, cl, false, nullptr, nullptr, 0);
      if (e != cudaSuccess) return e;
    }
  return cudaSuccess;
}

}  // namespace

cudaError_t init_bqr_attributes() {
  cudaError_t e = bqr_optin<float2>();
  return e != cudaSuccess ? e : bqr_optin<double2>();
}

bool bqr_fits(int m, int n, size_t elem, bool want_q, int cluster) {
  QrPlan p;
  return elem == sizeof(double2) ? qr_plan<double2>(m, n, want_q, cluster, p)
                                 : qr_plan<float2>(m, n, want_q, cluster, p);
}

cudaError_t launch_bqr(const float2* A, int m_all, int n, int rb, long long stride, float2* Q, float2* R, int cluster,
                       cudaStream_t s) {
  return bqr_t(A, m_all, n, rb, stride, false, Q, R, cluster, s);
}
cudaError_t launch_bqr(const double2* A, int m_all, int n, int rb, long long stride, double2* Q, double2* R,
                       int cluster, cudaStream_t s) {
  return bqr_t(A, m_all, n, rb, stride, false, Q, R, cluster, s);
}

cudaError_t launch_blq(float2* T, int n, int m, float2* R, cudaStream_t s) {
  return bqr_t<float2>(T, m, n, m, 0, true, T, R, 0, s);
}
cudaError_t launch_blq(double2* T, int n, int m, double2* R, cudaStream_t s) {
  return bqr_t<double2>(T, m, n, m, 0, true, T, R, 0, s);
}

}  // namespace bbp
