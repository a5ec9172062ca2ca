// Supernodal numeric factorization: assembly and the persistent task kernel.
//
// Tasks (Section III-A; Section IV labels a task by source and target):
//   POTRF(s)     F on the diagonal block of panel s: the dense Cholesky of
//                Algorithm 1 on a w x w block, always in FP64.
//   TRSM(s, k)   F on rows tile k below the diagonal block:
//                L21 = A21 L11^{-T} by forward substitution along each row.
//   UPD(s, t, k) U + A fused: C = L_s[rows k] L_s[rows in t]^T, subtracted
//                from panel t at the relative positions of those rows and
//                columns in t (the aggregate vector of Section III-A is
//                applied immediately, by atomic adds, instead of being kept).
// Dependencies (Section II-C): UPD(s, ., .) needs every TRSM tile of s;
// POTRF(t) needs every update tile targeting t.
#include <algorithm>
#include <climits>
#include <cstdint>

#include <cuda_bf16.h>

#include "device_common.cuh"
#include "kernels.hpp"
#include "sched.cuh"

namespace spchol {

namespace {

constexpr int kTrsmMaxW = 64;  // panels up to this width take the register-resident panel solve

struct FactorShared {
  int task;
  int skip;
  int flag;
  int base;
  int next;  // a diagonal task this CTA made ready and runs next (-1: none; thread 0)
  int hold;  // this CTA holds a high-priority slot, or is inside a subtree task: no continuation
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ Ring2 rings_of(const FactorArgs& a) {
  return Ring2{a.ring, a.ring + a.n_hi, a.n_hi, a.ntask - a.n_hi, a.ctrl, a.budget_ns};
}

// Panel s (w columns) has its rows below solved by its diagonal task (see
// kFuseWidth).
__device__ __forceinline__ bool fused_panel(const FactorArgs& a, int s, int w) {
  const int nb = a.pv.nrows[s] - w;
  return w <= a.fuse_w && a.ntrsm[s] == 1 && nb <= kFuseRows && w * w * nb <= kFuseWork;
}

template <typename T>
__device__ __forceinline__ T* panel_ptr(const FactorArgs& a, int s) {
  return reinterpret_cast<T*>(a.pool) + a.pv.valoff[s];
}

// ---------------------------------------------------------------- POTRF(s)
// Cholesky of the w x w diagonal block in shared memory (Algorithm 1),
// right-looking, two columns and one barrier per step.  Step c: the pivot warp
// finishes columns c and c + 1 (rows c .. c + 31; a second warp the rows
// below them) -- subtracts columns c - 2 and c - 1 from them and scales them --
// while the update warps subtract columns c - 2 and c - 1 from the columns
// beyond.  What bounds it: a warp-wide FP64 instruction holds one of the SM's
// four FP64 pipes for 64 clocks whatever its active lanes, warps issue in
// order, and a warp whose lanes are all predicated off still takes its turn.
// So the pivots' reciprocal square roots run on the integer pipe (seven FP64
// instructions per pair of columns are left on the chain), the update warps
// leave the pivot warps' sub-partitions to them as far as they can (warp 3
// comes last), and a warp branches around the pairs it has none of.  A w = 64
// block alone on an SM (clocks, w = 32 in parentheses): 75,800 (32,600) one
// column per step with the square root in FP64, 59,600 (24,800) this way; the
// chain alone is 49,700, the updates alone 39,700.
// The trailing entries are enumerated by the pair index p of the triangle in
// column-major order from its bottom-right corner, so that p < m (m + 1) / 2
// is exactly the triangle of order m and consecutive p touch consecutive rows;
// each thread decodes its first pairs once.
constexpr int kPivotWarp = 7;   // and kPivotWarp - 1: the rows from c + 32 on
constexpr int kUpdWarps = 6;    // warps 0, 1, 2, 4, 5 and 3
constexpr int kPairRegs = 10;   // pairs a thread keeps decoded: 10 x 192 >= 60 x 61 / 2 (w = 64)

__device__ __forceinline__ void tri_pair(int p, int& ei, int& ek) {
  int e = (int)((sqrtf((float)(8 * p + 1)) - 1.0f) * 0.5f);
  if ((e + 1) * (e + 2) / 2 <= p) ++e;
  if (e * (e + 1) / 2 > p) --e;
  ek = e;
  ei = p - e * (e + 1) / 2;
}

// d > 0 on the integer pipe (false for a NaN, as the comparison).
__device__ __forceinline__ bool pivot_positive(double d) {
  const long long b = __double_as_longlong(d);
  return b > 0 && b <= 0x7FF0000000000000ll;
}

// 1 / sqrt(d) for the pivot d > 0, in integers: one step of third order,
// y (1 + e / 2 + 3 e^2 / 8) with e = 1 - d y^2, from the single-precision
// approximate reciprocal square root y of d cut to single precision (|e| <
// 2^-20: the remainder 5/16 e^3 is below 2^-61).  With d = M 2^(E - 52) and y =
// Y 2^(F - 23), d y^2 = M Y^2 2^(E + 2F - 98), so e is the low part of -M Y^2
// taken from its bit 32 on (its high part is the power of two next to it), in
// units of 2^(E + 2F - 66); everything below is kept to 2^-57 and the result
// rounded to nearest (largest error seen over 1.5e8 values: 0.51 units of
// 2^-52 of a mantissa near 1).  Outside |exponent| < 120, the square root and
// the division.
__device__ __forceinline__ double pivot_rsqrt(double d) {
  const int hi = __double2hiint(d);
  const unsigned lo = (unsigned)__double2loint(d);
  if ((unsigned)(hi - (903 << 20)) < (unsigned)(240 << 20)) {
    float f;
    asm("rsqrt.approx.ftz.f32 %0, %1;"
        : "=f"(f)
        : "f"(__int_as_float(((hi - (896 << 20)) << 3) | (int)(lo >> 29))));
    const unsigned fb = __float_as_uint(f);
    const unsigned Y = (fb & 0x7fffffu) | 0x800000u;
    const int fe = (int)(fb >> 23);
    const unsigned long long Q = (unsigned long long)Y * Y;
    const unsigned mh = (hi & 0xFFFFF) | 0x100000, qh = (unsigned)(Q >> 32), ql = (unsigned)Q;
    unsigned long long t = (unsigned long long)mh * ql + __umulhi(lo, ql);
    t += (unsigned long long)lo * qh;
    t += (unsigned long long)(mh * qh) << 32;
    const long long e = (-(long long)t) >> (1283 - (hi >> 20) - 2 * fe);  // units of 2^-60
    const int eh = (int)(e >> 20);
    const long long c = (e >> 1) + (((long long)eh * eh * 3) >> 23);
    const unsigned long long y = ((unsigned long long)Y << 39) + (((long long)Y * c) >> 21);
    const int lz = __clzll((long long)y);
    const unsigned long long yn = y << lz;
    return __longlong_as_double(((long long)(fe + 896 - lz) << 52) + (long long)((yn >> 11) + ((yn >> 10) & 1)));
  }
  return 1.0 / sqrt(d);
}

// Columns c and c + 1 of rows i = row(lane) from columns c - 2 and c - 1 (c >
// 0): the entries before scaling.
__device__ __forceinline__ void pivot_load(const double* sm, int w, int c, int i, double& v2, double& v3) {
  const double* c2 = sm + c * w;
  const bool rv = i < w, two = c + 1 < w;
  v2 = rv ? c2[i] : 0.0;
  v3 = two && rv && i > c ? c2[w + i] : 0.0;
  if (c > 0) {
    const double *c1 = c2 - w, *c0 = c1 - w;
    const double a0 = rv ? c0[i] : 0.0, a1 = rv ? c1[i] : 0.0;
    const double e0 = two ? c0[c + 1] : 0.0, e1 = two ? c1[c + 1] : 0.0;
    v2 = fma(-a1, c1[c], fma(-a0, c0[c], v2));
    v3 = fma(-a1, e1, fma(-a0, e0, v3));
  }
}

// The pivot warps finish columns c and c + 1.  MAIN: rows c .. c + 31 and
// 1 / l_cc, 1 / l_c+1,c+1 in xd; else the rows from c + 32 on, lanes 30 and 31
// of the first pass repeating rows c and c + 1 for the pivots.  The main warp
// overwrites those two rows only after the other one has read them (both = the
// other one takes part).  A pivot that is not positive is reported; the
// columns after it are not meaningful and are not used.
template <bool MAIN>
__device__ __forceinline__ void pivot_pair(const FactorArgs& a, double* sm, double* xd, int w, int c, int f,
                                           bool both, FactorShared& sh) {
  const int lane = threadIdx.x & 31;
  const bool two = c + 1 < w;
  constexpr int kL = MAIN ? 0 : 30;  // the lanes that hold rows c and c + 1
  int i = MAIN ? c + lane : lane < 30 ? c + 32 + lane : c + lane - 30;
  double v2, v3;
  pivot_load(sm, w, c, i, v2, v3);
  if (!MAIN) {
    __syncwarp();
    asm volatile("bar.arrive 1, 64;" ::: "memory");
  }
  const double d2 = __shfl_sync(0xffffffffu, v2, kL);
  const double r2 = pivot_rsqrt(d2);
  double x2 = v2 * r2, x3 = 0.0, r3 = 0.0, d3 = 1.0;
  const double k32 = __shfl_sync(0xffffffffu, x2, kL + 1);
  if (two) {
    v3 = fma(-x2, k32, v3);
    d3 = __shfl_sync(0xffffffffu, v3, kL + 1);
    r3 = pivot_rsqrt(d3);
    x3 = v3 * r3;
  }
  if (MAIN) {
    if (both) asm volatile("bar.sync 1, 64;" ::: "memory");
    // an infinite pivot's root is infinite (r is 0, and inf * 0 no number)
    if (lane == 0 && __double2hiint(d2) == 0x7ff00000) x2 = d2;
    if (lane == 1 && __double2hiint(d3) == 0x7ff00000) x3 = d3;
    if (lane == 0) {
      xd[c] = r2;
      if (two) xd[c + 1] = r3;
      const bool bad2 = !pivot_positive(d2);
      if (bad2 || !pivot_positive(d3)) {
        atomicMin(&a.ctrl[kInfo], f + c + (bad2 ? 1 : 2));
        sh.flag = 1;
      }
    }
  }
  double* c2 = sm + c * w;
  if (MAIN || lane < 30) {
    if (i < w) {
      c2[i] = x2;
      if (two && i > c) c2[w + i] = x3;
    }
  }
  if (!MAIN) {
    for (i = c + 62 + lane; i - lane < w; i += 32) {
      pivot_load(sm, w, c, i, v2, v3);
      x2 = v2 * r2;
      if (i < w) {
        c2[i] = x2;
        if (two) c2[w + i] = fma(-x2, k32, v3) * r3;
      }
    }
  }
}

// The update warps subtract columns c - 2 and c - 1 from one trailing entry.
__device__ __forceinline__ void potrf_update(double* sm, int w, int c, int i, int k) {
  const double *c0 = sm + (c - 2) * w, *c1 = c0 + w;
  double* s = sm + i + k * w;
  *s = fma(-c1[i], c1[k], fma(-c0[i], c0[k], *s));
}

// X = L11^{-1} for the solves, off the critical path (the panel-solve tiles
// are already released), by block rows of 8: X_bc = inv(L_bb) (-L_b,: X_:,c).
// First every 8 x 8 diagonal block's inverse (a warp each), then the rows of
// L below the diagonal blocks are replaced by G_b = -inv(L_bb) L_b,: (in
// place: L11 is stored), then block row after block row X_b = G_b X, one
// barrier each, 8 rows x 4 columns per warp and dot products over the columns
// k >= c alone.  1600 warp-wide FP64 instructions for w = 64 against 2500 and
// 9 barriers against 63 for the substitution row by row it replaces.  X[i][c],
// i > c, lives in the upper triangle at (c, i); the diagonal is xd.
__device__ void invert_l11(double* sm, const double* xd, int w, double* __restrict__ X) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int li = lane & 7, lc = lane >> 3;
  const int nb = (w + 7) >> 3;
  for (int b = warp; b < nb; b += kFactorThreads / 32) {
    // lane (li, lc): row 8 b + li of columns 8 b + lc and 8 b + lc + 4.  With
    // the rows scaled by 1 / l_ii first, x_ic = -sum over q of l_iq x_qc
    const int r0 = 8 * b, i = r0 + li;
    const bool rv = i < w;
    const double ri = rv ? xd[i] : 0.0;
    double x0 = li == lc ? ri : 0.0, x1 = li == lc + 4 ? ri : 0.0;
#pragma unroll
    for (int q = 0; q < 7; ++q) {
      const double l = (rv && li > q) ? sm[i + (r0 + q) * w] * ri : 0.0;
      const double y0 = __shfl_sync(0xffffffffu, x0, (lane & 24) | q);
      const double y1 = __shfl_sync(0xffffffffu, x1, (lane & 24) | q);
      x0 = fma(-l, y0, x0);
      x1 = fma(-l, y1, x1);
    }
    __syncwarp();
    if (rv && li > lc) {
      sm[(r0 + lc) + i * w] = x0;
      X[i + (size_t)(r0 + lc) * w] = x0;
    }
    if (rv && li > lc + 4) {
      sm[(r0 + lc + 4) + i * w] = x1;
      X[i + (size_t)(r0 + lc + 4) * w] = x1;
    }
  }
  if (nb == 1) return;
  __syncthreads();
  // G_b for all block rows: group t of 4 columns of block row b (2 b of them)
  for (int g = warp; g < nb * (nb - 1); g += kFactorThreads / 32) {
    int b = 1, t = g;
    while (t >= 2 * b) {
      t -= 2 * b;
      ++b;
    }
    const int r0 = 8 * b, i = r0 + li, c = 4 * t + lc;
    const bool rv = i < w;
    const double* lcol = sm + r0 + c * w;
    double acc = rv ? xd[i] * lcol[li] : 0.0;
#pragma unroll
    for (int q = 0; q < 7; ++q) {
      const double x = (rv && li > q) ? sm[(r0 + q) + i * w] : 0.0;
      acc = fma(x, (rv && li > q) ? lcol[q] : 0.0, acc);
    }
    __syncwarp();
    if (rv) sm[i + c * w] = -acc;
  }
  __syncthreads();
  for (int b = 1; b < nb; ++b) {
    const int r0 = 8 * b, i = r0 + li;
    const bool rv = i < w;
    for (int r = 0; 8 * r < 2 * b; ++r) {
      // long and short columns alternate over the warps
      const int t = 8 * r + ((r & 1) ? 7 - warp : warp);
      if (t >= 2 * b) continue;
      const int c = 4 * t + lc;
      const double* G = sm + i;
      const double* Xc = sm + c;
      double a0 = 0.0, a1 = 0.0;
      if (rv) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int k = 4 * t + u;
          const double x = k < c ? 0.0 : k == c ? xd[c] : Xc[k * w];
          a0 = fma(G[k * w], x, a0);
        }
        int k = 4 * t + 4;
        for (; k < r0; k += 4) {  // r0 - 4 t is a multiple of 4
          a0 = fma(G[k * w], Xc[k * w], a0);
          a1 = fma(G[(k + 1) * w], Xc[(k + 1) * w], a1);
          a0 = fma(G[(k + 2) * w], Xc[(k + 2) * w], a0);
          a1 = fma(G[(k + 3) * w], Xc[(k + 3) * w], a1);
        }
        a0 += a1;
        sm[c + i * w] = a0;
        X[i + (size_t)c * w] = a0;
      }
    }
    __syncthreads();
  }
}

// L21 = A21 L11^{-T} for rows row0 .. row0 + cnt - 1 of a panel at most 8 NC
// wide, row by row: forward substitution along each row with the
// columns in registers.  Warp q takes 4-row strips 4 (q + 8 v); lane (lr, lc)
// holds row lr of the strip at columns lc + 8 cc.  Step c: the lane holding
// column c scales it by rinv[c] = 1 / l_cc, the value is broadcast within the 8
// lanes of the row, and every later column subtracts it times l_qc = Ls[q + ldl
// c] (read past row w only for columns that are not stored).
template <int NC, typename T>
__device__ __forceinline__ void trsm_strips(T* P, int ld, int row0, int cnt, int w, const T* Ls, int ldl,
                                            const T* rinv) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, lr = lane >> 3, lc = lane & 7;
  const int nstrip = (cnt + 3) >> 2;
  for (int st = warp; st < nstrip; st += kFactorThreads / 32) {
    const int rloc = 4 * st + lr;
    const bool rv = rloc < cnt;
    T* Pi = P + row0 + rloc;
    T x[NC];
#pragma unroll
    for (int cc = 0; cc < NC; ++cc) {
      const int c = lc + 8 * cc;
      x[cc] = (rv && c < w) ? ldcg(Pi + (size_t)c * ld) : T(0);
    }
#pragma unroll
    for (int cbk = 0; cbk < NC; ++cbk) {
      if (8 * cbk >= w) break;
      for (int c8 = 0; c8 < 8; ++c8) {
        const int c = 8 * cbk + c8;
        if (c >= w) break;
        if (lc == c8) x[cbk] *= rinv[c];
        const T xc = __shfl_sync(0xffffffffu, x[cbk], (lr << 3) | c8);
        const T* Lc = Ls + ldl * c;
        if (lc > c8) x[cbk] -= xc * Lc[lc + 8 * cbk];
#pragma unroll
        for (int cc = cbk + 1; cc < NC; ++cc) {
          if (8 * cc >= w) break;
          x[cc] -= xc * Lc[lc + 8 * cc];
        }
      }
    }
#pragma unroll
    for (int cc = 0; cc < NC; ++cc) {
      const int c = lc + 8 * cc;
      if (rv && c < w) Pi[(size_t)c * ld] = x[cc];
    }
  }
}

// Every row of panel s below its diagonal block is solved (published, and
// acquired by thread 0 before a barrier): its update tiles are ready.  Whole
// CTA.
__device__ __forceinline__ void release_updates(const FactorArgs& a, int s, FactorShared& sh) {
  const Ring2 q = rings_of(a);
  const int first = a.pv.ns + a.n_trsm + a.u_first[s], nhi = a.nu_hi[s];
  if (a.u_dep) {  // deterministic order: a tile also waits for its predecessor into the same target
    fence_gpu();
    for (int i = threadIdx.x; i < a.nu[s]; i += blockDim.x)
      if (count_down(&a.u_dep[a.u_first[s] + i])) ring2_push_one(q, i < nhi, first + i);
  } else {
    ring2_push_range(q, true, first, nhi, &sh.base);
    ring2_push_range(q, false, first + nhi, a.nu[s] - nhi, &sh.base);
  }
}

// W = L21 L11^{-1} for rows row0 .. row0 + cnt - 1 of a W panel (Plan::woff):
// each row w solves w L11 = l21 by back substitution, w_c = (l21_c - sum over
// q > c of w_q l_qc) / l_cc for c = w-1 .. 0, from the rows this panel-solve
// tile has just written and L11 (the inverse of the diagonal task is formed
// after the release of these tiles, so it is not read here).  The layout of
// the panel solve: warp q takes 4-row strips, lane (lr, lc) row lr at columns
// lc + 8 cc; L11 is restaged with leading dimension 65, so that the 8 lanes of
// a row read the entries l_c,lc+8cc of row c of L11 from distinct banks.
template <typename T>
__device__ void form_w_rows(const FactorArgs& a, int s, int row0, int cnt, double* smd) {
  using ct = T;
  constexpr int kLd = kTrsmMaxW + 1;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int w = a.pv.fcol[s + 1] - a.pv.fcol[s], ld = a.pv.ld[s];
  const T* P = panel_ptr<T>(a, s);
  T* W = reinterpret_cast<T*>(a.wbuf) + a.woff[s];
  ct* Ls = reinterpret_cast<ct*>(smd);  // Ls[q + kLd c] = l_qc for q > c
  ct* rinv = Ls + kLd * w;              // 1 / l_cc
  __syncthreads();                      // the panel solve is done with shared memory
  for (int idx = tid; idx < kTrsmMaxW * w; idx += nt) {
    const int qq = idx & (kTrsmMaxW - 1), c = idx >> 6;
    Ls[qq + kLd * c] = (qq < w && qq > c) ? (ct)ldcg(P + qq + (size_t)c * ld) : ct(0);
  }
  const double* Xd = a.inv + a.invoff[s];
  for (int c = tid; c < w; c += nt) rinv[c] = (ct)ldcg(Xd + c * (w + 1));
  __syncthreads();
  const int warp = tid >> 5, lane = tid & 31, lr = lane >> 3, lc = lane & 7;
  const int nstrip = (cnt + 3) >> 2;
  for (int st = warp; st < nstrip; st += nt >> 5) {
    const int rloc = 4 * st + lr;
    const bool rv = rloc < cnt;
    const T* Pi = P + row0 + rloc;
    ct x[8];
#pragma unroll
    for (int cc = 0; cc < 8; ++cc) {
      const int c = lc + 8 * cc;
      x[cc] = (rv && c < w) ? (ct)ldcg(Pi + (size_t)c * ld) : ct(0);
    }
#pragma unroll
    for (int cbk = 7; cbk >= 0; --cbk) {
      if (8 * cbk >= w) continue;
      for (int c8 = 7; c8 >= 0; --c8) {
        const int c = 8 * cbk + c8;
        if (c >= w) continue;
        if (lc == c8) x[cbk] *= rinv[c];
        const ct xc = __shfl_sync(0xffffffffu, x[cbk], (lr << 3) | c8);
        const ct* Lr = Ls + c;  // l_c,c' at Lr[kLd c'] for c' < c
        if (lc < c8) x[cbk] -= xc * Lr[kLd * (lc + 8 * cbk)];
#pragma unroll
        for (int cc = 0; cc < cbk; ++cc) x[cc] -= xc * Lr[kLd * (lc + 8 * cc)];
      }
    }
    T* Wi = W + row0 + rloc;
#pragma unroll
    for (int cc = 0; cc < 8; ++cc) {
      const int c = lc + 8 * cc;
      if (rv && c < w) Wi[(size_t)c * ld] = (T)x[cc];
    }
  }
}

template <typename T, bool FAN, bool FUSE>
__device__ void task_potrf(const FactorArgs& a, int s, double* sm, FactorShared& sh, bool skip, bool release = true) {
  const int tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  const int f = a.pv.fcol[s], w = a.pv.fcol[s + 1] - f, ld = a.pv.ld[s];
  T* P = panel_ptr<T>(a, s);
  double* xd = sm + w * w;  // 1 / l_jj, the diagonal of L11^{-1}
  double* X = a.inv + a.invoff[s];
  bool ok = true;
  const bool fuse = FUSE && fused_panel(a, s, w);
  if (!skip) {
    stage_lower<true>(P, w, ld, sm);  // lower triangle (what is above it is not read before L11^{-1} goes there)
    if (tid == 0) sh.flag = 0;  // 1: a failed pivot, whose columns are not used (a word of the CTA's own: the
                                // status word is a trip to L2 ahead of the release)
    const int uw = warp == 3 ? kUpdWarps - 1 : warp > 3 ? warp - 1 : warp;  // number among the update warps
    const int ut = uw * 32 + lane;
    constexpr int kStep = kUpdWarps * 32;
    int pair[kPairRegs];  // row << 16 | column
    if (warp < kPivotWarp - 1 && w > 4) {
#pragma unroll
      for (int q = 0; q < kPairRegs; ++q) {
        int ei, ek;
        tri_pair(ut + kStep * q, ei, ek);
        pair[q] = ((w - 1 - ei) << 16) | ((w - 1 - ek) & 0xffff);
      }
    }
    __syncthreads();
    for (int c = 0; c < w; c += 2) {
      if (warp == kPivotWarp) {
        pivot_pair<true>(a, sm, xd, w, c, f, w - c > 32, sh);
      } else if (warp == kPivotWarp - 1) {
        if (w - c > 32) pivot_pair<false>(a, sm, xd, w, c, f, true, sh);
      } else if (c > 0) {
        const int m = w - 2 - c;  // columns c + 2 .. w - 1
        const int np = m > 0 ? m * (m + 1) / 2 : 0;
#pragma unroll
        for (int q = 0; q < kPairRegs; ++q) {
          if (kStep * q + 32 * uw >= np) break;
          if (kStep * q + ut < np) potrf_update(sm, w, c, pair[q] >> 16, pair[q] & 0xffff);
        }
        for (int p = kStep * kPairRegs + ut; p < np; p += kStep) {  // w > 64
          int ei, ek;
          tri_pair(p, ei, ek);
          potrf_update(sm, w, c, w - 1 - ei, w - 1 - ek);
        }
      }
      __syncthreads();
    }
    if (FUSE && fuse) {  // the rows below, with L11 from shared memory (in the panel's type)
      const int nb = a.pv.nrows[s] - w;
      if constexpr (sizeof(T) == 8) {
        trsm_strips<kFuseWidth / 8>(P, ld, w, nb, w, sm, w, xd);
      } else {
        T *Lf = reinterpret_cast<T*>(xd + w), *rf = Lf + w * w;
        for (int idx = tid; idx < w * w; idx += blockDim.x) Lf[idx] = (T)sm[idx];
        for (int j = tid; j < w; j += blockDim.x) rf[j] = (T)xd[j];
        __syncthreads();
        trsm_strips<kFuseWidth / 8>(P, ld, w, nb, w, Lf, w, rf);
      }
    }
    for (int j = warp; j < w; j += kFactorThreads / 32)
      for (int i = j + lane; i < w; i += 32) P[i + (size_t)j * ld] = (T)sm[i + j * w];
    // the panel-solve tiles scale by 1 / l_jj
    for (int j = tid; j < w; j += blockDim.x) X[j + (size_t)j * w] = xd[j];
  }
  publish_cta_writes();
  ok = !skip && !sh.flag;
  if (FAN && release) {  // fan-in mode: a panel-solve tile also waits for its rows' gathers
    fence_gpu();
    for (int k = tid; k < a.ntrsm[s]; k += blockDim.x) {
      const int kt = a.trsm_first[s] + k;
      if (count_down(&a.tdep[kt])) ring2_push_one(rings_of(a), true, a.pv.ns + kt);
    }
  } else if (release) {
    if (FUSE && fuse)
      release_updates(a, s, sh);
    else
      ring2_push_range(rings_of(a), true, a.pv.ns + a.trsm_first[s], a.ntrsm[s], &sh.base);
  }
  if (ok) {
    invert_l11(sm, xd, w, X);
    if (FUSE && fuse && a.woff != nullptr && a.woff[s] >= 0) form_w_rows<T>(a, s, w, a.pv.nrows[s] - w, sm);
  }
}

// The same as a function of its own: inlined into the kernel of the BF16-split
// tiles it makes the registers of their hot loops spill (64^3: 140.1 -> 131.8
// ms; the other kernels are faster with it inlined, 64^3 FP64 383.5 against
// 386.9 ms, 64^2 0.437 against 0.477).
template <typename T, bool FAN>
__device__ __noinline__ void task_potrf_apart(const FactorArgs& a, int s, double* sm, FactorShared& sh, bool skip,
                                              bool release) {
  task_potrf<T, FAN, false>(a, s, sm, sh, skip, release);
}

// ---------------------------------------------------------------- FP64 operand slicing
// Error-free splitting of a row of L for the BF16 tensor cores (the splitting
// step of Ozaki, Ogita, Oishi and Rump, "Error-free transformations of matrix
// multiplication by using fast routines of matrix multiplication", Numer.
// Algorithms 2012).  With e the smallest integer such that every |x_k| of the
// row is below 2^e, x_k * 2^(56-e) is written as a 56-bit fixed-point integer
// q_k (truncated below 2^(e-56), a relative perturbation of the row of at most
// 2^-56) and cut into kSlices 8-bit digits; digit p carries weight
// 2^(e - 8(p+1)).  Each digit, with the sign of x_k, is an integer in
// [-255, 255] and is exact in BF16.  Products of two digit matrices summed over
// k <= 64 stay below 2^22 and are exact in the FP32 accumulator.
__device__ __forceinline__ int row_exponent_bits(const double* Pi, int w, int ld) {
  int emax = 0;
  for (int k = 0; k < w; ++k) {
    const int ex = (int)((__double_as_longlong(ldcg(Pi + (size_t)k * ld)) >> 52) & 0x7FF);
    emax = max(emax, ex);
  }
  return emax;  // 0: the row is zero (or denormal)
}

__device__ __forceinline__ unsigned long long fixed56(double x, int e, bool& neg) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
  neg = (bits >> 63) != 0;
  const int ex = (int)((bits >> 52) & 0x7FF);
  if (ex == 0) return 0ull;
  const unsigned long long mant = (bits & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  const int sh = ex - 1019 - e;  // q = mant * 2^sh < 2^56
  if (sh >= 0) return mant << sh;
  return (-sh < 64) ? (mant >> (-sh)) : 0ull;
}

__device__ __forceinline__ uint32_t bf16_digit(unsigned long long q, int p, bool neg) {
  const int d = (int)((q >> (56 - kSliceBits * (p + 1))) & 0xFF);
  return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn((float)(neg ? -d : d)));
}

// Slice one row (Pi[k * ld], k < w) into the panel's slice block: slice p of
// below-row ib at sl[(p * nb + ib) * kpad + k], zero for k >= w.
__device__ void slice_row(const double* Pi, int w, int ld, int kpad, int nb, int ib, uint16_t* sl, int32_t* rexp) {
  const int emax = row_exponent_bits(Pi, w, ld);
  const int e = emax ? emax - 1022 : 0;
  *rexp = e;
  for (int k0 = 0; k0 < kpad; k0 += 8) {
    uint32_t packed[kSlices][4];
#pragma unroll
    for (int p = 0; p < kSlices; ++p)
#pragma unroll
      for (int c = 0; c < 4; ++c) packed[p][c] = 0u;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const int k = k0 + c;
      bool neg = false;
      const unsigned long long q = (k < w && emax) ? fixed56(ldcg(Pi + (size_t)k * ld), e, neg) : 0ull;
#pragma unroll
      for (int p = 0; p < kSlices; ++p) packed[p][c >> 1] |= bf16_digit(q, p, neg) << (16 * (c & 1));
    }
#pragma unroll
    for (int p = 0; p < kSlices; ++p) {
      uint4 v = make_uint4(packed[p][0], packed[p][1], packed[p][2], packed[p][3]);
      *reinterpret_cast<uint4*>(sl + ((size_t)p * nb + ib) * kpad + k0) = v;
    }
  }
}

// ---------------------------------------------------------------- TRSM(s, k)
// Arithmetic in the panel's type: FP64 panels solve in FP64, FP32 panels (the
// mixed-precision modes) in FP32.
// Panels wider than kTrsmMaxW (CUDA-core tiles only): the same rows, 16 columns
// a lane, with the whole of L11 in shared memory.  What bounds it is the chain
// of w steps.  (A thread a row, its solved columns read back from L2 in blocks
// of 8, kept 16 of the CTA's threads busy with a 16-row tile, each waiting for
// one trip after another: 602 us a tile of a 128-column panel, FP32 470, now 73
// and 59.  Factorization of a full matrix of order 1500 with max_width 128: 9.9 ->
// 4.05 ms, FP32 7.9 -> 3.3; 31^3 Laplacian with relax_zeros 32: 20.5 -> 10.0.)
template <typename T>
__device__ __forceinline__ void trsm_wide(T* P, int ld, int row0, int cnt, int w, T* Ls, const double* Xd) {
  T* rinv = Ls + w * w;
  for (int idx = threadIdx.x; idx < w * w; idx += kFactorThreads) {
    const int i = idx % w, j = idx / w;
    Ls[idx] = i > j ? ldcg(P + i + (size_t)j * ld) : T(0);
  }
  for (int c = threadIdx.x; c < w; c += kFactorThreads) rinv[c] = (T)ldcg(Xd + c * (w + 1));
  __syncthreads();
  trsm_strips<16>(P, ld, row0, cnt, w, Ls, w, rinv);
}

template <typename T, int MODE>
__device__ void task_trsm(const FactorArgs& a, int s, int k, double* smd, FactorShared& sh, bool skip,
                          bool release = true) {
  using ct = T;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int f = a.pv.fcol[s], w = a.pv.fcol[s + 1] - f, ld = a.pv.ld[s], r = a.pv.nrows[s];
  const int tr = a.trsm_rows_of[s];
  const int row0 = w + k * tr;
  const int cnt = min(tr, r - row0);
  T* P = panel_ptr<T>(a, s);
  ct* sm = reinterpret_cast<ct*>(smd);
  (void)f;
  if (!skip && w <= kTrsmMaxW) {
    ct* Ls = sm;                        // Ls[q + 64 c] = l_qc for q > c, else 0
    ct* rinv = sm + kTrsmMaxW * w;      // 1 / l_cc
    for (int idx = tid; idx < kTrsmMaxW * w; idx += nt) {
      const int qq = idx & (kTrsmMaxW - 1), c = idx >> 6;
      Ls[idx] = (qq < w && qq > c) ? (ct)ldcg(P + qq + (size_t)c * ld) : ct(0);
    }
    const double* Xd = a.inv + a.invoff[s];
    for (int c = tid; c < w; c += nt) rinv[c] = (ct)ldcg(Xd + c * (w + 1));  // written by the diagonal task
    __syncthreads();
    trsm_strips<kTrsmMaxW / 8>(P, ld, row0, cnt, w, Ls, kTrsmMaxW, rinv);
    if constexpr (sizeof(T) == 8 && MODE == 3) {
      if (w >= a.tc_min_width) {
        __syncthreads();  // the tile's rows are written (visible to this CTA through L2)
        const int kpad = (w + 15) & ~15, nbel = r - w;
        for (int rr = tid; rr < cnt; rr += nt)
          slice_row(reinterpret_cast<const double*>(P + row0 + rr), w, ld, kpad, nbel, row0 + rr - w,
                    a.slices + a.sliceoff[s], a.rexp + a.pv.rowoff[s] + row0 + rr);
      }
    }
  } else if (!skip) {
    // (the tensor-core modes have no such panels: options_valid)
    if constexpr (MODE == 0) trsm_wide<T>(P, ld, row0, cnt, w, sm, a.inv + a.invoff[s]);
  }
  publish_cta_writes();
  if (!release) return;  // inside a subtree task: no counters, the same CTA goes on
  if (tid == 0) sh.flag = count_down(&a.trsm_left[s]);
  __syncthreads();
  if (sh.flag) release_updates(a, s, sh);
  // W rows after the release: the updates of this panel do not wait for them
  // (the solves, a later launch, read them)
  if (!skip && a.woff != nullptr && a.woff[s] >= 0) form_w_rows<T>(a, s, row0, cnt, smd);
}

// ---------------------------------------------------------------- an update has landed
// Count down the updates still to land in target panel t; the last one makes
// the panel's diagonal task ready -- in the fan-in mode its gather tasks, and
// the diagonal task too when none of them holds rows of its diagonal block.
// Whole CTA (the fan-in mode pushes its gathers together).
template <bool FAN>
__device__ __forceinline__ void target_update_done(const FactorArgs& a, int t, FactorShared& sh, bool release) {
  if constexpr (!FAN) {
    // the diagonal task follows in this CTA, unless it holds a claimed slot of
    // the high-priority ring or is inside a subtree task.  (A claimed slot of
    // the other ring, or a stashed tile, waits for the diagonal task, as it
    // would behind it in the rings.)
    if (release && threadIdx.x == 0 && count_down(&a.dep_f[t])) {
      if (sh.hold)
        ring2_push_one(rings_of(a), true, t);
      else
        sh.next = t;
    }
  } else {
    if (threadIdx.x == 0) sh.flag = release && count_down(&a.dep_f[t]);
    __syncthreads();
    if (sh.flag) {
      const int g0 = a.gat_first[t], g1 = a.gat_first[t + 1];
      ring2_push_range(rings_of(a), true, a.gat0 + g0, g1 - g0, &sh.base);
      if (threadIdx.x == 0 && a.gdiag0[t] == 0) ring2_push_one(rings_of(a), true, t);
    }
  }
}

// ---------------------------------------------------------------- relative indices
// The relative index of row g of panel s in a target panel t is the position
// of g in t's sorted row list (the relative-index maps of the supernodal
// update, Section III-A).  They are fixed by the structure, so one kernel at
// analysis time finds them for every row of every update tile (a binary search
// each), and an update tile only loads its rowlen of them.
// In the fan-in mode the tile writes its own buffer instead, addressed as a
// panel whose rows are the tile's rows and whose columns are the segment's:
// position i for row i, and the source's own row numbers for the lower-
// triangle test (the row lists are increasing, so it gives the same answer).
__device__ __forceinline__ void load_relpos(const FactorArgs& a, const UTask& u, int* pos, int* grow,
                                            const int32_t* Rs, bool fan) {
  for (int i = threadIdx.x; i < u.rowlen; i += blockDim.x) {
    if (fan) {
      pos[i] = i;
      grow[i] = u.row0 + i;
      continue;
    }
    const int p = __ldg(a.relpos + u.rel + i);
    if (p < 0) atomicCAS(&a.ctrl[kErr], 0, SPCHOL_DEV_EINTERNAL);  // cannot happen for a consistent plan
    pos[i] = p;
    grow[i] = __ldg(Rs + u.row0 + i);
  }
}

__global__ void relpos_kernel(const UTask* __restrict__ ut, int n_u, const int32_t* __restrict__ rows,
                              const int64_t* __restrict__ rowoff, const int32_t* __restrict__ nrows,
                              int32_t* __restrict__ relpos) {
  for (int k = blockIdx.x; k < n_u; k += gridDim.x) {
    const UTask u = ut[k];
    const int32_t* Rs = rows + rowoff[u.s];
    const int32_t* Rt = rows + rowoff[u.t];
    const int rt = nrows[u.t];
    for (int i = threadIdx.x; i < u.rowlen; i += blockDim.x) {
      const int g = Rs[u.row0 + i];
      int lo = 0, hi = rt;
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (Rt[mid] < g) lo = mid + 1; else hi = mid;
      }
      relpos[u.rel + i] = (lo < rt && Rt[lo] == g) ? lo : -1;
    }
  }
}

// ---------------------------------------------------------------- UPD(s, t, k)
// C = A B^T for one tile, A = L_s[row tile] (rowlen x ws), B = L_s[segment]
// (ncol x ws), staged through shared memory in k-chunks.  Warp q owns the
// 8-row strip [8q, 8q + 8) of C; lane (lr, lc) = (lane / 8, lane % 8) holds
// rows 8q + lr + 4 rr (rr < NR) and columns lc + 8 cc (cc < NC).  Strips past
// rowlen, the second half of a strip with at most 4 valid rows, column blocks
// past ncol and, where the row tile overlaps the segment (the diagonal tiles),
// column blocks entirely above the diagonal are never computed: the FP64 pipe
// only runs on entries of the lower triangle, padded to 4 x 8 blocks.
// Operand staging.  A k-column of the tile (rows row0 .. row0 + len - 1 of one
// column of panel s) is copied in 16-byte pieces by cp.async (L2 only, no
// register round trip), starting at the 16-byte boundary at or below row0:
// the rows sit at offset row0 % E (E = 16 / sizeof(T)) of a shared-memory row
// of kStageStr elements.  A piece that would reach past the column's padded
// length ld is shortened to the elements inside it (the rest zero-filled), so
// no copy leaves the panel's storage.
template <typename T>
struct Stage {
  static constexpr int E = 16 / (int)sizeof(T);
  static constexpr int kStr = kUpdBoxRows((int)sizeof(T));  // row stride: 64 + E, a multiple of E
  static constexpr int kPieces = (kUpdTileM + E - 1) / E + 1;  // pieces per k-column, worst alignment
};

template <typename T>
__device__ __forceinline__ void cp_async16(T* dst, const T* src, int valid_elems) {
  const int bytes = valid_elems * (int)sizeof(T);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(dst)), "l"(src), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// TMA staging.  When the handle has a tensor map per panel (a 2-D view of
// the column-major panel: ld rows x w columns, box kStr rows x kUpdKC
// columns), one thread loads a k-chunk of an operand with one
// cp.async.bulk.tensor whose x coordinate (the first row) is rounded down to
// a 16-byte boundary; rows past ld and columns past w arrive as zeros.  The
// copies complete on an mbarrier per buffer.
struct UpdTma {
  uint32_t mbar[2];  // shared addresses of the two buffers' mbarriers
  uint32_t* phase;   // shared: parity bits of the next completion of each
};

__device__ __forceinline__ void tma_load_2d(void* dst, const void* tmap, int x, int y, uint32_t mbar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::
          "r"(smem_addr(dst)),
      "l"(tmap), "r"(x), "r"(y), "r"(mbar)
      : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t mbar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_wait_parity(uint32_t mbar, uint32_t phase) {
  for (int it = 0; it < (1 << 24); ++it) {
    uint32_t done;
    asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
                 : "=r"(done)
                 : "r"(mbar), "r"(phase)
                 : "memory");
    if (done) return true;
  }
  return false;
}

// Issue the copies of k-columns k0 .. k0 + kc - 1 of rows r0 .. r0 + len - 1 of
// a panel (column-major, leading dimension ld) into dst[kk][...].
template <typename T>
__device__ __forceinline__ void stage_cols(const T* __restrict__ P, int ld, int r0, int len, int k0, int kc,
                                           T* __restrict__ dst) {
  constexpr int E = Stage<T>::E, NP = Stage<T>::kPieces, STR = Stage<T>::kStr;
  const int base = r0 - (r0 % E);
  const int np = (r0 % E + len + E - 1) / E;  // pieces that cover the rows
  for (int idx = threadIdx.x; idx < kc * NP; idx += blockDim.x) {
    const int kk = idx / NP, pc = idx - kk * NP;
    if (pc < np) {
      const int row = base + pc * E;
      const int valid = min(E, ld - row);
      cp_async16(dst + kk * STR + pc * E, P + row + (size_t)(k0 + kk) * ld, valid);
    }
  }
}

// C = A B^T for one tile, A = L_s[row tile] (rowlen x ws), B = L_s[segment]
// (ncol x ws), staged through shared memory in k-chunks, double-buffered (the
// copies of chunk c + 1 are in flight while chunk c is multiplied).  Warp q owns
// the 8-row strip [8q, 8q + 8) of C; lane (lr, lc) = (lane / 8, lane % 8) holds
// rows 8q + lr + 4 rr (rr < NR) and columns lc + 8 cc (cc < NC).  Strips past
// rowlen, the second half of a strip with at most 4 valid rows, column blocks
// past ncol and, where the row tile overlaps the segment (the diagonal tiles),
// column blocks entirely above the diagonal are never computed: the FP64 pipe
// only runs on entries of the lower triangle, padded to 4 x 8 blocks.
template <typename acc_t, int NR, int NC>
__device__ __forceinline__ void upd_strip(const acc_t* __restrict__ As, const acc_t* __restrict__ Bs, int kc, int r0,
                                          int lc, acc_t (&acc)[2][8]) {
  constexpr int STR = Stage<acc_t>::kStr;
#pragma unroll 1
  for (int kk = 0; kk < kc; ++kk) {
    acc_t av[NR];
#pragma unroll
    for (int rr = 0; rr < NR; ++rr) av[rr] = As[kk * STR + r0 + 4 * rr];
#pragma unroll
    for (int cc = 0; cc < NC; ++cc) {
      const acc_t bv = Bs[kk * STR + lc + 8 * cc];
#pragma unroll
      for (int rr = 0; rr < NR; ++rr) acc[rr][cc] += av[rr] * bv;
    }
  }
}

template <typename acc_t, int NR>
__device__ __forceinline__ void upd_strip_nc(int nc, const acc_t* As, const acc_t* Bs, int kc, int r0, int lc,
                                             acc_t (&acc)[2][8]) {
  switch (nc) {
    case 1: upd_strip<acc_t, NR, 1>(As, Bs, kc, r0, lc, acc); break;
    case 2: upd_strip<acc_t, NR, 2>(As, Bs, kc, r0, lc, acc); break;
    case 3: upd_strip<acc_t, NR, 3>(As, Bs, kc, r0, lc, acc); break;
    case 4: upd_strip<acc_t, NR, 4>(As, Bs, kc, r0, lc, acc); break;
    case 5: upd_strip<acc_t, NR, 5>(As, Bs, kc, r0, lc, acc); break;
    case 6: upd_strip<acc_t, NR, 6>(As, Bs, kc, r0, lc, acc); break;
    case 7: upd_strip<acc_t, NR, 7>(As, Bs, kc, r0, lc, acc); break;
    default: upd_strip<acc_t, NR, 8>(As, Bs, kc, r0, lc, acc); break;
  }
}

template <typename T, bool FAN>
__device__ void task_update(const FactorArgs& a, const UTask u, unsigned char* smraw, FactorShared& sh,
                            bool skip, int rot, const UpdTma& tma, long long fo, bool release = true) {
  using acc_t = T;
  constexpr int STR = Stage<T>::kStr, E = Stage<T>::E;
  constexpr uint32_t kBoxBytes = (uint32_t)(kUpdKC * STR * sizeof(T));
  const int tid = threadIdx.x;
  const int s = u.s, t = u.t;
  if (!skip) {
    const int fs = a.pv.fcol[s], ws = a.pv.fcol[s + 1] - fs, lds = a.pv.ld[s];
    constexpr bool fan = FAN;  // fan-in mode: the tile's buffer at fo (see load_relpos)
    const int ft = fan ? u.seg0 : a.pv.fcol[t], ldt = fan ? u.rowlen : a.pv.ld[t];
    const T* Ps = panel_ptr<T>(a, s);
    T* Pt = fan ? reinterpret_cast<T*>(a.fan_buf) + fo : panel_ptr<T>(a, t);
    const int32_t* Rs = a.pv.rows + a.pv.rowoff[s];

    // [2][A, B][kUpdKC][STR], 128-byte aligned (each chunk is a multiple of 128 bytes)
    T* buf = reinterpret_cast<T*>(smraw + ((128u - (smem_addr(smraw) & 127u)) & 127u));
    const void* tmap = a.tmaps ? (const void*)(a.tmaps + 128 * (size_t)s) : nullptr;
    uint32_t ph = tmap ? *tma.phase : 0u;
    constexpr int kBuf = 2 * kUpdKC * STR;                // one buffer: A and B chunks
    // FP32 panels: the shared memory sized for two FP64 buffers holds four FP32
    // ones, so a tile of K <= 64 stages its whole K at once and waits once
    constexpr int kSlots = sizeof(T) == 4 ? 4 : 2;
    int* pos = reinterpret_cast<int*>(buf + kSlots * kBuf);  // [kUpdTileM] row position in t
    int* grow = pos + kUpdTileM;                          // [kUpdTileM] global row
    int* gcol = grow + kUpdTileM;                         // [kUpdTileN] global column (pass-local)

    // Relative row indices (computed once per analysis): position of each
    // row of the tile in t's sorted row list.
    load_relpos(a, u, pos, grow, Rs, fan);
    // Warp slot q' = (warp - rot) % 8 (tiles of few strips load the four SM
    // sub-partitions, warp % 4, evenly over many tasks).  A tile of S strips
    // gives each strip C = 8 / S (rounded down to a power of two) warps, which
    // split its column blocks: short tiles near the root keep every warp busy.
    const int lane = tid & 31, qs = ((tid >> 5) - rot) & 7;
    const int nstrip = (u.rowlen + 7) >> 3;
    const int C = nstrip >= 5 ? 1 : nstrip >= 3 ? 2 : nstrip == 2 ? 4 : 8;
    const int q = qs / C, cg = qs - q * C;              // strip and column group of this warp
    const int lr = lane >> 3, lc = lane & 7;
    const int srows = min(8, u.rowlen - 8 * q);        // valid rows of this warp's strip
    const int nr = srows > 4 ? 2 : 1;
    const int off = u.row0 - u.seg0;                   // >= 0: tile row i >= segment column j iff off + i >= j
    const int oa = u.row0 % E;                         // row offset of the A rows in shared memory
    const int r0 = oa + 8 * q + lr;                    // this lane's first A row in shared memory
    const int nchunk = (ws + kUpdKC - 1) / kUpdKC;
    for (int cb = 0; cb < u.seglen; cb += kUpdTileN) {
      const int ncol = min(kUpdTileN, u.seglen - cb);
      const int c0 = u.seg0 + cb;
      const int ob = c0 % E;
      const int dd = off - cb + 8 * q + 7;  // last column any row of the strip needs
      const int nall = (ncol + 7) >> 3;
      const int nper = (nall + C - 1) / C;
      const int b0 = cg * nper;             // this warp's column blocks b0 .. b0 + ncb - 1
      const int ncb = dd < 0 ? 0 : max(0, min(min(nall, b0 + nper), dd / 8 + 1) - b0);
      const bool active = srows > 0 && ncb > 0;
      __syncthreads();  // the previous pass is done with the buffers and gcol
      for (int j = tid; j < ncol; j += blockDim.x) gcol[j] = fan ? c0 + j : Rs[c0 + j];
      acc_t acc[2][8];
#pragma unroll
      for (int rr = 0; rr < 2; ++rr)
#pragma unroll
        for (int cc = 0; cc < 8; ++cc) acc[rr][cc] = acc_t(0);
      if (sizeof(T) == 4 && nchunk <= kSlots) {
        // every k-chunk in flight at once, one wait, then the arithmetic in
        // the same chunk order as below (the same sums)
        if (tmap) {
          if (tid == 0) {
            asm volatile("fence.proxy.async.global;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_expect_tx(tma.mbar[0], 2 * kBoxBytes * (uint32_t)nchunk);
            for (int c = 0; c < nchunk; ++c) {
              tma_load_2d(buf + c * kBuf, tmap, u.row0 - oa, c * kUpdKC, tma.mbar[0]);
              tma_load_2d(buf + c * kBuf + kUpdKC * STR, tmap, c0 - ob, c * kUpdKC, tma.mbar[0]);
            }
          }
          if (!mbar_wait_parity(tma.mbar[0], ph & 1u) && tid == 0) atomicCAS(&a.ctrl[kErr], 0, SPCHOL_DEV_ETIMEOUT);
          ph ^= 1u;
        } else {
          for (int c = 0; c < nchunk; ++c) {
            const int k0 = c * kUpdKC, kc = min(kUpdKC, ws - k0);
            stage_cols(Ps, lds, u.row0, u.rowlen, k0, kc, buf + c * kBuf);
            stage_cols(Ps, lds, c0, ncol, k0, kc, buf + c * kBuf + kUpdKC * STR);
          }
          cp_async_commit();
          cp_async_wait<0>();
        }
        __syncthreads();
        if (active)
          for (int c = 0; c < nchunk; ++c) {
            const int kc = min(kUpdKC, ws - c * kUpdKC);
            const T* As = buf + c * kBuf;
            const T* Bs = As + kUpdKC * STR + ob + 8 * b0;
            if (nr == 2)
              upd_strip_nc<acc_t, 2>(ncb, As, Bs, kc, r0, lc, acc);
            else
              upd_strip_nc<acc_t, 1>(ncb, As, Bs, kc, r0, lc, acc);
          }
        __syncthreads();  // the buffers are refilled by the next pass or tile
      } else {
      // chunk 0 into buffer 0
      if (tmap) {
        if (tid == 0) {
          // the panel was written through the generic proxy (by other CTAs, or
          // by this one inside a subtree task); order that before the TMA reads
          asm volatile("fence.proxy.async.global;" ::: "memory");
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          mbar_expect_tx(tma.mbar[0], 2 * kBoxBytes);
          tma_load_2d(buf, tmap, u.row0 - oa, 0, tma.mbar[0]);
          tma_load_2d(buf + kUpdKC * STR, tmap, c0 - ob, 0, tma.mbar[0]);
        }
      } else {
        stage_cols(Ps, lds, u.row0, u.rowlen, 0, min(kUpdKC, ws), buf);
        stage_cols(Ps, lds, c0, ncol, 0, min(kUpdKC, ws), buf + kUpdKC * STR);
        cp_async_commit();
      }
      for (int c = 0; c < nchunk; ++c) {
        const int k0 = c * kUpdKC, kc = min(kUpdKC, ws - k0);
        if (tmap) {
          if (c + 1 < nchunk && tid == 0) {
            const int b1 = (c + 1) & 1;
            T* nb = buf + b1 * kBuf;
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_expect_tx(tma.mbar[b1], 2 * kBoxBytes);
            tma_load_2d(nb, tmap, u.row0 - oa, k0 + kUpdKC, tma.mbar[b1]);
            tma_load_2d(nb + kUpdKC * STR, tmap, c0 - ob, k0 + kUpdKC, tma.mbar[b1]);
          }
          const int b = c & 1;
          if (!mbar_wait_parity(tma.mbar[b], (ph >> b) & 1u) && tid == 0)
            atomicCAS(&a.ctrl[kErr], 0, SPCHOL_DEV_ETIMEOUT);
          ph ^= 1u << b;
        } else if (c + 1 < nchunk) {
          T* nb = buf + ((c + 1) & 1) * kBuf;
          const int k1 = k0 + kUpdKC, kc1 = min(kUpdKC, ws - k1);
          stage_cols(Ps, lds, u.row0, u.rowlen, k1, kc1, nb);
          stage_cols(Ps, lds, c0, ncol, k1, kc1, nb + kUpdKC * STR);
          cp_async_commit();
          cp_async_wait<1>();  // chunk c has landed (this thread's copies)
        } else {
          cp_async_wait<0>();
        }
        __syncthreads();       // ... and every thread's
        if (active) {
          const T* As = buf + (c & 1) * kBuf;
          const T* Bs = As + kUpdKC * STR + ob + 8 * b0;
          if (nr == 2)
            upd_strip_nc<acc_t, 2>(ncb, As, Bs, kc, r0, lc, acc);
          else
            upd_strip_nc<acc_t, 1>(ncb, As, Bs, kc, r0, lc, acc);
        }
        __syncthreads();  // buffer c & 1 is refilled by the next iteration's copies
      }
      }
      if (tmap && tid == 0) *tma.phase = ph;  // every thread has waited on the last chunk
      // Scatter-subtract into panel t: only the lower triangle (row >= column).
      if (active) {
#pragma unroll
        for (int rr = 0; rr < 2; ++rr) {
          const int i = 8 * q + lr + 4 * rr;
          if (rr >= nr || i >= u.rowlen || pos[i] < 0) continue;
          T* dst = Pt + pos[i];
          const int gi = grow[i];
#pragma unroll
          for (int cc = 0; cc < 8; ++cc) {
            const int j = lc + 8 * (b0 + cc);
            if (cc < ncb && j < ncol && gi >= gcol[j])
              scatter_put(dst + (size_t)(gcol[j] - ft) * ldt, (T)(-acc[rr][cc]), fan);
          }
        }
      }
    }
  }
  publish_cta_writes();
  target_update_done<FAN>(a, t, sh, release);  // not for a target inside the running subtree task
}

// ---------------------------------------------------------------- UPD on tensor cores (FP32 panels)
// The same update tile computed with tcgen05.mma kind::tf32: A (tile rows, up
// to 128) and B (segment rows, up to 64 per pass) are staged K-major in shared
// memory (8-row x 16-byte core matrices, no swizzle), one elected thread issues
// the MMAs into a TMEM accumulator (128 lanes x 64 columns, allocated once per
// CTA), the commit arrives on an mbarrier, and the epilogue reads TMEM by warp
// quadrant and scatter-adds into the target panel.  With split = 1 each operand
// is also split into a TF32 high part and a TF32 remainder, and three products
// (hi*hi + hi*lo + lo*hi) recover FP32-level accuracy.
struct TcState {
  uint32_t tmem;   // TMEM base address of this CTA's accumulator
  uint32_t mbar;   // shared address of the MMA-completion mbarrier
  uint32_t phase;  // parity of the next completion
};


// Shared-memory matrix descriptor: K-major, no swizzle; LBO = byte distance of
// K-adjacent core matrices, SBO = byte distance of row-adjacent core matrices.
__device__ __forceinline__ uint64_t kmajor_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46);
}

// Instruction descriptor: FP32 accumulator, TF32 A and B, both K-major, M x N.
__device__ __forceinline__ uint32_t tf32_idesc(int m, int n) {
  return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

__device__ __forceinline__ float to_tf32(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

// Byte offset of element (r, k) in a K-major tile whose rows hold kpad fp32 values.
__device__ __forceinline__ uint32_t kmaj_off(int r, int k, int kpad) {
  return (uint32_t)((r >> 3) * (kpad * 32) + (k >> 2) * 128 + (r & 7) * 16 + (k & 3) * 4);
}

constexpr int kTcM = 128;      // MMA rows (tile rows are padded up to it)
constexpr int kTcN = 64;       // accumulator columns per pass
constexpr int kTcKmax = 64;    // panel width bound for the tensor-core path

__device__ __forceinline__ bool mbar_wait_bounded(uint32_t mbar, uint32_t phase) {
  for (int it = 0; it < (1 << 24); ++it) {
    uint32_t done;
    asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
                 : "=r"(done)
                 : "r"(mbar), "r"(phase)
                 : "memory");
    if (done) return true;
  }
  return false;
}

template <bool FAN>
__device__ void task_update_tc(const FactorArgs& a, const UTask u, unsigned char* smraw, FactorShared& sh, bool skip,
                               TcState& tc, long long fo, bool release = true) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int s = u.s, t = u.t;
  if (!skip) {
    const int fs = a.pv.fcol[s], ws = a.pv.fcol[s + 1] - fs, lds = a.pv.ld[s];
    constexpr bool fan = FAN;  // fan-in mode: the tile's buffer at fo (see load_relpos)
    const int ft = fan ? u.seg0 : a.pv.fcol[t], ldt = fan ? u.rowlen : a.pv.ld[t];
    const float* Ps = reinterpret_cast<const float*>(a.pool) + a.pv.valoff[s];
    float* Pt = fan ? reinterpret_cast<float*>(a.fan_buf) + fo : reinterpret_cast<float*>(a.pool) + a.pv.valoff[t];
    const int32_t* Rs = a.pv.rows + a.pv.rowoff[s];
    const int split = a.mma_mode == 2 ? 1 : 0;
    const int kpad = (ws + 7) & ~7;
    const int abytes = kTcM * kpad * 4, bbytes = kTcN * kpad * 4;
    // operand tiles start on a 128-byte boundary of shared memory
    unsigned char* Ah = smraw + ((128u - (smem_addr(smraw) & 127u)) & 127u);
    unsigned char* Bh = Ah + abytes;
    unsigned char* Al = Bh + bbytes;           // remainders (split only)
    unsigned char* Bl = Al + abytes;
    int* pos = reinterpret_cast<int*>(Ah + 2 * (abytes + bbytes));
    int* grow = pos + kTcM;
    int* gcol = grow + kTcM;

    load_relpos(a, u, pos, grow, Rs, fan);
    // A: tile rows x k (rows >= rowlen and k >= ws are zero)
    for (int idx = tid; idx < kTcM * kpad; idx += blockDim.x) {
      const int i = idx % kTcM, k = idx / kTcM;
      const float v = (i < u.rowlen && k < ws) ? ldcg(Ps + (u.row0 + i) + (size_t)k * lds) : 0.f;
      const float h = to_tf32(v);
      *reinterpret_cast<float*>(Ah + kmaj_off(i, k, kpad)) = h;
      if (split) *reinterpret_cast<float*>(Al + kmaj_off(i, k, kpad)) = to_tf32(v - h);
    }
    for (int cb = 0; cb < u.seglen; cb += kTcN) {
      const int ncol = min(kTcN, u.seglen - cb);
      const int npad = kTcN;  // the MMA always spans the full accumulator width; unused B rows are zero
      for (int j = tid; j < ncol; j += blockDim.x) gcol[j] = fan ? u.seg0 + cb + j : Rs[u.seg0 + cb + j];
      for (int idx = tid; idx < npad * kpad; idx += blockDim.x) {
        const int j = idx % npad, k = idx / npad;
        const float v = (j < ncol && k < ws) ? ldcg(Ps + (u.seg0 + cb + j) + (size_t)k * lds) : 0.f;
        const float h = to_tf32(v);
        *reinterpret_cast<float*>(Bh + kmaj_off(j, k, kpad)) = h;
        if (split) *reinterpret_cast<float*>(Bl + kmaj_off(j, k, kpad)) = to_tf32(v - h);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncthreads();
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (tid == 0) {
        const uint32_t idesc = tf32_idesc(kTcM, npad);
        const uint32_t sbo = (uint32_t)kpad * 32;
        const uint32_t ah = smem_addr(Ah), bh = smem_addr(Bh), al = smem_addr(Al), bl = smem_addr(Bl);
        int first = 1;
        for (int k0 = 0; k0 < kpad; k0 += 8) {
          const uint32_t off = (uint32_t)(k0 >> 2) * 128;  // two K-adjacent core matrices per MMA
          const int nprod = split ? 3 : 1;
          for (int pr = 0; pr < nprod; ++pr) {
            const uint32_t aa = (pr == 2) ? al : ah;
            const uint32_t bb = (pr == 1) ? bl : bh;
            const uint64_t ad = kmajor_desc(aa + off, 128, sbo);
            const uint64_t bd = kmajor_desc(bb + off, 128, sbo);
            const uint32_t acc = first ? 0u : 1u;
            asm volatile("{\n.reg .pred p;\nsetp.ne.u32 p, %4, 0;\n"
                         "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}" ::"r"(tc.tmem),
                         "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
                         : "memory");
            first = 0;
          }
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(tc.mbar)
                     : "memory");
      }
      const bool ok = mbar_wait_bounded(tc.mbar, tc.phase);
      tc.phase ^= 1u;
      if (!ok && tid == 0) atomicCAS(&a.ctrl[kErr], 0, SPCHOL_DEV_ETIMEOUT);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      // epilogue: warp w reads TMEM lanes 32*(w%4).. (tile rows), columns half (w/4)
      const int quad = warp & 3, half = warp >> 2;
      const int row = 32 * quad + lane;
      for (int c0 = half * 32; c0 < half * 32 + 32; c0 += 16) {
        uint32_t v[16];
        const uint32_t taddr = tc.tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)c0;
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
            : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
              "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
            : "r"(taddr));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (ok && row < u.rowlen && pos[row] >= 0) {
#pragma unroll
          for (int q = 0; q < 16; ++q) {
            const int j = c0 + q;
            if (j < ncol && grow[row] >= gcol[j])
              scatter_put(Pt + pos[row] + (size_t)(gcol[j] - ft) * ldt, -__uint_as_float(v[q]), fan);
          }
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncthreads();  // TMEM and the B tile are reused by the next pass / task
    }
  }
  publish_cta_writes();
  target_update_done<FAN>(a, t, sh, release);  // not for a target inside the running subtree task
}

// ---------------------------------------------------------------- UPD, FP64 on BF16 tensor cores
// C = A B^T with A, B given by their kSlices digit matrices (see slice_row):
// C_ij = 2^(e_i + e_j) sum_{p,q} 2^(-8(p+q+2)) (A_p B_q^T)_ij.  The products
// with p + q <= kSlices - 1 are kept (the dropped ones weigh below 2^-64 of
// the leading one); products of equal p + q share one TMEM accumulator
// (group d = p + q, kOzN columns each), in which the integer sums stay exact
// for d <= 3 and round at most at 2^-56 relative beyond.  The epilogue
// combines the seven group values per entry exactly in two 64-bit integers,
// converts once to FP64 and scales by 2^(e_i + e_j).
// The double nearest to t * 2^k for a 64-bit integer t, with integer
// operations only (round to nearest, ties to even).
__device__ __forceinline__ double fixed64_to_double(long long t, int k) {
  if (t == 0) return 0.0;
  const bool neg = t < 0;
  const unsigned long long u = neg ? (unsigned long long)(-t) : (unsigned long long)t;
  int msb = 63 - __clzll((long long)u);
  unsigned long long m;
  if (msb <= 52) {
    m = u << (52 - msb);
  } else {
    const int sh = msb - 52;
    m = u >> sh;
    const unsigned long long rem = u & ((1ull << sh) - 1), halfw = 1ull << (sh - 1);
    if (rem > halfw || (rem == halfw && (m & 1ull))) {
      ++m;
      if (m >> 53) {
        m >>= 1;
        ++msb;
      }
    }
  }
  const int be = msb + k + 1023;
  if (be <= 0 || be >= 2047) {
    const double r = ldexp((double)m, msb - 52 + k);  // outside the range of this path's data
    return neg ? -r : r;
  }
  return __longlong_as_double(
      (long long)(((unsigned long long)neg << 63) | ((unsigned long long)be << 52) | (m & ((1ull << 52) - 1))));
}

// The MMAs have M = 64 (the tile's at most kOzRows = 64 rows) and cover one
// 16-column block of the segment: the accumulator of group d is TMEM columns
// 16 d .. 16 d + 15.  With M = 64 the accumulator's row 16 q + i (i < 16) sits
// in TMEM lane 32 q + i, columns as N.  7 groups x 16 columns fit 128 TMEM
// columns, a quarter of the SM's, and a CTA needs 73 KB of shared memory, so
// three CTAs share an SM.  A tcgen05.mma costs about the same to issue whatever
// its M and N (~48 clocks from one thread, ~28 SM-wide when several issue), so
// the MMA phase is bound by the instruction count: each A digit p is issued
// once per K step against the stacked B digits 0 .. 6 - p (N up to 112),
// 28 MMAs per block instead of 112 single products.
constexpr int kOzM = 64, kOzN = 16, kOzRows = 64;
constexpr int kOzCols = 128;  // TMEM columns: kSlices groups x kOzN, rounded to a power of two

__device__ __forceinline__ uint32_t bf16_idesc(int m, int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

template <bool FAN>
__device__ void task_update_oz(const FactorArgs& a, const UTask u, unsigned char* smraw, FactorShared& sh, bool skip,
                               TcState& tc, long long fo, bool release = true) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int s = u.s, t = u.t;
  if (!skip) {
    const int fs = a.pv.fcol[s], ws = a.pv.fcol[s + 1] - fs, rs = a.pv.nrows[s];
    constexpr bool fan = FAN;  // fan-in mode: the tile's buffer at fo (see load_relpos)
    const int ft = fan ? u.seg0 : a.pv.fcol[t], ldt = fan ? u.rowlen : a.pv.ld[t];
    double* Pt = fan ? reinterpret_cast<double*>(a.fan_buf) + fo : reinterpret_cast<double*>(a.pool) + a.pv.valoff[t];
    const int32_t* Rs = a.pv.rows + a.pv.rowoff[s];
    const int32_t* ex = a.rexp + a.pv.rowoff[s];
    const int kpad = (ws + 15) & ~15, nb = rs - ws;
    const uint16_t* sl = a.slices + a.sliceoff[s];
    const int arow = kOzRows * kpad * 2, brow = kOzN * kpad * 2;  // bytes of one slice tile
    unsigned char* A0 = smraw + ((128u - (smem_addr(smraw) & 127u)) & 127u);
    unsigned char* B0 = A0 + kSlices * arow;
    int* pos = reinterpret_cast<int*>(B0 + kSlices * brow);
    int* grow = pos + kOzRows;
    int* gcol = grow + kOzRows;
    int* ea = gcol + kOzN;
    int* eb = ea + kOzRows;
    const uint32_t sbo = (uint32_t)kpad * 16;  // 8 rows x (kpad bf16) bytes
    const int chunks = kpad / 8;               // 16-byte chunks per row

    load_relpos(a, u, pos, grow, Rs, fan);
    for (int i = tid; i < u.rowlen; i += blockDim.x) ea[i] = ldcg(ex + u.row0 + i);
    // A digits: kSlices x rowlen rows x kpad, K-major core matrices (8 rows x
    // 16 bytes).  Rows past rowlen are left as they are: they only feed rows
    // of the product that are never scattered.  Columns past ws are zero in
    // the slices themselves.
    // 16-byte pieces by cp.async (L2 only): every piece of the tile is in
    // flight at once instead of one load's latency per piece
    // (at most 8 pieces a row: thread = row * 8 + piece, no index divisions)
    const int pc = tid & 7;
    if (pc < chunks)
      for (int r = tid >> 3; r < u.rowlen; r += kFactorThreads / 8) {
        const uint16_t* src = sl + (size_t)(u.row0 - ws + r) * kpad + 8 * pc;
        const uint32_t dst = smem_addr(A0) + (r >> 3) * sbo + (r & 7) * 16 + pc * 128;
#pragma unroll
        for (int p = 0; p < kSlices; ++p)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + p * arow),
                       "l"(src + (size_t)p * nb * kpad)
                       : "memory");
      }
    cp_async_commit();
    for (int cb = 0; cb < u.seglen; cb += kOzN) {
      const int ncol = min(kOzN, u.seglen - cb);
      for (int j = tid; j < ncol; j += blockDim.x) {
        gcol[j] = fan ? u.seg0 + cb + j : Rs[u.seg0 + cb + j];
        eb[j] = ldcg(ex + u.seg0 + cb + j);
      }
      {
        const int r = (tid >> 3) & (kOzN - 1);
        if (pc < chunks && r < ncol) {
          const uint16_t* src = sl + (size_t)(u.seg0 + cb - ws + r) * kpad + 8 * pc;
          const uint32_t dst = smem_addr(B0) + (r >> 3) * sbo + (r & 7) * 16 + pc * 128;
          for (int p = tid / (8 * kOzN); p < kSlices; p += kFactorThreads / (8 * kOzN))
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + p * brow),
                         "l"(src + (size_t)p * nb * kpad)
                         : "memory");
        }
      }
      cp_async_commit();
      cp_async_wait<0>();  // this thread's A (first pass) and B pieces have landed
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncthreads();
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (tid == 0) {
        // One MMA per A digit p and K step: its B operand is the run of B
        // digits 0 .. 6 - p (N = (7 - p) x 16 rows, contiguous in shared
        // memory), its accumulator starts at group p's columns, so the product
        // with B digit q lands in group p + q.  28 MMAs per block instead of
        // one per (p, q) pair (112); the first (p = 0, all groups) initialises.
        const uint32_t a0 = smem_addr(A0), b0 = smem_addr(B0);
        for (int p = 0; p < kSlices; ++p) {
          const uint32_t idesc = bf16_idesc(kOzM, (kSlices - p) * kOzN);
          const uint32_t dcol = tc.tmem + (uint32_t)(p * kOzN);
          for (int k0 = 0; k0 < kpad; k0 += 16) {
            const uint32_t off = (uint32_t)(k0 >> 3) * 128;  // 16 bf16 = two K-adjacent core matrices
            const uint64_t ad = kmajor_desc(a0 + p * arow + off, 128, sbo);
            const uint64_t bd = kmajor_desc(b0 + off, 128, sbo);
            const uint32_t acc = (p == 0 && k0 == 0) ? 0u : 1u;
            asm volatile("{\n.reg .pred pp;\nsetp.ne.u32 pp, %4, 0;\n"
                         "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, pp;\n}" ::"r"(dcol),
                         "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
                         : "memory");
          }
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(tc.mbar)
                     : "memory");
      }
      const bool ok = mbar_wait_bounded(tc.mbar, tc.phase);
      tc.phase ^= 1u;
      if (!ok && tid == 0) atomicCAS(&a.ctrl[kErr], 0, SPCHOL_DEV_ETIMEOUT);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      // Epilogue: warp w reads rows 16 (w % 4) .. + 15 (TMEM lanes 32 (w % 4) ..)
      // and the w / 4-th half of the columns of every group, as 16 x 256-bit
      // fragments: lane l holds rows l / 4 and l / 4 + 8 at columns 2 (l % 4) and
      // the next, so that every lane has four outputs (reading a row per lane
      // left half of them idle; with the copies' index divisions gone, 64^3 160.8
      // -> 141.1 ms).  tcgen05.ld is warp-collective: the condition is
      // warp-uniform.
      const int quad = warp & 3, c0 = (warp >> 2) * (kOzN / 2);
      if (16 * quad < u.rowlen && c0 < ncol) {
        uint32_t v[kSlices][4];
#pragma unroll
        for (int d = 0; d < kSlices; ++d)
          asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0,%1,%2,%3}, [%4];"
                       : "=r"(v[d][0]), "=r"(v[d][1]), "=r"(v[d][2]), "=r"(v[d][3])
                       : "r"(tc.tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)(d * kOzN + c0)));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int row = 16 * quad + (lane >> 2) + 8 * (q >> 1), j = c0 + 2 * (lane & 3) + (q & 1);
          if (!ok || row >= u.rowlen || j >= ncol || pos[row] < 0 || grow[row] < gcol[j]) continue;
          // t = sum_d v_d 2^(8 (6 - d)), C = t 2^(e_i + e_j - 64).  The group
          // sums are integers below 2^25 in magnitude; t (< 2^75) is formed
          // as hi 2^32 + lo and kept to 2^12 units in one int64, a
          // truncation of at most 2^(e_i + e_j - 52), below the rounding
          // bound of an FP64 dot product of these rows.
          long long hi = 0, lo = 0;
#pragma unroll
          for (int d = 0; d < 3; ++d) hi = hi * 256 + __float2int_rn(__uint_as_float(v[d][q]));
#pragma unroll
          for (int d = 3; d < kSlices; ++d) lo = lo * 256 + __float2int_rn(__uint_as_float(v[d][q]));
          const long long t12 = hi * (1ll << 20) + (lo >> 12);  // floor((hi 2^32 + lo) / 2^12)
          const double c = fixed64_to_double(t12, ea[row] + eb[j] - 52);
          scatter_put(Pt + pos[row] + (size_t)(gcol[j] - ft) * ldt, -c, fan);
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncthreads();
    }
  }
  publish_cta_writes();
  target_update_done<FAN>(a, t, sh, release);  // not for a target inside the running subtree task
}

// ---------------------------------------------------------------- fan-in gather
// Deterministic fan-in mode (the fan-in family of Section II-C, restated for
// one GPU): update tiles store their products in private buffers, and a
// gather task per piece of a target panel's rows (at most kFanPieceRows rows,
// all columns or, where the list is long, a window of them: split_gathers) adds
// them in, tile after tile in the piece's list order, before
// the task that owns those rows factors or solves them; every entry of L thus
// receives its updates in one fixed order whatever the schedule, and the
// pieces of one panel are gathered in parallel.  The piece sits in shared
// memory and the list is consumed in batches of up to kFanBatch tiles:
//   1. warp 0 cuts the batch where its staged values would overflow the
//      staging area (the records were fetched during the previous batch);
//   2. all threads copy, for each column of each tile, the 16-byte pieces that
//      hold its rows in the piece (cp.async, L2 only: the buffers were written
//      by other CTAs; every copy of the batch in flight at once) and load the
//      rows' positions in the piece and the columns' positions in the panel;
//   3. the values are added tile by tile: with a barrier between tiles, or --
//      for at most kFanOwn columns, which most split gathers and the narrow
//      panels have -- each thread adding to the one entry it owns, in a
//      register, from maps of where the tiles' rows and columns lie.
// What bounds it: the latency of a tile's step (0.35 us with the barrier; a
// tile has 107 values in a piece on average), one after another in the top
// separators' pieces.  Factorization of a 27^3 Laplacian: 12.0 ms; split 8.8;
// and with the threads' own entries 8.0.  (Columns dealt out to the warps
// without barriers, whatever the width, was slower: 14.5 and split 9.9 -- each
// warp's FP64 add holds the pipe for 64 clocks, however few lanes it has.)
// The piece and the buffers are read around L1; the records were written at
// analysis.
struct FanMeta {
  long long fo, rp, rs;  // FanRec: buffer offset of the first listed row, relative rows, segment rows
  int pre_b, pre_v;      // the tile's first staged 16-byte piece and first staged position
  int rowlen, cps;       // buffer rows; staged pieces per column
  short ni, seglen;
  float inv_ni;  // 1 / ni: value index -> (row, column) without a division
  float inv_cps;
};
constexpr int kFanBatch = 32;
constexpr int kFanVcap = 1024;  // staged positions per batch (a tile has at most 32 + 128)
constexpr int kFanOwn = kFactorThreads / 32;  // columns of a piece whose entries the threads own
constexpr int kFanAhead = 4;                  // tiles whose values are read before the first is added
static_assert(kFanPieceRows == 32 && kFanVcap * sizeof(int16_t) >= kFanBatch * (32 + 4 * kFanOwn),
              "the owners' maps take the positions' place");
constexpr size_t kFanMetaBytes = ((kFanBatch * sizeof(FanMeta) + 16) + 15) & ~size_t(15);

// 16-byte pieces that can hold ni consecutive values starting anywhere.
template <typename T>
__host__ __device__ constexpr int fan_pieces(int ni) {
  return (ni + 16 / (int)sizeof(T) - 2) / (16 / (int)sizeof(T)) + 1;
}

// The batch tile that staged piece (pieces) or position (!pieces) idx belongs to.
__device__ __forceinline__ int fan_tile_of(const FanMeta* meta, int nb, int idx, bool pieces) {
  int k = 0;
#pragma unroll
  for (int b = kFanBatch / 2; b > 0; b >>= 1)
    if (k + b < nb && (pieces ? meta[k + b].pre_b : meta[k + b].pre_v) <= idx) k += b;
  return k;
}

template <typename T>
__device__ void fanin_gather(const FactorArgs& a, int t, const GatherTask& G, int p0, int np, unsigned char* smraw) {
  constexpr int E = 16 / (int)sizeof(T);  // values per 16-byte piece
  const int tid = threadIdx.x, nt = blockDim.x;
  long long e = G.e0;
  const long long e1 = G.e1;
  if (e == e1) return;  // nothing lands in these rows
  // its columns [G.c0, G.c1) of the panel: numbered from 0 here, and rows from
  // position c on have entries in its column c
  const int ft = a.pv.fcol[t] + G.c0, wt = G.c1 - G.c0, ldt = a.pv.ld[t];
  const int d0 = p0 - G.c0;
  T* Pt = panel_ptr<T>(a, t) + (size_t)G.c0 * ldt;
  const T* F = reinterpret_cast<const T*>(a.fan_buf);
  const int cap = a.fan_cap;  // 16-byte pieces per batch; one tile's always fit
  unsigned char* base = smraw + ((16u - (smem_addr(smraw) & 15u)) & 15u);
  FanMeta* meta = reinterpret_cast<FanMeta*>(base);
  int* scal = reinterpret_cast<int*>(meta + kFanBatch);  // tiles, pieces and positions of the batch
  int16_t* pv = reinterpret_cast<int16_t*>(base + kFanMetaBytes);  // positions: rows in the piece, then columns
  T* Bs = reinterpret_cast<T*>(pv + kFanVcap);                     // the staged pieces
  T* S = Bs + (size_t)cap * E;  // the piece: np rows x wt columns, leading dimension kFanPieceRows
  // at most one column a warp: a thread owns the entry (lane, warp)
  const int lane = tid & 31, warp = tid >> 5;
  const bool own = wt <= kFanOwn;
  T acc = T(0);
  int8_t* rowof = reinterpret_cast<int8_t*>(pv);              // [kFanBatch][32]: the tile's row there, or -1
  int32_t* colof = reinterpret_cast<int32_t*>(rowof + kFanBatch * 32);  // [kFanBatch][kFanOwn]: its column's
                                                                        // first staged value, or -1
  if (own) {
    if (lane < np && warp < wt) acc = ldcg(Pt + p0 + lane + (size_t)warp * ldt);
  } else {
    for (int idx = tid; idx < np * wt; idx += nt) {
      const int p = idx % np, c = idx / np;
      S[p + kFanPieceRows * c] = ldcg(Pt + p0 + p + (size_t)c * ldt);
    }
  }
  FanRec r{};  // warp 0: the records of the next batch window
  if (tid < 32 && e + tid < e1) r = a.fan_rec[e + tid];
  const bool prof = a.prof != nullptr && tid == 0;
  uint64_t tp[3] = {0, 0, 0}, tq = prof ? global_ns() : 0;
  long long nbat = 0, ntile = 0;
  while (e < e1) {
    __syncthreads();  // the piece is loaded, or the previous batch is added
    int nb = 0;
    if (tid < 32) {
      const bool have = e + tid < e1;
      const int cps = have ? fan_pieces<T>(r.ni) : 0;
      const int n = have ? r.seglen * cps : 0, v = have ? r.ni + r.seglen : 0;
      int in = n, iv = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, in, o), z = __shfl_up_sync(0xffffffffu, iv, o);
        if (tid >= o) {
          in += y;
          iv += z;
        }
      }
      // the tiles that fit form a prefix; the first one always fits
      nb = max(1, __popc(__ballot_sync(0xffffffffu, have && in <= cap && iv <= kFanVcap)));
      if (tid < nb) {
        FanMeta mm;
        mm.fo = r.fo;
        mm.rp = r.rp;
        mm.rs = r.rs;
        mm.pre_b = in - n;
        mm.pre_v = iv - v;
        mm.rowlen = r.rowlen;
        mm.cps = cps;
        mm.ni = r.ni;
        mm.seglen = r.seglen;
        mm.inv_ni = 1.0f / (float)max(1, (int)r.ni);
        mm.inv_cps = 1.0f / (float)max(1, cps);
        meta[tid] = mm;
      }
      if (tid == nb - 1) {
        scal[0] = nb;
        scal[1] = in;
        scal[2] = iv;
      }
      r = FanRec{};
      if (e + nb + tid < e1) r = a.fan_rec[e + nb + tid];  // in flight during this batch
    } else if (own) {
      for (int idx = tid - 32; idx < kFanBatch * (8 + kFanOwn); idx += nt - 32) reinterpret_cast<int32_t*>(rowof)[idx] = -1;
    }
    __syncthreads();
    if (prof) {
      const uint64_t tn = global_ns();
      tp[0] += tn - tq;
      tq = tn;
    }
    nb = scal[0];
    int npc = scal[1], npos = scal[2];
    if (npc > cap || npos > kFanVcap) {  // cannot happen for a consistent plan
      if (tid == 0) atomicCAS(&a.ctrl[kErr], 0, SPCHOL_DEV_EINTERNAL);
      npc = npos = 0;
    }
    // 2. the pieces that hold each column's rows (the 16-byte piece at or below
    // its first value, and on), and the positions
    for (int idx = tid; idx < npc; idx += nt) {
      const FanMeta& mk = meta[fan_tile_of(meta, nb, idx, true)];
      const int lp = idx - mk.pre_b;
      // lp / cps exactly: lp < 2^12 and cps <= 17 leave a margin of 1 / 34 for rounding
      const int j = (int)(((float)lp + 0.5f) * mk.inv_cps), q = lp - j * mk.cps;
      const long long g0 = mk.fo + (long long)j * mk.rowlen;  // the column's first value
      const long long a0 = (g0 & ~(long long)(E - 1)) + (long long)q * E;
      if (a0 < g0 + mk.ni)  // a piece past the column's last value holds nothing it needs
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(Bs + (size_t)idx * E)),
                     "l"(F + a0)
                     : "memory");
    }
    cp_async_commit();
    for (int idx = tid; idx < npos; idx += nt) {
      const int k = fan_tile_of(meta, nb, idx, false);
      const FanMeta& mk = meta[k];
      const int lv = idx - mk.pre_v;
      int q;
      bool ok;
      if (lv < mk.ni) {
        q = __ldg(a.relpos + mk.rp + lv) - p0;
        ok = q >= 0 && q < np;
      } else {
        q = __ldg(a.pv.rows + mk.rs + (lv - mk.ni)) - ft;
        ok = q >= 0 && q < wt;
      }
      if (!ok) atomicCAS(&a.ctrl[kErr], 0, SPCHOL_DEV_EINTERNAL);  // outside the piece: an inconsistent plan
      if (!own) {
        pv[idx] = ok ? (int16_t)q : (int16_t)-1;
      } else if (ok) {
        const int j = lv - mk.ni;
        if (j < 0)
          rowof[k * 32 + q] = (int8_t)lv;
        else
          colof[k * kFanOwn + q] =
              (mk.pre_b + j * mk.cps) * E + (int)((mk.fo + (long long)j * mk.rowlen) & (E - 1));
      }
    }
    cp_async_wait<0>();
    __syncthreads();
    if (prof) {
      const uint64_t tn = global_ns();
      tp[1] += tn - tq;
      tq = tn;
    }
    // 3. tile by tile: an entry's updates land in list order
    if (own && warp < wt && d0 + np > warp) {  // (the warp's column has rows in the lower triangle)
      for (int k0 = 0; k0 < nb; k0 += kFanAhead) {
        int col[kFanAhead], row[kFanAhead];
        T x[kFanAhead];
#pragma unroll
        for (int u = 0; u < kFanAhead; ++u) {
          col[u] = k0 + u < nb ? colof[(k0 + u) * kFanOwn + warp] : -1;  // the same in every lane
          row[u] = k0 + u < nb && d0 + lane >= warp ? rowof[(k0 + u) * 32 + lane] : -1;
        }
#pragma unroll
        for (int u = 0; u < kFanAhead; ++u) x[u] = col[u] >= 0 && row[u] >= 0 ? Bs[col[u] + row[u]] : T(0);
#pragma unroll
        for (int u = 0; u < kFanAhead; ++u)
          if (col[u] >= 0) {
            const T y = acc + x[u];
            if (row[u] >= 0) acc = y;
          }
      }
    }
    for (int k = 0; !own && k < nb; ++k) {
      const FanMeta& mk = meta[k];
      const int ni = mk.ni, n = ni * mk.seglen;
      for (int idx = tid; idx < n; idx += nt) {
        // idx / ni exactly: idx < 2^12 and ni <= 32 leave a margin of 1 / 64 for rounding
        const int j = (int)(((float)idx + 0.5f) * mk.inv_ni), ii = idx - j * ni;
        const int p = pv[mk.pre_v + ii], c = pv[mk.pre_v + ni + j];
        // lower triangle of the target (rows below its diagonal block always are)
        if (p >= 0 && c >= 0 && d0 + p >= c) {
          const int sub = (int)((mk.fo + (long long)j * mk.rowlen) & (E - 1));
          S[p + kFanPieceRows * c] += Bs[(size_t)(mk.pre_b + j * mk.cps) * E + sub + ii];
        }
      }
      __syncthreads();
    }
    if (prof) {
      const uint64_t tn = global_ns();
      tp[2] += tn - tq;
      tq = tn;
      ++nbat;
      ntile += nb;
    }
    e += nb;
  }
  if (own) {
    if (lane < np && warp < wt) Pt[p0 + lane + (size_t)warp * ldt] = acc;
  } else {
    for (int idx = tid; idx < np * wt; idx += nt) {
      const int p = idx % np, c = idx / np;
      Pt[p0 + p + (size_t)c * ldt] = S[p + kFanPieceRows * c];
    }
  }
  if (prof) {
    for (int k = 0; k < 3; ++k) atomicAdd(&a.prof[10 + k], (unsigned long long)tp[k]);
    atomicAdd(&a.prof[13], (unsigned long long)nbat);
    atomicAdd(&a.prof[14], (unsigned long long)ntile);
  }
  __syncthreads();  // the task reads these rows next, and reuses the shared memory
}

// ---------------------------------------------------------------- warp-level subtree tasks
// A subtree task whose panels are all at most kWarpSubW columns wide
// (FactorArgs::wsub) runs on one warp, before the warps of its CTA join the
// task loop: the many small subtrees of a batch of small matrices, or the
// leaves of a large one, then advance kWarpExec per CTA side by side with warp
// barriers only, where a CTA subtree task runs one of them with CTA barriers
// at every column and step.  What bounds them: a warp-wide FP64 instruction
// holds an SM sub-partition's pipe for 64 clocks whatever its active lanes,
// and every dependent trip to L2 costs 600.  So each step spreads its entries
// over the lanes, and a panel that fits the warp's shared memory (97 % of
// those of 512 2D grids; 6.9 columns and 17.6 rows below them on average) is
// loaded once, factored with its rows below in place, and subtracted from its
// ancestors over the flattened triangle of its rows below, not tile by tile:
//   * column by column, the pivot's reciprocal square root on the integer
//     pipe, the trailing rectangle one entry per lane and pass;
//   * the inverse of the diagonal block by substitution on scaled rows; FP32
//     panels solve their rows below by it, in FP32 (a substitution with L11
//     rounded to FP32 refined to errors 10 % larger);
//   * the updates kWarpOuts outputs per lane at a time: into panels inside the
//     subtree by plain read-modify-write (no other task touches them), into the
//     others by atomics.
// A panel that does not fit has its diagonal block and inverse in shared
// memory, the rows below solved by that inverse (l_rc = sum_{k <= c} a_rk
// X_ck, one output per lane and pass) and its update tiles one after another.
// The panel's tiles are then counted down on their targets outside.
// After a failed pivot (here or anywhere) the rest of the subtree skips its
// arithmetic but still counts its outside targets down.
// Launch over the 512 grids, before -> now: FP64 8.0 -> 5.0 ms, FP32 5.7 -> 3.9 ms.
constexpr int kWarpLd = kWarpSubW + 1;
constexpr int kWarpExec = 4;                                   // warps of a CTA that run them
constexpr int kWarpSmem = kWarpSubW * kWarpLd + kWarpSubW;     // doubles per warp
constexpr int kWarpOuts = 4;                                   // update outputs in flight per lane

// Entry p of a lower triangle numbered row by row (p = a (a + 1) / 2 + b,
// 0 <= b <= a): row a, column b.  The float square root is exact at the
// triangular numbers; the two corrections absorb its rounding elsewhere.
__device__ __forceinline__ void tri_decode(int p, int& ra, int& cb) {
  int t = (int)((sqrtf(8.0f * (float)p + 1.0f) - 1.0f) * 0.5f);
  if ((t + 1) * (t + 2) / 2 <= p) ++t;
  if (t * (t + 1) / 2 > p) --t;
  ra = t;
  cb = p - t * (t + 1) / 2;
}

// p / m for p < 2^12, m >= 1, inv = 1 / m: the margin of 1 / (2 m) is far above the rounding.
__device__ __forceinline__ int quick_div(int p, float inv) { return (int)(((float)p + 0.5f) * inv); }

// Cholesky of the R x w columns at A (leading dimension la, R >= w): L11 and,
// for R > w, the rows below it, and xd[j] = 1 / l_jj.  The upper triangle is
// overwritten.  One warp; false at a pivot that is not positive, with its
// column in *bad.
__device__ __forceinline__ bool warp_factor(double* A, int la, int R, int w, double* xd, int* bad) {
  const int lane = threadIdx.x & 31;
  for (int j = 0; j < w; ++j) {
    double* cj = A + j * la;
    const double d = cj[j];
    __syncwarp();  // every lane has read the pivot
    if (!pivot_positive(d)) {
      *bad = j;
      return false;
    }
    const double y = pivot_rsqrt(d);
    if (lane == 0) xd[j] = y;
    for (int i = j + lane; i < R; i += 32) cj[i] *= y;
    if (lane == 0 && __double2hiint(d) == 0x7ff00000) cj[j] = d;  // (y is 0, and inf * 0 no number)
    __syncwarp();
    const int m = R - j - 1, nc = w - j - 1;
    if (nc > 0) {
      const float inv = 1.0f / (float)m;
      for (int p = lane; p < m * nc; p += 32) {
        const int q = quick_div(p, inv), k = j + 1 + q, i = j + 1 + p - q * m;
        A[i + k * la] = fma(-cj[i], cj[k], A[i + k * la]);
      }
    }
    __syncwarp();
  }
  return true;
}

// X = L11^{-1} from L11 at A, by substitution row by row: with the rows below
// the diagonal scaled by 1 / l_ii first (in place: L11 is stored), step kk
// adds -l_ik X_kc to every X_ic with c <= kk < i, one per lane and pass.  X_ic,
// i > c, in the upper triangle at (c, i); the diagonal is xd.
__device__ __forceinline__ void warp_invert(double* A, int la, int w, const double* xd, double* __restrict__ X) {
  const int lane = threadIdx.x & 31;
  const float inv_w = 1.0f / (float)w;
  for (int p = lane; p < w * w; p += 32) {
    const int j = quick_div(p, inv_w), i = p - j * w;
    if (i > j)
      A[i + j * la] *= xd[i];
    else if (i < j)
      A[i + j * la] = 0.0;
  }
  __syncwarp();
  for (int kk = 0; kk < w - 1; ++kk) {
    const int nc = kk + 1, n = nc * (w - kk - 1);
    const float inv = 1.0f / (float)nc;
    for (int p = lane; p < n; p += 32) {
      const int q = quick_div(p, inv), c = p - q * nc, i = kk + 1 + q;
      const double x = c == kk ? xd[kk] : A[c + kk * la];
      A[c + i * la] = fma(-A[i + kk * la], x, A[c + i * la]);
    }
    __syncwarp();
  }
  for (int p = lane; p < w * w; p += 32) {
    const int j = quick_div(p, inv_w), i = p - j * w;
    if (i >= j) X[p] = i == j ? xd[j] : A[j + i * la];
  }
}

// Panel s of the subtree ending at panel hi, in shared memory: false (nothing
// done) if it does not fit.
template <typename T>
__device__ __forceinline__ bool warp_panel(const FactorArgs& a, int s, int hi, double* ws, bool& skip) {
  constexpr bool D64 = sizeof(T) == 8;
  const int lane = threadIdx.x & 31;
  const int f = a.pv.fcol[s], w = a.pv.fcol[s + 1] - f, ld = a.pv.ld[s], r = a.pv.nrows[s], nb = r - w;
  const int R = D64 ? r : w, la = R | 1, ls = D64 ? la : nb | 1;
  // shared memory: the columns, 1 / l_jj, two words per row below; FP32 panels: the rows below, X in FP32
  const int need = la * w + w + 2 * nb + (D64 ? 0 : (ls * w + w * w + 1) / 2);
  if (need > kWarpSmem) return false;
  double* A = ws;
  double* xd = A + la * w;
  long long* ro = reinterpret_cast<long long*>(xd + w);  // where column j's entries start in its target, with row 0's offset out
  long long* rp = ro + nb;                               // its relative indices: offset of row 0's | outside the subtree
  T* S = D64 ? reinterpret_cast<T*>(A + w) : reinterpret_cast<T*>(rp + nb);
  float* xf = D64 ? nullptr : reinterpret_cast<float*>(rp + nb) + ls * w;  // X in FP32: X_ck at xf[k + c w]
  T* P = panel_ptr<T>(a, s);
  const float inv_r = 1.0f / (float)r;
#pragma unroll 4
  for (int p = lane; p < r * w; p += 32) {
    const int j = quick_div(p, inv_r), i = p - j * r;
    const T v = i >= j ? ldcg(P + i + (size_t)j * ld) : T(0);
    if (D64 || i < w)
      A[i + j * la] = (double)v;
    else
      S[i - w + j * ls] = v;
  }
  // each target's first tile tells where the columns of its segment go (the
  // relative indices of its later row tiles follow it)
  const int32_t* Rs = a.pv.rows + a.pv.rowoff[s];
  for (int q = lane; q < a.nu[s]; q += 32) {
    const UTask u = a.ut[a.u_first[s] + q];
    if (u.row0 != u.seg0) continue;
    const long long base = a.pv.valoff[u.t] - (long long)a.pv.fcol[u.t] * a.pv.ld[u.t];
    const long long rel = 2 * (u.rel - (u.row0 - w)) + (u.t > hi ? 1 : 0);
    for (int jj = 0; jj < u.seglen; ++jj) {
      ro[u.seg0 - w + jj] = base + (long long)Rs[u.seg0 + jj] * a.pv.ld[u.t];
      rp[u.seg0 - w + jj] = rel;
    }
  }
  __syncwarp();
  int bad = 0;
  if (!warp_factor(A, la, R, w, xd, &bad)) {
    if (lane == 0) atomicMin(&a.ctrl[kInfo], f + bad + 1);
    skip = true;
    return true;
  }
  const float inv_R = 1.0f / (float)R;
  for (int p = lane; p < R * w; p += 32) {
    const int j = quick_div(p, inv_R), i = p - j * R;
    if (i >= j) P[i + (size_t)j * ld] = (T)A[i + j * la];
  }
  __syncwarp();
  warp_invert(A, la, w, xd, a.inv + a.invoff[s]);
  if (!D64) {
    const float inv_w = 1.0f / (float)w;
    for (int p = lane; p < w * w; p += 32) {
      const int c = quick_div(p, inv_w), k = p - c * w;
      if (k <= c) xf[p] = (float)(k == c ? xd[c] : A[k + c * la]);
    }
    __syncwarp();
    for (int i = lane; i < nb; i += 32)  // l_ic = sum over k <= c of a_ik X_ck, highest column first
      for (int c = w - 1; c >= 0; --c) {
        T v = T(0);
        for (int k = 0; k <= c; ++k) v = fma(S[i + k * ls], (T)xf[k + c * w], v);
        S[i + c * ls] = v;
        P[w + i + (size_t)c * ld] = v;
      }
    __syncwarp();
  }
  // entry (i, j), i >= j, of the rows below's triangle, consecutive i on consecutive lanes
  T* pool = reinterpret_cast<T*>(a.pool);
  const int ntri = nb * (nb + 1) / 2;
  for (int o0 = 0; o0 < ntri; o0 += 32 * kWarpOuts) {
    T* dst[kWarpOuts];
    T old[kWarpOuts];
    int ij[kWarpOuts];  // row << 16 | column, bit 15: outside
#pragma unroll
    for (int q = 0; q < kWarpOuts; ++q) {
      const int o = o0 + 32 * q + lane;
      dst[q] = nullptr;
      ij[q] = 0;
      if (o < ntri) {
        int ra, cb;
        tri_decode(o, ra, cb);
        const int j = nb - 1 - ra, i = nb - 1 - cb;
        const long long e = rp[j];
        const int pos = __ldg(a.relpos + (e >> 1) + i);
        if (pos < 0) atomicCAS(&a.ctrl[kErr], 0, SPCHOL_DEV_EINTERNAL);  // cannot happen for a consistent plan
        dst[q] = pos < 0 ? nullptr : pool + ro[j] + pos;
        ij[q] = (i << 16) | ((int)(e & 1) << 15) | j;
      }
    }
#pragma unroll
    for (int q = 0; q < kWarpOuts; ++q) old[q] = dst[q] && !(ij[q] & 0x8000) ? *dst[q] : T(0);
#pragma unroll
    for (int q = 0; q < kWarpOuts; ++q) {
      if (o0 + 32 * q >= ntri) break;
      // the products are summed before they meet the entry: one rounding at
      // the entry's size, not one per column
      const T* si = S + (ij[q] >> 16);
      const T* sj = S + (ij[q] & 0x7fff);
      T acc = T(0);
      if (D64) {
        for (int k = 0; k < w; ++k) acc = fma(si[k * ls], sj[k * ls], acc);
      } else {
        T acc1 = T(0);
        int k = 0;
        for (; k + 1 < w; k += 2) {
          acc = fma(si[k * ls], sj[k * ls], acc);
          acc1 = fma(si[(k + 1) * ls], sj[(k + 1) * ls], acc1);
        }
        if (k < w) acc = fma(si[k * ls], sj[k * ls], acc);
        acc += acc1;
      }
      if (dst[q]) {
        if (ij[q] & 0x8000)
          red_add(dst[q], -acc);
        else
          *dst[q] = old[q] - acc;
      }
    }
  }
  return true;
}

// A panel that does not fit.
template <typename T>
__device__ void warp_panel_wide(const FactorArgs& a, int s, int hi, double* ws, bool& skip) {
  const int lane = threadIdx.x & 31;
  const int f = a.pv.fcol[s], w = a.pv.fcol[s + 1] - f, ld = a.pv.ld[s], r = a.pv.nrows[s];
  double* xd = ws + kWarpSubW * kWarpLd;
  T* P = panel_ptr<T>(a, s);
  for (int idx = lane; idx < w * w; idx += 32) {
    const int i = idx % w, j = idx / w;
    ws[i + j * kWarpLd] = i >= j ? (double)ldcg(P + i + (size_t)j * ld) : 0.0;
  }
  __syncwarp();
  int bad = 0;
  if (!warp_factor(ws, kWarpLd, w, w, xd, &bad)) {
    if (lane == 0) atomicMin(&a.ctrl[kInfo], f + bad + 1);
    skip = true;
    return;
  }
  for (int idx = lane; idx < w * w; idx += 32) {
    const int i = idx % w, j = idx / w;
    if (i >= j) P[i + (size_t)j * ld] = (T)ws[i + j * kWarpLd];
  }
  __syncwarp();
  warp_invert(ws, kWarpLd, w, xd, a.inv + a.invoff[s]);
  // L21 = A21 L11^{-T} by the inverse, in the panels' precision, columns in
  // decreasing order, so that a_rc is overwritten only after every output that
  // reads it (its row's higher columns: an earlier pass, or this one, whose
  // reads all precede its writes)
  using ct = T;
  const int rb = r - w, nout = rb * w;
  for (int o0 = 0; o0 < nout; o0 += 32) {
    const int o = o0 + lane;
    const bool ov = o < nout;
    const int c = ov ? w - 1 - o / rb : 0, rr = ov ? o % rb : 0;
    T* Pr = P + w + rr;
    ct acc = ct(0);
    if (ov)
      for (int k = 0; k <= c; ++k)
        acc = fma((ct)ldcg(Pr + (size_t)k * ld), k == c ? (ct)xd[c] : (ct)ws[k + c * kWarpLd], acc);
    __syncwarp();
    if (ov) Pr[(size_t)c * ld] = (T)acc;
  }
  __syncwarp();  // the rows below are written before the update tiles read them
  const int32_t* Rs = a.pv.rows + a.pv.rowoff[s];
  for (int ui = a.u_first[s]; ui < a.u_first[s] + a.nu[s]; ++ui) {
    const UTask u = a.ut[ui];
    const int ft = a.pv.fcol[u.t], ldt = a.pv.ld[u.t];
    T* Pt = panel_ptr<T>(a, u.t);
    const int nout = u.rowlen * u.seglen;
    for (int o = lane; o < nout; o += 32) {
      const int i = o % u.rowlen, j = o / u.rowlen;
      const int gi = Rs[u.row0 + i], gj = Rs[u.seg0 + j];
      if (gi < gj) continue;  // the upper part of a target's diagonal block
      const T* ai = P + u.row0 + i;
      const T* bj = P + u.seg0 + j;
      T c0 = T(0), c1 = T(0);
      int kk = 0;
      for (; kk + 1 < w; kk += 2) {
        c0 = fma(ai[(size_t)kk * ld], bj[(size_t)kk * ld], c0);
        c1 = fma(ai[(size_t)(kk + 1) * ld], bj[(size_t)(kk + 1) * ld], c1);
      }
      if (kk < w) c0 = fma(ai[(size_t)kk * ld], bj[(size_t)kk * ld], c0);
      const int p = __ldg(a.relpos + u.rel + i);
      if (p < 0) {  // cannot happen for a consistent plan
        atomicCAS(&a.ctrl[kErr], 0, SPCHOL_DEV_EINTERNAL);
        continue;
      }
      T* dst = Pt + p + (size_t)(gj - ft) * ldt;
      if (u.t > hi)
        red_add(dst, -(c0 + c1));
      else
        *dst -= c0 + c1;
    }
  }
}

template <typename T>
__device__ void warp_subtree(const FactorArgs& a, int k, double* ws) {
  const int lane = threadIdx.x & 31;
  const int lo = a.sub_lo[k], hi = a.sub_hi[k];
  bool skip = ld_relaxed(&a.ctrl[kInfo]) != INT_MAX;
  const Ring2 q = rings_of(a);
  for (int s = lo; s <= hi; ++s) {
    if (!skip && !warp_panel<T>(a, s, hi, ws, skip)) warp_panel_wide<T>(a, s, hi, ws, skip);
    // publish the warp's atomics, then count the panel's tiles down on their
    // targets outside the subtree, one per lane
    __syncwarp();
    bool fenced = false;
    for (int ui = a.u_first[s] + lane; ui < a.u_first[s] + a.nu[s]; ui += 32) {
      const int t = a.ut[ui].t;
      if (t <= hi) continue;
      if (!fenced) fence_gpu();
      fenced = true;
      if (count_down(&a.dep_f[t])) ring2_push_one(q, true, t);
    }
    __syncwarp();  // the next panel reads what this one's tiles wrote into it
  }
}

// MODE: 0 = CUDA-core update tiles (DFMA / FFMA), 1 = TF32 tensor cores (FP32
// panels, split or not), 3 = BF16 tensor cores on split FP64 operands.
// Five CTAs per SM (48 registers a thread; a few live values of the update
// tile's epilogue spill to L1) for the DFMA mode, six (40 registers) for FP32
// panels on FFMA, whose tasks are shortest: more resident CTAs hide each
// other's latencies (measured: FP32 factor -12 %, FP64 -0.8 % for five against
// four).  The TF32 mode runs two CTAs per SM and the BF16-split mode three, as
// their operand tiles' shared memory allows (a BF16-split CTA holds 128 of the
// SM's 512 TMEM columns).  The fan-in mode's CUDA-core kernels run four: the
// gather's staging area takes a quarter of the SM's shared memory.
// FUSE: the diagonal tasks of narrow panels solve the rows below them
// (kFuseWidth).
template <typename T, int MODE, bool FAN, bool FUSE>
__global__ void __launch_bounds__(kFactorThreads, MODE == 3 ? 3 : MODE != 0 ? 2 : FAN ? 4 : sizeof(T) == 4 ? 6 : 5)
    factor_kernel(FactorArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ FactorShared sh;
  double* smd = reinterpret_cast<double*>(smem_raw);
  const Ring2 q = rings_of(a);
  __shared__ int pend[3];  // claimed, not yet taken ring slots (thread 0)
  if (threadIdx.x == 0) {
    pend[0] = pend[1] = pend[2] = -1;
    sh.next = -1;
  }
  // per-CTA task timing (thread 0 only, in shared memory so that no register
  // stays live across the tasks), flushed once at exit: [0..4] busy ns per task
  // type ([3]: tensor-core update tiles, [4]: subtree tasks), [5..9] counts,
  // [10] wait ns, [11] start of the current task
  __shared__ unsigned long long tprof[12];
  if (threadIdx.x == 0)
    for (int k = 0; k < 12; ++k) tprof[k] = 0ull;
  // TMA staging of the CUDA-core update tiles: one mbarrier per operand buffer
  __shared__ __align__(8) uint64_t upd_mbar[2];
  __shared__ uint32_t upd_phase;
  UpdTma utma{{smem_addr(&upd_mbar[0]), smem_addr(&upd_mbar[1])}, &upd_phase};
  if (a.tmaps && threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(utma.mbar[0]), "r"(1) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(utma.mbar[1]), "r"(1) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    upd_phase = 0u;
  }
  __syncthreads();
  // tensor-core state (FP32 panels with mma_mode 1 / 2): TMEM accumulator + mbarrier
  __shared__ __align__(8) uint64_t tc_mbar;
  __shared__ uint32_t tc_tmem;
  TcState tc{0u, 0u, 0u};
  constexpr bool use_tc = MODE != 0;
  constexpr uint32_t tmem_cols = MODE == 3 ? kOzCols : kTcN;
  if (use_tc) {
    if (threadIdx.x < 32) {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tc_tmem)),
                   "r"(tmem_cols)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(&tc_mbar)), "r"(1) : "memory");
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    tc.tmem = tc_tmem;
    tc.mbar = smem_addr(&tc_mbar);
  }
  // Thread 0: a normal-priority slot claimed ahead while the ring is deep, so
  // that the claim's round trip overlaps the current task; it joins pend[1] at
  // the next claim (a deep ring fills it long before).  Two adjacent slots are
  // claimed ahead at a time: the next claim reads both in one round trip and
  // the second task (the stash) then runs without a claim of its own.
  int ahead = -1, stash = -1;
  bool deep = false;
  // Subtree task cursor (thread 0): a claimed subtree task is run as a
  // sequence of panel-level steps through the same dispatch as the ring's
  // tasks -- diagonal, panel-solve tiles, update tiles of each panel in
  // postorder -- with counters only for targets outside the subtree.
  __shared__ int cur_task, cur_lo, cur_hi, cur_s, cur_ph, cur_i, cur_skip;
  __shared__ int step_kind, step_s, step_i, step_release, step_last;
  if (threadIdx.x == 0) cur_task = -1;
  const int sub0 = a.pv.ns + a.n_trsm + a.n_u;  // first subtree task id
  for (;;) {
    if (threadIdx.x == 0) {
      const bool timed = a.prof || a.trace;
      if (cur_task < 0) {
        const uint64_t t0 = timed ? global_ns() : 0;
        const bool idle = pend[1] < 0 && pend[2] < 0;
        if (sh.next >= 0) {  // made ready by this CTA's last task
          sh.task = sh.next;
          sh.next = -1;
        } else if (stash >= 0) {  // acquired by the previous claim
          sh.task = stash;
          stash = -1;
          if (deep && idle) ahead = atomicAdd(&q.ctrl[kHead], 2);
        } else {
          if (ahead >= 0) {
            pend[1] = ahead < q.n_lo ? ahead : -1;
            pend[2] = ahead + 1 < q.n_lo ? ahead + 1 : -1;
            ahead = -1;
          }
          int lo_ready;
          sh.task = ring2_claim(q, pend, &lo_ready, a.ntask_done, &stash);
          deep = lo_ready > 4 * (int)gridDim.x;
          if (sh.task >= 0 && pend[1] < 0 && pend[2] < 0 && stash < 0 && deep) ahead = atomicAdd(&q.ctrl[kHead], 2);
        }
        // The failure word is read after the claim's acquire: a task whose
        // inputs were skipped by tasks that saw a failed pivot (their release
        // precedes this claim) then sees it too and skips as well.  Read
        // before the claim, a diagonal task could factor a panel missing
        // skipped updates and report a pivot failure that is not there.
        sh.skip = (ld_relaxed(&a.ctrl[kInfo]) != INT_MAX);
        if (timed) {
          const uint64_t t1 = global_ns();
          tprof[10] += t1 - t0;
          tprof[11] = t1;
        }
        if (sh.task >= sub0 && (!FAN || sh.task < a.gat0)) {
          const int k = sh.task - sub0;
          cur_task = sh.task;
          cur_lo = a.sub_lo[k];
          cur_hi = a.sub_hi[k];
          cur_s = cur_lo;
          cur_ph = 0;
          cur_i = 0;
          cur_skip = sh.skip;
        }
      }
      // a CTA that holds a high-priority slot takes no continuation: that
      // slot's task would wait for it
      sh.hold = cur_task >= 0 || pend[0] >= 0;
      if (cur_task >= 0) {  // the next step of the subtree, then advance the cursor
        const int s = cur_s;
        step_kind = cur_ph;
        step_s = s;
        step_i = cur_i;
        step_release = cur_ph == 2 ? (a.ut[a.u_first[s] + cur_i].t > cur_hi) : 0;
        sh.skip = cur_skip;
        sh.task = cur_task;
        int ph = cur_ph, i = cur_i + 1;
        if (ph == 0) {
          ph = FUSE && fused_panel(a, s, a.pv.fcol[s + 1] - a.pv.fcol[s]) ? 2 : 1;
          i = 0;
        }
        if (ph == 1 && i >= a.ntrsm[s]) {
          ph = 2;
          i = 0;
        }
        step_last = 0;
        if (ph == 2 && i >= a.nu[s]) {
          if (s < cur_hi) {
            cur_s = s + 1;
            ph = 0;
            i = 0;
          } else {
            step_last = 1;
          }
        }
        cur_ph = ph;
        cur_i = i;
      } else if (sh.task >= 0) {  // a task of the rings
        const int task = sh.task;
        step_release = 1;
        step_last = 1;
        if (task < a.pv.ns) {
          step_kind = 0;
          step_s = task;
          step_i = 0;
        } else if (task < a.pv.ns + a.n_trsm) {
          const int kt = task - a.pv.ns;
          step_kind = 1;
          step_s = a.trsm_sn[kt];
          step_i = kt - a.trsm_first[step_s];
        } else if (FAN && task >= a.gat0) {
          step_kind = 4;  // a gather task (fan-in mode)
          step_s = -1;
          step_i = task - a.gat0;
        } else {
          step_kind = 3;  // an update tile by its global index
          step_s = -1;
          step_i = task - a.pv.ns - a.n_trsm;
        }
      }
    }
    __syncthreads();
    const int task = sh.task;
    if (task < 0) break;
    const bool skip = sh.skip != 0;
    const int kind = step_kind, s = step_s, si = step_i;
    const bool release = step_release != 0;
    int type;
    if (FAN && kind == 4) {
      // fan-in mode: a gather task adds the buffered updates of one row piece
      // of a panel, then counts down the task that owns those rows
      type = 0;
      const GatherTask G = a.gat[si];
      const int pc = G.pc, o = a.pc_owner[pc];
      const int t = o < a.pv.ns ? o : a.trsm_sn[o - a.pv.ns];
      const int w = a.pv.fcol[t + 1] - a.pv.fcol[t];
      int p0, p1;
      if (o < a.pv.ns) {
        p0 = (pc - a.fan_task[t]) * kFanPieceRows;
        p1 = min(w, p0 + kFanPieceRows);
      } else {
        const int tr = a.trsm_rows_of[t], r0 = w + (o - a.pv.ns - a.trsm_first[t]) * tr;
        p0 = r0 + (pc - a.fan_task[o]) * kFanPieceRows;
        p1 = min(min(a.pv.nrows[t], r0 + tr), p0 + kFanPieceRows);
      }
      if (!skip) fanin_gather<T>(a, t, G, p0, p1 - p0, smem_raw);
      publish_cta_writes();
      if (threadIdx.x == 0) {
        if (o < a.pv.ns) {
          if (count_down(&a.gdiag[t])) ring2_push_one(rings_of(a), true, t);
        } else if (count_down(&a.tdep[o - a.pv.ns])) {
          ring2_push_one(rings_of(a), true, o);
        }
      }
    } else if (kind == 0) {
      type = 0;
      if constexpr (MODE == 3)
        task_potrf_apart<T, FAN>(a, s, smd, sh, skip, release);
      else
        task_potrf<T, FAN, FUSE>(a, s, smd, sh, skip, release);
    } else if (kind == 1) {
      type = 1;
      task_trsm<T, MODE>(a, s, si, smd, sh, skip, release);
    } else {
      type = 2;
      const int ui = kind == 2 ? a.u_first[s] + si : si;
      const UTask u = a.ut[ui];
      const long long fo = FAN ? (long long)a.fan_off[ui] : -1ll;  // fan-in: the tile's buffer
      if constexpr (MODE == 3) {
        if (a.pv.fcol[u.s + 1] - a.pv.fcol[u.s] >= a.tc_min_width) {
          type = 3;
          task_update_oz<FAN>(a, u, smem_raw, sh, skip, tc, fo, release);
        } else {
          task_update<T, FAN>(a, u, smem_raw, sh, skip, ui & 7, utma, fo, release);
        }
      } else if constexpr (MODE == 1) {
        task_update_tc<FAN>(a, u, smem_raw, sh, skip, tc, fo, release);
      } else {
        task_update<T, FAN>(a, u, smem_raw, sh, skip, ui & 7, utma, fo, release);
      }
      // deterministic order: the next tile into the same target may start
      // (the tile's scatter-adds were published before its own release)
      if (a.u_next && release && threadIdx.x == 0) {
        const int nx = a.u_next[ui];
        if (nx >= 0 && count_down(&a.u_dep[nx])) {
          const int sx = a.ut[nx].s;
          ring2_push_one(rings_of(a), nx - a.u_first[sx] < a.nu_hi[sx], a.pv.ns + a.n_trsm + nx);
        }
      }
    }
    if (threadIdx.x == 0) {
      const bool in_sub = cur_task >= 0;
      if (in_sub) {
        type = 4;
        // after a failed pivot the rest of the subtree skips its arithmetic
        if (kind == 0 && ld_relaxed(&a.ctrl[kInfo]) != INT_MAX) cur_skip = 1;
      }
      if (step_last) {
        atomicAdd(&a.ctrl[kDone], 1);
        if (a.trace) {
          a.trace[2 * (size_t)task] = tprof[11];
          a.trace[2 * (size_t)task + 1] = global_ns();
        }
        if (a.prof) {
          tprof[type] += global_ns() - tprof[11];
          tprof[5 + type] += 1;
        }
        if (in_sub) cur_task = -1;
      }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0 && a.prof) {
    for (int k = 0; k < 3; ++k) {
      atomicAdd(&a.prof[k], tprof[k] + (k == 2 ? tprof[3] : 0ull));
      atomicAdd(&a.prof[4 + k], tprof[5 + k] + (k == 2 ? tprof[8] : 0ull));
    }
    atomicAdd(&a.prof[3], tprof[10]);
    atomicAdd(&a.prof[7], tprof[3]);   // tensor-core share of the update tiles
    atomicAdd(&a.prof[8], tprof[4]);   // subtree tasks
    atomicAdd(&a.prof[9], tprof[9]);
  }
  if (use_tc) {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (threadIdx.x < 32)
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tc.tmem), "r"(tmem_cols) : "memory");
  }
}

// The warp-level subtree tasks, launched before the task loop's kernel (on the
// same stream, after the ring reset): kWarpExec warps per CTA, each taking
// the next subtree from a counter until none is left.  The tiles they count
// down push ready tasks into the rings, which the task loop's kernel then
// finds there; every subtree adds one to the completed-task count.
template <typename T>
__global__ void __launch_bounds__(32 * kWarpExec) warp_subtree_kernel(FactorArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double* ws = reinterpret_cast<double*>(smem_raw) + warp * kWarpSmem;
  const int sub0 = a.pv.ns + a.n_trsm + a.n_u;  // first subtree task id
  for (;;) {
    int e = 0;
    if (lane == 0) e = atomicAdd(&a.ctrl[kWarpNext], 1);
    e = __shfl_sync(0xffffffffu, e, 0);
    if (e >= a.n_wsub) break;
    const int k = a.wsub[e];
    const unsigned long long t0 = a.trace && lane == 0 ? global_ns() : 0ull;
    warp_subtree<T>(a, k, ws);
    if (lane == 0) {
      atomicAdd(&a.ctrl[kDone], 1);
      if (a.trace) {
        a.trace[2 * (size_t)(sub0 + k)] = t0;
        a.trace[2 * (size_t)(sub0 + k) + 1] = global_ns();
      }
    }
  }
}

template <typename T>
__global__ void assemble_kernel(const double* __restrict__ values, const int64_t* __restrict__ dest,
                                int64_t nnz, T* __restrict__ pool) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nnz; e += (int64_t)gridDim.x * blockDim.x)
    pool[dest[e]] = (T)values[e];
}

}  // namespace

size_t warp_subtree_smem_bytes() { return (size_t)kWarpExec * kWarpSmem * sizeof(double); }

static const void* warp_subtree_fn(bool fp32) {
  return fp32 ? (const void*)warp_subtree_kernel<float> : (const void*)warp_subtree_kernel<double>;
}

cudaError_t warp_subtree_configure(bool fp32, int* blocks_per_sm) {
  const size_t smem = warp_subtree_smem_bytes();
  cudaError_t e = ensure_smem_limit(warp_subtree_fn(fp32), smem);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, warp_subtree_fn(fp32), 32 * kWarpExec, smem);
}

cudaError_t launch_warp_subtrees(bool fp32, const FactorArgs& a, int grid, cudaStream_t st) {
  if (a.n_wsub == 0) return cudaSuccess;
  void* args[] = {const_cast<FactorArgs*>(&a)};
  return cudaLaunchKernel(warp_subtree_fn(fp32), dim3(grid), dim3(32 * kWarpExec), args, warp_subtree_smem_bytes(),
                          st);
}

size_t factor_smem_bytes(int max_w, int mma_mode) {
  // POTRF: the block and 1 / l_jj; TRSM: L11 with 64-row columns and 1 / l_cc.
  size_t tri = ((size_t)max_w * max_w + (size_t)max_w) * sizeof(double);
  // (+ 1: the W rows of W panels restage L11 with leading dimension 65)
  if (max_w <= kTrsmMaxW) tri = std::max(tri, (size_t)(kTrsmMaxW + 2) * max_w * sizeof(double));
  if (mma_mode == 3) {
    const size_t kpad = ((size_t)max_w + 15) & ~size_t(15);
    const size_t oz = (size_t)kSlices * (kOzRows + kOzN) * kpad * 2 + (3 * kOzRows + 2 * kOzN) * sizeof(int) + 1024;
    if (oz > tri) tri = oz;
  } else if (mma_mode != 0) {
    const size_t kpad = ((size_t)max_w + 7) & ~size_t(7);
    const size_t tcb = 2 * (kTcM + kTcN) * kpad * 4 + (2 * kTcM + kTcN) * sizeof(int) + 1024;
    if (tcb > tri) tri = tcb;
  }
  // update tiles: two FP64 chunk buffers, or four FP32 ones (A and B each),
  // then the row positions, rows and columns
  const size_t bufs = std::max((size_t)2 * 2 * kUpdKC * Stage<double>::kStr * sizeof(double),
                               (size_t)4 * 2 * kUpdKC * Stage<float>::kStr * sizeof(float));
  size_t upd = bufs + 128 + (size_t)(2 * kUpdTileM + kUpdTileN) * sizeof(int);
  return tri > upd ? tri : upd;
}

size_t fanin_smem_bytes(int max_w, bool fp32, int* cap) {
  const size_t es = fp32 ? sizeof(float) : sizeof(double);
  const int per_col = fp32 ? fan_pieces<float>(kFanPieceRows) : fan_pieces<double>(kFanPieceRows);
  const int c = std::max(2048, per_col * max_w);  // 32 KB of pieces, and never less than one tile
  if (cap) *cap = c;
  return 16 + kFanMetaBytes + kFanVcap * sizeof(int16_t) + (size_t)c * 16 + (size_t)kFanPieceRows * max_w * es;
}

// The fan-in mode has kernels of its own, so that the other modes' update
// tiles and dispatch carry none of its code.
template <bool FAN>
static const void* factor_fn_of(bool fp32, int mma_mode) {
  if (fp32)
    return mma_mode == 0 ? (const void*)factor_kernel<float, 0, FAN, false>
                         : (const void*)factor_kernel<float, 1, FAN, false>;
  return mma_mode == 3 ? (const void*)factor_kernel<double, 3, FAN, false>
                       : (const void*)factor_kernel<double, 0, FAN, false>;
}

static const void* factor_fn(bool fp32, int mma_mode, bool fan, bool fuse) {
  if (fuse) return fp32 ? (const void*)factor_kernel<float, 0, false, true> : (const void*)factor_kernel<double, 0, false, true>;
  return fan ? factor_fn_of<true>(fp32, mma_mode) : factor_fn_of<false>(fp32, mma_mode);
}

cudaError_t factor_configure(bool fp32, int mma_mode, bool fan, bool fuse, size_t smem, int* blocks_per_sm) {
  const void* fn = factor_fn(fp32, mma_mode, fan, fuse);
  cudaError_t e = ensure_smem_limit(fn, smem);
  if (e != cudaSuccess) return e;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, fn, kFactorThreads, smem);
  if (e != cudaSuccess || mma_mode == 0) return e;
  // The runtime's occupancy query reports one block per SM for the kernels
  // that allocate TMEM, while their registers and shared memory allow more
  // (the profiler's launch statistics agree).  Count those limits directly,
  // capped by the TMEM columns a CTA holds (512 per SM; the BF16-split mode's
  // shared-memory request, over a third of the SM, also keeps a third CTA out).
  cudaFuncAttributes fa{};
  int dev = 0, regs_sm = 0, smem_sm = 0;
  if ((e = cudaFuncGetAttributes(&fa, fn)) != cudaSuccess || (e = cudaGetDevice(&dev)) != cudaSuccess ||
      (e = cudaDeviceGetAttribute(&regs_sm, cudaDevAttrMaxRegistersPerMultiprocessor, dev)) != cudaSuccess ||
      (e = cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev)) != cudaSuccess)
    return e;
  const int regs_cta = ((fa.numRegs + 7) / 8) * 8 * kFactorThreads;
  const size_t smem_cta = smem + fa.sharedSizeBytes + 1024;  // + the driver's per-block reserve
  const int by_regs = regs_cta > 0 ? regs_sm / regs_cta : 0;
  const int by_smem = (int)((size_t)smem_sm / smem_cta);
  const int by_tmem = 512 / (mma_mode == 3 ? kOzCols : kTcN);
  const int direct = std::min(by_tmem, std::min(by_regs, by_smem));
  if (direct > *blocks_per_sm) *blocks_per_sm = direct;
  return cudaSuccess;
}

cudaError_t launch_relpos(const UTask* ut, int n_u, const int32_t* rows, const int64_t* rowoff,
                          const int32_t* nrows, int32_t* relpos, cudaStream_t st) {
  if (n_u <= 0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int grid = std::max(1, std::min(n_u, 32 * std::max(sms, 1)));
  relpos_kernel<<<grid, 64, 0, st>>>(ut, n_u, rows, rowoff, nrows, relpos);
  return cudaGetLastError();
}

cudaError_t launch_assemble(bool fp32, const double* values, const int64_t* dest, int64_t nnz, void* pool,
                            cudaStream_t st) {
  if (nnz <= 0) return cudaSuccess;
  int grid = (int)((nnz + 255) / 256);
  if (grid > 152 * 16) grid = 152 * 16;
  if (fp32)
    assemble_kernel<float><<<grid, 256, 0, st>>>(values, dest, nnz, (float*)pool);
  else
    assemble_kernel<double><<<grid, 256, 0, st>>>(values, dest, nnz, (double*)pool);
  return cudaGetLastError();
}

__global__ void fanrec_kernel(const FanEnt* __restrict__ ent, int64_t n, const UTask* __restrict__ ut,
                              const int64_t* __restrict__ fan_off, const int64_t* __restrict__ rowoff,
                              FanRec* __restrict__ rec) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    const FanEnt fe = ent[k];
    const UTask u = ut[fe.u];
    FanRec r;
    r.fo = fan_off[fe.u] + fe.i0 + (int64_t)fe.j0 * u.rowlen;
    r.rp = u.rel + fe.i0;
    r.rs = rowoff[u.s] + u.seg0 + fe.j0;
    r.rowlen = u.rowlen;
    r.ni = (int16_t)(fe.i1 - fe.i0);
    r.seglen = (int16_t)(fe.j1 - fe.j0);
    rec[k] = r;
  }
}

cudaError_t launch_fanrec(const FanEnt* ent, int64_t n, const UTask* ut, const int64_t* fan_off,
                          const int64_t* rowoff, FanRec* rec, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const int grid = (int)std::min<int64_t>((n + 255) / 256, 152 * 16);
  fanrec_kernel<<<grid, 256, 0, st>>>(ent, n, ut, fan_off, rowoff, rec);
  return cudaGetLastError();
}

cudaError_t launch_factor(bool fp32, const FactorArgs& a, int grid, size_t smem, cudaStream_t st) {
  void* args[] = {const_cast<FactorArgs*>(&a)};
  return cudaLaunchKernel(factor_fn(fp32, a.mma_mode, a.gat != nullptr, a.fuse_w > 0), dim3(grid), dim3(kFactorThreads), args,
                          smem, st);
}

}  // namespace spchol
