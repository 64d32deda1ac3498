// Per-row and per-block arithmetic shared by the one-solve kernels and their batched forms
// (internal).  Both kinds of launch call these functions, so a row, a partial sum or a CG
// scalar comes out with the same bits whichever launch computes it.
#pragma once

#include "csr.cuh"

namespace saamg {
namespace rows {

__device__ __forceinline__ double ldv(const double* p, size_t i) { return p[i]; }
__device__ __forceinline__ float ldv(const float* p, size_t i) { return p[i]; }
__device__ __forceinline__ float ldv(const __nv_bfloat16* p, size_t i) {
  return __bfloat162float(p[i]);
}

// (double)f with integer operations: the conversion instruction holds the FP64 pipe as long as a
// multiply-add (64 clocks a warp), and the vector passes of the mixed modes are bound by that
// pipe (solve at 256^3 with the FP32 V-cycle: 15.4 -> 14.9 ms).  Zeros, subnormals, infinities and NaN convert.
__device__ __forceinline__ double widen(float f) {
  const unsigned u = __float_as_uint(f);
  if (((u >> 23) & 0xffu) - 1u >= 254u) {
    if ((u << 1) == 0u) return __hiloint2double((int)u, 0);
    return (double)f;
  }
  return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)),
                          (int)(u << 29));
}
__device__ __forceinline__ double widen(double f) { return f; }

// (float)v the same way: the bits below the float's are rounded off to even; a result that is not a
// normal number or an overflow converts.
__device__ __forceinline__ float narrow(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const unsigned e = (unsigned)(b >> 52) & 0x7ffu;
  if (e - 897u > 1150u - 897u) {
    if ((b << 1) == 0ull) return __uint_as_float((unsigned)(b >> 32));
    return (float)v;
  }
  const unsigned long long m = (b & 0x7fffffffffffffffull) - (896ull << 52);
  const unsigned r = (unsigned)((m + 0x0fffffffull + ((m >> 29) & 1ull)) >> 29);
  return __uint_as_float(r | ((unsigned)(b >> 32) & 0x80000000u));
}

// --- CSR, G lanes per row ---------------------------------------------------------------
// Lane gl of the row's group sums entries gl, gl + G, ... (four loads in flight), the group
// combines its sums with shuffles (all 32 lanes of the warp take part), and lane 0 of the
// group applies MODE.  A row past n (active false) only joins the shuffles.
template <class TV, class TM, int G, int MODE>
__device__ __forceinline__ void csr_group_row(int row, bool active, int gl,
                                              const int* __restrict__ rowptr,
                                              const int* __restrict__ col,
                                              const TM* __restrict__ val,
                                              const TV* __restrict__ x, TV* __restrict__ y,
                                              const TV* __restrict__ b, TV* __restrict__ d,
                                              const TV* __restrict__ invd, TV c1, TV c2,
                                              double& dacc, TV* __restrict__ y2 = nullptr) {
  TV acc = TV(0);
  if (MODE != CSR_CHEB0 && active) {
    const int p0 = rowptr[row], p1 = rowptr[row + 1];
    int p = p0 + gl;
    for (; p + 7 * G < p1; p += 8 * G) {
      int kk[8];
      TV a[8], xv[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        kk[u] = col[p + u * G];
        a[u] = (TV)ldv(val, p + u * G);
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) xv[u] = x[kk[u]];
#pragma unroll
      for (int u = 0; u < 8; ++u) acc += a[u] * xv[u];
    }
    for (; p + 3 * G < p1; p += 4 * G) {
      const int k0 = col[p], k1 = col[p + G], k2 = col[p + 2 * G], k3 = col[p + 3 * G];
      const TV a0 = (TV)ldv(val, p), a1 = (TV)ldv(val, p + G), a2 = (TV)ldv(val, p + 2 * G),
               a3 = (TV)ldv(val, p + 3 * G);
      const TV x0 = x[k0], x1 = x[k1], x2 = x[k2], x3 = x[k3];
      acc += a0 * x0;
      acc += a1 * x1;
      acc += a2 * x2;
      acc += a3 * x3;
    }
    for (; p < p1; p += G) acc += (TV)ldv(val, p) * x[col[p]];
  }
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o, G);
  if (active && gl == 0) {
    if (MODE == CSR_SPMV) {
      y[row] = acc;
    } else if (MODE == CSR_RESID) {
      y[row] = b[row] - acc;
    } else if (MODE == CSR_ADD) {
      y[row] = y[row] + acc;
    } else if (MODE == CSR_CHEB) {
      // written with explicit fma so that the compiler cannot contract it differently in
      // different kernels (c1 = 0: d is not read)
      const TV t = invd[row] * (b[row] - acc);
      const TV dv = (c1 == TV(0)) ? c2 * t : fma(c2, t, c1 * d[row]);
      d[row] = dv;
      y[row] = x[row] + dv;
    } else if (MODE == CSR_SPMV_CHEB0) {
      const TV dv = c2 * (invd[row] * acc);
      y[row] = acc;
      d[row] = dv;
      y2[row] = dv;
    } else if (MODE == CSR_CHEB0) {
      const TV dv = c2 * (invd[row] * b[row]);
      d[row] = dv;
      y[row] = dv;
    } else {  // CSR_SPMV_DINV_DOT: c2 carries the scale of x
      const TV w = (c2 * invd[row]) * acc;
      y[row] = w;
      dacc += (double)w * (double)w;
    }
  }
}

// Up to four rows of a group at a time, as csr_group_row computes each, G (2 .. 32) known at run time:
// the rows' bounds, two entries of every lane and row, their x and the update's operands are loaded
// for all rows before the first is summed, and lane q of the group applies MODE to row q (the
// butterfly leaves the same sum in every lane; with G = 2 the caller passes two rows).  A warp
// that takes many short rows of many matrices waits for one chain of loads instead of four.
template <class TV, class TM, int MODE>
__device__ __forceinline__ void csr_group_rows(const int row[4], const bool active[4], int gl, int G,
                                               const int* __restrict__ rowptr,
                                               const int* __restrict__ col,
                                               const TM* __restrict__ val,
                                               const TV* __restrict__ x, TV* __restrict__ y,
                                               const TV* __restrict__ b, TV* __restrict__ d,
                                               const TV* __restrict__ invd, TV c1, TV c2,
                                               TV* __restrict__ y2) {
  constexpr int NR = 4, E = 2;
  int p[NR], p1[NR], er = -1;
#pragma unroll
  for (int q = 0; q < NR; ++q) {
    p[q] = active[q] ? rowptr[row[q]] + gl : 0;
    p1[q] = active[q] ? rowptr[row[q] + 1] : 0;
    if (gl == q && active[q]) er = row[q];
  }
  TV bv = TV(0), dv = TV(0), iv = TV(0), xv = TV(0);
  if (er >= 0) {
    if (MODE == CSR_RESID || MODE == CSR_CHEB) bv = b[er];
    if (MODE == CSR_CHEB) {
      iv = invd[er];
      xv = x[er];
      if (c1 != TV(0)) dv = d[er];
    }
    if (MODE == CSR_ADD) xv = y[er];
    if (MODE == CSR_SPMV_CHEB0) iv = invd[er];
  }
  TV acc[NR];
#pragma unroll
  for (int q = 0; q < NR; ++q) acc[q] = TV(0);
  for (bool more = true; more;) {
    int k[NR][E];
    TV a[NR][E];
#pragma unroll
    for (int q = 0; q < NR; ++q)
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int pe = p[q] + e * G;
        const bool on = pe < p1[q];
        k[q][e] = on ? col[pe] : -1;
        a[q][e] = on ? (TV)ldv(val, pe) : TV(0);
      }
    more = false;
#pragma unroll
    for (int q = 0; q < NR; ++q) {
      TV xe[E];
#pragma unroll
      for (int e = 0; e < E; ++e) xe[e] = k[q][e] >= 0 ? x[k[q][e]] : TV(0);
#pragma unroll
      for (int e = 0; e < E; ++e)
        if (k[q][e] >= 0) acc[q] += a[q][e] * xe[e];
      p[q] += E * G;
      more |= p[q] < p1[q];
    }
  }
  __syncwarp();
  for (int o = G >> 1; o > 0; o >>= 1)
#pragma unroll
    for (int q = 0; q < NR; ++q) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], o);
  TV s = acc[0];
#pragma unroll
  for (int q = 1; q < NR; ++q)
    if (gl == q) s = acc[q];
  if (er < 0) return;
  if (MODE == CSR_SPMV) {
    y[er] = s;
  } else if (MODE == CSR_SPMV_CHEB0) {
    const TV w = c2 * (iv * s);
    y[er] = s;
    d[er] = w;
    y2[er] = w;
  } else if (MODE == CSR_RESID) {
    y[er] = bv - s;
  } else if (MODE == CSR_ADD) {
    y[er] = xv + s;
  } else {  // CSR_CHEB
    const TV t = iv * (bv - s);
    const TV w = (c1 == TV(0)) ? c2 * t : fma(c2, t, c1 * dv);
    d[er] = w;
    y[er] = xv + w;
  }
}

// --- CSR, a thread per short row ------------------------------------------------------------
constexpr int kShortWin = 6;

template <class TV, class TM, int MODE>
__device__ __forceinline__ void csr_short_row(int row, const int* __restrict__ rowptr,
                                              const int* __restrict__ col,
                                              const TM* __restrict__ val,
                                              const TV* __restrict__ x, TV* __restrict__ y) {
  const int p0 = rowptr[row], p1 = rowptr[row + 1];
  const TV y0 = MODE == CSR_ADD ? y[row] : TV(0);
  int k[kShortWin];
  TV a[kShortWin];
#pragma unroll
  for (int q = 0; q < kShortWin; ++q) {
    const bool on = p0 + q < p1;
    k[q] = on ? col[p0 + q] : 0;
    a[q] = on ? (TV)ldv(val, p0 + q) : TV(0);
  }
  // the sum starts from y: the six predicated steps and an addition would be seven FP64
  // instructions a row, and FP64 issue binds the level-0 prolongation
  TV acc = y0;
#pragma unroll
  for (int q = 0; q < kShortWin; ++q)
    if (p0 + q < p1) acc += a[q] * x[k[q]];
  for (int p = p0 + kShortWin; p < p1; ++p) acc += (TV)ldv(val, p) * x[col[p]];
  y[row] = acc;
}

// --- SELL-32, a thread per row of slice s ---------------------------------------------------
constexpr int kSellCheb1 = 6;  // CSR_CHEB with c1 = 0: d is not read

template <class TV, class TM, int MODE, bool REL>
__device__ __forceinline__ void sell_row(int s, int lane, int n, const int* __restrict__ perm,
                                         const int* __restrict__ soff,
                                         const int* __restrict__ col,
                                         const short* __restrict__ dcol,
                                         const TM* __restrict__ val, const TV* __restrict__ x,
                                         TV* __restrict__ y, const TV* __restrict__ b,
                                         TV* __restrict__ d, const TV* __restrict__ invd, TV c1,
                                         TV c2, double& dacc) {
  const int p = 32 * s + lane;
  if (p >= n) return;
  const int row = perm[p];
  TV acc = TV(0);
  if (MODE != CSR_CHEB0) {
    const int e0 = soff[s] + lane, w = (soff[s + 1] - soff[s]) >> 5;
    int k = 0;
    // eight independent (column, value, x) loads in flight per lane
    for (; k + 8 <= w; k += 8) {
      const int e = e0 + 32 * k;
      int kk[8];
      TV a[8], xv[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        kk[u] = REL ? row + dcol[e + 32 * u] : col[e + 32 * u];
        a[u] = (TV)ldv(val, e + 32 * u);
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) xv[u] = x[kk[u]];
#pragma unroll
      for (int u = 0; u < 8; ++u) acc = fma(a[u], xv[u], acc);
    }
    for (; k + 4 <= w; k += 4) {
      const int e = e0 + 32 * k;
      const int k0 = REL ? row + dcol[e] : col[e];
      const int k1 = REL ? row + dcol[e + 32] : col[e + 32];
      const int k2 = REL ? row + dcol[e + 64] : col[e + 64];
      const int k3 = REL ? row + dcol[e + 96] : col[e + 96];
      const TV a0 = (TV)ldv(val, e), a1 = (TV)ldv(val, e + 32), a2 = (TV)ldv(val, e + 64),
               a3 = (TV)ldv(val, e + 96);
      const TV x0 = x[k0], x1 = x[k1], x2 = x[k2], x3 = x[k3];
      acc = fma(a0, x0, acc);
      acc = fma(a1, x1, acc);
      acc = fma(a2, x2, acc);
      acc = fma(a3, x3, acc);
    }
    for (; k < w; ++k) {
      const int e = e0 + 32 * k;
      acc = fma((TV)ldv(val, e), x[REL ? row + dcol[e] : col[e]], acc);
    }
  }
  if (MODE == CSR_SPMV) {
    y[row] = acc;
  } else if (MODE == CSR_RESID) {
    y[row] = b[row] - acc;
  } else if (MODE == CSR_ADD) {
    y[row] = y[row] + acc;
  } else if (MODE == CSR_CHEB) {
    const TV dv = fma(c1, d[row], c2 * (invd[row] * (b[row] - acc)));
    d[row] = dv;
    y[row] = x[row] + dv;
  } else if (MODE == kSellCheb1) {
    const TV dv = c2 * (invd[row] * (b[row] - acc));
    d[row] = dv;
    y[row] = x[row] + dv;
  } else if (MODE == CSR_CHEB0) {
    const TV dv = c2 * (invd[row] * b[row]);
    d[row] = dv;
    y[row] = dv;
  } else {  // CSR_SPMV_DINV_DOT: c2 carries the scale of x
    const TV w = (c2 * invd[row]) * acc;
    y[row] = w;
    dacc += (double)w * (double)w;
  }
}

// --- coarse solve: row i of the explicit inverse times b, a warp per row -------------------
template <class TV>
__device__ __forceinline__ void gemv_row(int i, int n, int lane, const double* __restrict__ inv,
                                         const TV* __restrict__ b, TV* __restrict__ x) {
  const double* row = inv + (size_t)i * n;
  double acc = 0.0;
#pragma unroll 8  // that many loads in flight, added in order
  for (int c = lane; c < n; c += 32) acc += row[c] * widen(b[c]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) x[i] = (TV)acc;
}

// --- reductions -----------------------------------------------------------------------------
// The tail of a reduction is a chain of dependent FP64 additions (66 clocks each) and barriers (40):
// shuffles inside the warps, one barrier, shuffles over the warps' sums.
__device__ __forceinline__ double warp_tree(double v, int width) {
  for (int o = width / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum over the block (a power of two of warps), valid in the threads of warp 0.
__device__ __forceinline__ double block_sum(double v) {
  __shared__ double sh[32];
  const int nw = (int)(blockDim.x >> 5);
  v = warp_tree(v, 32);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x < 32) t = warp_tree((int)threadIdx.x < nw ? sh[threadIdx.x] : 0.0, nw);
  return t;
}

// Ordered sum of `count` partials by one block, valid in the threads of warp 0.  The partials are
// read through L2: blocks of the same launch may have written them.
__device__ __forceinline__ double sum_fixed(const double* part, int count) {
  double acc = 0.0;
#pragma unroll 4
  for (int i = threadIdx.x; i < count; i += blockDim.x) acc += __ldcg(part + i);
  __syncthreads();  // block_sum's shared array may still be read from an earlier sum
  return block_sum(acc);
}

// Block `blk` of a fixed grid of kRedBlocks x kRedThreads: its partial of sum a_i b_i (loads
// of four grid strides in flight, the multiply-adds in index order).  Valid in thread 0.
template <class TA, class TB>
__device__ __forceinline__ double dot_block(int blk, int n, const TA* __restrict__ a,
                                            const TB* __restrict__ b) {
  double acc = 0.0;
  const int st = kRedBlocks * kRedThreads;
  int i = blk * kRedThreads + threadIdx.x;
  for (; i + 3 * st < n; i += 4 * st) {
    const double a0 = widen(a[i]), a1 = widen(a[i + st]), a2 = widen(a[i + 2 * st]),
                 a3 = widen(a[i + 3 * st]);
    const double b0 = widen(b[i]), b1 = widen(b[i + st]), b2 = widen(b[i + 2 * st]),
                 b3 = widen(b[i + 3 * st]);
    acc += a0 * b0;
    acc += a1 * b1;
    acc += a2 * b2;
    acc += a3 * b3;
  }
  for (; i < n; i += st) acc += widen(a[i]) * widen(b[i]);
  return block_sum(acc);
}

// r'z and z'q of block `blk` in one sweep; the same per-thread order and block tree as two
// dot_block calls.
template <class TZ>
__device__ __forceinline__ void dot2_block(int blk, int n, const double* __restrict__ r,
                                           const TZ* __restrict__ z,
                                           const double* __restrict__ q, double& t1,
                                           double& t2) {
  double a1 = 0.0, a2 = 0.0;
  const int st = kRedBlocks * kRedThreads;
  int i = blk * kRedThreads + threadIdx.x;
  // loads of four grid strides in flight (the fixed grid holds half the warps an SM can)
  for (; i + 3 * st < n; i += 4 * st) {
    double zz[4], rr[4], qq[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      zz[u] = widen(z[i + u * st]);
      rr[u] = r[i + u * st];
      qq[u] = q[i + u * st];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      a1 += rr[u] * zz[u];
      a2 += zz[u] * qq[u];
    }
  }
  for (; i < n; i += st) {
    const double zi = widen(z[i]);
    a1 += r[i] * zi;
    a2 += zi * q[i];
  }
  t1 = block_sum(a1);
  __syncthreads();  // block_sum's shared array is reused
  t2 = block_sum(a2);
}

// x += alpha p; r -= alpha q; r32 = (float) r; block `blk`'s partial of r'r (thread 0).
__device__ __forceinline__ double update_block(int blk, int n, double a, double* __restrict__ x,
                                               double* __restrict__ r,
                                               const double* __restrict__ p,
                                               const double* __restrict__ q,
                                               float* __restrict__ r32) {
  double acc = 0.0;
  const int st = kRedBlocks * kRedThreads;
  int i = blk * kRedThreads + threadIdx.x;
  // two grid strides per step, every load before the stores
  for (; i + st < n; i += 2 * st) {
    const double x0 = x[i], x1 = x[i + st], p0 = p[i], p1 = p[i + st];
    const double rv0 = r[i], rv1 = r[i + st], q0 = q[i], q1 = q[i + st];
    x[i] = x0 + a * p0;
    const double ri0 = rv0 - a * q0;
    r[i] = ri0;
    if (r32) r32[i] = narrow(ri0);
    acc += ri0 * ri0;
    x[i + st] = x1 + a * p1;
    const double ri1 = rv1 - a * q1;
    r[i + st] = ri1;
    if (r32) r32[i + st] = narrow(ri1);
    acc += ri1 * ri1;
  }
  for (; i < n; i += st) {
    x[i] = x[i] + a * p[i];
    double ri = r[i] - a * q[i];
    r[i] = ri;
    if (r32) r32[i] = narrow(ri);
    acc += ri * ri;
  }
  return block_sum(acc);
}

// --- the same blocks emulated by one warp ---------------------------------------------------
// A warp can stand in for a block of kRedThreads = 8 x 32 threads: lane l holds the accumulators
// of the block's threads 32 w + l (w = 0..7, the block's warps), every accumulator is reduced by
// the warp's xor tree (the block's per-warp reduction), and the eight sums by the block's tree
// over its warps.  The result has the bits of the block's partial, in every
// lane, without shared memory or barriers, and eight of these run side by side in a block.
constexpr int kVirtWarps = kRedThreads / 32;

// The eight xor trees (16, 8, 4, 2, 1) at once: at the first three levels a lane keeps half of its
// accumulators and passes the other half on, so a tree level is 4, 2, 1, 1, 1 additions for all
// eight instead of 8 each (an FP64 instruction holds a quarter of the SM for 64 clocks, whatever
// its lanes do); each sum adds the same two numbers as the plain tree.  Lane bits 4, 3 and 2 then
// hold the warp's number, and three more levels are the block's sum over its warps.
__device__ __forceinline__ double warp_tree8(const double v[kVirtWarps], int lane) {
  double u[4], w[2];
  const bool h16 = lane & 16, h8 = lane & 8, h4 = lane & 4;
#pragma unroll
  for (int q = 0; q < 4; ++q)
    u[q] = (h16 ? v[q + 4] : v[q]) + __shfl_xor_sync(0xffffffffu, h16 ? v[q] : v[q + 4], 16);
#pragma unroll
  for (int q = 0; q < 2; ++q)
    w[q] = (h8 ? u[q + 2] : u[q]) + __shfl_xor_sync(0xffffffffu, h8 ? u[q] : u[q + 2], 8);
  double s = (h4 ? w[1] : w[0]) + __shfl_xor_sync(0xffffffffu, h4 ? w[0] : w[1], 4);
#pragma unroll
  for (int o : {2, 1, 16, 8, 4}) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

// f(i, w) for every element i of the block's threads 32 w + lane, in each thread's order
template <class F>
__device__ __forceinline__ void virt_block(int blk, int n, int lane, F&& f) {
  for (int base = blk * kRedThreads; base < n; base += kRedBlocks * kRedThreads) {
#pragma unroll
    for (int w = 0; w < kVirtWarps; ++w) {
      if (base + 32 * w >= n) break;  // uniform
      const int i = base + 32 * w + lane;
      if (i < n) f(i, w);
    }
  }
}

template <class TA, class TB>
__device__ __forceinline__ double dot_block_warp(int blk, int n, const TA* __restrict__ a,
                                                 const TB* __restrict__ b, int lane) {
  double acc[kVirtWarps] = {};
  virt_block(blk, n, lane, [&](int i, int w) { acc[w] += widen(a[i]) * widen(b[i]); });
  return warp_tree8(acc, lane);
}

template <class TZ>
__device__ __forceinline__ void dot2_block_warp(int blk, int n, const double* __restrict__ r,
                                                const TZ* __restrict__ z,
                                                const double* __restrict__ q, int lane,
                                                double& t1, double& t2) {
  double a1[kVirtWarps] = {}, a2[kVirtWarps] = {};
  virt_block(blk, n, lane, [&](int i, int w) {
    const double zi = widen(z[i]);
    a1[w] += r[i] * zi;
    a2[w] += zi * q[i];
  });
  t1 = warp_tree8(a1, lane);
  t2 = warp_tree8(a2, lane);
}

__device__ __forceinline__ double update_block_warp(int blk, int n, double a,
                                                    double* __restrict__ x,
                                                    double* __restrict__ r,
                                                    const double* __restrict__ p,
                                                    const double* __restrict__ q,
                                                    float* __restrict__ r32, int lane) {
  double acc[kVirtWarps] = {};
  virt_block(blk, n, lane, [&](int i, int w) {
    x[i] = x[i] + a * p[i];
    const double ri = r[i] - a * q[i];
    r[i] = ri;
    if (r32) r32[i] = narrow(ri);
    acc[w] += ri * ri;
  });
  return warp_tree8(acc, lane);
}

}  // namespace rows
}  // namespace saamg
