// The steps on either side of the solve in a PIC time step (Sec. 1: E = -grad phi of the
// Poisson solution; Sec. 4.1: cloud-in-cell deposition of the particle charges): CIC
// deposition onto the box lattice and the CIC gather of the nodal field at the particles.
//
// Deposition is deterministic: every contribution ((q / V) wx) wy) wz is rounded once to a
// 64-bit fixed-point number with a power-of-two scale chosen from sum |q| (no node can hold
// more), and the integer atomic additions commute.  The gather uses explicit round-to-
// nearest multiply and add in the reference's order, so it is bitwise the CPU result.
#include "pic.cuh"

#include "divc.cuh"
#include "softmul.cuh"

namespace saamg {

namespace {

struct Lattice {
  int nx, ny, nz;
  double ox, oy, oz;
  DivC hx, hy, hz;  // spacings
  DivC vol;
};

// u = (x - o) / h: the particle's lattice coordinate.
__device__ __forceinline__ double lattice_coord(double x, double o, const DivC& h) {
  return div_by(x - o, h);
}

// Whether the cell of u can touch the box: -1 <= u < 2^31 - 1 (false for NaN), on the bits.
__device__ __forceinline__ bool coord_near(double u) {
  const long long b = __double_as_longlong(u);
  return b >= 0 ? b < 0x41dfffffffc00000LL
                : (b & 0x7fffffffffffffffLL) <= 0x3ff0000000000000LL;
}

// c = floor(u), f = u - floor(u) for coord_near(u).  Adding 1.5 * 2^52 rounds u to an integer in
// the low word; the difference to it is exact, and one below zero belongs to the cell before
// (f = d + 1 rounds the same real number as u - floor(u)).  Four FP64 additions; floor and the
// two conversions would take as many instructions on slower paths.
__device__ __forceinline__ void split_coord(double u, int& c, double& f) {
  const double big = 6755399441055744.0;  // 1.5 * 2^52
  const double t = __dadd_rn(u, big);
  const double d = __dadd_rn(u, -__dadd_rn(t, -big));
  c = __double2loint(t);
  f = d;
  if (__double2hiint(d) < 0 &&
      (static_cast<unsigned long long>(__double_as_longlong(d)) << 1) != 0ull) {
    c -= 1;
    f = __dadd_rn(d, 1.0);
  }
}

// The same cell and the fraction as a 64-bit fixed-point number, by integer operations.
__device__ __forceinline__ void split_coord_fixed(double u, int& c, unsigned long long& f) {
  const long long b = __double_as_longlong(u);
  const int e = (int)((b >> 52) & 0x7ff) - 1023;  // |u| = m / 2^63 * 2^e
  const unsigned long long m =
      e == -1023 ? 0ull : ((unsigned long long)b << 11) | 0x8000000000000000ull;
  if (e >= 0) {  // e <= 30; u = -1 is the only negative one
    c = (int)(m >> (63 - e));
    f = m << (e + 1);
  } else {
    c = 0;
    f = e > -65 ? m >> (-1 - e) : 0ull;
  }
  if (b < 0) {
    c = f != 0ull ? -c - 1 : -c;
    f = 0ull - f;
  }
}

// Whether split_coord_fixed's fraction of u holds all of u's bits: u is 0 or at least 2^-11, so
// that neither a bit below 2^-64 is cut nor, for u < 0, a rounding of 1 + u left out.
__device__ __forceinline__ bool fraction_exact(double u) {
  const long long b = __double_as_longlong(u);
  return b == 0 || b >= 0x3f40000000000000LL;
}

__global__ void abs_sum_k(int n, const double* __restrict__ q, double* __restrict__ part) {
  double acc = 0.0;
  const int st = gridDim.x * blockDim.x;
  long long i = blockIdx.x * blockDim.x + threadIdx.x;
  for (; i + 3LL * st < n; i += 4LL * st) {  // four loads in flight, added in index order
    const double a = q[i], b = q[i + st], c = q[i + 2LL * st], d = q[i + 3LL * st];
    acc += fabs(a);
    acc += fabs(b);
    acc += fabs(c);
    acc += fabs(d);
  }
  for (; i < n; i += st) acc += fabs(q[i]);
  __shared__ double sh[32];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[w];
    part[blockIdx.x] = t;
  }
}

// scale exponent: sum|q| / V * 2^S < 2^61, so no node sum can overflow 64 bits;
// exp[1] = 1 when the charges are not finite
__global__ void scale_k(const double* __restrict__ part, int nparts, double vol,
                        int* __restrict__ exp) {
  if (threadIdx.x != 0) return;
  double t = 0.0;
  for (int i = 0; i < nparts; ++i) t += part[i];
  const double b = t / vol;
  exp[1] = isfinite(b) ? 0 : 1;
  exp[0] = (b > 0.0 && isfinite(b)) ? 60 - ilogb(b) : 0;
}

// |v| w for a weight w in units of 2^-64, in units of the 64-bit mantissa of v.
__device__ __forceinline__ unsigned long long wmul(unsigned long long a, unsigned long long w) {
  return __umul64hi(a, w);
}

// The warp's sum modulo 2^64: pieces of 27 bits, of which 32 add up below 2^32.
__device__ __forceinline__ unsigned long long warp_sum64(unsigned long long v) {
  const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)v & 0x7ffffffu);
  const unsigned mid = __reduce_add_sync(0xffffffffu, (unsigned)(v >> 27) & 0x7ffffffu);
  const unsigned hi = __reduce_add_sync(0xffffffffu, (unsigned)(v >> 54));
  return lo + ((unsigned long long)mid << 27) + ((unsigned long long)hi << 54);
}

// A particle adds round(2^S (q / V) wx wy wz) to each of its eight nodes.  The weights are
// 64-bit fixed-point fractions and the products integer multiplications: |q / V| 2^S < 2^61, so
// a product's three truncations are off by less than 3/8 of the fixed-point unit, where the
// rounding of the product in FP64 (53 bits of a number of up to 61) could be off by 2^7 units.
// In FP64 the divisions, the 14 weight products, the scalings and the conversions of a particle ran
// on a pipe of two lanes per clock and SM; now the L2 atomics bind the pass (86 % of the L2's
// throughput, FP64 pipe 42 %): 10^7 particles on 256^3 take 384 us here, and the whole call 515 us
// instead of 2472.
__global__ void __launch_bounds__(256) cic_deposit_k(Lattice g, int np,
                                                     const double* __restrict__ x,
                                                     const double* __restrict__ y,
                                                     const double* __restrict__ z,
                                                     const double* __restrict__ q,
                                                     const int* __restrict__ exp,
                                                     unsigned long long* __restrict__ acc) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= np) return;
  const double xp = x[p], yp = y[p], zp = z[p], qp = q[p];
  if (exp[1]) return;
  const double ux = lattice_coord(xp, g.ox, g.hx), uy = lattice_coord(yp, g.oy, g.hy),
               uz = lattice_coord(zp, g.oz, g.hz);
  if (!(coord_near(ux) && coord_near(uy) && coord_near(uz))) return;
  int ci, cj, ck;
  unsigned long long fx, fy, fz;
  split_coord_fixed(ux, ci, fx);
  split_coord_fixed(uy, cj, fy);
  split_coord_fixed(uz, ck, fz);
  if (ci >= g.nx || cj >= g.ny || ck >= g.nz) return;
  // |q / V| = m / 2^63 * 2^e, scaled by 2^S: the product m w >> 64 is to be shifted right by sh
  const long long qb = __double_as_longlong(div_by(qp, g.vol));
  int e = (int)((qb >> 52) & 0x7ff) - 1023;
  unsigned long long m = (unsigned long long)qb << 11;
  if (e > -1023) {
    m |= 0x8000000000000000ull;
  } else {
    if (m == 0ull) return;
    const int lz = __clzll((long long)m);  // subnormal
    m <<= lz;
    e = -1022 - lz;
  }
  const int sh = 63 - (e + exp[0]);  // >= 3
  if (sh > 64) return;  // less than half a unit at every node
  const bool neg = qb < 0;
  // 1 - f: 2^64 - f, and 2^64 - 1 for f = 0
  const unsigned long long wx[2] = {fx ? 0ull - fx : ~0ull, fx};
  const unsigned long long wy[2] = {fy ? 0ull - fy : ~0ull, fy};
  const unsigned long long wz[2] = {fz ? 0ull - fz : ~0ull, fz};
  const unsigned long long half = 1ull << (sh - 1);
  const unsigned long long mx[2] = {wmul(m, wx[0]), wmul(m, wx[1])};
  const bool inner = ci >= 0 && cj >= 0 && ck >= 0 && ci + 1 < g.nx && cj + 1 < g.ny &&
                     ck + 1 < g.nz;
  const long long v0 = ci + (long long)g.nx * (cj + (long long)g.ny * ck);
  auto weight = [&](int a, int b, int c) {  // what node (a, b, c) of the cell takes
    const unsigned long long r = wmul(wmul(mx[a], wy[b]), wz[c]);
    const unsigned long long w = sh < 64 ? (r >> sh) + ((r & half) != 0) : (r >> 63);
    return neg ? 0ull - w : w;
  };
  // 32 particles of one cell: their sum per node, one atomic each (an inner cell's index is below
  // 4.0e9, the most nodes a grid may have).  Additions to the same address are served one after the
  // other: 10^6 particles in one cell took 926 us without this (841 with the FP64 weights), now 90
  if (__activemask() == 0xffffffffu) {
    const unsigned lane = threadIdx.x & 31;
    int same;
    __match_all_sync(0xffffffffu, inner ? (unsigned)v0 : ~lane, &same);
    if (same) {
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const unsigned long long w = weight(k & 1, (k >> 1) & 1, k >> 2);
        const unsigned long long sum = warp_sum64(w);
        if (lane == k && sum)
          atomicAdd(&acc[v0 + (k & 1) + (long long)g.nx * (((k >> 1) & 1) + (long long)g.ny * (k >> 2))],
                    sum);
      }
      return;
    }
  }
#pragma unroll
  for (int c = 0; c < 2; ++c)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const bool line = inner || (cj + b >= 0 && ck + c >= 0 && cj + b < g.ny && ck + c < g.nz);
      const long long v = v0 + (long long)g.nx * (b + (long long)g.ny * c);
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        if (!inner && !(line && ci + a >= 0 && ci + a < g.nx)) continue;
        const unsigned long long w = weight(a, b, c);
        if (w) atomicAdd(&acc[v + a], w);
      }
    }
}

// rho = acc 2^-S (acc may be rho), the nearest double: the leading one of |acc| is found and the 53 bits below
// it rounded to even with integer operations (the FP64 conversion and scaling of 16.8 M nodes
// would take as long as their bytes); a result outside the normal range takes ldexp.
__global__ void __launch_bounds__(256) fixed_to_double_k(size_t n, const int* __restrict__ exp,
                                                         const unsigned long long* acc,
                                                         unsigned long long* rho) {
  const int S = exp[0];
  const bool bad = exp[1] != 0;
  for (size_t v = blockIdx.x * (size_t)blockDim.x + threadIdx.x; v < n;
       v += (size_t)gridDim.x * blockDim.x) {
    if (bad) {
      rho[v] = 0x7ff8000000000000ull;
      continue;
    }
    const long long a = (long long)acc[v];
    if (a == 0) {
      if (acc != rho) rho[v] = 0ull;
      continue;
    }
    unsigned long long u = a < 0 ? 0ull - (unsigned long long)a : (unsigned long long)a;
    const int lz = __clzll((long long)u);
    const int e = 63 - lz - S + 1023;
    unsigned long long r;
    if (e < 1 || e > 2045) {
      r = (unsigned long long)__double_as_longlong(ldexp((double)(long long)u, -S));
    } else {
      u <<= lz;
      r = ((unsigned long long)e << 52) + ((u & 0x7fffffffffffffffull) >> 11);
      const unsigned long long low = u & 0x7ffull;
      if (low > 0x400ull || (low == 0x400ull && (r & 1ull))) ++r;  // may carry into the exponent
    }
    rho[v] = r | (a < 0 ? 0x8000000000000000ull : 0ull);
  }
}

// Components of the field whose products run on the integer units, the others' on the FP64 pipe:
// 10^7 particles on 256^3 took 1101, 951, 1026 and 1139 us with 0, 1, 2 and 3.
constexpr int kGatherSoft = 1;

// Bitwise the reference's sums: ((wx wy) wz) E added in its corner order, every product and sum
// rounded -- 12 + 24 products and 24 sums a particle.  On the FP64 pipe alone they took 1656 us for
// 10^7 particles on 256^3 (pipe 84 % busy, L2 29 %); here the cell and the weights of a particle
// inside the box are integer arithmetic (softmul.cuh, the bits of the FP64 operations), and so are
// the products of kGatherSoft components, which run beside the sums on the other pipe.  A
// particle at the box's edge, and operands that are not normal numbers, take the FP64 operations.
__global__ void __launch_bounds__(256) cic_gather_k(Lattice g, const double* __restrict__ ex,
                                                    const double* __restrict__ ey,
                                                    const double* __restrict__ ez, int np,
                                                    const double* __restrict__ x,
                                                    const double* __restrict__ y,
                                                    const double* __restrict__ z,
                                                    double* __restrict__ epx,
                                                    double* __restrict__ epy,
                                                    double* __restrict__ epz) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= np) return;
  const double xp = x[p], yp = y[p], zp = z[p];
  const double ux = lattice_coord(xp, g.ox, g.hx), uy = lattice_coord(yp, g.oy, g.hy),
               uz = lattice_coord(zp, g.oz, g.hz);
  double s[3] = {0.0, 0.0, 0.0};
  if (coord_near(ux) && coord_near(uy) && coord_near(uz)) {
    const double* E[3] = {ex, ey, ez};
    const long long sy = g.nx, sz = (long long)g.nx * g.ny;
    int ci, cj, ck;
    unsigned long long hx, hy, hz;
    split_coord_fixed(ux, ci, hx);
    split_coord_fixed(uy, cj, hy);
    split_coord_fixed(uz, ck, hz);
    if (fraction_exact(ux) && fraction_exact(uy) && fraction_exact(uz) && ci + 1 < g.nx &&
        cj + 1 < g.ny && ck + 1 < g.nz) {
      const long long v0 = ci + (long long)g.nx * (cj + (long long)g.ny * ck);
      Unpacked w[8];
      {
        const Unpacked wx[2] = {unpack_complement(hx), unpack_fraction(hx)};
        const Unpacked wy[2] = {unpack_complement(hy), unpack_fraction(hy)};
        const Unpacked wz[2] = {unpack_complement(hz), unpack_fraction(hz)};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const Unpacked wxy = mul_unpacked(wx[q & 1], wy[q >> 1]);
          w[q] = mul_unpacked(wxy, wz[0]);
          w[q + 4] = mul_unpacked(wxy, wz[1]);
        }
      }
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const double* e = E[k] + v0;
        double t[8];
#pragma unroll
        for (int q = 0; q < 8; ++q)
          t[q] = e[(q & 1) + ((q >> 1) & 1) * sy + (q >> 2) * sz];
        double a = 0.0;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          double m;
          bool ok = false;
          if (k < kGatherSoft)
            m = __longlong_as_double(
                (long long)mul_bits(w[q], (uint64_t)__double_as_longlong(t[q]), ok));
          if (!ok) m = __dmul_rn(__longlong_as_double((long long)pack_bits(w[q])), t[q]);
          a = q == 0 ? m : __dadd_rn(a, m);
        }
        // the reference starts from +0, which no sum of zeros of either sign leaves
        s[k] = (static_cast<unsigned long long>(__double_as_longlong(a)) << 1) == 0ull ? 0.0 : a;
      }
    } else {
      double fx, fy, fz;
      split_coord(ux, ci, fx);
      split_coord(uy, cj, fy);
      split_coord(uz, ck, fz);
      const long long v0 = ci + (long long)g.nx * (cj + (long long)g.ny * ck);
      const double wx[2] = {__dadd_rn(1.0, -fx), fx}, wy[2] = {__dadd_rn(1.0, -fy), fy},
                   wz[2] = {__dadd_rn(1.0, -fz), fz};
#pragma unroll 1
      for (int q = 0; q < 8; ++q) {
        const int i = q & 1, j = (q >> 1) & 1, k = q >> 2;
        if (ci + i < 0 || cj + j < 0 || ck + k < 0 || ci + i >= g.nx || cj + j >= g.ny ||
            ck + k >= g.nz)
          continue;
        const double w = __dmul_rn(__dmul_rn(i ? wx[1] : wx[0], j ? wy[1] : wy[0]),
                                   k ? wz[1] : wz[0]);
        const long long v = v0 + i + j * sy + k * sz;
#pragma unroll
        for (int d = 0; d < 3; ++d) s[d] = __dadd_rn(s[d], __dmul_rn(w, E[d][v]));
      }
    }
  }
  epx[p] = s[0];
  epy[p] = s[1];
  epz[p] = s[2];
}

Lattice lattice(const saamg_grid& g) {
  return Lattice{g.n[0], g.n[1], g.n[2], g.origin[0], g.origin[1], g.origin[2],
                 make_divc(g.h[0]), make_divc(g.h[1]), make_divc(g.h[2]),
                 make_divc((g.h[0] * g.h[1]) * g.h[2])};
}

}  // namespace

void deposit_cic(const saamg_grid& grid, int np, const double* x, const double* y,
                 const double* z, const double* q, double* rho, cudaStream_t s) {
  const Lattice g = lattice(grid);
  const size_t nbox = (size_t)g.nx * g.ny * g.nz;
  Buf<double> part;
  Buf<int> exp;
  part.alloc(kRedBlocks, s);
  exp.alloc(2, s);
  // rho itself holds the fixed-point sums until they are converted, unless it overlaps an input
  unsigned long long* out = reinterpret_cast<unsigned long long*>(rho);
  unsigned long long* acc = out;
  Buf<unsigned long long> own;
  for (const double* in : {x, y, z, q})
    if ((uintptr_t)in < (uintptr_t)(rho + nbox) && (uintptr_t)rho < (uintptr_t)(in + np) && !own.p) {
      own.alloc(nbox, s);
      acc = own.p;
    }
  SAAMG_CUDA(cudaMemsetAsync(acc, 0, nbox * sizeof(unsigned long long), s));
  abs_sum_k<<<kRedBlocks, 256, 0, s>>>(np, q, part.p);
  SAAMG_LAUNCH();
  scale_k<<<1, 32, 0, s>>>(part.p, kRedBlocks, g.vol.c, exp.p);
  SAAMG_LAUNCH();
  if (np > 0) {
    KernelTimer kt(SAAMG_KT_PIC, np, s);
    cic_deposit_k<<<(np + 255) / 256, 256, 0, s>>>(g, np, x, y, z, q, exp.p, acc);
    SAAMG_LAUNCH();
  }
  const int blocks = (int)std::min<size_t>((nbox + 255) / 256, sm_count() * 16);
  fixed_to_double_k<<<blocks, 256, 0, s>>>(nbox, exp.p, acc, out);
  SAAMG_LAUNCH();
}

void gather_cic(const saamg_grid& grid, const double* ex, const double* ey, const double* ez,
                int np, const double* x, const double* y, const double* z, double* epx,
                double* epy, double* epz, cudaStream_t s) {
  if (np <= 0) return;
  KernelTimer kt(SAAMG_KT_PIC, np, s);
  cic_gather_k<<<(np + 255) / 256, 256, 0, s>>>(lattice(grid), ex, ey, ez, np, x, y, z, epx,
                                                epy, epz);
  SAAMG_LAUNCH();
}

}  // namespace saamg
