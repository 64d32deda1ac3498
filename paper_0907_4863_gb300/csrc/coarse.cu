// Coarsest-level direct solver (Sec. 3.2, "Coarse level solver"; Algorithm 1,
// DirectSolve).  The paper factors A_L with KLU; here A_L is small (<= max_coarse) and its
// inverse is formed once, densely in FP64, by Gauss-Jordan elimination with the pivoting of
// an LU with partial pivoting (largest |a_ik|, lowest row on ties), so that every V-cycle
// applies x = A_L^-1 b as one dense product.
// The elimination works on column-major arrays, a(i, j) at [j * n + i]; the finished inverse
// is stored by rows, A_L^-1(i, j) at [i * n + j], for the per-cycle product.
#include "coarse.cuh"
#include "rows.cuh"

#include <cooperative_groups.h>

#include <utility>

namespace saamg {

namespace {

__global__ void densify_k(int n, const int* __restrict__ rowptr, const int* __restrict__ col,
                          const double* __restrict__ val, double* __restrict__ a) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  for (int p = rowptr[i]; p < rowptr[i + 1]; ++p) a[(size_t)col[p] * n + i] = val[p];
}

// --- explicit inverse by blocked Gauss-Jordan elimination ------------------------------
// Step k picks the pivot among the rows not yet pivoted (largest |a_ik|, lowest row on ties; rows
// are never exchanged), scales that row p by 1 / a_pk to r, and takes a_ik r off every other row;
// column k becomes 1 / a_pk in row p and -a_ik / a_pk elsewhere.  After n steps with pivot rows
// p_k the inverse is inv(k, p_j) = a(p_k, j).
// B steps make a panel.  gj_panel_k factors the panel's B columns on one cluster of 16 blocks, each
// with a range of rows in its shared memory, and leaves the multipliers c_s(i) = a_ik of its steps
// (B x n); gj_update_k applies the B steps to the whole matrix: per column the B values r_s by a
// forward substitution over the pivot rows, then x_i - sum_s c_s(i) r_s on every row, an FP64
// contraction of depth B that runs on all SMs from registers.  The update reads one copy of the
// matrix and writes the other, so a tile never reads a pivot row that another tile has overwritten.
// The panel of the next steps needs only its own columns of the updated matrix: gj_panel_k applies
// the pending panel to them itself and runs beside the update.  It is launched first and lets the
// update start once its blocks are resident (programmatic dependent launch); their shared-memory
// requests keep the two off the same SM, where the update's warps would queue before every FP64
// instruction of the panel's serial chain (n = 1250: 70 instead of 52 us a panel).
// What the update reads was written by the launches before the panel beside it, and a programmatic
// dependent has no order with those but through griddepcontrol.wait, which would have it wait for
// the panel as well.  The panel has waited for them: it says so by a release store before it lets
// the update start, and the update's blocks read that with an acquire load (or wait, if they do not
// see it).
constexpr int kGjB = 16;           // steps of a panel
constexpr int kGjCluster = 16;     // blocks of the panel kernel (an opt-in size)
constexpr int kGjThreads = 256;    // panel kernel: two of the panel's columns per warp
constexpr int kGjMaxRows = 16384 / kGjCluster;  // rows per panel block at the largest n
constexpr int kGjUpdThreads = 512;
constexpr int kGjUpdCols = 32;     // most columns of an update tile, two per warp
// dynamic shared memory: a panel block's rows at the largest n, and enough on either side that a
// panel block and an update block do not fit one SM (228 KB)
constexpr size_t kGjRowBytes = kGjB * sizeof(double) + sizeof(int);
constexpr size_t kGjPanelSmem = 192u << 10, kGjUpdSmem = 36u << 10;
static_assert(kGjMaxRows * kGjRowBytes <= kGjPanelSmem, "the panel's rows fit a block");
static_assert(kGjThreads / 32 * 2 == kGjB && kGjUpdThreads / 32 * 2 == kGjUpdCols && kGjB == 16,
              "a half-warp per column in the forward substitutions");

// What a panel leaves for its update beside the multipliers: the pivot rows, their pivots'
// reciprocals and l[t][s] = c_s(p_t) / pivot_s for s < t.
struct GjPanel {
  double ip[kGjB];
  double l[kGjB][kGjB];
  int row[kGjB];
};

// Pivot keys order like |v| as integers, so the search runs on the integer units instead of the
// FP64 pipe: 0 for no row, 1 for a NaN (it loses against every number), 2 + the bits of |v|.
__device__ __forceinline__ unsigned long long pivot_key(double v) {
  const unsigned long long b =
      (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
  return b > 0x7ff0000000000000ull ? 1ull : b + 2ull;
}

// (key, index) maximum over a warp, lowest index on ties, by three integer warp reductions (a
// butterfly of 64-bit shuffles takes five times as long); every lane holds the result
__device__ __forceinline__ void gj_warp_argmax(unsigned long long& key, int& idx) {
  const unsigned hi = (unsigned)(key >> 32), lo = (unsigned)key;
  const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
  const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
  idx = (int)__reduce_min_sync(0xffffffffu, hi == mh && lo == ml ? (unsigned)idx : 0x7fffffffu);
  key = ((unsigned long long)mh << 32) | ml;
}

// r_t of one column in lane t of a half-warp, from the column's value x in pivot row t; the steps
// s <= s0 and s >= bw do not apply.  A step is one shuffle and one FP64 instruction (a warp's
// FP64 instruction holds its quarter of the SM for 64 clocks: a thread per column would take 136).
__device__ __forceinline__ double gj_forward(double x, int t, const GjPanel& pn, int s0, int bw) {
  if (t <= s0 || t >= bw) x = 0.0;
#pragma unroll
  for (int s = 0; s < kGjB - 1; ++s) {
    const double xs = __shfl_sync(0xffffffffu, x, s, kGjB);
    if (t > s && t < bw && t > s0) x = fma(-pn.l[t][s], xs, x);
  }
  return t > s0 && t < bw ? x * pn.ip[t] : 0.0;
}

// Factors the panel of columns k0 .. k0 + bw - 1 after applying the pending panel (pend = 0: none)
// to them (pstep: the rows' steps before it, NULL for none).  A step's chain -- the next column's update and pivot search, the exchange of the
// blocks' candidates through distributed shared memory, one division -- is what bounds the kernel:
// the candidate's own row is brought up to date by one instruction per panel column, and the rest
// of the panel is updated while the cluster barrier is on its way.
__global__ void __launch_bounds__(kGjThreads)
    gj_panel_k(int n, int k0, int rpb, const double* __restrict__ a, int pend,
               const GjPanel* __restrict__ ppn, const double* __restrict__ pc,
               GjPanel* __restrict__ opn, double* __restrict__ oc, const int* __restrict__ pstep,
               int* __restrict__ step, int* __restrict__ prow, int* __restrict__ err, int seq,
               int* ready) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  asm volatile("griddepcontrol.wait;" ::: "memory");  // the update before
  if (threadIdx.x == 0) {                             // the update beside this panel
    if (blockIdx.x == 0)
      asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(ready), "r"(seq) : "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  }
  constexpr int B = kGjB;
  struct Cand {
    double v[B];
    unsigned long long key;
    int row;
  };
  extern __shared__ double pan[];  // B columns of the block's rpb rows
  __shared__ Cand cand[2][kGjCluster];
  __shared__ unsigned long long sv[kGjThreads / 32];
  __shared__ int si[kGjThreads / 32];
  __shared__ double s_r[2][B];
  __shared__ GjPanel pn;       // the pending panel, then this one
  __shared__ double rr[B][B];  // pending r_s of each panel column j: rr[s][j]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int me = (int)cluster.block_rank();
  const int bw = min(B, n - k0);
  const int i0 = me * rpb, rows = max(0, min(rpb, n - i0));
  // threads by (row, column group): G groups of rp threads
  int rp = 32;
  while (rp < rows && rp < kGjThreads) rp <<= 1;
  const int G = kGjThreads / rp, gi = tid & (rp - 1), gg = tid / rp;
  // the pivot step of every own row so far sits behind the panel
  int* own = reinterpret_cast<int*>(pan + (size_t)B * rpb);
  for (int i = tid; i < rows; i += kGjThreads) own[i] = pstep ? pstep[i0 + i] : -1;
  if (pend > 0) {
    const double* src = reinterpret_cast<const double*>(ppn);
    double* dst = reinterpret_cast<double*>(&pn);
    for (int e = tid; e < (int)(sizeof(GjPanel) / 8); e += kGjThreads) dst[e] = src[e];
    __syncthreads();
    const int j = 2 * warp + (lane >> 4), t = lane & 15;
    const double x = j < bw && t < pend ? a[(size_t)(k0 + j) * n + pn.row[t]] : 0.0;
    rr[t][j] = gj_forward(x, t, pn, -1, pend);
  }
  __syncthreads();
  for (int i = gi; i < rows; i += rp) {
    const int kp = own[i] - (k0 - pend);  // its step in the pending panel, if any
    double c[B];
    if (pend > 0) {
#pragma unroll
      for (int s = 0; s < B; ++s) c[s] = s < pend ? pc[(size_t)s * n + i0 + i] : 0.0;
    }
    for (int j = gg; j < bw; j += G) {
      double x = a[(size_t)(k0 + j) * n + i0 + i];
      if (pend > 0) {
        if (kp >= 0) x = rr[kp][j];
#pragma unroll
        for (int s = 0; s < B; ++s) x = fma(-c[s], rr[s][j], x);
      }
      pan[(size_t)j * rpb + i] = x;
    }
  }
  cluster.sync();  // every block runs before the first one writes into another's shared memory
  int p = -1;         // pivot row of the current step
  double myip = 0.0;  // warp 0, lane s: 1 / pivot of step s
  for (int s = -1; s < bw - 1; ++s) {
    // step s (none for -1) on column s + 1, and the pivot search there
    const int jn = s + 1;
    const double* r = s_r[s & 1];
    unsigned long long best = 0;
    int bi = n;
    for (int i = tid; i < rows; i += kGjThreads) {
      double v = pan[(size_t)jn * rpb + i];
      if (s >= 0) {
        const bool isp = i0 + i == p;
        if (isp) own[i] = k0 + s;
        v = isp ? r[jn] : fma(-pan[(size_t)s * rpb + i], r[jn], v);
        pan[(size_t)jn * rpb + i] = v;
      }
      if (own[i] < 0) {
        const unsigned long long key = pivot_key(v);
        if (key > best) {
          best = key;
          bi = i0 + i;
        }
      }
    }
    gj_warp_argmax(best, bi);
    if (lane == 0) {
      sv[warp] = best;
      si[warp] = bi;
    }
    __syncthreads();
    if (warp == 0) {
      // the block's candidate with its row of the panel (multipliers up to s, the values after
      // step s beyond) goes to every block of the cluster, a half-warp a block
      best = lane < kGjThreads / 32 ? sv[lane] : 0ull;
      bi = lane < kGjThreads / 32 ? si[lane] : n;
      gj_warp_argmax(best, bi);
      const int j = lane & 15;
      double v = 0.0;
      if (best > 0ull && j < bw) {
        v = pan[(size_t)j * rpb + (bi - i0)];
        if (s >= 0 && j > jn) v = fma(-pan[(size_t)s * rpb + (bi - i0)], r[j], v);
      }
#pragma unroll
      for (int q = 0; q < kGjCluster; q += 2)
        cluster.map_shared_rank(&cand[jn & 1][me], q + (lane >> 4))->v[j] = v;
      if (lane < kGjCluster) {
        Cand* to = cluster.map_shared_rank(&cand[jn & 1][me], lane);
        to->key = best;
        to->row = bi;
      }
    }
    __syncthreads();  // the candidate's row has been read
    auto token = cluster.barrier_arrive();
    if (s >= 0) {
      for (int i = gi; i < rows; i += rp) {
        const bool isp = i0 + i == p;
        const double c = -pan[(size_t)s * rpb + i];
        for (int j = s + 2 + gg; j < bw; j += G) {
          const double v = pan[(size_t)j * rpb + i];
          pan[(size_t)j * rpb + i] = isp ? r[j] : fma(c, r[j], v);
        }
      }
    }
    cluster.barrier_wait(std::move(token));
    const Cand* cd = cand[jn & 1];
    // rows ascend with the blocks: the lowest block wins a tie
    unsigned long long key = lane < kGjCluster ? cd[lane].key : 0ull;
    int w = lane;
    gj_warp_argmax(key, w);
    p = cd[w].row;
    if (warp == 0) {
      const double ip = 1.0 / cd[w].v[jn];
      const double v = lane < B ? cd[w].v[lane] : 0.0;
      if (lane < B) s_r[jn & 1][lane] = v * ip;
      if (lane == jn) myip = ip;
      if (lane < jn) pn.l[jn][lane] = v * myip;
      if (lane == 0) {
        pn.ip[jn] = ip;
        pn.row[jn] = p;
        // a zero or NaN column: flagged, and the pivot stays a valid row
        if (me == 0 && key <= 2ull) atomicOr(err, 1);
      }
    }
    __syncthreads();
  }
  for (int i = tid; i < rows; i += kGjThreads) {
    if (i0 + i == p) own[i] = k0 + bw - 1;
    // multipliers: a pivot row of this panel starts from its r_s, so its steps up to s are 0
    const int ks = own[i] - k0;
    for (int t = 0; t < bw; ++t)
      oc[(size_t)t * n + i0 + i] = ks >= t ? 0.0 : pan[(size_t)t * rpb + i];
    step[i0 + i] = own[i];
  }
  if (me == 0) {
    double* dst = reinterpret_cast<double*>(opn);
    const double* src = reinterpret_cast<const double*>(&pn);
    for (int e = tid; e < (int)(sizeof(GjPanel) / 8); e += kGjThreads) dst[e] = src[e];
    if (tid < bw) prow[k0 + tid] = pn.row[tid];
  }
}

// dst = src after the steps of the panel at k0: a tile of cpb columns and rpt rows per block.
// seq > 0: launched beside the panel that stores seq to *ready (the inputs are not __restrict__:
// they must not be read through the non-coherent path or ahead of that).
__global__ void __launch_bounds__(kGjUpdThreads) gj_update_k(int n, int k0, int cpb, int rpt,
                                                             const GjPanel* gpn, const double* cc,
                                                             const int* step, const double* src,
                                                             double* __restrict__ dst, int seq,
                                                             const int* ready) {
  constexpr int B = kGjB;
  __shared__ GjPanel pn;
  __shared__ double rr[kGjUpdCols][B];
  const int tid = threadIdx.x, lane = tid & 31;
  const int bw = min(B, n - k0);
  const int c0 = blockIdx.x * cpb, nc = min(cpb, n - c0);
  const int r0 = blockIdx.y * rpt, r1 = min(n, r0 + rpt);
  if (seq > 0) {
    if (tid == 0) {
      int seen;
      asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(seen) : "l"(ready) : "memory");
      if (seen != seq) asm volatile("griddepcontrol.wait;" ::: "memory");
    }
    __syncthreads();
  }
  {
    const double* g = reinterpret_cast<const double*>(gpn);
    double* d = reinterpret_cast<double*>(&pn);
    for (int e = tid; e < (int)(sizeof(GjPanel) / 8); e += kGjUpdThreads) d[e] = g[e];
  }
  __syncthreads();
  if (2 * (tid >> 5) < nc) {
    // a panel column s0 starts after its own step: 1 / pivot in its pivot row, -c_s0(i) / pivot
    // elsewhere
    const int u = 2 * (tid >> 5) + (lane >> 4), t = lane & 15;
    const int j = c0 + u, s0 = j >= k0 && j < k0 + bw ? j - k0 : -1;
    double x = 0.0;
    if (u < nc && t < bw && t > s0)
      x = s0 < 0 ? src[(size_t)j * n + pn.row[t]] : -pn.l[t][s0];
    rr[u][t] = gj_forward(x, t, pn, s0, bw);
  }
  __syncthreads();
  for (int i = r0 + tid; i < r1; i += kGjUpdThreads) {
    const int ks = step[i] - k0;  // >= 0: a pivot row of this panel
    double c[B];
#pragma unroll
    for (int s = 0; s < B; ++s) c[s] = s < bw ? cc[(size_t)s * n + i] : 0.0;
    auto start = [&](int t) {
      const int j = c0 + t, s0 = j >= k0 && j < k0 + bw ? j - k0 : -1;
      if (ks > s0) return rr[t][ks];
      if (s0 < 0) return src[(size_t)j * n + i];
      return ks == s0 ? pn.ip[s0] : -cc[(size_t)s0 * n + i] * pn.ip[s0];
    };
    int t = 0;
    for (; t + 8 <= nc; t += 8) {
      double x[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) x[u] = start(t + u);
#pragma unroll
      for (int s = 0; s < B; ++s)
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = fma(-c[s], rr[t + u][s], x[u]);
#pragma unroll
      for (int u = 0; u < 8; ++u) dst[(size_t)(c0 + t + u) * n + i] = x[u];
    }
    for (; t < nc; ++t) {
      double x = start(t);
#pragma unroll
      for (int s = 0; s < B; ++s) x = fma(-c[s], rr[t][s], x);
      dst[(size_t)(c0 + t) * n + i] = x;
    }
  }
  // the grid ends after the panel beside it, so that the next launch follows both
  if (blockIdx.x == 0 && blockIdx.y == 0) pdl_wait();
}

// inverse(k, p_j) = w(p_k, j), stored by rows: a 32 x 32 tile read along the work's columns and
// written along the inverse's rows through shared memory (step, prow NULL: a plain transpose)
__global__ void __launch_bounds__(256) gj_gather_k(int n, const double* __restrict__ w,
                                                   const int* __restrict__ step,
                                                   const int* __restrict__ prow,
                                                   double* __restrict__ inv) {
  __shared__ double tile[32][33];
  const int i0 = blockIdx.x * 32, j0 = blockIdx.y * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int jj = ty; jj < 32; jj += 8) {
    const int j = j0 + jj, i = i0 + tx;
    if (j < n && i < n) tile[jj][tx] = w[(size_t)j * n + i];
  }
  __syncthreads();
  for (int ii = ty; ii < 32; ii += 8) {
    const int i = i0 + ii, j = j0 + tx;
    if (i < n && j < n)
      inv[(size_t)(step ? step[i] : i) * n + (prow ? prow[j] : j)] = tile[tx][ii];
  }
}

// x_i = sum_c inv(i, c) b_c, FP64 accumulation: one warp per row (the row is contiguous, so
// every load is coalesced), lane l summing the columns c = l mod 32, the lanes' partial sums
// added by a fixed butterfly
constexpr int kGemvWarps = 8;

template <class TV>
__global__ void __launch_bounds__(32 * kGemvWarps) coarse_apply_k(int n,
                                                                  const double* __restrict__ inv,
                                                                  const TV* __restrict__ b,
                                                                  TV* __restrict__ x) {
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const int i = blockIdx.x * kGemvWarps + (threadIdx.x >> 5);
  if (i >= n) return;  // whole warps leave together
  rows::gemv_row<TV>(i, n, lane, inv, b, x);
}

// --- Gauss-Seidel (one CTA) ---------------------------------------------------------
constexpr int kGsThreads = 1024;
constexpr int kGsMaxColours = 256;

__device__ __forceinline__ uint32_t fmix32_gs(uint32_t h) {  // MurmurHash3 finaliser
  h ^= h >> 16;
  h *= 0x85ebca6bu;
  h ^= h >> 13;
  h *= 0xc2b2ae35u;
  h ^= h >> 16;
  return h;
}

__device__ __forceinline__ unsigned long long gs_key(const unsigned* ids, int v) {
  const uint32_t id = ids ? ids[v] : (uint32_t)v;
  return ((unsigned long long)fmix32_gs(id ^ 0x2545F491u) << 32) | id;
}

// Colouring by synchronous rounds, then a stable sort of the rows by colour (order, coff).
// pick: n bytes of scratch.  err: set when more than kGsMaxColours colours are needed.
__global__ void __launch_bounds__(kGsThreads) gs_colour_k(int n, const int* __restrict__ rowptr,
                                                          const int* __restrict__ col,
                                                          const unsigned* __restrict__ ids,
                                                          int* __restrict__ colour,
                                                          unsigned char* __restrict__ pick,
                                                          int* __restrict__ order,
                                                          int* __restrict__ coff,
                                                          int* __restrict__ ncol_out) {
  __shared__ int left, wcount[kGsThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int i = tid; i < n; i += blockDim.x) colour[i] = -1;
  if (tid == 0) left = n;
  __syncthreads();
  int c = 0;
  while (left > 0 && c < kGsMaxColours) {
    for (int i = tid; i < n; i += blockDim.x) {
      unsigned char pk = 0;
      if (colour[i] < 0) {
        const unsigned long long ki = gs_key(ids, i);
        pk = 1;
        for (int p = rowptr[i]; p < rowptr[i + 1]; ++p) {
          const int j = col[p];
          if (j != i && colour[j] < 0 && gs_key(ids, j) > ki) pk = 0;
        }
      }
      pick[i] = pk;
    }
    __syncthreads();
    int got = 0;
    for (int i = tid; i < n; i += blockDim.x)
      if (pick[i]) {
        colour[i] = c;
        ++got;
      }
    got = __reduce_add_sync(0xffffffffu, got);
    if (lane == 0 && got) atomicSub(&left, got);
    ++c;
    __syncthreads();
  }
  const int ncol = left > 0 ? -1 : c;
  if (tid == 0) *ncol_out = ncol;
  if (ncol < 0) return;
  // stable partition by colour: for each colour, rows in ascending order
  int base = 0;
  for (int cc = 0; cc < ncol; ++cc) {
    if (tid == 0) coff[cc] = base;
    for (int b0 = 0; b0 < n; b0 += blockDim.x) {
      const int i = b0 + tid;
      const bool f = i < n && colour[i] == cc;
      const unsigned bal = __ballot_sync(0xffffffffu, f);
      if (lane == 0) wcount[warp] = __popc(bal);
      __syncthreads();
      int before = 0, total = 0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
        before += w < warp ? wcount[w] : 0;
        total += wcount[w];
      }
      if (f) order[base + before + __popc(bal & ((1u << lane) - 1u))] = i;
      base += total;
      __syncthreads();
    }
  }
  if (tid == 0) coff[ncol] = base;
}

// `steps` symmetric sweeps from x = 0; x and b in shared memory (FP64); warp per row,
// lanes over the row's entries, shuffle reduction in a fixed order.
template <class TV>
__global__ void __launch_bounds__(kGsThreads) gs_apply_k(int n, const int* __restrict__ rowptr,
                                                         const int* __restrict__ col,
                                                         const double* __restrict__ val,
                                                         const double* __restrict__ invd,
                                                         const int* __restrict__ order,
                                                         const int* __restrict__ coff, int ncol,
                                                         int steps, const TV* __restrict__ b,
                                                         TV* __restrict__ x) {
  extern __shared__ double gs_sm[];
  double* xs = gs_sm;
  double* bs = gs_sm + n;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = blockDim.x >> 5;
  for (int i = tid; i < n; i += blockDim.x) {
    xs[i] = 0.0;
    bs[i] = (double)b[i];
  }
  __syncthreads();
  for (int st = 0; st < steps; ++st)
    for (int half = 0; half < 2; ++half)
      for (int cc = 0; cc < ncol; ++cc) {
        const int c = half == 0 ? cc : ncol - 1 - cc;
        for (int k = coff[c] + warp; k < coff[c + 1]; k += nwarp) {
          const int i = order[k];
          double acc = 0.0;
          for (int p = rowptr[i] + lane; p < rowptr[i + 1]; p += 32) {
            const int j = col[p];
            if (j != i) acc += val[p] * xs[j];
          }
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
          if (lane == 0) xs[i] = (bs[i] - acc) * invd[i];
        }
        __syncthreads();
      }
  for (int i = tid; i < n; i += blockDim.x) x[i] = (TV)xs[i];
}

}  // namespace

void coarse_gs_setup(const DevCsr& A, const double* invd, const unsigned* ids, int steps,
                     CoarseSolver& cs, cudaStream_t s) {
  const int n = A.n;
  if (n > kCoarseGsMax) fail(SAAMG_UNIMPLEMENTED, "Gauss-Seidel coarse level above 12288 rows");
  cs.kind = SAAMG_COARSE_GS;
  cs.n = n;
  cs.steps = steps;
  cs.rowptr = A.rowptr.p;
  cs.col = A.col.p;
  cs.val = A.val.p;
  cs.invd = invd;
  // shared-memory opt-in for the largest coarse level (set outside any stream capture)
  const int smax = (int)(2 * kCoarseGsMax * sizeof(double));
  SAAMG_CUDA(cudaFuncSetAttribute(gs_apply_k<double>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  smax));
  SAAMG_CUDA(cudaFuncSetAttribute(gs_apply_k<float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  smax));
  cs.colour.alloc(n, s);
  cs.order.alloc(n, s);
  cs.coff.alloc(kGsMaxColours + 1, s);
  if (n == 0) return;
  Buf<unsigned char> pick;
  Buf<int> ncol;
  pick.alloc(n, s);
  ncol.alloc(1, s);
  gs_colour_k<<<1, kGsThreads, 0, s>>>(n, A.rowptr.p, A.col.p, ids, cs.colour.p, pick.p,
                                       cs.order.p, cs.coff.p, ncol.p);
  SAAMG_LAUNCH();
  int h = 0;
  d2h_sync(&h, ncol.p, sizeof(int), s);
  if (h <= 0) fail(SAAMG_NUMERICAL, "coarse-level colouring needs more than 256 colours");
  cs.ncolours = h;
}

// A^-1 by Gauss-Jordan elimination of the column-major n x n work array w (overwritten),
// written by rows to inv; synchronises to read the zero-pivot flag
static void gauss_jordan_inverse(int n, const Buf<double>& w, double* inv, cudaStream_t s) {
  constexpr int B = kGjB;
  // one array for everything: panels, multipliers, the second matrix, then the integers (an array
  // for each took a call at n <= 3 from 49 to 55 us)
  constexpr size_t kPanel = sizeof(GjPanel) / sizeof(double);
  static_assert(sizeof(GjPanel) == kPanel * sizeof(double), "panels lie among doubles");
  const size_t nn = (size_t)n * n, nb = (size_t)B * n;
  Buf<double> work;
  work.alloc(2 * (kPanel + nb) + nn + (3 * (size_t)n + 3) / 2, s);
  GjPanel* const pn[2] = {reinterpret_cast<GjPanel*>(work.p),
                          reinterpret_cast<GjPanel*>(work.p + kPanel)};
  double* const c[2] = {work.p + 2 * kPanel, work.p + 2 * kPanel + nb};
  double *src = w.p, *dst = work.p + 2 * (kPanel + nb);
  int* const err = reinterpret_cast<int*>(dst + nn);  // zero pivot, last panel that has begun
  int* const prow = err + 2;
  int* const step[2] = {prow + n, prow + 2 * (size_t)n};
  SAAMG_CUDA(cudaMemsetAsync(err, 0, 2 * sizeof(int), s));
  const int rpb = (n + kGjCluster - 1) / kGjCluster;
  SAAMG_CUDA(cudaFuncSetAttribute(gj_panel_k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)kGjPanelSmem));
  SAAMG_CUDA(cudaFuncSetAttribute(gj_panel_k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  // tile of the update: the fewest clocks of the busiest SM beside the panel's, a tile costing its
  // multiply-adds (two a clock) and about 6000 clocks of start-up and forward substitution
  const int nsm = std::max(1, sm_count() - kGjCluster);
  int cpb = 1, rt = 1;
  double least = -1.0;
  for (int r = 1; r <= 16; ++r)
    for (int k = 1; k <= kGjUpdCols; ++k) {
      const long long tiles = (long long)((n + k - 1) / k) * r;
      const double rows = (double)((n + r - 1) / r);
      const double cost = (double)((tiles + nsm - 1) / nsm) * (k * rows * B / 2.0 + 6000.0);
      if (least < 0.0 || cost < least) {
        least = cost;
        cpb = k;
        rt = r;
      }
    }
  const int rpt = (n + rt - 1) / rt;
  const dim3 ugrid((n + cpb - 1) / cpb, rt);
  // panel q reads the matrix before update q - 1 and the panel q - 1; update q the same matrix as
  // panel q + 1, and the panel q.  Panel q waits at its entry for the launch before it, update
  // q - 2, which ends after panel q - 1 beside it: everything before has finished.  Update q starts
  // once panel q + 1 has passed that wait, so update q - 1 and panel q have finished, and takes their
  // writes from panel q + 1 through err[1].
  const int panels = (n + B - 1) / B;
  auto panel = [&](int q) {
    const int pq = (q & 1) ^ 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = kGjCluster;
    cfg.blockDim = kGjThreads;
    cfg.dynamicSmemBytes = kGjPanelSmem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kGjCluster;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = pdl_enabled() ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    SAAMG_CUDA(cudaLaunchKernelEx(&cfg, gj_panel_k, n, q * B, rpb, (const double*)src,
                                  q > 0 ? B : 0, (const GjPanel*)pn[pq], (const double*)c[pq],
                                  pn[q & 1], c[q & 1], (const int*)(q > 0 ? step[pq] : nullptr),
                                  step[q & 1], prow, err, q, err + 1));
    SAAMG_LAUNCH();
  };
  panel(0);
  for (int q = 0; q < panels; ++q) {
    const bool beside = q + 1 < panels;
    if (beside) panel(q + 1);
    auto args = [&](auto&& launch) {
      launch(n, q * B, cpb, rpt, (const GjPanel*)pn[q & 1], (const double*)c[q & 1],
             (const int*)step[q & 1], (const double*)src, dst, beside ? q + 1 : 0,
             (const int*)(err + 1));
    };
    args([&](auto... a) {
      if (beside) launch_pdl(gj_update_k, ugrid, kGjUpdThreads, kGjUpdSmem, s, a...);
      else gj_update_k<<<ugrid, kGjUpdThreads, kGjUpdSmem, s>>>(a...);
    });
    SAAMG_LAUNCH();
    std::swap(src, dst);
  }
  const dim3 tiles((n + 31) / 32, (n + 31) / 32);
  gj_gather_k<<<tiles, 256, 0, s>>>(n, src, step[(panels - 1) & 1], prow, inv);
  SAAMG_LAUNCH();
  int herr = 0;
  d2h_sync(&herr, err, sizeof(int), s);
  if (herr) fail(SAAMG_NUMERICAL, "zero pivot in the coarse factorisation");
}

void coarse_factor(const DevCsr& A, CoarseSolver& cs, cudaStream_t s) {
  const int n = A.n;
  cs.n = n;
  cs.inv.alloc((size_t)n * n, s);
  if (n == 0) return;
  Buf<double> w;
  w.alloc((size_t)n * n, s);
  SAAMG_CUDA(cudaMemsetAsync(w.p, 0, sizeof(double) * (size_t)n * n, s));
  densify_k<<<(n + 255) / 256, 256, 0, s>>>(n, A.rowptr.p, A.col.p, A.val.p, w.p);
  SAAMG_LAUNCH();
  gauss_jordan_inverse(n, w, cs.inv.p, s);
}

void dense_inverse(int n, const double* a, double* inv, cudaStream_t s) {
  if (n == 0) return;
  Buf<double> w;
  w.alloc((size_t)n * n, s);
  const dim3 tiles((n + 31) / 32, (n + 31) / 32);
  gj_gather_k<<<tiles, 256, 0, s>>>(n, a, nullptr, nullptr, w.p);  // rows of a -> columns of w
  SAAMG_LAUNCH();
  gauss_jordan_inverse(n, w, inv, s);
}

template <class TV>
void coarse_apply(const CoarseSolver& cs, const TV* b, TV* x, cudaStream_t s) {
  if (cs.n == 0) return;
  if (cs.kind == SAAMG_COARSE_GS) {
    const size_t sm = 2 * (size_t)cs.n * sizeof(double);
    gs_apply_k<TV><<<1, kGsThreads, sm, s>>>(cs.n, cs.rowptr, cs.col, cs.val, cs.invd,
                                             cs.order.p, cs.coff.p, cs.ncolours, cs.steps, b, x);
    SAAMG_LAUNCH();
    return;
  }
  launch_pdl(coarse_apply_k<TV>, (cs.n + kGemvWarps - 1) / kGemvWarps, 32 * kGemvWarps, 0, s,
             cs.n, cs.inv.p, b, x);
  SAAMG_LAUNCH();
}

template void coarse_apply<double>(const CoarseSolver&, const double*, double*, cudaStream_t);
template void coarse_apply<float>(const CoarseSolver&, const float*, float*, cudaStream_t);

}  // namespace saamg
