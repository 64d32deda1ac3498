// Conjugate-gradient recursion (Sec. 3.1) on the scaled system: fused axpy + norm,
// direction update, dot products.  Every reduction writes one partial per block of a
// fixed grid and one block adds the partials in index order, so a run is
// reproducible bit for bit.  The CG scalars stay on the device.
#include <algorithm>

#include "pcg.cuh"
#include "rows.cuh"

namespace saamg {

namespace {

using rows::sum_fixed;

// Blocks of the vector reductions of n elements: those of the fixed grid that hold any (the
// partials of the others are 0; a short vector has few, and each costs a fence and an atomic).
inline int red_blocks(int n) {
  return std::max(1, std::min(kRedBlocks, (n + kRedThreads - 1) / kRedThreads));
}

// Loads of four grid strides are issued before their (in-order) multiply-adds: the sum is
// the same sequence of operations as the plain strided loop, with more bytes in flight.
template <class TA, class TB>
__global__ void __launch_bounds__(kRedThreads) dot_k(int n, const TA* __restrict__ a,
                                                        const TB* __restrict__ b,
                                                        double* __restrict__ part) {
  pdl_wait();
  const double t = rows::dot_block<TA, TB>(blockIdx.x, n, a, b);
  if (threadIdx.x == 0) part[blockIdx.x] = t;
}

// r'z (and z'q in the same sweep) and, in the last block, beta
template <class TZ, bool PR>
__global__ void __launch_bounds__(kRedThreads) beta_k(int n, const double* __restrict__ r,
                                                         const TZ* __restrict__ z,
                                                         const double* __restrict__ q,
                                                         double* part_rz, double* part_zq,
                                                         PcgCtl* ctl) {
  pdl_wait();
  double t1, t2 = 0.0;
  if (PR) rows::dot2_block<TZ>(blockIdx.x, n, r, z, q, t1, t2);
  else t1 = rows::dot_block<double, TZ>(blockIdx.x, n, r, z);
  if (threadIdx.x == 0) {
    part_rz[blockIdx.x] = t1;
    if (PR) part_zq[blockIdx.x] = t2;
  }
  if (!last_block(&ctl->tick[0])) return;
  const BetaIn in(ctl);
  const double rz = sum_fixed(part_rz, gridDim.x);
  const double zq = PR ? sum_fixed(part_zq, gridDim.x) : 0.0;
  if (threadIdx.x == 0) finish_beta(ctl, rz, zq, PR ? 1 : 0, in);
}

// r32 (mixed precision): the FP32 copy of the new residual, the next V-cycle's input
__global__ void __launch_bounds__(kRedThreads) update_k(int n, double* __restrict__ x,
                                                           double* __restrict__ r,
                                                           const double* __restrict__ p,
                                                           const double* __restrict__ q,
                                                           PcgCtl* ctl, double* part,
                                                           float* __restrict__ r32,
                                                           cudaGraphConditionalHandle cond,
                                                           int has_cond, int maxit) {
  pdl_wait();
  const double t = rows::update_block(blockIdx.x, n, ctl->alpha, x, r, p, q, r32);
  if (threadIdx.x == 0) part[blockIdx.x] = t;
  if (!last_block(&ctl->tick[2])) return;
  const double rr = sum_fixed(part, gridDim.x);
  if (threadIdx.x == 0) {
    const bool go = finish_check(ctl, rr, maxit);
    if (has_cond) cudaGraphSetConditional(cond, go ? 1u : 0u);
  }
}

template <class TZ>
__global__ void direction_k(int n, const TZ* __restrict__ z, double* __restrict__ p,
                            const PcgCtl* __restrict__ ctl) {
  pdl_wait();
  const double b = ctl->beta;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    p[i] = rows::widen(z[i]) + b * p[i];
}

__global__ void init_k(const double* __restrict__ part_bb, const double* __restrict__ part_rr,
                       int count, PcgCtl* ctl, cudaGraphConditionalHandle cond, int has_cond,
                       int maxit) {
  pdl_wait();
  const double bb = sum_fixed(part_bb, count);
  const double rr = sum_fixed(part_rr, count);
  if (threadIdx.x == 0) {
    const bool go = finish_init(ctl, bb, rr, maxit);
    if (has_cond) cudaGraphSetConditional(cond, go ? 1u : 0u);
  }
}

__global__ void zero_if_rhs_zero_k(double* __restrict__ x, int n, const PcgCtl* __restrict__ ctl) {
  pdl_wait();
  if (ctl->bb != 0.0) return;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) x[i] = 0.0;
}

__global__ void store_true_k(const double* __restrict__ part, int count, PcgCtl* ctl) {
  pdl_wait();
  const double rr = sum_fixed(part, count);
  if (threadIdx.x == 0) ctl->rr_true = rr;
}

inline int vec_blocks(int n) {
  int b = (n + 255) / 256;
  return b < sm_count() * 8 ? (b > 0 ? b : 1) : sm_count() * 8;
}

}  // namespace

template <class TA, class TB>
void dot_partials(int n, const TA* a, const TB* b, double* partials, cudaStream_t s) {
  launch_pdl(dot_k<TA, TB>, red_blocks(n), kRedThreads, 0, s, n, a, b, partials);
  SAAMG_LAUNCH();
}
template void dot_partials<double, double>(int, const double*, const double*, double*, cudaStream_t);

template <class TZ>
void pcg_beta(int n, const double* r, const TZ* z, const double* q, double* part_rz,
              double* part_zq, int rule, PcgCtl* ctl, cudaStream_t s) {
  if (rule == 1)
    launch_pdl(beta_k<TZ, true>, red_blocks(n), kRedThreads, 0, s, n, r, z, q, part_rz, part_zq,
               ctl);
  else
    launch_pdl(beta_k<TZ, false>, red_blocks(n), kRedThreads, 0, s, n, r, z, q, part_rz, part_zq,
               ctl);
  SAAMG_LAUNCH();
}
template void pcg_beta<double>(int, const double*, const double*, const double*, double*, double*,
                               int, PcgCtl*, cudaStream_t);
template void pcg_beta<float>(int, const double*, const float*, const double*, double*, double*,
                              int, PcgCtl*, cudaStream_t);

template <class TZ>
void pcg_direction(int n, const TZ* z, double* p, const PcgCtl* ctl, cudaStream_t s) {
  launch_pdl(direction_k<TZ>, vec_blocks(n), 256, 0, s, n, z, p, ctl);
  SAAMG_LAUNCH();
}
template void pcg_direction<double>(int, const double*, double*, const PcgCtl*, cudaStream_t);
template void pcg_direction<float>(int, const float*, double*, const PcgCtl*, cudaStream_t);

void pcg_update(int n, double* x, double* r, const double* p, const double* q, PcgCtl* ctl,
                double* partials, float* r32, const cudaGraphConditionalHandle* cond, int maxit,
                cudaStream_t s) {
  launch_pdl(update_k, red_blocks(n), kRedThreads, 0, s, n, x, r, p, q, ctl, partials, r32,
             cond ? *cond : cudaGraphConditionalHandle{}, cond ? 1 : 0, maxit);
  SAAMG_LAUNCH();
}

void pcg_init(const double* part_bb, const double* part_rr, PcgCtl* ctl,
              const cudaGraphConditionalHandle* cond, int maxit, double* x, int n, cudaStream_t s) {
  launch_pdl(init_k, 1, kRedThreads, 0, s, part_bb, part_rr, red_blocks(n), ctl,
             cond ? *cond : cudaGraphConditionalHandle{}, cond ? 1 : 0, maxit);
  SAAMG_LAUNCH();
  launch_pdl(zero_if_rhs_zero_k, vec_blocks(n), 256, 0, s, x, n, ctl);
  SAAMG_LAUNCH();
}

void pcg_store_true(const double* partials, int n, PcgCtl* ctl, cudaStream_t s) {
  launch_pdl(store_true_k, 1, kRedThreads, 0, s, partials, red_blocks(n), ctl);
  SAAMG_LAUNCH();
}

}  // namespace saamg
