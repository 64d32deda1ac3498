// Conjugate-gradient vector kernels (internal).
#pragma once

#include "common.cuh"

namespace saamg {

// Scalars of the CG recursion, kept on the device between kernels.
struct PcgCtl {
  double rtol;    // stopping tolerance (device-loop solves read it here)
  double bb;      // ||b||^2
  double rr_true; // ||b - A x||^2 at exit
  double rz;      // r'z of the current direction
  double alpha;
  double beta;
  double pq;
  double rr;      // ||r||^2 after the last update
  double rz_new;
  double zq;
  double tol2;    // (rtol ||b||)^2
  int iters;
  int converged;
  int breakdown;
  unsigned tick[3];  // blocks of r'z, A p and the update that have stored their partials
};

// --- CG scalars, on the device -------------------------------------------------------------
// alpha = rz / pq (breakdown flag on 0/NaN); rz: ctl->rz
__device__ __forceinline__ void finish_alpha(PcgCtl* ctl, double pq, double rz) {
  ctl->pq = pq;
  double a = rz / pq;
  if (!(pq != 0.0) || !isfinite(a)) {
    ctl->breakdown = 1;
    a = 0.0;
  }
  ctl->alpha = a;
}
// beta: 0 on the first pass (p = z), else rz_new / rz (rule 0) or -alpha zq / rz (rule 1)
struct BetaIn {  // read before the sums
  int iters;
  double alpha, rz;
  __device__ __forceinline__ explicit BetaIn(const PcgCtl* c)
      : iters(c->iters), alpha(c->alpha), rz(c->rz) {}
};
__device__ __forceinline__ void finish_beta(PcgCtl* ctl, double rz, double zq, int rule,
                                            const BetaIn& in) {
  double b = 0.0;
  if (in.iters > 0) b = (rule == 1) ? (-in.alpha * zq) / in.rz : rz / in.rz;
  if (!isfinite(b) || !isfinite(rz)) {
    ctl->breakdown = 1;
    b = 0.0;
  }
  ctl->rz_new = rz;
  ctl->zq = zq;
  ctl->beta = b;
  ctl->rz = rz;
}
// end of a pass: rr, iters, converged; whether the loop goes on
__device__ __forceinline__ bool finish_check(PcgCtl* ctl, double rr, int maxit) {
  ctl->rr = rr;
  ctl->iters += 1;
  if (!isfinite(rr)) ctl->breakdown = 1;
  ctl->converged = rr <= ctl->tol2;
  return !ctl->converged && !ctl->breakdown && ctl->iters < maxit;
}
// The scalars from ||b||^2 and the first ||r||^2; whether the loop runs at all
__device__ __forceinline__ bool finish_init(PcgCtl* ctl, double bb, double rr, int maxit) {
  ctl->bb = bb;
  ctl->rr = rr;
  ctl->tol2 = (ctl->rtol * ctl->rtol) * bb;
  ctl->iters = 0;
  ctl->breakdown = !(isfinite(bb) && isfinite(rr));
  ctl->converged = (bb == 0.0) || rr <= ctl->tol2;
  ctl->rz = 0.0;
  ctl->alpha = 0.0;
  ctl->beta = 0.0;
  for (int k = 0; k < 3; ++k) ctl->tick[k] = 0;
  return !ctl->converged && !ctl->breakdown && maxit > 0;
}

// True in every thread of the launch's last block to get here, after thread 0 of every block has
// stored its partial: that block adds the partials (in index order, so which block it is does
// not matter) and forms the scalar that the next launch reads.  A launch of one block for each
// scalar cost three of a pass's launches, 3 to 5 us each.  *tick is left 0.
__device__ __forceinline__ bool last_block(unsigned* tick) {
  __shared__ int last;
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(tick, 1u) == gridDim.x - 1;
    if (last) {
      *tick = 0;
      __threadfence();
    }
  }
  __syncthreads();
  return last != 0;
}

// partials[blockIdx] of sum a_i b_i (fixed grid kRedBlocks, of which the blocks with elements run)
template <class TA, class TB>
void dot_partials(int n, const TA* a, const TB* b, double* partials, cudaStream_t s);

// A pass of the loop, in order: r'z (and z'q for rule 1, in one sweep) and beta; p = z + beta p;
// A p with p'q and alpha (stencil_apply with ctl); x += alpha p, r -= alpha q, r32 (if not
// null) = FP32 copy of r, r'r and the convergence test.  cond (if given): the loop condition of the
// graph, cleared when the loop ends.
template <class TZ>
void pcg_beta(int n, const double* r, const TZ* z, const double* q, double* part_rz,
              double* part_zq, int rule, PcgCtl* ctl, cudaStream_t s);
template <class TZ>
void pcg_direction(int n, const TZ* z, double* p, const PcgCtl* ctl, cudaStream_t s);
void pcg_update(int n, double* x, double* r, const double* p, const double* q, PcgCtl* ctl,
                double* partials, float* r32, const cudaGraphConditionalHandle* cond, int maxit,
                cudaStream_t s);

// prologue: ctl from ||b||^2 and ||r||^2 (partials) and the rtol in ctl; the loop condition; x is
// zeroed when b = 0
void pcg_init(const double* part_bb, const double* part_rr, PcgCtl* ctl,
              const cudaGraphConditionalHandle* cond, int maxit, double* x, int n, cudaStream_t s);
// ctl->rr_true = sum of the partials of n elements
void pcg_store_true(const double* partials, int n, PcgCtl* ctl, cudaStream_t s);

}  // namespace saamg
