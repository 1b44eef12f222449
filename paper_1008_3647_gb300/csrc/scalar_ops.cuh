// Krylov scalar updates on the device (one thread) and the block reductions that feed them; used
// by the single-CTA scalar kernels and, in batched solves, by the last CTA of a producing kernel
// (last_block_update), which then needs no separate launch.
#pragma once
#include <cuda_runtime.h>

#include "blas.cuh"

namespace ufg {

constexpr int SCAL_NT = 256;  // threads of every CTA that runs these reductions

// Sums of a and b over the warp with one addition per step after the first: lanes 0-15 go on with
// a, lanes 16-31 with b (the pairing of the xor butterfly, so the sums keep their bits; an FP64
// warp instruction takes 16 cycles of the SM's pipe).  a in lane 0, b in lane 16.
static __device__ __forceinline__ double warp_sum2(double a, double b) {
  const bool hi = (threadIdx.x & 16) != 0;
  double v = hi ? b : a;
  v += __shfl_xor_sync(0xffffffffu, hi ? a : b, 16);
#pragma unroll
  for (int off = 8; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

static __device__ __forceinline__ bool bad(double v) { return !isfinite(v); }

// The four sums (pairs [i0, i1) of part, pairs [j0, j1) of part2) in one sweep: each thread adds
// its strided share, the warps fold with shuffles and thread 0 adds the warp results in order
// (a fixed, launch-independent order: the result is deterministic).  Valid in thread 0.
// NT: threads of the calling CTA (SCAL_NT unless a kernel says otherwise).
template <int NT = SCAL_NT>
static __device__ void block_sums4(const double* part, int i0, int i1, const double* part2, int j0,
                            int j1, double (&out)[4]) {
  __shared__ double red[NT / 32][4];
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  if (part != nullptr)
    for (int i = i0 + (int)threadIdx.x; i < i1; i += NT) {
      s[0] += part[2 * i];
      s[1] += part[2 * i + 1];
    }
  if (part2 != nullptr)
    for (int i = j0 + (int)threadIdx.x; i < j1; i += NT) {
      s[2] += part2[2 * i];
      s[3] += part2[2 * i + 1];
    }
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s[k] += __shfl_xor_sync(0xffffffffu, s[k], off);
  if ((threadIdx.x & 31) == 0)
#pragma unroll
    for (int k = 0; k < 4; ++k) red[threadIdx.x >> 5][k] = s[k];
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      double t = 0.0;
      for (int w = 0; w < NT / 32; ++w) t += red[w][k];
      out[k] = t;
    }
  }
}

static __device__ __forceinline__ void bi_rho(DevScalars* sc, double rho, double rr) {
  if (fabs(rho) <= sc->restart_cos * sqrt(sc->rhatn2 * rr)) {
    sc->done = 2;  // near-breakdown: the host restarts from the true residual
    return;
  }
  sc->iters += 1;
  sc->rho = rho;
  sc->beta = (rho / sc->rho_old) * (sc->alpha / sc->omega);
  if (bad(sc->beta)) sc->done = 4;
}

// |v| against a bound from v.v: no square root on the one thread's chain (FP64 divisions and roots
// take hundreds of cycles here)
static __device__ __forceinline__ bool within(double vv, double bound) { return vv <= bound * bound; }
static __device__ __forceinline__ bool diverged(const DevScalars* sc, double vv) {
  if (!(sc->div_limit > 0)) return false;
  const double lim = sc->div_limit * sc->bn;
  return vv > lim * lim;
}

static __device__ __forceinline__ void bi_rcheck(DevScalars* sc, double rr, double tb) {
  sc->rr = rr;
  sc->rho_old = sc->rho;
  if (bad(rr)) sc->done = 4;
  else if (within(rr, tb)) sc->done = 1;
  else if (diverged(sc, rr)) sc->done = 6;
  else if (sc->omega == 0.0) sc->done = 2;
  else if (sc->iters >= sc->maxit) sc->done = 5;
}

// One thread.  The scalars are read at once, updated in registers and written back at once (read
// where needed, each field was a dependent load from L2).
static __device__ __noinline__ void scalar_update(int op, DevScalars* gsc, const double* part, double a0, double a1,
                              const double* part2, double b0, double b1) {
  DevScalars local = *gsc;
  DevScalars* const sc = &local;
  if ((op == OP_CG_INIT || op == OP_BI_INIT_RHO) && part2 != nullptr)
    sc->bn = sqrt(b1);  // rhs.rhs
  const double tb = sc->tol * sc->bn;
  switch (op) {
    case OP_CG_INIT:  // part = (r.z, r.r), part2 = (-, rhs.rhs)
      sc->rz = a0;
      sc->rr = a1;
      sc->done = 0;
      if (bad(a0) || bad(a1)) sc->done = 4;
      else if (within(a1, tb)) sc->done = 1;
      break;
    case OP_CG_ALPHA:  // part = slice partials (p.q, -)
      sc->pq = a0;
      sc->alpha = sc->rz / a0;
      if (bad(sc->alpha)) sc->done = 4;
      break;
    case OP_CG_CHECK_BETA:
    case OP_CG_CHECK:  // part = (-, r.r)
      sc->iters += 1;
      sc->rr = a1;
      if (bad(a1)) sc->done = 4;
      else if (within(a1, tb)) sc->done = 1;
      else if (diverged(sc, a1)) sc->done = 6;
      else if (sc->iters >= sc->maxit) sc->done = 5;
      if (op == OP_CG_CHECK_BETA && sc->done == 0) {
        sc->beta = a1 / sc->rz;
        sc->rz = a1;
        if (bad(sc->beta)) sc->done = 4;
      }
      break;
    case OP_CG_BETA:  // part = (r.z, -)
      sc->beta = a0 / sc->rz;
      sc->rz = a0;
      if (bad(sc->beta)) sc->done = 4;
      break;
    case OP_BI_INIT_RHO:  // part = (rhat.r, r.r), part2 = (rhat.rhat, rhs.rhs); the first
                          // iteration's rho from the same partials
      sc->rho = a0;
      sc->rr = a1;
      sc->rhatn2 = b0;
      sc->rho_old = 1.0;
      sc->alpha = 1.0;
      sc->omega = 1.0;
      sc->done = 0;
      if (bad(a0) || bad(a1)) sc->done = 4;
      else if (within(a1, tb)) sc->done = 1;
      else bi_rho(sc, a0, a1);
      break;
    case OP_BI_RHO_REDO:  // part = (rhat.r, r.r) of the replaced residual
      sc->rr = a1;
      if (fabs(a0) <= sc->restart_cos * sqrt(sc->rhatn2 * a1)) {
        sc->done = 2;
        break;
      }
      sc->rho = a0;
      sc->beta = (a0 / sc->rho_old) * (sc->alpha / sc->omega);
      sc->done = bad(sc->beta) ? 4 : 0;
      break;
    case OP_BI_ALPHA:  // part = slice partials (v.rhat, -)
      sc->alpha = sc->rho / a0;
      if (bad(sc->alpha)) sc->done = 4;
      break;
    case OP_BI_SCHECK:  // part = (-, s.s)
      sc->ss = a1;
      if (bad(a1)) sc->done = 4;
      else if (within(a1, tb)) sc->done = 1;
      else if (diverged(sc, a1)) sc->done = 6;
      break;
    case OP_BI_OMEGA:  // part = slice partials (t.s, t.t)
      sc->omega = a1 > 0.0 ? a0 / a1 : 0.0;
      if (bad(sc->omega)) sc->done = 4;
      break;
    case OP_NORM2:  // part = (-, v.v)
      sc->rr = a1;
      break;
    case OP_BI_RCHECK_RHO:  // part = (rhat.r, r.r): the iteration's check, then (still
                            // running) the next one's rho
      bi_rcheck(sc, a1, tb);
      if (sc->done == 0) bi_rho(sc, a0, a1);
      break;
  }
  *gsc = local;
}

// Called by every thread of a CTA of a producer whose thread 0 has just written the CTA's
// partial pair into `part`: the CTA that completes a problem's set [i0, i1) (counted on
// `counter`, left at 0 for the next producer) sums the set in fixed order and applies `op` to
// that problem's scalars.  Partials reach the summing CTA through thread 0's fence before its
// count (only thread 0 wrote them, so only it fences).
// NT: threads of the CTA, 0 where they are not known at compile time (whole warps, at most 1024).
template <int NT = SCAL_NT>
static __device__ __forceinline__ void last_block_update(int op, DevScalars* sc, const double* part,
                                                        int i0, int i1, unsigned* counter) {
  const int nt = NT > 0 ? NT : (int)blockDim.x;
  __shared__ int is_last;
  if (threadIdx.x == 0) {
    __threadfence();
    is_last = atomicAdd(counter, 1u) == (unsigned)(i1 - i0 - 1);
  }
  __syncthreads();
  if (!is_last) return;
  __threadfence();
  __shared__ double red[NT > 0 ? NT / 32 : 32][2];
  double s0 = 0.0, s1 = 0.0;
  for (int i = i0 + (int)threadIdx.x; i < i1; i += nt) {
    s0 += part[2 * i];
    s1 += part[2 * i + 1];
  }
  const double v = warp_sum2(s0, s1);
  if ((threadIdx.x & 15) == 0) red[threadIdx.x >> 5][(threadIdx.x >> 4) & 1] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    s0 = s1 = 0.0;
    for (int w = 0; w < nt / 32; ++w) {
      s0 += red[w][0];
      s1 += red[w][1];
    }
    scalar_update(op, sc, part, s0, s1, nullptr, 0.0, 0.0);
    *counter = 0u;
  }
}

}  // namespace ufg
