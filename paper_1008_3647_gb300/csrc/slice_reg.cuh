// FP32 fused momentum-space kernels (FAM_M1W, see slice_tma.cuh for the operators) for the
// lattice extents below 16, on the plan of the FP64 ones (slice_fix.cuh): a warp owns PW
// whole z-planes, lanes = (plane, x); the first line of each thread comes straight from global
// memory and the last goes straight back, both with consecutive x.
//
//   y, x (inverse)   within the warp's planes of shared memory, no CTA barrier
//   z                column (y, x): inverse pass, site multiplier and forward pass in registers
//   x, y (forward)   within the warp's planes again, epilogue from registers
//
// Two CTA barriers and four exchanges for six passes (the TMA-staged kernel: six and five, plus
// the staging), no copies to wait for.  Rows are padded to N + 1 words.  Latency-bound: a batch's
// extent has a few hundred CTAs.  With these kernels the batched and single solves of every
// extent below 32 iterate in the momentum basis; before, at N_x = 4 .. 12, each preconditioner
// application took seven transforms instead of two of these kernels: 96-problem mixed batch 60 ->
// 39 ms.  At N = 16 the TMA-staged kernel stays: M1 term 27.8 against 28.5-29.4 us, full
// operator with dot 45 against 50 us (8 x 16^3 x 256).
#pragma once
#include <cuda_runtime.h>

#include <cstring>

#include "slice_fix.cuh"

namespace ufg {

template <int N>
struct RegM1wArgs {
  // one copy of the line operators per pass: constant-bank operands (see TmaArgs)
  LineCoef<N, float> iy, ix, iz, fz, fx, fy;
  const float* in;
  const float* site;  // s or w
  const float* bk;    // per-mode factor
  float* out;
  double a;
  const int* done;
  int exec_if;
  const BatchTile* tiles;
  const BatchProb* probs;
  int scale_by_A;
  int ntau, spc;
  const float* U;
  const float* dotP;
  double full_scale, bU;
  int want_dotP, want_self;
  double* partials;
  int fop;
  DevScalars* scs;
  unsigned* counters;
  int part_base;
  int* err;
  int expire;  // test hook (ufg_test_expire_waits)
};

template <int N, int DIR, bool FULL>
__global__ void __launch_bounds__(FixShape<N>::NT, 2)
slice_reg_m1w_kernel(const __grid_constant__ RegM1wArgs<N> A) {
  pdl_begin();
  using S = FixShape<N>;
  static_assert(S::C == 1, "one CTA holds whole slices");
  constexpr int NN = N * N, VOL = N * NN, P = S::P, PL = S::PL;
  extern __shared__ __align__(16) unsigned char fix_smem[];
  __shared__ alignas(8) uint64_t bar2;
  const FixPos<N> p = fix_pos<N>();
  const int unit = blockIdx.x;
  const FixUnit u = fix_unit<N>(A, unit, p.s);
  if (!u.run) return;
  if (A.expire && threadIdx.x == 0) mbar_expire_one_wait(&bar2, 256u, A.err);
  const bool on = p.on && u.have;
  float* const sm = reinterpret_cast<float*>(fix_smem) + (size_t)p.s * S::SLOT;
  float* const mine = sm + p.line * PL;  // plane z = line
  const int t_in = DIR == 0 ? (u.t_out == 0 ? u.ntau - 1 : u.t_out - 1)
                            : (u.t_out == u.ntau - 1 ? 0 : u.t_out + 1);
  const float sgn = (DIR == 0 ? u.t_out != 0 : u.t_out != u.ntau - 1) ? -1.0f : 1.0f;
  const int t_s = DIR == 0 ? t_in : u.t_out;  // slice of the site multiplier
  const int m0 = p.line * NN + p.lx;          // first mode of this thread's (plane, x) line
  float v[N];
  if (on) {  // inverse y-pass: mode line (plane, x)
    const float* gi = A.in + u.off + (size_t)t_in * VOL + m0;
#pragma unroll
    for (int y = 0; y < N; ++y) v[y] = __ldg(gi + y * N);
    if constexpr (DIR == 1) {
#pragma unroll
      for (int y = 0; y < N; ++y) v[y] *= __ldg(A.bk + m0 + y * N);
    }
    line_op<N, float, true, false>(v, A.iy, [&](int i, float r) { mine[i * P + p.lx] = r; });
  }
  __syncwarp();
  if (on) {  // inverse x-pass: row (plane, y = lx), in place
    float* const row = mine + p.lx * P;
#pragma unroll
    for (int x = 0; x < N; ++x) v[x] = row[x];
    line_op<N, float, true, false>(v, A.ix, [&](int i, float r) { row[i] = r; });
  }
  __syncthreads();
  if (on) {  // column (y = line, x): inverse z-pass, site multiplier, forward z-pass, in place
    float* const col = sm + p.line * P + p.lx;
    const float* gs = A.site + u.off + (size_t)t_s * VOL + p.line * N + p.lx;
    const float f1 = DIR == 1 ? sgn * (float)u.acoef : 1.0f;
    float w[N];
#pragma unroll
    for (int z = 0; z < N; ++z) v[z] = col[z * PL];
    line_op<N, float, true, false>(
        v, A.iz, [&](int z, float r) { w[z] = (f1 * __ldg(gs + z * NN)) * r; });
    line_op<N, float, false, true>(w, A.fz, [&](int i, float r) { col[i * PL] = r; });
  }
  __syncthreads();
  if (on) {  // forward x-pass: row (plane, y = lx), in place
    float* const row = mine + p.lx * P;
#pragma unroll
    for (int x = 0; x < N; ++x) v[x] = row[x];
    line_op<N, float, false, true>(v, A.fx, [&](int i, float r) { row[i] = r; });
  }
  __syncwarp();
  float acc_dot = 0.0f, acc_self = 0.0f;
  if (on) {  // forward y-pass and epilogue: modes (plane, y, x)
#pragma unroll
    for (int y = 0; y < N; ++y) v[y] = mine[y * P + p.lx];
    const float f2 = DIR == 0 ? sgn * (float)u.acoef : 1.0f;
    const size_t so = u.off + (size_t)u.t_out * VOL;
    const float fs = (float)A.full_scale, bU = (float)A.bU;
    line_op<N, float, false, true>(v, A.fy, [&](int y, float r) {
      const int g = m0 + y * N;
      float o = f2 * r;
      if constexpr (DIR == 0) o *= __ldg(A.bk + g);
      if constexpr (FULL) {
        o = fs * (o + __ldg(A.in + so + g));
        if (A.U != nullptr) o = fmadd(bU, A.U[so + g], o);  // U may be out
      }
      A.out[so + g] = o;
      if constexpr (FULL) {
        if (A.want_dotP) acc_dot = fmadd(o, __ldg(A.dotP + so + g), acc_dot);
        if (A.want_self) acc_self = fmadd(o, o, acc_self);
      }
    });
  }
  if constexpr (FULL) {
    if (A.want_dotP || A.want_self)
      fix_partials((double)acc_dot, (double)acc_self, A.partials, A.fop, A.tiles, unit, A.probs,
                   A.scs, A.counters, A.part_base);
  }
}

template <int N, int DIR, bool FULL>
inline cudaError_t reg_m1w_launch(const SliceCall& c, cudaStream_t st) {
  if (c.in == nullptr || c.pre == nullptr || c.out == nullptr || c.coef == nullptr ||
      c.coef2 == nullptr || (DIR == 1 ? c.bkpre : c.bkpost) == nullptr)
    return cudaErrorInvalidValue;
  RegM1wArgs<N> a;
  std::memset(&a, 0, sizeof(a));
  a.iy = *static_cast<const LineCoef<N, float>*>(c.coef);
  a.ix = a.iy;
  a.iz = a.iy;
  a.fz = *static_cast<const LineCoef<N, float>*>(c.coef2);
  a.fx = a.fz;
  a.fy = a.fz;
  fix_common<N>(a, c, st);
  a.site = static_cast<const float*>(c.pre);
  a.bk = static_cast<const float*>(DIR == 1 ? c.bkpre : c.bkpost);
  a.full_scale = c.full_scale;
  static int configured = 0;
  return fix_launch<N, float>(slice_reg_m1w_kernel<N, DIR, FULL>, &configured, a, c, st);
}

template <int N>
inline cudaError_t slice_reg_m1w_try(const SliceCall& c, cudaStream_t st) {
  if constexpr (N < 16) {
    if (c.shift < 0)
      return c.m1w_full ? reg_m1w_launch<N, 0, true>(c, st) : reg_m1w_launch<N, 0, false>(c, st);
    if (c.shift > 0)
      return c.m1w_full ? reg_m1w_launch<N, 1, true>(c, st) : reg_m1w_launch<N, 1, false>(c, st);
  }
  return cudaErrorNotSupported;
}

}  // namespace ufg
