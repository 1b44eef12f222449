// The normal-equation operator Q = M^T M (Eq. 1) in one kernel per output slice.
//
// With B_t = e^{-tau K} w_t (Sec. 1; T = e^{-tau K} applied by the line operators, w the
// potential) and the antiperiodic signs of Eq. MatrixM,
//   y_s = (M x)_s = x_s + sm(s) T(w_{s-1} x_{s-1}),      sm(s) = -1 except sm(0) = +1,
//   q_t = (M^T y)_t = y_t + st(t) w_t T(y_{t+1}),        st(t) = -1 except st(N_tau - 1) = +1,
// so q_t needs x at t-1, t and t+1 (cyclically).  One CTA per output slice holds those three
// slices as TMA boxes and runs three kinetic stages in place:
//   A: X0 <- x_t + sm(t) T(w_{t-1} X0)          (= y_t)
//   B: X2 <- X2 + sm(t+1) T(w_t X1)             (= y_{t+1})
//   C: q_t = a (X0 + st(t) w_t T(X2)) + bU U + cV V, with the dot partials of the slice kernels.
// Three kinetic stages per slice instead of the two of M followed by M^T, in exchange for one
// launch instead of two and no intermediate vector in memory: at 16^3 the two launches are
// bound by latency (one CTA per slice, few CTAs per SM), not by their bytes.  The multiplier
// rows of the x-passes come from global memory (16-byte loads), the epilogue's w_t per site.
// Stages A and B run side by side in the two halves of the CTA, and the multiplier rows are
// requested before the boxes arrive: back to back 13.3 -> 8.0 us at 16^3 x 256 with programmatic
// dependent launch, which apply_op uses for this kernel (CG + Chebyshev 16, mixed: 195 -> 183 us per
// iteration of 17 Q, 9 of them launched that way; without it the launch gaps hid the gain).  Latency-bound: 256 CTAs on
// 152 SMs, issue 27 %.
// Built for FP32 16^3 slices; slice_q_supported says where it runs.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstring>

#include "slice_tma.cuh"

namespace ufg {

template <int N>
struct QArgs {
  CUtensorMap tm_in;  // [rows][N] view of x, box = one slice
  // the kinetic line operator once per pass direction (constant-bank operands, see TmaArgs)
  LineCoef<N, float> cx, cy, cz;
  const float* w;  // the potential w = 1 + A sin(sigma) [S]
  float* out;
  const float* U;
  const float* V;
  const float* dotP;
  double a, bU, cV;
  double* partials;
  int want_dotP, want_self;
  const int* done;
  int exec_if;
  int ntau;
  int fop;  // scalar op of the grid's last CTA (-1: none), see SliceCall
  DevScalars* scs;
  unsigned* counters;
  int* err;
  int expire;  // test hook, see TmaArgs
};

// Stages A and B (see above) share no output, so two halves of the CTA run them side by side: six
// passes in a row instead of nine (x_t is loaded twice, once per half).
constexpr int Q_NT = 2 * TMA_NT;

// x-pass in place, row r: times the multiplier row w when MUL
template <int N, bool MUL, class CF>
__device__ __forceinline__ void q_xpass(float* X, int r, const float (&w)[N], const CF& cf) {
  using G = SwzGeom<N, float>;
  constexpr int CPR = G::RB / 16, EPC = 16 / (int)sizeof(float);
  float v[N];
#pragma unroll
  for (int c = 0; c < CPR; ++c) {
    const int o = G::chunk(r, c);
    float vc[EPC], wc[EPC];
#pragma unroll
    for (int e = 0; e < EPC; ++e) {
      vc[e] = X[o + e];
      wc[e] = w[c * EPC + e];
    }
    if constexpr (MUL) mul_chunk(vc, wc);
#pragma unroll
    for (int e = 0; e < EPC; ++e) v[c * EPC + e] = vc[e];
  }
  swz_store_row<N, float>(X, r, v, cf, false, false);
}

// y-pass in place, column l = (plane, x)
template <int N, class CF>
__device__ __forceinline__ void q_ypass(float* X, int l, const CF& cf) {
  using G = SwzGeom<N, float>;
  const int p = l / N, x = l - (l / N) * N;
  float v[N];
#pragma unroll
  for (int y = 0; y < N; ++y) v[y] = X[G::off(p * N + y, x)];
  line_op<N, float, false, false>(v, cf, [&](int i, float val) { X[G::off(p * N + i, x)] = val; });
}

template <int N, bool UV, bool DOT>
__global__ void __launch_bounds__(Q_NT, 2)
slice_q_kernel(const __grid_constant__ QArgs<N> A) {
  pdl_begin();
  using G = SwzGeom<N, float>;
  constexpr int NN = N * N;
  constexpr int VOL = N * NN;
  static_assert(NN == TMA_NT, "one row, line and column per thread of a half");
  extern __shared__ __align__(1024) unsigned char tma_smem[];
  __shared__ double red[Q_NT / 32][2];
  __shared__ alignas(8) uint64_t bar, bar2;
  const int tid = threadIdx.x;
  const int t = blockIdx.x;
  const int ntau = A.ntau;
  if (A.done != nullptr && A.exec_if >= 0 && *A.done != A.exec_if) return;
  const int tm = t == 0 ? ntau - 1 : t - 1;
  const int tp = t == ntau - 1 ? 0 : t + 1;
  const float sA = t != 0 ? float(-1) : float(1);          // sm(t)
  const float sB = tp != 0 ? float(-1) : float(1);         // sm(t+1)
  const float sC = t != ntau - 1 ? float(-1) : float(1);   // st(t)
  unsigned char* const base = tma_smem + ((1024u - (smem_addr(tma_smem) & 1023u)) & 1023u);
  float* const X0 = reinterpret_cast<float*>(base);
  float* const X1 = X0 + VOL;
  float* const X2 = X1 + VOL;
  float* const X3 = X2 + VOL;  // x_t again, for stage A's epilogue
  if (tid == 0) {
    mbar_init(&bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    mbar_expect_tx(&bar, (uint32_t)(4 * VOL * sizeof(float)));
    tma_load_rows(X0, &A.tm_in, tm * NN, &bar);
    tma_load_rows(X1, &A.tm_in, t * NN, &bar);
    tma_load_rows(X2, &A.tm_in, tp * NN, &bar);
    tma_load_rows(X3, &A.tm_in, t * NN, &bar);
  }
  // this thread's multiplier row of its first x-pass, while the boxes are in flight
  const float* const w_tm = A.w + (size_t)tm * VOL;
  const float* const w_t = A.w + (size_t)t * VOL;
  float wrow[N];
  {
    constexpr int EPC = 16 / (int)sizeof(float);
    const float* src = (tid >= NN ? w_t + (size_t)(tid - NN) * N : w_tm + (size_t)tid * N);
#pragma unroll
    for (int c = 0; c < N / EPC; ++c) {
      float w4[EPC];
      ld16(src + c * EPC, w4);
#pragma unroll
      for (int e = 0; e < EPC; ++e) wrow[c * EPC + e] = w4[e];
    }
  }
  __syncthreads();
  mbar_wait_bounded(&bar, 0u, TMA_WAIT_LIMIT, A.err);
  if (A.expire && tid == 0) mbar_expire_one_wait(&bar2, EXPIRE_LIMIT, A.err);
  // ---- A: X0 <- x_t + sm(t) T(w_{t-1} x_{t-1});  B: X2 <- x_{t+1} + sm(t+1) T(w_t x_t) ----
  {
    const bool second = tid >= NN;
    const int l = second ? tid - NN : tid;
    float* const X = second ? X1 : X0;
    q_xpass<N, true>(X, l, wrow, A.cx);
    __syncthreads();
    q_ypass<N>(X, l, A.cy);
    __syncthreads();
    const float* const id = second ? X2 : X3;
    float* const dst = second ? X2 : X0;
    const float sg = second ? sB : sA;
    const int y = l / N, x = l - (l / N) * N;
    float v[N];
#pragma unroll
    for (int z = 0; z < N; ++z) v[z] = X[G::off(z * N + y, x)];
    line_op<N, float, false, false>(v, A.cz, [&](int zp, float val) {
      const int o = G::off(zp * N + y, x);
      dst[o] = fmadd(sg, val, id[o]);
    });
  }
  __syncthreads();
  // ---- C: q_t = a (y_t + st(t) w_t T(y_{t+1})) + bU U + cV V ----
  if (tid < NN) q_xpass<N, false>(X2, tid, wrow, A.cx);
  __syncthreads();
  if (tid < NN) q_ypass<N>(X2, tid, A.cy);
  __syncthreads();
  const size_t obase0 = (size_t)t * VOL;
  const float ra = float(A.a), rbU = float(A.bU), rcV = float(A.cV);
  float acc_dot = float(0), acc_self = float(0);
  if (tid < NN) {
    const int q = tid;
    const int y = q / N, x = q - (q / N) * N;
    float v[N];
#pragma unroll
    for (int z = 0; z < N; ++z) v[z] = X2[G::off(z * N + y, x)];
    const size_t obase = obase0 + q;
    line_op<N, float, false, false>(v, A.cz, [&](int zp, float val) {
      const size_t g = obase + (size_t)zp * NN;
      const int o = G::off(zp * N + y, x);
      float r = ra * fmadd(sC * __ldg(w_t + zp * NN + q), val, X0[o]);
      if constexpr (UV) {
        if (A.U != nullptr) r = fmadd(rbU, __ldg(A.U + g), r);
        if (A.V != nullptr) r = fmadd(rcV, __ldg(A.V + g), r);
      }
      A.out[g] = r;
      if constexpr (DOT) {
        if (A.want_dotP) acc_dot = fmadd(r, __ldg(A.dotP + g), acc_dot);
        if (A.want_self) acc_self = fmadd(r, r, acc_self);
      }
    });
  }
  if constexpr (DOT) {  // one partial pair per CTA, as the slice kernels
    double pd = (double)acc_dot, ps = (double)acc_self;
#pragma unroll
    for (int o2 = 16; o2 > 0; o2 >>= 1) {
      pd += __shfl_xor_sync(0xffffffffu, pd, o2);
      ps += __shfl_xor_sync(0xffffffffu, ps, o2);
    }
    if ((tid & 31) == 0) {
      red[tid >> 5][0] = pd;
      red[tid >> 5][1] = ps;
    }
    __syncthreads();
    if (tid == 0) {
      double d = 0.0, q2 = 0.0;
      for (int wi = 0; wi < Q_NT / 32; ++wi) {
        d += red[wi][0];
        q2 += red[wi][1];
      }
      A.partials[2 * blockIdx.x] = d;
      A.partials[2 * blockIdx.x + 1] = q2;
    }
    if (A.fop >= 0) last_block_update<0>(A.fop, A.scs, A.partials, 0, (int)gridDim.x, A.counters);
  }
}

template <int N, bool UV, bool DOT>
inline cudaError_t q_launch(const SliceCall& c, cudaStream_t st) {
  constexpr int VOL = N * N * N;
  QArgs<N> a;
  std::memset(&a, 0, sizeof(a));
  if (c.in == nullptr || c.pre == nullptr || c.out == nullptr || c.coef == nullptr ||
      c.ntau < 3 || c.tiles != nullptr || (c.want_dotP && c.dotP == nullptr) ||
      ((c.want_dotP || c.want_self) && c.partials == nullptr) ||
      (c.fop >= 0 && (!DOT || c.scs == nullptr || c.counters == nullptr)))
    return cudaErrorInvalidValue;
  if (encode_rows<float>(&a.tm_in, c.in, (long long)c.ntau * VOL, N, N * N) != cudaSuccess)
    return cudaErrorNotSupported;
  a.cx = *reinterpret_cast<const LineCoef<N, float>*>(c.coef);
  a.cy = a.cx;
  a.cz = a.cx;
  a.w = static_cast<const float*>(c.pre);
  a.out = static_cast<float*>(c.out);
  a.U = static_cast<const float*>(c.U);
  a.V = static_cast<const float*>(c.V);
  a.dotP = static_cast<const float*>(c.dotP);
  a.a = c.a;
  a.bU = c.bU;
  a.cV = c.cV;
  a.partials = c.partials;
  a.want_dotP = c.want_dotP;
  a.want_self = c.want_self;
  a.done = c.done;
  a.exec_if = c.exec_if;
  a.ntau = c.ntau;
  a.fop = c.fop;
  a.scs = c.scs;
  a.counters = c.counters;
  a.err = c.err;
  a.expire = take_expired_wait(st);
  const size_t smem = 4 * (size_t)VOL * sizeof(float) + 1024;
  auto kern = slice_q_kernel<N, UV, DOT>;
  static int configured = 0;
  if (!configured) {
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)smem);
    if (err != cudaSuccess) return err;
    err = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                               cudaSharedmemCarveoutMaxShared);
    if (err != cudaSuccess) return err;
    configured = 1;
  }
  if (c.grid_out) *c.grid_out = c.ntau;
  return launch_k(kern, dim3(c.ntau), dim3(Q_NT), smem, st, 1, a);
}

template <int N>
inline cudaError_t q_launch_epi(const SliceCall& c, cudaStream_t st) {
  const bool uv = c.U != nullptr || c.V != nullptr;
  const bool dot = c.want_dotP || c.want_self;
  if (uv) return dot ? q_launch<N, true, true>(c, st) : q_launch<N, true, false>(c, st);
  return dot ? q_launch<N, false, true>(c, st) : q_launch<N, false, false>(c, st);
}

// The fused Q for FP32 16^3 slices, where the one-CTA TMA boxes hold one slice.
template <int N>
cudaError_t slice_q_try(const SliceCall& c, cudaStream_t st) {
  if constexpr (N == 16) {
    if (c.prec == 1) return q_launch_epi<16>(c, st);
  }
  return cudaErrorNotSupported;
}

}  // namespace ufg
