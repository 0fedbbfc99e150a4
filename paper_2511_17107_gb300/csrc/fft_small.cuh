// The apply (and T0) of a whole complex64 vector by one CTA, for N = 8 and 16.
//
// At these sizes a vector (12 KB and 98 KB) fits the shared memory of an SM,
// while each of the five passes of fft_kernels.cuh has one or two CTAs per
// vector and costs a launch: a single 16^3 vector took 37.5 us in five launches,
// 21 us in this one (back to back: 34.8 and 16.3); 256 vectors 158 and 37.5 us,
// 1000 8^3 vectors 401 and 21 us.  A thread transforms one line of one
// component in registers per axis; the vector goes through shared memory
// between the axes and through global memory once each way, and gamma kappa.x
// stays in registers from the first step to the last.  The arithmetic is that
// of the five passes, step by step (same results).  What bounds a single
// vector is the latency of its eight steps on one SM.
#pragma once

#include "fft_kernels.cuh"

namespace pcx {
namespace fftk {

template <int N>
struct SmallTile {
  static constexpr int N2 = N * N, N3 = N2 * N;
  static constexpr int THREADS = 3 * N2;              // one line each
  static constexpr int SX = N + 1, SZ = N * SX;       // row and plane strides: lines along x hit distinct banks
  static constexpr int CS = N * SZ;                   // component stride
  static constexpr int MODES = (N3 + THREADS - 1) / THREADS;   // modes per thread in the pointwise steps
  static constexpr size_t entries() { return 3 * CS + 3 * N + 3 * N2; }   // tile, kappa tables
};

template <int N, bool T0>
__global__ void __launch_bounds__(SmallTile<N>::THREADS) apply_small_kernel(PassArgs a) {
  using ST = SmallTile<N>;
  using F = cx<float>;
  constexpr int N2 = ST::N2, N3 = ST::N3;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  F* s = reinterpret_cast<F*>(smem_raw);
  F* ka = s + 3 * ST::CS;   // [3][N]
  F* kb = ka + 3 * N;       // [N2][3]
  float* mtab = reinterpret_cast<float*>(kb + 3 * N2);   // [n_mat][9]
  const size_t v = blockIdx.x;
  const F* in = static_cast<const F*>(a.in) + v * 3 * N3;
  F* out = static_cast<F*>(a.out) + v * 3 * N3;
  KParams kp = a.kp;
  if (a.kps) kp = a.kps[(a.v_base + (int)v) / a.vec_per_k];
  auto at = [](int e) { return (e / N2) * ST::SZ + ((e / N) % N) * ST::SX + e % N; };   // mode or cell e = (z N + y) N + x

  // this thread's modes, their loads in flight while the tables are built
  F x[ST::MODES][3];
#pragma unroll
  for (int i = 0; i < ST::MODES; ++i) {
    const int e = threadIdx.x + i * ST::THREADS;
    if (e < N3) {
#pragma unroll
      for (int c = 0; c < 3; ++c) x[i][c] = in[c * N3 + e];
    }
  }
  kappa_tables<float, N, N2, ST::THREADS>(static_cast<const F*>(a.lam), kp, 0, ka, kb);
  if (a.mid)
    for (int i = threadIdx.x; i < 9 * a.n_mat; i += ST::THREADS) mtab[i] = static_cast<const float*>(a.mtab)[i];
  __syncthreads();
  const float gam = (float)kp.gamma, igam = (float)(1.0 / kp.gamma);
  F sk[ST::MODES];
#pragma unroll
  for (int i = 0; i < ST::MODES; ++i) {
    const int e = threadIdx.x + i * ST::THREADS;
    if (e < N3) {
      pre_point<float, T0>(x[i][0], x[i][1], x[i][2], sk[i], ka + e % N, N, kb + 3 * (e / N), kp, gam, igam);
#pragma unroll
      for (int c = 0; c < 3; ++c) s[c * ST::CS + at(e)] = x[i][c];
    }
  }
  __syncthreads();
  // line (c, p, q) of this thread: along x at (z, y) = (p, q), along y at
  // (z, x), along z at (y, x)
  const int c = threadIdx.x / N2, p = (threadIdx.x / N) % N, q = threadIdx.x % N;
  F* lx = s + c * ST::CS + p * ST::SZ + q * ST::SX;
  F* ly = s + c * ST::CS + p * ST::SZ + q;
  F* lz = s + c * ST::CS + p * ST::SX + q;
  auto line = [&](F* l, int stride, auto dir) {
    F r[N];
#pragma unroll
    for (int n = 0; n < N; ++n) r[n] = l[n * stride];
    dft<N, decltype(dir)::value>(r);
#pragma unroll
    for (int n = 0; n < N; ++n) l[n * stride] = r[n];
    __syncthreads();
  };
  const std::integral_constant<int, +1> inv{};
  const std::integral_constant<int, -1> fwd{};
  line(lx, 1, inv);
  line(ly, ST::SX, inv);
  line(lz, ST::SZ, inv);
  const uchar4* mid = static_cast<const uchar4*>(a.mid);
#pragma unroll
  for (int i = 0; i < ST::MODES; ++i) {
    const int e = threadIdx.x + i * ST::THREADS;
    if (e < N3) {
      F w[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) w[k] = s[k * ST::CS + at(e)];
      cell_point<float, N, T0>(w, mid ? mid + e : nullptr, mtab, static_cast<const float*>(a.M), e,
                               (float)(1.0 / (double)N3));
#pragma unroll
      for (int k = 0; k < 3; ++k) s[k * ST::CS + at(e)] = w[k];
    }
  }
  __syncthreads();
  line(lz, ST::SZ, fwd);
  line(ly, ST::SX, fwd);
  line(lx, 1, fwd);
#pragma unroll
  for (int i = 0; i < ST::MODES; ++i) {
    const int e = threadIdx.x + i * ST::THREADS;
    if (e < N3) {
      F w[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) w[k] = s[k * ST::CS + at(e)];
      post_point<float, T0>(w, sk[i], ka + e % N, N, kb + 3 * (e / N), out[e], out[N3 + e], out[2 * N3 + e]);
    }
  }
}

template <typename T, int N, bool T0>
cudaError_t launch_small(const PassArgs& a, int nv, cudaStream_t st) {
  using ST = SmallTile<N>;
  const auto kern = apply_small_kernel<N, T0>;
  const size_t smem = ST::entries() * sizeof(cx<float>) + (size_t)9 * a.n_mat * sizeof(float);
  cudaError_t e = raise_dyn_smem(reinterpret_cast<const void*>(kern), smem);
  if (e != cudaSuccess) return e;
  kern<<<(unsigned)nv, ST::THREADS, smem, st>>>(a);
  return cudaGetLastError();
}

}  // namespace fftk
}  // namespace pcx
