// Block kernels of the Rayleigh-Ritz eigensolver (Sec. 4: LOBPCG): Gram
// products of tall-skinny blocks, the tall x small update, residuals and
// their norms (eq. exp_relativeresidual), random initial blocks and the
// k = 0 deflation of the constant fields (Prop. 2.5).
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstdint>

#include "cx.cuh"
#include "dfloat.cuh"
#include "pcx_internal.h"

namespace pcx {
namespace {

// ---------------------------------------------------------------------------
// Gram: G[i][j] = sum_l conj(A_i[l]) B_j[l], FP64 output.
// CTA tile: 32 x 32 outputs, 256 threads each owning a 2 x 2 output block.
// The row range [l0, l1) of one CTA is walked in chunks of GL rows staged in
// shared memory; products accumulate in T within a chunk and in FP64 across
// chunks; CTA partials are added to G with FP64 atomics.
// ---------------------------------------------------------------------------
constexpr int GT = 32;
constexpr int GL = 32;
// Default complex64 Gram path by shape, from CUDA-event timings of both
// kernels at L = 3 * 128^3 on GB300 (ms, tensor cores / FP32 pipes):
// 16x16 0.73 / 0.52, 16x32 1.46 / 0.84, 16x48 1.88 / 1.25, 32x48 2.12 / 2.06,
// 48x48 2.37 / 3.65; A^H A: 16 0.76 / 0.34, 32 0.91 / 0.86, 48 1.11 / 2.21.
// The FMA count grows with na nb while the tensor-core kernel's cost is
// dominated by its per-element hi/lo conversion, so small products go to the
// FP32 pipes.
bool gram_fp32_pipes_faster(bool herm, int na, int nb) { return herm ? na <= 32 : na * nb <= 32 * 48; }

template <typename T>
__global__ void __launch_bounds__(256) gram_kernel(const cx<T>* __restrict__ A, int na, const cx<T>* __restrict__ B,
                                                   int nb, size_t L, size_t rows_per_cta, double* __restrict__ G) {
  __shared__ cx<T> sa[GL][GT + 1];
  __shared__ cx<T> sb[GL][GT + 1];
  const int ti = blockIdx.x * GT, tj = blockIdx.y * GT;
  const size_t l0 = (size_t)blockIdx.z * rows_per_cta;
  const size_t l1 = (l0 + rows_per_cta < L) ? l0 + rows_per_cta : L;
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;   // output block (2ty.., 2tx..)
  double acc[2][2][2] = {};
  for (size_t base = l0; base < l1; base += GL) {
    // stage GL rows of 32 columns of A and B (row index fastest across threads)
    for (int e = threadIdx.x; e < GL * GT; e += 256) {
      const int r = e % GL, col = e / GL;
      const size_t l = base + r;
      const bool ok = l < l1;
      sa[r][col] = (ok && ti + col < na) ? A[(size_t)(ti + col) * L + l] : mk((T)0, (T)0);
      sb[r][col] = (ok && tj + col < nb) ? B[(size_t)(tj + col) * L + l] : mk((T)0, (T)0);
    }
    __syncthreads();
    cx<T> part[2][2];
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b) part[a][b] = mk((T)0, (T)0);
#pragma unroll 8
    for (int r = 0; r < GL; ++r) {
      cx<T> av[2] = {sa[r][2 * ty], sa[r][2 * ty + 1]};
      cx<T> bv[2] = {sb[r][2 * tx], sb[r][2 * tx + 1]};
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) part[a][b] = cfma_conj(av[a], bv[b], part[a][b]);
    }
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        acc[a][b][0] += (double)part[a][b].x;
        acc[a][b][1] += (double)part[a][b].y;
      }
    __syncthreads();
  }
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int i = ti + 2 * ty + a, j = tj + 2 * tx + b;
      if (i < na && j < nb) {
        atomicAdd(&G[2 * ((size_t)i * nb + j)], acc[a][b][0]);
        atomicAdd(&G[2 * ((size_t)i * nb + j) + 1], acc[a][b][1]);
      }
    }
}

// ---------------------------------------------------------------------------
// Combine: Y_j = sum_i S_i C[i][j] (+ beta Y_j), one row per thread, up to
// CY output columns per sweep; C staged in shared memory in T.
// ---------------------------------------------------------------------------
constexpr int CY = 16;

template <typename T>
__global__ void __launch_bounds__(256) combine_kernel(const cx<T>* __restrict__ S, int ns, const double* __restrict__ Cm,
                                                      int ny, int j0, double beta, cx<T>* __restrict__ Y, size_t L) {
  extern __shared__ __align__(16) unsigned char csm[];
  cx<T>* c = reinterpret_cast<cx<T>*>(csm);   // [ns][CY]
  const int nyl = (ny - j0 < CY) ? ny - j0 : CY;
  for (int e = threadIdx.x; e < ns * CY; e += blockDim.x) {
    const int i = e / CY, j = e % CY;
    c[e] = (j < nyl) ? mk((T)Cm[2 * ((size_t)i * ny + j0 + j)], (T)Cm[2 * ((size_t)i * ny + j0 + j) + 1])
                     : mk((T)0, (T)0);
  }
  __syncthreads();
  for (size_t l = (size_t)blockIdx.x * blockDim.x + threadIdx.x; l < L; l += (size_t)gridDim.x * blockDim.x) {
    cx<T> acc[CY];
#pragma unroll
    for (int j = 0; j < CY; ++j) acc[j] = mk((T)0, (T)0);
    for (int i = 0; i < ns; ++i) {
      const cx<T> sv = S[(size_t)i * L + l];
#pragma unroll
      for (int j = 0; j < CY; ++j) acc[j] = cfma(sv, c[i * CY + j], acc[j]);
    }
#pragma unroll
    for (int j = 0; j < CY; ++j) {
      if (j < nyl) {
        cx<T>* yp = Y + (size_t)(j0 + j) * L + l;
        cx<T> r = acc[j];
        if (beta != 0.0) r = r + scale(*yp, (T)beta);
        *yp = r;
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Combine of complex64 columns with even L and 16-byte aligned columns: two
// rows l per thread (one 16-byte load of S_i per thread and i).  A product
// s c adds s.re (c.re, c.im) and s.im (-c.im, c.re) to the pair (re, im), two
// packed FMAs; the coefficients sit in shared memory as those two pairs, one
// 16-byte load for the four packed FMAs of both rows.  Packed FMAs halve the
// issue slots.  The entries arrive by cp.async in a ring of RING slots per
// thread (private to it, so no barrier), which keeps that many loads in flight
// across columns and rows without registers.  Measured at 48 -> 16 columns of
// 3 128^3 rows: 1.18 ms with four loads in registers and scalar FMAs, 1.13
// with packed ones, 0.83 with the ring (FMA pipes alone 0.52 ms, HBM 0.47).
// ADD64: Y is complex128 and the FP32 sums are added to it (combine_add32);
// otherwise Y = sum (+ beta Y).
// ---------------------------------------------------------------------------
constexpr int RING = 8;
template <bool ADD64>
__global__ void __launch_bounds__(256, 2) combine2_kernel(const float4* __restrict__ S, int ns,
                                                          const double* __restrict__ Cm, int ny, int j0, double beta,
                                                          void* __restrict__ Yv, size_t L2) {
  extern __shared__ __align__(16) unsigned char csm[];
  float4* ring = reinterpret_cast<float4*>(csm);   // [RING][256]
  float4* c = ring + RING * 256;                   // [ns][CY]: (re, im, -im, re)
  const int nyl = (ny - j0 < CY) ? ny - j0 : CY;
  for (int e = threadIdx.x; e < ns * CY; e += 256) {
    const int i = e / CY, j = e % CY;
    float re = 0.f, im = 0.f;
    if (j < nyl) {
      const double* ci = Cm + 2 * ((size_t)i * ny + j0 + j);
      re = (float)ci[0];
      im = (float)ci[1];
    }
    c[e] = make_float4(re, im, -im, re);
  }
  const size_t f0 = (size_t)blockIdx.x * 256 + threadIdx.x, stride = (size_t)gridDim.x * 256;
  const unsigned slot0 = (unsigned)__cvta_generic_to_shared(ring + threadIdx.x);
  // the next entry to fetch: column pi of row pair pf
  size_t pf = f0;
  int pi = 0;
  auto fetch = [&](int k) {
    if (pf < L2) {
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(slot0 + (unsigned)k * 4096u),
                   "l"(S + (size_t)pi * L2 + pf)
                   : "memory");
      if (++pi == ns) {
        pi = 0;
        pf += stride;
      }
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
#pragma unroll
  for (int k = 0; k < RING; ++k) fetch(k);
  __syncthreads();
  const float fb = (float)beta;
  int k = 0;
  for (size_t f = f0; f < L2; f += stride) {
    float2 a0[CY], a1[CY];   // rows 2f and 2f + 1
#pragma unroll
    for (int j = 0; j < CY; ++j) a0[j] = a1[j] = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int i = 0; i < ns; ++i) {
      asm volatile("cp.async.wait_group %0;\n" ::"n"(RING - 1) : "memory");
      const float4 sv = ring[k * 256 + threadIdx.x];
      const float4* ci = c + i * CY;
      const float2 r0 = make_float2(sv.x, sv.x), m0 = make_float2(sv.y, sv.y);
      const float2 r1 = make_float2(sv.z, sv.z), m1 = make_float2(sv.w, sv.w);
#pragma unroll
      for (int j = 0; j < CY; ++j) {
        const float4 cc = ci[j];
        const float2 cn = make_float2(cc.x, cc.y), cr = make_float2(cc.z, cc.w);
        fma2(a0[j], r0, cn);
        fma2(a0[j], m0, cr);
        fma2(a1[j], r1, cn);
        fma2(a1[j], m1, cr);
      }
      fetch(k);   // into the slot just read
      k = (k + 1) % RING;
    }
#pragma unroll
    for (int j = 0; j < CY; ++j) {
      if (j < nyl) {
        if constexpr (ADD64) {
          double2* yp = static_cast<double2*>(Yv) + (size_t)(j0 + j) * 2 * L2 + 2 * f;
          double2 y0 = yp[0], y1 = yp[1];
          y0.x += (double)a0[j].x;
          y0.y += (double)a0[j].y;
          y1.x += (double)a1[j].x;
          y1.y += (double)a1[j].y;
          yp[0] = y0;
          yp[1] = y1;
          if (j % 4 == 3) asm volatile("" ::: "memory");   // not all 32 loads at once
        } else {
          float4* yp = static_cast<float4*>(Yv) + (size_t)(j0 + j) * L2 + f;
          float4 r = make_float4(a0[j].x, a0[j].y, a1[j].x, a1[j].y);
          if (beta != 0.0) {
            const float4 o = *yp;
            r.x = fmaf(fb, o.x, r.x);
            r.y = fmaf(fb, o.y, r.y);
            r.z = fmaf(fb, o.z, r.z);
            r.w = fmaf(fb, o.w, r.w);
          }
          *yp = r;
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Combine for complex128 on the FP32 pipes (GB300's FP64 rate is a small
// fraction of its FP32 rate): entries and coefficients split into FP32 hi + lo
// and sums kept as double-float pairs (dfloat.cuh).  Entries must stay inside
// the FP32 exponent range.  Each row's entries are split once (integer
// operations) for the CT outputs of the sweep; C is split once per CTA into
// shared memory.  Packed operations take half the issue slots of scalar ones
// and leave room for the splits; their pairs are the same part of two outputs,
// so that a coefficient is read once for the real and the imaginary sums (with
// (re, im) as the pair the reads of C took as long as the arithmetic).  Bound
// by the FP32 pipes.
// CT = 4, 8, 12 or 16 outputs, so that narrow sweeps (few active columns) don't
// pay for 16.  Measured at 16 -> 16 columns of 3 128^3 rows: 3.09 ms with
// scalar operations of the textbook form (13 a product; entries split by
// truncation, whose error is a third larger), 2.54 now (FP32 pipes alone 1.9,
// HBM 0.47); at 3 32^3 rows 72 -> 56 us, for 3 outputs 74 -> 25.
// ---------------------------------------------------------------------------
template <int CT>
__global__ void __launch_bounds__(256) combine_ff_kernel(const double2* __restrict__ S, int ns,
                                                                   const double* __restrict__ Cm, int ny, int j0,
                                                                   int nyl, double beta, double2* __restrict__ Y,
                                                                   size_t L) {
  extern __shared__ __align__(16) unsigned char csm[];
  float4* c = reinterpret_cast<float4*>(csm);   // [ns][CT / 2][2]: hi re, re', im, im'; lo the same
  for (int e = threadIdx.x; e < ns * CT / 2; e += blockDim.x) {
    const int i = e / (CT / 2), j = 2 * (e % (CT / 2));
    float h[2][2] = {}, t[2][2] = {};   // [part][output]
#pragma unroll
    for (int o = 0; o < 2; ++o)
      if (j + o < nyl)
#pragma unroll
        for (int p = 0; p < 2; ++p) dfloat::split_rn(Cm[2 * ((size_t)i * ny + j0 + j + o) + p], h[p][o], t[p][o]);
    c[2 * e] = make_float4(h[0][0], h[0][1], h[1][0], h[1][1]);
    c[2 * e + 1] = make_float4(t[0][0], t[0][1], t[1][0], t[1][1]);
  }
  __syncthreads();
  for (size_t l = (size_t)blockIdx.x * blockDim.x + threadIdx.x; l < L; l += (size_t)gridDim.x * blockDim.x) {
    float2 re[CT / 2], im[CT / 2], rr[CT / 2], ir[CT / 2];   // sums of two outputs and their compensations
#pragma unroll
    for (int j = 0; j < CT / 2; ++j) re[j] = im[j] = rr[j] = ir[j] = make_float2(0.f, 0.f);
    double2 next = S[l];
#pragma unroll 1
    for (int i = 0; i < ns; ++i) {
      const double2 sv = next;
      if (i + 1 < ns) next = S[(size_t)(i + 1) * L + l];
      float h, t;
      dfloat::split_rn(sv.x, h, t);
      const float2 xh = make_float2(h, h), xl = make_float2(t, t);
      dfloat::split_rn(sv.y, h, t);
      const float2 yh = make_float2(h, h), yl = make_float2(t, t), nh = make_float2(-h, -h), nl = make_float2(-t, -t);
#pragma unroll
      for (int j = 0; j < CT / 2; ++j) {
        const float4 ch = c[(i * (CT / 2) + j) * 2], cl = c[(i * (CT / 2) + j) * 2 + 1];
        const float2 rh = make_float2(ch.x, ch.y), ih = make_float2(ch.z, ch.w);
        const float2 rl = make_float2(cl.x, cl.y), il = make_float2(cl.z, cl.w);
        dfloat::mac_pair(re[j], rr[j], xh, xl, rh, rl);
        dfloat::mac_pair(re[j], rr[j], nh, nl, ih, il);
        dfloat::mac_pair(im[j], ir[j], xh, xl, ih, il);
        dfloat::mac_pair(im[j], ir[j], yh, yl, rh, rl);
      }
    }
#pragma unroll
    for (int j = 0; j < CT; ++j) {
      if (j < nyl) {
        double2* yp = Y + (size_t)(j0 + j) * L + l;
        const float2 a = re[j / 2], b = im[j / 2], ar = rr[j / 2], br = ir[j / 2];
        double2 v = j % 2 ? make_double2((double)a.y + (double)ar.y, (double)b.y + (double)br.y)
                          : make_double2((double)a.x + (double)ar.x, (double)b.x + (double)br.x);
        if (beta != 0.0) {
          const double2 y0 = *yp;
          v.x += beta * y0.x;
          v.y += beta * y0.y;
        }
        *yp = v;
      }
    }
  }
}

template <int CT>
cudaError_t run_combine_ff(const void* S, int ns, const double* C, int ny, int j0, int nyl, double beta, void* Y,
                           size_t L, cudaStream_t s) {
  const size_t smem = (size_t)ns * CT * sizeof(float4);
  if (smem > 48 * 1024) {
    cudaError_t e = raise_dyn_smem(reinterpret_cast<const void*>(combine_ff_kernel<CT>), smem);
    if (e != cudaSuccess) return e;
  }
  // CTAs of 64 threads even out the short columns (32^3 has 20 warps of rows
  // per SM); with many columns S_i the coefficients of a CTA leave room for few
  // CTAs, so these are larger.  24 CTAs of 64 per SM divide evenly over any
  // usual number of resident ones.
  const unsigned threads = smem > 32 * 1024 ? 256 : 64;
  const unsigned blocks = (unsigned)std::min<size_t>((L + threads - 1) / threads, 152u * 24u * 64u / threads);
  combine_ff_kernel<CT><<<blocks, threads, smem, s>>>(static_cast<const double2*>(S), ns, C, ny, j0, nyl, beta,
                                                         static_cast<double2*>(Y), L);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Y64_j += sum_i S32_i C[i][j]: a combination of complex64 columns evaluated
// in FP32 and added into complex128 columns (the small correction part of a
// mixed-precision update).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) combine_add32_kernel(const cx<float>* __restrict__ S, int ns,
                                                            const double* __restrict__ Cm, int ny, int j0,
                                                            double2* __restrict__ Y, size_t L) {
  extern __shared__ __align__(16) unsigned char csm[];
  cx<float>* c = reinterpret_cast<cx<float>*>(csm);
  const int nyl = (ny - j0 < CY) ? ny - j0 : CY;
  for (int e = threadIdx.x; e < ns * CY; e += blockDim.x) {
    const int i = e / CY, j = e % CY;
    c[e] = (j < nyl) ? mk((float)Cm[2 * ((size_t)i * ny + j0 + j)], (float)Cm[2 * ((size_t)i * ny + j0 + j) + 1])
                     : mk(0.f, 0.f);
  }
  __syncthreads();
  for (size_t l = (size_t)blockIdx.x * blockDim.x + threadIdx.x; l < L; l += (size_t)gridDim.x * blockDim.x) {
    cx<float> acc[CY];
#pragma unroll
    for (int j = 0; j < CY; ++j) acc[j] = mk(0.f, 0.f);
    for (int i = 0; i < ns; ++i) {
      const cx<float> sv = S[(size_t)i * L + l];
#pragma unroll
      for (int j = 0; j < CY; ++j) acc[j] = cfma(sv, c[i * CY + j], acc[j]);
    }
#pragma unroll
    for (int j = 0; j < CY; ++j) {
      if (j < nyl) {
        double2* yp = Y + (size_t)(j0 + j) * L + l;
        double2 y = *yp;
        y.x += (double)acc[j].x;
        y.y += (double)acc[j].y;
        *yp = y;
      }
    }
  }
}

// total += eight FP32 squares: gathered in a double-float pair on the FP32 pipes
// (the pair rounds at 2^-48, each square at 2^-24) and added once.  Squares that
// take the pair beyond the FP32 range, or are Inf or NaN themselves, are added one
// by one, so the sum has the range of FP64 and infinities stay infinite.
__device__ __forceinline__ void add_squares(double& total, const float q[8]) {
  dfloat::DF p{q[0], 0.f};
#pragma unroll
  for (int u = 1; u < 8; ++u) dfloat::add(p, q[u], 0.f);
  if (p.s <= 3.402823466e38f) {
    total += (double)p.s + (double)p.c;
  } else {
    for (int u = 0; u < 8; ++u) total += (double)q[u];
  }
}

// ---------------------------------------------------------------------------
// Residual R_j = AX_j - theta_j X_j with ||R_j||^2 and ||X_j||^2 (FP64).
// BATCH (complex64): eight entries of a thread at a time.
// ---------------------------------------------------------------------------
template <typename T, bool BATCH>
__global__ void __launch_bounds__(256) residual_kernel(const cx<T>* __restrict__ X, const cx<T>* AX, const double* theta,
                                                       cx<T>* R, double* norms, int nvec, size_t L) {
  const int j = blockIdx.y;
  const T th = (T)theta[j];
  // squares summed per thread in FP64.  complex64: two FP64 conversions and
  // additions per entry bound the kernel at 0.80 ms for 16 columns of 3 128^3;
  // eight entries at a time it takes 0.37 (columns of at least as many a thread).
  double rr = 0.0, xx = 0.0;
  const cx<T>* x = X + (size_t)j * L;
  const cx<T>* ax = AX + (size_t)j * L;
  cx<T>* r = R + (size_t)j * L;
  const size_t first = (size_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (size_t)gridDim.x * blockDim.x;
  if constexpr (BATCH) {
    for (size_t l0 = first; l0 < L; l0 += 8 * stride) {
      cx<T> xv[8], av[8];   // R may be AX: all eight are read before any is written
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const size_t l = l0 + u * stride;
        xv[u] = l < L ? x[l] : mk((T)0, (T)0);
        av[u] = l < L ? ax[l] : mk((T)0, (T)0);
      }
      float qr[8], qx[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const size_t l = l0 + u * stride;
        const cx<T> rv = mk(fma(-th, xv[u].x, av[u].x), fma(-th, xv[u].y, av[u].y));
        if (l < L) r[l] = rv;
        qr[u] = l < L ? norm2(rv) : 0.f;   // theta may be Inf or NaN
        qx[u] = norm2(xv[u]);
      }
      add_squares(rr, qr);
      add_squares(xx, qx);
    }
  } else {
    for (size_t l = first; l < L; l += stride) {
      const cx<T> xv = x[l], av = ax[l];
      const cx<T> rv = mk(fma(-th, xv.x, av.x), fma(-th, xv.y, av.y));
      r[l] = rv;
      if constexpr (sizeof(T) == 4) {
        rr += (double)norm2(rv);
        xx += (double)norm2(xv);
      } else {
        rr = fma(rv.x, rv.x, fma(rv.y, rv.y, rr));
        xx = fma(xv.x, xv.x, fma(xv.y, xv.y, xx));
      }
    }
  }
  __shared__ double red[2][32];
  for (int o = 16; o > 0; o >>= 1) {
    rr += __shfl_down_sync(0xffffffffu, rr, o);
    xx += __shfl_down_sync(0xffffffffu, xx, o);
  }
  const int lane = threadIdx.x % 32, wid = threadIdx.x / 32;
  if (lane == 0) {
    red[0][wid] = rr;
    red[1][wid] = xx;
  }
  __syncthreads();
  if (wid == 0) {
    const int nw = blockDim.x / 32;
    rr = lane < nw ? red[0][lane] : 0.0;
    xx = lane < nw ? red[1][lane] : 0.0;
    for (int o = 16; o > 0; o >>= 1) {
      rr += __shfl_down_sync(0xffffffffu, rr, o);
      xx += __shfl_down_sync(0xffffffffu, xx, o);
    }
    if (lane == 0) {
      atomicAdd(&norms[j], rr);
      atomicAdd(&norms[nvec + j], xx);
    }
  }
}

// ---------------------------------------------------------------------------
// The residual of the mixed-precision refinement, R_j = AX_j - theta_j X_j,
// from the FP64 X and AX, stored rounded to complex64, with X_j rounded to
// complex64 alongside and ||R_j||^2, ||X_j||^2 summed from the rounded
// values (FP32 within a thread, FP64 across threads).  The difference is
// formed in double-float on the FP32 pipes: every FP64 operand split into
// FP32 hi + lo, theta x as TwoProd of the hi parts plus the cross terms,
// ax - theta x by TwoSum (Knuth), about 2^-48 of |ax| before the final
// rounding to FP32, the same as FP64 for a result stored in FP32 (GB300's
// FP64 pipes made the FP64 form three times slower than the memory traffic).
// ---------------------------------------------------------------------------
__device__ __forceinline__ float dd_residual(float ah, float al, float th, float tl, float xh, float xl) {
  const float p = __fmul_rn(th, xh);
  float e = fmaf(th, xh, -p);   // p + e == th * xh exactly
  e = fmaf(th, xl, e);
  e = fmaf(tl, xh, e);
  const float sm = __fsub_rn(ah, p);   // TwoSum(ah, -p)
  const float bb = __fsub_rn(sm, ah);
  const float err = __fadd_rn(__fsub_rn(ah, __fsub_rn(sm, bb)), __fsub_rn(-p, bb));
  const float lo = __fadd_rn(__fsub_rn(al, e), err);
  return __fadd_rn(sm, lo);
}

__global__ void __launch_bounds__(256) residual_mixed_kernel(const double2* __restrict__ X, const double2* AX,
                                                             const double* theta, float2* R32, float2* X32,
                                                             double* norms, int nvec, size_t L) {
  const int j = blockIdx.y;
  float th, tl;
  dfloat::split(theta[j], th, tl);
  float rrf = 0.f, xxf = 0.f;
  const double2* x = X + (size_t)j * L;
  const double2* ax = AX + (size_t)j * L;
  float2* r = R32 + (size_t)j * L;
  float2* x32 = X32 + (size_t)j * L;
  for (size_t l = (size_t)blockIdx.x * blockDim.x + threadIdx.x; l < L; l += (size_t)gridDim.x * blockDim.x) {
    const double2 xv = x[l], av = ax[l];
    float xh, xl, yh, yl, ah, al, bh, bl;
    dfloat::split(xv.x, xh, xl);
    dfloat::split(xv.y, yh, yl);
    dfloat::split(av.x, ah, al);
    dfloat::split(av.y, bh, bl);
    const float rx = dd_residual(ah, al, th, tl, xh, xl), ry = dd_residual(bh, bl, th, tl, yh, yl);
    const float x0 = __fadd_rn(xh, xl), x1 = __fadd_rn(yh, yl);
    r[l] = make_float2(rx, ry);
    x32[l] = make_float2(x0, x1);
    rrf = fmaf(rx, rx, fmaf(ry, ry, rrf));
    xxf = fmaf(x0, x0, fmaf(x1, x1, xxf));
  }
  double rr = rrf, xx = xxf;
  __shared__ double red[2][32];
  for (int o = 16; o > 0; o >>= 1) {
    rr += __shfl_down_sync(0xffffffffu, rr, o);
    xx += __shfl_down_sync(0xffffffffu, xx, o);
  }
  const int lane = threadIdx.x % 32, wid = threadIdx.x / 32;
  if (lane == 0) {
    red[0][wid] = rr;
    red[1][wid] = xx;
  }
  __syncthreads();
  if (wid == 0) {
    const int nw = blockDim.x / 32;
    rr = lane < nw ? red[0][lane] : 0.0;
    xx = lane < nw ? red[1][lane] : 0.0;
    for (int o = 16; o > 0; o >>= 1) {
      rr += __shfl_down_sync(0xffffffffu, rr, o);
      xx += __shfl_down_sync(0xffffffffu, xx, o);
    }
    if (lane == 0) {
      atomicAdd(&norms[j], rr);
      atomicAdd(&norms[nvec + j], xx);
    }
  }
}

// ---------------------------------------------------------------------------
// Seeded complex Gaussian fill: SplitMix64 hash of (seed, index) -> two
// uniforms -> Box-Muller (uses the CUDA math library's log, sqrt, sincos).
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint64_t splitmix(uint64_t z) {
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

template <typename T>
__global__ void fill_random_kernel(cx<T>* X, size_t total, uint64_t seed) {
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const uint64_t h1 = splitmix(seed ^ splitmix(2 * e)), h2 = splitmix(seed ^ splitmix(2 * e + 1));
    const double u1 = ((h1 >> 11) + 1) * (1.0 / 9007199254740993.0);   // (0, 1]
    const double u2 = (h2 >> 11) * (1.0 / 9007199254740992.0);
    const double rad = sqrt(-2.0 * log(u1));
    double sn, cs;
    sincospi(2.0 * u2, &sn, &cs);
    X[e] = mk((T)(rad * cs), (T)(rad * sn));
  }
}

template <typename T>
__global__ void deflate_kernel(cx<T>* X, int nvec, size_t n3) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < 3 * nvec) X[(size_t)i * n3] = mk((T)0, (T)0);   // mode p = 0 of component i % 3 of vector i / 3
}

template <typename S, typename D>
__global__ void convert_kernel(const S* __restrict__ src, D* __restrict__ dst, size_t count) {
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < count; e += (size_t)gridDim.x * blockDim.x)
    dst[e] = (D)src[e];
}

// columns of even length starting on 16-byte boundaries (pairs of complex64
// entries load as one float4)
bool pair_ok(const void* S, const void* Y, size_t L) {
  return L % 2 == 0 && (reinterpret_cast<uintptr_t>(S) & 15) == 0 && (reinterpret_cast<uintptr_t>(Y) & 15) == 0;
}

// CTAs per column of the residual kernels: eight entries a thread where the
// columns are short (each CTA ends with two FP64 atomics on its column's
// norms; one entry a thread at 32^3 made 384 CTAs of them per column: 16
// complex128 columns 53 -> 27 us, 16 of 64^3 181 -> 163)
unsigned residual_grid(size_t L, int nvec) {
  const size_t fill = (152u * 4u + nvec - 1) / nvec, want = (L + 8 * 256 - 1) / (8 * 256);
  return (unsigned)std::max<size_t>(std::min<size_t>((L + 255) / 256, fill), std::min<size_t>(want, 152u * 4u));
}

unsigned grid_for(size_t work, int threads, unsigned cap = 152u * 32u) {
  return (unsigned)std::max<size_t>(1, std::min<size_t>((work + threads - 1) / threads, cap));
}

}  // namespace

namespace {
std::atomic<int> g_gram_path{0};
}  // namespace

void set_gram_path(int path) { g_gram_path.store(path); }
int get_gram_path() { return g_gram_path.load(); }

cudaError_t launch_gram(const void* A, int na, const void* B, int nb, size_t L, int precision, double* G,
                        cudaStream_t s) {
  if (precision == PCX_FP64) return launch_gram_digits(A, na, B, PCX_FP64, nb, L, G, s);
  const int path = g_gram_path.load();
  const bool cc = L > 0 && gram_cc_supported(A, B, na, nb, L);
  const bool tc = L > 0 && gram_tc_supported(na, nb, L);
  if (cc && (path == 2 || (path == 0 && gram_fp32_pipes_faster(A == B && na == nb, na, nb))))
    return launch_gram_cc(A, na, B, nb, L, G, s);
  if (tc && path != 2) return launch_gram_tc(A, na, B, nb, L, G, s);
  if (cc) return launch_gram_cc(A, na, B, nb, L, G, s);
  return launch_gram_cuda_cores(A, na, B, nb, L, G, s);
}

cudaError_t launch_gram_cuda_cores(const void* A, int na, const void* B, int nb, size_t L, double* G, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(G, 0, sizeof(double) * 2 * (size_t)na * nb, s);
  if (e != cudaSuccess) return e;
  if (L == 0) return cudaSuccess;
  const int tile = GT;
  const int rows_step = GL;
  const unsigned gx = (na + tile - 1) / tile, gy = (nb + tile - 1) / tile;
  // enough CTAs to fill the GPU several times over
  const size_t want = std::max<size_t>(1, (size_t)152 * 8 / (gx * gy));
  size_t rows = (L + want - 1) / want;
  rows = ((rows + rows_step - 1) / rows_step) * rows_step;
  const unsigned gz = (unsigned)((L + rows - 1) / rows);
  dim3 grid(gx, gy, gz);
  gram_kernel<float><<<grid, 256, 0, s>>>(static_cast<const cx<float>*>(A), na, static_cast<const cx<float>*>(B), nb,
                                          L, rows, G);
  return cudaGetLastError();
}

cudaError_t launch_combine(const void* S, int ns, const double* C, int ny, double beta, void* Y, size_t L,
                           int precision, cudaStream_t s) {
  if (L == 0) return cudaSuccess;
  if (precision == PCX_FP64) {
    // sweeps of equal width, at most 16 outputs each
    const int sweeps = (ny + 15) / 16, width = sweeps ? (ny + sweeps - 1) / sweeps : 0;
    for (int j0 = 0; j0 < ny; j0 += width) {
      const int nyl = std::min(width, ny - j0);
      auto run = nyl <= 4 ? run_combine_ff<4> : nyl <= 8 ? run_combine_ff<8> : nyl <= 12 ? run_combine_ff<12>
                                                                                        : run_combine_ff<16>;
      cudaError_t e = run(S, ns, C, ny, j0, nyl, beta, Y, L, s);
      if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
  }
  const int threads = 256;
  const unsigned blocks = grid_for(L, threads, 152u * 8u);
  for (int j0 = 0; j0 < ny; j0 += CY) {
    if (pair_ok(S, Y, L)) {
      const size_t smem = (size_t)(RING * 256 + ns * CY) * sizeof(float4);
      cudaError_t e = raise_dyn_smem(reinterpret_cast<const void*>(combine2_kernel<false>), smem);
      if (e != cudaSuccess) return e;
      combine2_kernel<false><<<grid_for(L / 2, threads, 152u * 2u), threads, smem, s>>>(
          static_cast<const float4*>(S), ns, C, ny, j0, beta, Y, L / 2);
    } else {
      const size_t smem = (size_t)ns * CY * sizeof(cx<float>);
      combine_kernel<float><<<blocks, threads, smem, s>>>(static_cast<const cx<float>*>(S), ns, C, ny, j0, beta,
                                                          static_cast<cx<float>*>(Y), L);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_combine_add32(const void* S32, int ns, const double* C, int ny, void* Y64, size_t L,
                                cudaStream_t s) {
  if (L == 0) return cudaSuccess;
  const unsigned blocks = grid_for(L, 256, 152u * 8u);
  const bool pairs = pair_ok(S32, Y64, L);
  for (int j0 = 0; j0 < ny; j0 += CY) {
    cudaError_t e = cudaSuccess;
    if (pairs) {
      const size_t smem = (size_t)(RING * 256 + ns * CY) * sizeof(float4);
      if ((e = raise_dyn_smem(reinterpret_cast<const void*>(combine2_kernel<true>), smem)) != cudaSuccess) return e;
      combine2_kernel<true><<<grid_for(L / 2, 256, 152u * 2u), 256, smem, s>>>(static_cast<const float4*>(S32), ns,
                                                                              C, ny, j0, 0.0, Y64, L / 2);
    } else {
      combine_add32_kernel<<<blocks, 256, (size_t)ns * CY * sizeof(cx<float>), s>>>(
          static_cast<const cx<float>*>(S32), ns, C, ny, j0, static_cast<double2*>(Y64), L);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_residual(const void* X, const void* AX, const double* theta, void* R, double* norms, int nvec,
                            size_t L, int precision, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(norms, 0, sizeof(double) * 2 * nvec, s);
  if (e != cudaSuccess || nvec == 0) return e;
  dim3 grid(std::max(1u, residual_grid(L, nvec)), nvec);
  if (precision == PCX_FP64) {
    residual_kernel<double, false><<<grid, 256, 0, s>>>(static_cast<const cx<double>*>(X),
                                                        static_cast<const cx<double>*>(AX), theta,
                                                        static_cast<cx<double>*>(R), norms, nvec, L);
  } else {
    const auto kern = L >= (size_t)8 * 256 * grid.x ? residual_kernel<float, true> : residual_kernel<float, false>;
    kern<<<grid, 256, 0, s>>>(static_cast<const cx<float>*>(X), static_cast<const cx<float>*>(AX), theta,
                              static_cast<cx<float>*>(R), norms, nvec, L);
  }
  return cudaGetLastError();
}

cudaError_t launch_residual_mixed(const void* X, const void* AX, const double* theta, void* R32, void* X32,
                                  double* norms, int nvec, size_t L, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(norms, 0, sizeof(double) * 2 * nvec, s);
  if (e != cudaSuccess || nvec == 0) return e;
  dim3 grid(std::max(1u, residual_grid(L, nvec)), nvec);
  residual_mixed_kernel<<<grid, 256, 0, s>>>(static_cast<const double2*>(X), static_cast<const double2*>(AX), theta,
                                             static_cast<float2*>(R32), static_cast<float2*>(X32), norms, nvec, L);
  return cudaGetLastError();
}

cudaError_t launch_fill_random(void* X, int nvec, size_t L, uint64_t seed, int precision, cudaStream_t s) {
  const size_t total = (size_t)nvec * L;
  if (total == 0) return cudaSuccess;
  if (precision == PCX_FP64)
    fill_random_kernel<double><<<grid_for(total, 256), 256, 0, s>>>(static_cast<cx<double>*>(X), total, seed);
  else
    fill_random_kernel<float><<<grid_for(total, 256), 256, 0, s>>>(static_cast<cx<float>*>(X), total, seed);
  return cudaGetLastError();
}

cudaError_t launch_deflate_p0(void* X, int nvec, int n, int precision, cudaStream_t s) {
  if (nvec == 0) return cudaSuccess;
  const size_t n3 = (size_t)n * n * n;
  const unsigned blocks = (3 * nvec + 127) / 128;
  if (precision == PCX_FP64)
    deflate_kernel<double><<<blocks, 128, 0, s>>>(static_cast<cx<double>*>(X), nvec, n3);
  else
    deflate_kernel<float><<<blocks, 128, 0, s>>>(static_cast<cx<float>*>(X), nvec, n3);
  return cudaGetLastError();
}

cudaError_t launch_convert(const void* src, int src_prec, void* dst, int dst_prec, size_t count, cudaStream_t s) {
  // count = number of complex entries
  const size_t reals = 2 * count;
  if (reals == 0) return cudaSuccess;
  const unsigned blocks = grid_for(reals, 256);
  if (src_prec == PCX_FP32 && dst_prec == PCX_FP64)
    convert_kernel<float, double><<<blocks, 256, 0, s>>>(static_cast<const float*>(src), static_cast<double*>(dst), reals);
  else if (src_prec == PCX_FP64 && dst_prec == PCX_FP32)
    convert_kernel<double, float><<<blocks, 256, 0, s>>>(static_cast<const double*>(src), static_cast<float*>(dst), reals);
  else
    return cudaMemcpyAsync(dst, src, reals * (src_prec == PCX_FP64 ? 8 : 4), cudaMemcpyDeviceToDevice, s);
  return cudaGetLastError();
}

}  // namespace pcx
