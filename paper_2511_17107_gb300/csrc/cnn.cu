// Kernels of the learned preconditioner correction, which acts next to eps
// inside the curl-sandwich base preconditioner T0:
//
//   T(r) = T0 r + K_A F3_3^H g(F3_3 K_A^H r / |k|^2) / |k|^2
//
// with g a three-layer circular 3D convolution net (3 x 3 x 3 taps) on the
// real-space field, its hidden channels gated by sigmoid convolutions of the
// 9 reals of the per-cell blocks of M (Sec. 3.2.1).  The net acts on the real
// and imaginary parts of the complex field with shared weights, so T is
// complex-linear.  The paper has no learned component; the operator pieces
// it wraps are eqs. matrixfree_diagP / matrixfree_finalform (K_P^{-1}) and
// the Fourier basis x = F3_3^H H of Sec. 2.4.
//
// Arithmetic and accumulation are FP32; the convolutions optionally round
// their weights to BF16 as they load them (the learned form's BF16 flag).  A convolution CTA
// produces an 8 x 8 x 8 tile of output voxels for every output channel of
// one sample, from a 10 x 10 x 10 halo tile of all input channels staged in
// shared memory (periodic wrap on load; rows of 10 padded to 12 floats, so
// that a row loads in 16-byte pieces).  The weight gradient is a per-CTA sum
// over tiles written to scratch and reduced in a fixed order.
//
// Both convolutions wait for shared memory: counters at 64^3 (2 vectors, 8 -> 8
// channels) show the forward kernel at 79% of the shared-memory pipe and 24% of the
// FMA pipe, the weight gradient at 53% and 46% with a quarter of the warps
// resident.  So both make the loads per FMA few: the forward kernel keeps four voxels of a row for every output
// channel in registers (8 loads per 96 FMAs; two voxels took 10 per 48), the
// weight gradient nine taps of one (output, input) channel pair while it
// walks down the rows of a plane (5 loads per 72 FMAs; one thread per weight
// took 2 per FMA).  Halo rows are staged whole (two 16-byte loads and two
// edges) rather than voxel by voxel.  Measured at 64^3, 16 samples, 8 -> 8
// channels: forward 464 -> 358 us, weight gradient 2,569 -> 423 us; the
// gradient of 8 vectors in the Hermitian form 14.9 -> 6.1 ms.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "cnn.h"
#include "cx.cuh"
#include "pcx_internal.h"

namespace pcx {
namespace cnn {
namespace {

constexpr int TS = 8;                 // output tile edge
constexpr int HS = TS + 2;            // halo tile edge
constexpr int HV = HS * HS * HS;      // halo voxels
constexpr int TV = TS * TS * TS;      // tile voxels
constexpr int CT = 128;               // threads per forward CTA (4 voxels of a row each)
constexpr int XR = 12;                // floats per staged row
constexpr int XC = HS * HS * XR + 4;  // floats per staged channel: channels 20 banks apart

__device__ __forceinline__ long long voff(const View& t, int b, int ch, long long v) {
  return (long long)(b / t.split) * t.s_hi + (long long)(b % t.split) * t.s_lo + (long long)ch * t.sc + v * t.sv;
}

__device__ __forceinline__ void tile_origin(int tile, int n, int& z0, int& y0, int& x0) {
  const int tpa = n / TS;
  z0 = (tile / (tpa * tpa)) * TS;
  y0 = ((tile / tpa) % tpa) * TS;
  x0 = (tile % tpa) * TS;
}

// four consecutive voxels of a channel (16-byte access where the view allows it)
__device__ __forceinline__ bool quads(const View& t) {
  return t.sv == 1 && ((reinterpret_cast<unsigned long long>(t.p) & 15) | ((t.s_hi | t.s_lo | t.sc) & 3)) == 0;
}
__device__ __forceinline__ float4 load4(const View& t, int b, int ch, long long v, bool quad) {
  const float* p = t.p + voff(t, b, ch, v);
  if (quad) return *reinterpret_cast<const float4*>(p);
  return make_float4(p[0], p[t.sv], p[2 * t.sv], p[3 * t.sv]);
}
__device__ __forceinline__ void store4(const View& t, int b, int ch, long long v, bool quad, float4 r) {
  float* p = t.p + voff(t, b, ch, v);
  if (quad) {
    *reinterpret_cast<float4*>(p) = r;
  } else {
    p[0] = r.x;
    p[t.sv] = r.y;
    p[2 * t.sv] = r.z;
    p[3 * t.sv] = r.w;
  }
}

// Stage channels [0, CIN) of sample b around the tile at (z0, y0, x0), by
// NT threads, a row of ten voxels each: channel ci's voxel (hz, hy, hx) at
// sx[ci XC + (hz HS + hy) XR + hx].
template <int CIN, int NT>
__device__ __forceinline__ void load_halo(float* sx, const View& in, int b, int n, int z0, int y0, int x0) {
  const int mask = n - 1;   // n is a power of two
  const float* p = in.p + voff(in, b, 0, 0);
  const bool quad = quads(in);
  const int xl = (x0 - 1) & mask, xr = (x0 + TS) & mask;
#pragma unroll 2
  for (int e = threadIdx.x; e < CIN * HS * HS; e += NT) {
    const int ci = e / (HS * HS), hz = (e / HS) % HS, hy = e % HS;
    const int gz = (z0 - 1 + hz) & mask, gy = (y0 - 1 + hy) & mask;
    const float* row = p + (long long)ci * in.sc + ((long long)gz * n + gy) * n * in.sv;
    float* d = sx + ci * XC + (hz * HS + hy) * XR;
    float v[TS];
    if (quad) {
      const float4 q0 = *reinterpret_cast<const float4*>(row + x0), q1 = *reinterpret_cast<const float4*>(row + x0 + 4);
      v[0] = q0.x, v[1] = q0.y, v[2] = q0.z, v[3] = q0.w;
      v[4] = q1.x, v[5] = q1.y, v[6] = q1.z, v[7] = q1.w;
    } else {
#pragma unroll
      for (int i = 0; i < TS; ++i) v[i] = row[(x0 + i) * in.sv];
    }
    d[0] = row[xl * in.sv];
    d[TS + 1] = row[xr * in.sv];
#pragma unroll
    for (int i = 0; i < TS; ++i) d[1 + i] = v[i];
  }
}

// out[b][co] = conv(in[b], w)[co]            (MODE_PLAIN), times out_scale
// out[b][co] = conv(in[b], w)[co] * gate[co] (MODE_GATE; pre-gate value to pre)
// out[b][co] = sigmoid(conv(in[b], w)[co] + bias[co])   (MODE_SIGMOID)
template <int CIN, int COUT, int MODE>
__global__ void __launch_bounds__(CT) conv_fwd_kernel(View in, View out, const float* __restrict__ w,
                                                      const float* __restrict__ bias, View gate, View pre, int n,
                                                      float out_scale, int wbf16) {
  // Each thread produces four neighbouring voxels along x for every output
  // channel.  The weights sit in shared memory as [ci][tap][co] (co padded
  // to a multiple of 4), so one 16-byte broadcast load feeds 16 FMAs, and
  // the six input values of a halo row serve the three x taps of the voxels.
  // Output channels go in pairs through the packed FMA.
  constexpr int CP = (COUT + 3) / 4 * 4;
  static_assert(TV == 4 * CT, "four voxels per thread");
  extern __shared__ __align__(16) float cf_smem[];
  float* sx = cf_smem;               // [CIN][XC]
  float* sw = cf_smem + CIN * XC;    // [CIN][27][CP]
  const int b = blockIdx.y;
  int z0, y0, x0;
  tile_origin(blockIdx.x, n, z0, y0, x0);
  for (int i = threadIdx.x; i < CIN * 27 * CP; i += CT) {
    const int co = i % CP, t = (i / CP) % 27, ci = i / (CP * 27);
    float wv = co < COUT ? w[(co * CIN + ci) * 27 + t] : 0.f;
    if (wbf16) wv = __bfloat162float(__float2bfloat16_rn(wv));   // BF16 weights, FP32 accumulation
    sw[i] = wv;
  }
  load_halo<CIN, CT>(sx, in, b, n, z0, y0, x0);
  __syncthreads();
  const int lz = threadIdx.x / (TS * TS / 4), ly = (threadIdx.x / (TS / 4)) % TS, lx = 4 * (threadIdx.x % (TS / 4));
  float2 a[4][CP / 2];
#pragma unroll
  for (int v = 0; v < 4; ++v)
#pragma unroll
    for (int q = 0; q < CP / 2; ++q) a[v][q] = make_float2(0.f, 0.f);
#pragma unroll 1
  for (int ci = 0; ci < CIN; ++ci) {
#pragma unroll
    for (int dz = 0; dz < 3; ++dz)
#pragma unroll
      for (int dy = 0; dy < 3; ++dy) {
        const float* row = sx + ci * XC + ((lz + dz) * HS + (ly + dy)) * XR + lx;
        const float4 r4 = *reinterpret_cast<const float4*>(row);
        const float2 r2 = *reinterpret_cast<const float2*>(row + 4);
        const float2 xr[6] = {make_float2(r4.x, r4.x), make_float2(r4.y, r4.y), make_float2(r4.z, r4.z),
                              make_float2(r4.w, r4.w), make_float2(r2.x, r2.x), make_float2(r2.y, r2.y)};
#pragma unroll
        for (int dx = 0; dx < 3; ++dx) {
          const float4* wt = reinterpret_cast<const float4*>(&sw[(ci * 27 + dz * 9 + dy * 3 + dx) * CP]);
#pragma unroll
          for (int q = 0; q < CP / 4; ++q) {
            const float4 w4 = wt[q];
            const float2 w01 = make_float2(w4.x, w4.y), w23 = make_float2(w4.z, w4.w);
#pragma unroll
            for (int v = 0; v < 4; ++v) {
              fma2(a[v][2 * q], w01, xr[dx + v]);
              fma2(a[v][2 * q + 1], w23, xr[dx + v]);
            }
          }
        }
      }
  }
  const long long gv = ((long long)(z0 + lz) * n + (y0 + ly)) * n + (x0 + lx);
  const bool qo = quads(out), qg = MODE == MODE_GATE && quads(gate), qp = MODE == MODE_GATE && pre.p && quads(pre);
#pragma unroll
  for (int co = 0; co < COUT; ++co) {
    float4 r = co & 1 ? make_float4(a[0][co / 2].y, a[1][co / 2].y, a[2][co / 2].y, a[3][co / 2].y)
                      : make_float4(a[0][co / 2].x, a[1][co / 2].x, a[2][co / 2].x, a[3][co / 2].x);
    if constexpr (MODE == MODE_SIGMOID) {
      const float bc = bias[co];
      r.x = 1.f / (1.f + expf(-(r.x + bc)));
      r.y = 1.f / (1.f + expf(-(r.y + bc)));
      r.z = 1.f / (1.f + expf(-(r.z + bc)));
      r.w = 1.f / (1.f + expf(-(r.w + bc)));
    } else if constexpr (MODE == MODE_GATE) {
      if (pre.p) store4(pre, b, co, gv, qp, r);
      const float4 g4 = load4(gate, b, co, gv, qg);
      r.x *= g4.x;
      r.y *= g4.y;
      r.z *= g4.z;
      r.w *= g4.w;
    }
    r.x *= out_scale;
    r.y *= out_scale;
    r.z *= out_scale;
    r.w *= out_scale;
    store4(out, b, co, gv, qo, r);
  }
}

// partial[blockIdx.x][co][ci][t] = sum over the CTA's (sample, tile) jobs of
// sum_v dy[b][co][v] x[b][ci][v + offset_t].  Thread (pair, g): the 27 taps of
// one channel pair (co, ci) over the planes g, g + WG, ... of every tile; a
// plane's products are summed on their own before they join the thread's
// totals, and the WG totals of a pair are added at the end.
constexpr int DC = TV + 4;   // floats per staged channel of dy
template <int CIN, int COUT>
struct WGrad {
  static constexpr int PAIRS = CIN * COUT;
  static constexpr int WG = PAIRS <= 32 ? 8 : (PAIRS <= 64 ? 4 : 2);   // thread groups (planes in flight)
  static constexpr int NT = PAIRS * WG;
  static constexpr int TILE = CIN * XC + COUT * DC;                                       // floats
  static constexpr int SMEM = TILE > PAIRS * WG * 27 ? TILE : PAIRS * WG * 27;            // floats
};
template <int CIN, int COUT>
__global__ void __launch_bounds__(WGrad<CIN, COUT>::NT, 2) conv_wgrad_kernel(View dy, View x, int nb, int n,
                                                                            float* __restrict__ partial) {
  using W = WGrad<CIN, COUT>;
  extern __shared__ __align__(16) float wg_smem[];
  float* sx = wg_smem;              // [CIN][XC]
  float* sd = wg_smem + CIN * XC;   // [COUT][DC]
  const int tiles = (n / TS) * (n / TS) * (n / TS);
  const int pair = threadIdx.x % W::PAIRS, g = threadIdx.x / W::PAIRS;
  const int co = pair % COUT, ci = pair / COUT;
  float tot[27];
#pragma unroll
  for (int t = 0; t < 27; ++t) tot[t] = 0.f;
  for (long long job = blockIdx.x; job < (long long)nb * tiles; job += gridDim.x) {
    const int b = (int)(job / tiles), tile = (int)(job % tiles);
    int z0, y0, x0;
    tile_origin(tile, n, z0, y0, x0);
    __syncthreads();   // the previous job's tiles are consumed
    load_halo<CIN, W::NT>(sx, x, b, n, z0, y0, x0);
    const float* dp = dy.p + voff(dy, b, 0, 0);
    const bool quad = quads(dy);
    for (int e = threadIdx.x; e < COUT * TS * TS; e += W::NT) {
      const int c = e / (TS * TS), lz = (e / TS) % TS, ly = e % TS;
      const float* row = dp + (long long)c * dy.sc + (((long long)(z0 + lz) * n + (y0 + ly)) * n + x0) * dy.sv;
      float4 q0, q1;
      if (quad) {
        q0 = *reinterpret_cast<const float4*>(row);
        q1 = *reinterpret_cast<const float4*>(row + 4);
      } else {
        const int v = dy.sv;
        q0 = make_float4(row[0], row[v], row[2 * v], row[3 * v]);
        q1 = make_float4(row[4 * v], row[5 * v], row[6 * v], row[7 * v]);
      }
      float4* d = reinterpret_cast<float4*>(sd + c * DC + (lz * TS + ly) * TS);
      d[0] = q0;
      d[1] = q1;
    }
    __syncthreads();
#pragma unroll 1
    for (int z = g; z < TS; z += W::WG) {
      const float* dz_row = sd + co * DC + z * TS * TS;
#pragma unroll
      for (int tz = 0; tz < 3; ++tz) {
        const float* plane = sx + ci * XC + (z + tz) * HS * XR;
        float acc[9];
#pragma unroll
        for (int t = 0; t < 9; ++t) acc[t] = 0.f;
        float row[3][HS];
        auto load_row = [&](float* r, int y) {
          const float4 p0 = *reinterpret_cast<const float4*>(plane + y * XR);
          const float4 p1 = *reinterpret_cast<const float4*>(plane + y * XR + 4);
          const float2 p2 = *reinterpret_cast<const float2*>(plane + y * XR + 8);
          r[0] = p0.x, r[1] = p0.y, r[2] = p0.z, r[3] = p0.w;
          r[4] = p1.x, r[5] = p1.y, r[6] = p1.z, r[7] = p1.w;
          r[8] = p2.x, r[9] = p2.y;
        };
        load_row(row[0], 0);
        load_row(row[1], 1);
#pragma unroll
        for (int y = 0; y < TS; ++y) {
          load_row(row[(y + 2) % 3], y + 2);
          const float4 d0 = *reinterpret_cast<const float4*>(dz_row + y * TS);
          const float4 d1 = *reinterpret_cast<const float4*>(dz_row + y * TS + 4);
          const float d[TS] = {d0.x, d0.y, d0.z, d0.w, d1.x, d1.y, d1.z, d1.w};
#pragma unroll
          for (int ty = 0; ty < 3; ++ty)
#pragma unroll
            for (int tx = 0; tx < 3; ++tx)
#pragma unroll
              for (int v = 0; v < TS; ++v) acc[3 * ty + tx] = fmaf(d[v], row[(y + ty) % 3][v + tx], acc[3 * ty + tx]);
        }
#pragma unroll
        for (int t = 0; t < 9; ++t) tot[9 * tz + t] += acc[t];
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int t = 0; t < 27; ++t) wg_smem[(g * W::PAIRS + pair) * 27 + t] = tot[t];
  __syncthreads();
  for (int e = threadIdx.x; e < W::PAIRS * 27; e += W::NT) {
    const int c = e / (CIN * 27), i = (e / 27) % CIN, t = e % 27;   // output order [co][ci][t]
    float r = 0.f;
#pragma unroll
    for (int k = 0; k < W::WG; ++k) r += wg_smem[(k * W::PAIRS + i * COUT + c) * 27 + t];
    partial[(size_t)blockIdx.x * W::PAIRS * 27 + e] = r;
  }
}

// out[e] (+)= sum_c partial[c][e], summed in FP64 in a fixed order: 32 entries
// per CTA, its eight warps striding over the partials.
constexpr int RP = 8;
__global__ void __launch_bounds__(32 * RP) reduce_partials_kernel(const float* __restrict__ partial, int nparts, int ne,
                                                                  float* __restrict__ out, int accumulate) {
  __shared__ double red[RP][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, e = blockIdx.x * 32 + lane;
  double s = 0.0;
  if (e < ne)
    for (int c = w; c < nparts; c += RP) s += (double)partial[(size_t)c * ne + e];
  red[w][lane] = s;
  __syncthreads();
  if (w == 0 && e < ne) {
    s = 0.0;
#pragma unroll
    for (int k = 0; k < RP; ++k) s += red[k][lane];
    out[e] = accumulate ? (float)((double)out[e] + s) : (float)s;
  }
}

// wt[ci][co][26 - t] = w[co][ci][t]: the weights of the adjoint convolution
__global__ void adjoint_weights_kernel(const float* __restrict__ w, int cout, int cin, float* __restrict__ wt) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= cout * cin * 27) return;
  const int co = e / (cin * 27), ci = (e / 27) % cin, t = e % 27;
  wt[(ci * cout + co) * 27 + (26 - t)] = w[e];
}

// dz[c][v] = (sum_b dh[b][c][v] a[b][c][v]) g (1 - g);  dh[b][c][v] *= g
__global__ void gate_backward_kernel(View dh, View a, const float* __restrict__ g, int nb, int c, size_t n3,
                                     float* __restrict__ dz) {
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < (size_t)c * n3;
       e += (size_t)gridDim.x * blockDim.x) {
    const int ch = (int)(e / n3);
    const long long v = (long long)(e % n3);
    const float gg = g[e];
    float s = 0.f;
    for (int b = 0; b < nb; ++b) {
      const long long o = voff(dh, b, ch, v);
      const float d = dh.p[o];
      s = fmaf(d, a.p[voff(a, b, ch, v)], s);
      dh.p[o] = d * gg;
    }
    dz[e] = s * gg * (1.f - gg);
  }
}

// part[ch][blockIdx.x] = sum of a stretch of dz[ch], FP64; bias_sum_kernel adds
// the stretches in a fixed order: db[ch] (+)= sum_v dz[ch][v]
constexpr int BP = 32;   // stretches per channel
__global__ void __launch_bounds__(256) bias_grad_kernel(const float* __restrict__ dz, size_t n3, double* __restrict__ part) {
  __shared__ double red[8];
  const int ch = blockIdx.y;
  double s = 0.0;
  for (size_t v = (size_t)blockIdx.x * 256 + threadIdx.x; v < n3; v += (size_t)BP * 256) s += (double)dz[(size_t)ch * n3 + v];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += red[w];
    part[ch * BP + blockIdx.x] = t;
  }
}
__global__ void bias_sum_kernel(const double* __restrict__ part, int c, float* __restrict__ db, int accumulate) {
  const int ch = threadIdx.x;
  if (ch >= c) return;
  double t = 0.0;
  for (int k = 0; k < BP; ++k) t += part[ch * BP + k];
  db[ch] = accumulate ? (float)((double)db[ch] + t) : (float)t;
}

// dY = 2 w_v (Y - T); loss += sum w_v |Y - T|^2  (complex64 blocks, floats)
__global__ void loss_grad_kernel(const float* __restrict__ Y, const float* __restrict__ T,
                                 const double* __restrict__ wv, size_t per_vec, size_t total, float* __restrict__ dY,
                                 double* __restrict__ loss) {
  __shared__ double red[32];
  double s = 0.0;
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const double w = wv[e / per_vec];
    const float d = Y[e] - T[e];
    dY[e] = (float)(2.0 * w) * d;
    s += w * (double)d * (double)d;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    atomicAdd(loss, t);
  }
}

// f[0..8][v]: d1, d2, d3, Re/Im M_12, Re/Im M_13, Re/Im M_23 of cell v
__global__ void features_kernel(const uchar4* __restrict__ mid, const float* __restrict__ mtab,
                                const float* __restrict__ dense, size_t n3, float* __restrict__ f) {
  for (size_t v = (size_t)blockIdx.x * blockDim.x + threadIdx.x; v < n3; v += (size_t)gridDim.x * blockDim.x) {
    if (mid) {
      const uchar4 id = mid[v];
      f[v] = mtab[9 * id.x];
      f[n3 + v] = mtab[9 * id.y + 1];
      f[2 * n3 + v] = mtab[9 * id.z + 2];
#pragma unroll
      for (int j = 3; j < 9; ++j) f[j * n3 + v] = mtab[9 * id.w + j];
    } else {
#pragma unroll
      for (int j = 0; j < 9; ++j) f[j * n3 + v] = dense[j * n3 + v];
    }
  }
}

__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, int np, float lr, float b1, float b2, float eps, float c1,
                            float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= np) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// SplitMix64 (Steele, Lea, Flood 2014) of the counter, two uniforms, Box-Muller
__device__ __forceinline__ unsigned long long mix64(unsigned long long z) {
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__global__ void init_kernel(float* __restrict__ p, unsigned long long seed) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= NPARAMS) return;
  const unsigned long long h1 = mix64(seed ^ mix64(2ull * (unsigned long long)i));
  const unsigned long long h2 = mix64(seed ^ mix64(2ull * (unsigned long long)i + 1ull));
  const double u1 = ((double)(h1 >> 11) + 0.5) * (1.0 / 9007199254740992.0);
  const double u2 = (double)(h2 >> 11) * (1.0 / 9007199254740992.0);
  const double z = sqrt(-2.0 * log(u1)) * cos(6.283185307179586 * u2);
  double scale;
  if (i < OFF_W2) scale = 1.0 / sqrt(3.0 * 27.0);
  else if (i < OFF_W3) scale = 1.0 / sqrt((double)HIDDEN * 27.0);
  else if (i < OFF_V1) scale = 0.0;   // the correction starts at zero: T = K_P^{-1}
  else if (i < OFF_C1) scale = 1.0 / sqrt(9.0 * 27.0);
  else if (i < OFF_V2) scale = 0.0;
  else if (i < OFF_C2) scale = 1.0 / sqrt(9.0 * 27.0);
  else scale = 0.0;
  p[i] = (float)(scale * z);
}

__global__ void lincomb_kernel(const float* __restrict__ x, float alpha, const float* __restrict__ y, float beta,
                               float* __restrict__ z, size_t n) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    z[i] = y ? fmaf(alpha, x[i], beta * y[i]) : alpha * x[i];
}

__global__ void col_dots_kernel(const float2* __restrict__ a, const float2* __restrict__ b, size_t len,
                                double* __restrict__ dots) {
  __shared__ double red[2][32];
  const int v = blockIdx.y;
  const float2* av = a + (size_t)v * len;
  const float2* bv = b + (size_t)v * len;
  double re = 0.0, im = 0.0;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < len; i += (size_t)gridDim.x * blockDim.x) {
    const float2 x = av[i], y = bv[i];
    re += (double)x.x * y.x + (double)x.y * y.y;
    im += (double)x.x * y.y - (double)x.y * y.x;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    re += __shfl_xor_sync(0xffffffffu, re, o);
    im += __shfl_xor_sync(0xffffffffu, im, o);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = re;
    red[1][threadIdx.x >> 5] = im;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double tr = 0.0, ti = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      tr += red[0][w];
      ti += red[1][w];
    }
    atomicAdd(dots + 2 * v, tr);
    atomicAdd(dots + 2 * v + 1, ti);
  }
}

__global__ void col_axpby_kernel(const double* __restrict__ alpha, const float2* __restrict__ x,
                                 const double* __restrict__ beta, float2* __restrict__ y, size_t len) {
  const int v = blockIdx.y;
  const float al = (float)alpha[v], be = (float)beta[v];
  const float2* xv = x + (size_t)v * len;
  float2* yv = y + (size_t)v * len;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < len; i += (size_t)gridDim.x * blockDim.x) {
    const float2 a = xv[i], b = yv[i];
    yv[i] = make_float2(fmaf(al, a.x, be * b.x), fmaf(al, a.y, be * b.y));
  }
}

unsigned grid_for(size_t n, int threads, unsigned cap) {
  size_t b = (n + threads - 1) / threads;
  if (b < 1) b = 1;
  return (unsigned)(b > cap ? cap : b);
}

}  // namespace

// ---- host launchers ---------------------------------------------------------

#define PCX_CONV_CASE(CI, CO, MD)                                                                          \
  if (cin == CI && cout == CO && mode == MD) {                                                             \
    const size_t smem = (size_t)(CI * XC + CI * 27 * ((CO + 3) / 4 * 4)) * sizeof(float);                  \
    cudaError_t e = raise_dyn_smem(reinterpret_cast<const void*>(conv_fwd_kernel<CI, CO, MD>), smem);      \
    if (e != cudaSuccess) return e;                                                                        \
    conv_fwd_kernel<CI, CO, MD><<<grid, CT, smem, s>>>(in, out, w, bias, gate, pre, n, out_scale, wbf16); \
    return cudaGetLastError();                                                                             \
  }

cudaError_t conv_fwd(int cin, int cout, int mode, const View& in, const View& out, const float* w, const float* bias,
                     const View& gate, const View& pre, int nb, int n, float out_scale, cudaStream_t s, int wbf16) {
  if (n < TS || (n & (n - 1)) != 0 || nb < 1 || nb > 65535) return cudaErrorInvalidValue;
  const dim3 grid((unsigned)((n / TS) * (n / TS) * (n / TS)), (unsigned)nb);
  PCX_CONV_CASE(3, HIDDEN, MODE_GATE)
  PCX_CONV_CASE(HIDDEN, HIDDEN, MODE_GATE)
  PCX_CONV_CASE(HIDDEN, 3, MODE_PLAIN)
  PCX_CONV_CASE(9, HIDDEN, MODE_SIGMOID)
  PCX_CONV_CASE(3, HIDDEN, MODE_PLAIN)
  PCX_CONV_CASE(HIDDEN, HIDDEN, MODE_PLAIN)
  return cudaErrorInvalidValue;
}
#undef PCX_CONV_CASE

size_t wgrad_scratch_floats(int cin, int cout) { return (size_t)4 * 152 * cout * cin * 27; }

template <int CIN, int COUT>
static cudaError_t wgrad_t(const View& dy, const View& x, int nb, int n, float* dw, int accumulate, float* scratch,
                           cudaStream_t s) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const long long jobs = (long long)nb * (n / TS) * (n / TS) * (n / TS);
  long long grid = 2LL * (sms < 152 ? sms : 152);
  if (grid > jobs) grid = jobs;
  const size_t smem = (size_t)WGrad<CIN, COUT>::SMEM * sizeof(float);
  if ((e = raise_dyn_smem(reinterpret_cast<const void*>(conv_wgrad_kernel<CIN, COUT>), smem)) != cudaSuccess) return e;
  conv_wgrad_kernel<CIN, COUT><<<(unsigned)grid, WGrad<CIN, COUT>::NT, smem, s>>>(dy, x, nb, n, scratch);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  constexpr int NE = COUT * CIN * 27;
  reduce_partials_kernel<<<(NE + 31) / 32, 32 * RP, 0, s>>>(scratch, (int)grid, NE, dw, accumulate);
  return cudaGetLastError();
}

cudaError_t conv_wgrad(int cin, int cout, const View& dy, const View& x, int nb, int n, float* dw, int accumulate,
                       float* scratch, cudaStream_t s) {
  if (n < TS || (n & (n - 1)) != 0 || nb < 1) return cudaErrorInvalidValue;
  if (cin == HIDDEN && cout == 3) return wgrad_t<HIDDEN, 3>(dy, x, nb, n, dw, accumulate, scratch, s);
  if (cin == HIDDEN && cout == HIDDEN) return wgrad_t<HIDDEN, HIDDEN>(dy, x, nb, n, dw, accumulate, scratch, s);
  if (cin == 3 && cout == HIDDEN) return wgrad_t<3, HIDDEN>(dy, x, nb, n, dw, accumulate, scratch, s);
  if (cin == 9 && cout == HIDDEN) return wgrad_t<9, HIDDEN>(dy, x, nb, n, dw, accumulate, scratch, s);
  return cudaErrorInvalidValue;
}

cudaError_t adjoint_weights(const float* w, int cout, int cin, float* wt, cudaStream_t s) {
  const int ne = cout * cin * 27;
  adjoint_weights_kernel<<<(ne + 255) / 256, 256, 0, s>>>(w, cout, cin, wt);
  return cudaGetLastError();
}

cudaError_t gate_backward(const View& dh, const View& a, const float* g, int nb, int c, size_t n3, float* dz,
                          cudaStream_t s) {
  gate_backward_kernel<<<grid_for((size_t)c * n3, 256, 152u * 16u), 256, 0, s>>>(dh, a, g, nb, c, n3, dz);
  return cudaGetLastError();
}

cudaError_t bias_grad(const float* dz, int c, size_t n3, float* db, int accumulate, float* scratch, cudaStream_t s) {
  double* part = reinterpret_cast<double*>(scratch);
  bias_grad_kernel<<<dim3(BP, (unsigned)c), 256, 0, s>>>(dz, n3, part);
  bias_sum_kernel<<<1, 32, 0, s>>>(part, c, db, accumulate);
  return cudaGetLastError();
}

cudaError_t loss_grad(const void* Y, const void* T, const double* wv, int nvec, size_t n3, void* dY, double* loss,
                      cudaStream_t s) {
  const size_t per = 6 * n3, total = per * (size_t)nvec;
  loss_grad_kernel<<<grid_for(total, 256, 152u * 8u), 256, 0, s>>>(static_cast<const float*>(Y),
                                                                   static_cast<const float*>(T), wv, per, total,
                                                                   static_cast<float*>(dY), loss);
  return cudaGetLastError();
}

cudaError_t features(const pcx_ctx* c, float* f, cudaStream_t s) {
  const size_t n3 = (size_t)c->n * c->n * c->n;
  const uchar4* mid = static_cast<const uchar4*>(c->dev.mid);
  features_kernel<<<grid_for(n3, 256, 152u * 16u), 256, 0, s>>>(mid, static_cast<const float*>(c->dev.mtab32),
                                                                static_cast<const float*>(c->dev.m32), n3, f);
  return cudaGetLastError();
}

cudaError_t adam(float* p, const float* g, float* m, float* v, int np, int step, float lr, float b1, float b2, float eps,
                 cudaStream_t s) {
  const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
  adam_kernel<<<(np + 255) / 256, 256, 0, s>>>(p, g, m, v, np, lr, b1, b2, eps, c1, c2);
  return cudaGetLastError();
}

cudaError_t init_params(float* p, unsigned long long seed, cudaStream_t s) {
  init_kernel<<<(NPARAMS + 255) / 256, 256, 0, s>>>(p, seed);
  return cudaGetLastError();
}

cudaError_t lincomb(const float* x, float alpha, const float* y, float beta, float* z, size_t nfloat, cudaStream_t s) {
  lincomb_kernel<<<grid_for(nfloat, 256, 152u * 16u), 256, 0, s>>>(x, alpha, y, beta, z, nfloat);
  return cudaGetLastError();
}

cudaError_t col_dots(const void* a, const void* b, int nvec, size_t len, double* dots, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(dots, 0, sizeof(double) * 2 * (size_t)nvec, s);
  if (e != cudaSuccess || nvec == 0) return e;
  const dim3 grid(grid_for(len, 256, 152u * 4u), (unsigned)nvec);
  col_dots_kernel<<<grid, 256, 0, s>>>(static_cast<const float2*>(a), static_cast<const float2*>(b), len, dots);
  return cudaGetLastError();
}

cudaError_t col_axpby(const double* alpha, const void* x, const double* beta, void* y, int nvec, size_t len,
                      cudaStream_t s) {
  if (nvec == 0) return cudaSuccess;
  const dim3 grid(grid_for(len, 256, 152u * 4u), (unsigned)nvec);
  col_axpby_kernel<<<grid, 256, 0, s>>>(alpha, static_cast<const float2*>(x), beta, static_cast<float2*>(y), len);
  return cudaGetLastError();
}

}  // namespace cnn
}  // namespace pcx
