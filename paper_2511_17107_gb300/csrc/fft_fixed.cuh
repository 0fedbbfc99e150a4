// The complex128 passes of the apply with their 1D transforms in 64-bit
// fixed point.
//
// GB300 issues 2 FP64 operations per clock and SM against 64 integer
// multiply-adds and about 90 64-bit integer additions, and the FFTs are two
// thirds of the passes' FP64 operations.  A line (one pencil of one component)
// is converted to integers relative to its largest entry, transformed, and
// converted back; the work per mode and per cell between the transforms (C^H,
// M, C w + gamma conj(kappa)(kappa.x)) stays in FP64.
//
// Line format.  No partial sum of a transform is larger than the sum of the
// moduli of the line's entries, so the scale comes from that sum: E is the
// line's largest biased exponent (|re|, |im| < 2^(E - 1022)), S >= sum(|re| +
// |im|) is taken to 21 bits below 2^E, b = bit length of S in those units, and
// an entry becomes round(v 2^(61 - (E - 1022 - 21 + b))).  Every partial sum
// then stays below 2^61 (its real and imaginary part added or subtracted,
// below 2^61.5), no stage scales or overflows, and additions are exact.  What
// is lost is half a unit per entry of the input, and at most 1.8 (rms 0.5)
// units per twiddle product.  Against extended precision, lines of 16 to 256
// points: 0.35 to 0.6 of the error of the same transform in FP64, whether the
// entries are even, fall off with the index (powers 1, 2, 4) or are one large
// among small ones.  (A scale from the largest entry and N alone, one step
// shorter, wastes what the growth does not use: 1.0 to 7.5 times the error of
// FP64 at 256 points, up to 2.8 times at 128.)
//
// Twiddles are 2^61 cos and 2^61 sin split into signed limbs of 31 bits; a
// complex product is 12 wide multiply-adds (the products of two low limbs, up
// to a unit each, are left out).  A line with Inf or NaN gives NaN throughout.
#pragma once

#include "fft_kernels.cuh"

namespace pcx {
namespace fftk {
namespace fixed {

using ll = long long;
using cxl = cx<ll>;

struct Twid {
  int ch, cl, sh, sl;   // 2^61 cos = ch 2^31 + cl, 2^61 sin = sh 2^31 + sl
};
__device__ __forceinline__ void limbs(ll v, int& h, int& l) {
  l = (int)((unsigned)v << 1) >> 1;
  h = (int)((v - l) >> 31);
}
__device__ __forceinline__ Twid make_twid(cx<double> w) {
  Twid t;
  limbs(__double2ll_rn(w.x * 2305843009213693952.0), t.ch, t.cl);
  limbs(__double2ll_rn(w.y * 2305843009213693952.0), t.sh, t.sl);
  return t;
}

__device__ __forceinline__ ll wide(int a, int b) { return (ll)a * b; }
// (hi 2^62 + mid 2^31) 2^-61, rounded
__device__ __forceinline__ ll join(ll hi, ll mid) { return 2 * hi + ((mid + (1ll << 29)) >> 30); }

// v * (cos + i DIR sin), |v| < 2^62
template <int DIR>
__device__ __forceinline__ cxl rotate(cxl v, const Twid& t) {
  const int xh = (int)(v.x >> 31), xl = (int)(v.x & 0x7fffffff);
  const int yh = (int)(v.y >> 31), yl = (int)(v.y & 0x7fffffff);
  const int sh = DIR > 0 ? t.sh : -t.sh, sl = DIR > 0 ? t.sl : -t.sl;
  const int nh = -sh, nl = -sl;
  cxl r;
  r.x = join(wide(xh, t.ch) + wide(yh, nh), wide(xh, t.cl) + wide(xl, t.ch) + wide(yh, nl) + wide(yl, nh));
  r.y = join(wide(xh, sh) + wide(yh, t.ch), wide(xh, sl) + wide(xl, sh) + wide(yh, t.cl) + wide(yl, t.ch));
  return r;
}
// v sqrt(1/2)
__device__ __forceinline__ ll root_half(ll v) {
  constexpr int H = 759250125, L = -12858223;   // 2^61 sqrt(1/2) = H 2^31 + L
  const int h = (int)(v >> 31), l = (int)(v & 0x7fffffff);
  return join(wide(h, H), wide(h, L) + wide(l, H));
}
// v exp(DIR 2 pi i M / 8)
template <int DIR, int M>
__device__ __forceinline__ cxl rot8(cxl v) {
  if constexpr (M == 0) return v;
  else if constexpr (M == 2) return DIR > 0 ? mk<ll>(-v.y, v.x) : mk<ll>(v.y, -v.x);
  else {
    const ll a = DIR > 0 ? v.x - v.y : v.x + v.y;   // sqrt(2) times the real part of the rotation by pi / 4
    const ll b = DIR > 0 ? v.x + v.y : v.y - v.x;   // and the imaginary part
    const cxl r = mk<ll>(root_half(a), root_half(b));
    if constexpr (M == 1) return r;
    else return DIR > 0 ? mk<ll>(-r.y, r.x) : mk<ll>(r.y, -r.x);   // M = 3: another quarter turn
  }
}
// in-register DFT of length R = 4 or 8 (as dft in cx.cuh)
template <int R, int DIR>
__device__ __forceinline__ void dft_fixed(cxl* v) {
  static_assert(R == 4 || R == 8, "radix");
  constexpr int B = ilog2(R);
  cxl t[R];
  static_for<R>([&](auto i) { t[decltype(i)::value] = v[bitrev(decltype(i)::value, B)]; });
  static_for<B>([&](auto lg) {
    constexpr int LEN = 2 << decltype(lg)::value;
    static_for<R / LEN>([&](auto blk) {
      static_for<LEN / 2>([&](auto kk) {
        constexpr int K = decltype(kk)::value;
        constexpr int A = decltype(blk)::value * LEN + K;
        const cxl a = t[A];
        const cxl b = rot8<DIR, K * (8 / LEN)>(t[A + LEN / 2]);
        t[A] = a + b;
        t[A + LEN / 2] = a - b;
      });
    });
  });
  static_for<R>([&](auto i) { v[decltype(i)::value] = t[decltype(i)::value]; });
}

__device__ __forceinline__ int exp_bits(cx<double> v) {
  const uint32_t x = (uint32_t)(__double_as_longlong(v.x) >> 32) & 0x7fffffffu;
  const uint32_t y = (uint32_t)(__double_as_longlong(v.y) >> 32) & 0x7fffffffu;
  return (int)((x > y ? x : y) >> 20);
}
// A line's scale: its largest biased exponent e >= 1, and the sum of its
// entries' parts in units of 2^(e - 1043), each rounded up.
struct __align__(8) Line {
  int e;
  unsigned sum;
};
__device__ __forceinline__ unsigned coarse(double v, int E) {
  const uint32_t hi = (uint32_t)(__double_as_longlong(v) >> 32) & 0x7fffffffu;
  const int e = (int)(hi >> 20);
  const uint32_t m = (hi & 0xfffffu) | (e ? 0x100000u : 0u);
  return (m >> min(E - (e ? e : 1), 31)) + 1u;
}
// K = e + b - 21: an entry is v 2^(1083 - K), below 2^61
__device__ __forceinline__ int line_scale(Line l) { return l.e + 11 - __clz((int)l.sum); }
// round(v 2^(1083 - K))
__device__ __forceinline__ ll to_fixed(double v, int K) {
  const ll b = __double_as_longlong(v);
  const int e = (int)(b >> 52) & 0x7ff;
  const unsigned long long m = ((unsigned long long)b & 0xfffffffffffffull) | (e ? 0x10000000000000ull : 0ull);
  const int d = min(K - (e ? e : 1), 63);
  const ll q = (ll)(((m << 9) >> d) + 1) >> 1;
  const ll s = b >> 63;
  return (q ^ s) - s;
}
// v 2^e rounded to a double
__device__ __forceinline__ double to_double(ll v, int e) {
  const ll s = v >> 63;
  const unsigned long long m = (unsigned long long)((v ^ s) - s);
  const int lz = __clzll((ll)m);
  const unsigned long long n = (m << (lz & 63)) + 0x400ull;   // leading bit at 63, half a unit added; m < 2^62
  const int carry = n < 0x400ull;                             // all ones rounded up
  const int ex = 1023 + 63 + e - lz + carry;
  unsigned long long bits = ((unsigned long long)(unsigned)ex << 52) | (((n << carry) >> 11) & 0xfffffffffffffull);
  if (ex >= 2047) bits = 0x7ffull << 52;
  if (ex <= 0) {   // below the normal range: a multiple of 2^-1074
    const int d = -1074 - e;
    bits = d > 0 ? ((m >> (d - 1)) + 1) >> 1 : m << -d;
  }
  if (m == 0) bits = 0;
  return __longlong_as_double((ll)bits | (s & (ll)(1ull << 63)));
}
// an entry of a line as doubles, times 2^SHIFT
template <int SHIFT = 0>
__device__ __forceinline__ cx<double> line_value(cxl v, Line l) {
  const double bad = __longlong_as_double(0x7ff8000000000000ll);
  if (l.e == 2047) return mk(bad, bad);
  const int e = line_scale(l) - 1083 + SHIFT;
  return mk(to_double(v.x, e), to_double(v.y, e));
}

// One Stockham stage (as fftk::stage).  SRC: 0 fixed-point tile; 1 global
// memory, 2 tile holding doubles (first stage: finds the lines' scales and
// converts).  DST: 0 fixed-point tile, 1 global memory (last stage: converts
// back).  line[c TP + t]: the scale of line t of component c.
template <int N, int AXIS, int R, int DIR, int SRC, int DST>
__device__ __forceinline__ void stage_fixed(cxl* s, const Twid* tw, Line* line, int Ns, const cx<double>* gin,
                                            cx<double>* gout, int qb) {
  using C = Cfg<double, N>;
  using TL = Tile<double, N, AXIS>;
  constexpr int NB = N / R, PER = C::E / R, N3 = N * N * N, TP = C::TP;
  constexpr int NL = NB < 32 ? NB : 32;   // lanes of a line (x tiles: neighbours)
  cxl v[PER][R];
  if constexpr (SRC == 0) {
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      int t, j, c;
      TL::item(threadIdx.x + i * C::THREADS, NB, t, j, c);
#pragma unroll
      for (int r = 0; r < R; ++r) v[i][r] = s[TL::sidx(c, t, j + r * NB)];
    }
    if constexpr (DST == 0) __syncthreads();
  } else {
    cx<double> d[PER][R];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      int t, j, c;
      TL::item(threadIdx.x + i * C::THREADS, NB, t, j, c);
      int e = 1;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if constexpr (SRC == 1) d[i][r] = gin[c * N3 + TL::gidx(qb + t, j + r * NB)];
        else d[i][r] = reinterpret_cast<const cx<double>*>(s)[TL::sidx(c, t, j + r * NB)];
      }
#pragma unroll
      for (int r = 0; r < R; ++r) e = max(e, exp_bits(d[i][r]));
      if constexpr (AXIS == 0) {
#pragma unroll
        for (int o = NL / 2; o > 0; o >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
        if (j % NL == 0) atomicMax(&line[c * TP + t].e, e);
      } else {
        atomicMax(&line[c * TP + t].e, e);
      }
    }
    __syncthreads();   // exponents (and every read of a tile of doubles)
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      int t, j, c;
      TL::item(threadIdx.x + i * C::THREADS, NB, t, j, c);
      const int E = line[c * TP + t].e;
      unsigned sum = 0;   // 2 R parts of at most 2^21, 2 N <= 512 of them in a line
#pragma unroll
      for (int r = 0; r < R; ++r) sum += coarse(d[i][r].x, E) + coarse(d[i][r].y, E);
      if constexpr (AXIS == 0) {
#pragma unroll
        for (int o = NL / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (j % NL == 0) atomicAdd(&line[c * TP + t].sum, sum);
      } else {
        atomicAdd(&line[c * TP + t].sum, sum);
      }
    }
    __syncthreads();   // sums
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      int t, j, c;
      TL::item(threadIdx.x + i * C::THREADS, NB, t, j, c);
      const int K = line_scale(line[c * TP + t]);
#pragma unroll
      for (int r = 0; r < R; ++r) v[i][r] = mk(to_fixed(d[i][r].x, K), to_fixed(d[i][r].y, K));
    }
  }
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    int t, j, c;
    TL::item(threadIdx.x + i * C::THREADS, NB, t, j, c);
    const int k = j % Ns;
    if (SRC == 0 && Ns > 1) {
      const int step = N / (Ns * R);
#pragma unroll
      for (int r = 1; r < R; ++r) v[i][r] = rotate<-DIR>(v[i][r], tw[r * k * step]);   // tw: exp(-2 pi i m / N)
    }
    dft_fixed<R, DIR>(v[i]);
    const int base = (j / Ns) * Ns * R + k;
    if constexpr (DST == 1) {
      const Line l = line[c * TP + t];
      cx<double>* g = gout + (c * N3 + TL::gidx(qb + t, base));
#pragma unroll
      for (int r = 0; r < R; ++r) g[r * Ns * TL::GSTRIDE] = line_value(v[i][r], l);
    } else {
#pragma unroll
      for (int r = 0; r < R; ++r) s[TL::sidx(c, t, base + r * Ns)] = v[i][r];
    }
  }
  if constexpr (DST == 0) __syncthreads();
}

template <int N, int AXIS, int DIR, int SRC, int DST>
__device__ __forceinline__ void fft_fixed(cxl* s, const Twid* tw, Line* line, const cx<double>* gin, cx<double>* gout,
                                          int qb) {
  using P = typename Cfg<double, N>::P;
  if constexpr (P::NST == 1) {
    stage_fixed<N, AXIS, P::R0, DIR, SRC, DST>(s, tw, line, 1, gin, gout, qb);
  } else if constexpr (P::NST == 2) {
    stage_fixed<N, AXIS, P::R0, DIR, SRC, 0>(s, tw, line, 1, gin, gout, qb);
    stage_fixed<N, AXIS, P::R1, DIR, 0, DST>(s, tw, line, P::R0, gin, gout, qb);
  } else {
    stage_fixed<N, AXIS, P::R0, DIR, SRC, 0>(s, tw, line, 1, gin, gout, qb);
    stage_fixed<N, AXIS, P::R1, DIR, 0, 0>(s, tw, line, P::R0, gin, gout, qb);
    stage_fixed<N, AXIS, P::R2, DIR, 0, DST>(s, tw, line, P::R0 * P::R1, gin, gout, qb);
  }
}

// The passes of pass_kernel (fft_kernels.cuh) for complex128: the same tiles,
// tables and pointwise arithmetic, the transforms by fft_fixed.
template <int N, int AXIS, int OP>
__global__ void __launch_bounds__(Cfg<double, N>::THREADS, 2) pass_fixed_kernel(PassArgs a) {
  using C = Cfg<double, N>;
  using TL = Tile<double, N, AXIS>;
  using D = cx<double>;
  constexpr int TP = C::TP, N2 = N * N, N3 = N2 * N;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cxl* s = reinterpret_cast<cxl*>(smem_raw);
  D* sd = reinterpret_cast<D*>(s);
  Twid* tw = reinterpret_cast<Twid*>(s + 3 * C::CS);
  D* ka = reinterpret_cast<D*>(tw + N);   // [3][N], then [TP][3] (see pass_kernel)
  D* kb = ka + 3 * N;
  double* mtab = reinterpret_cast<double*>(kb + 3 * TP);   // z sandwich: material table, ids; x POST: scratch tile
  __shared__ Line line[2][3 * TP];

  const size_t q0 = (size_t)blockIdx.x * TP;
  const size_t v = q0 / N2;
  const int qb = (int)(q0 % N2);
  const D* in = static_cast<const D*>(a.in) + v * 3 * N3;
  D* out = static_cast<D*>(a.out) + v * 3 * N3;

  const D* gtw = static_cast<const D*>(a.tw);
  for (int i = threadIdx.x; i < N; i += C::THREADS) tw[i] = make_twid(gtw[i]);
  for (int i = threadIdx.x; i < 2 * 3 * TP; i += C::THREADS) line[0][i] = Line{1, 0u};
  KParams kp = a.kp;
  if (AXIS == 0 && a.kps) kp = a.kps[(a.v_base + (int)v) / a.vec_per_k];
  if constexpr (AXIS == 0 && OP != OP_PLAIN_INV && OP != OP_PLAIN_FWD)
    pass_kappa_tables<double, N>(static_cast<const D*>(a.lam), kp, qb, ka, kb);
  if constexpr (OP == OP_SANDWICH || OP == OP_SANDWICH_EPS) {
    if (a.mid) {
      const double* gt = static_cast<const double*>(a.mtab);
      for (int i = threadIdx.x; i < 9 * a.n_mat; i += C::THREADS) mtab[i] = gt[i];
    }
  }

  if constexpr (OP == OP_PLAIN_INV || OP == OP_PLAIN_FWD || OP == OP_INV || OP == OP_FWD) {
    __syncthreads();
    fft_fixed<N, AXIS, OP == OP_PLAIN_INV || OP == OP_INV ? +1 : -1, 1, 1>(s, tw, line[0], in, out, qb);
  } else if constexpr (OP == OP_PRE || OP == OP_PRE_T0) {
    for (int e = threadIdx.x; e < TP * N; e += C::THREADS) {
      const int t = e / N, n = e % N;
      const int g = TL::gidx(qb + t, n);
#pragma unroll
      for (int c = 0; c < 3; ++c) cp_async_cx<double>(&sd[TL::sidx(c, t, n)], &in[c * N3 + g]);
    }
    cp_async_commit_wait_all();
    __syncthreads();
    D* sb = static_cast<D*>(a.sbuf) + v * N3;
    const double gam = kp.gamma, igam = 1.0 / kp.gamma;
    for (int e = threadIdx.x; e < TP * N; e += C::THREADS) {
      const int t = e / N, n = e % N;
      pre_point<double, OP == OP_PRE_T0>(sd[TL::sidx(0, t, n)], sd[TL::sidx(1, t, n)], sd[TL::sidx(2, t, n)],
                                         sb[TL::gidx(qb + t, n)], ka + n, N, kb + 3 * t, kp, gam, igam);
    }
    __syncthreads();
    fft_fixed<N, 0, +1, 2, 1>(s, tw, line[0], nullptr, out, qb);
  } else if constexpr (OP == OP_POST || OP == OP_POST_T0) {
    const D* sb = static_cast<const D*>(a.sbuf) + v * N3;
    D* ssb = kb + 3 * TP;   // [TP * N]
    for (int e = threadIdx.x; e < TP * N; e += C::THREADS) {
      const int t = e / N, n = e % N;
      cp_async_cx<double>(&ssb[e], &sb[TL::gidx(qb + t, n)]);
    }
    __syncthreads();   // twiddles, scales
    fft_fixed<N, 0, -1, 1, 0>(s, tw, line[0], in, nullptr, qb);
    cp_async_commit_wait_all();
    __syncthreads();
    for (int e = threadIdx.x; e < TP * N; e += C::THREADS) {
      const int t = e / N, n = e % N;
      D w[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) w[c] = line_value(s[TL::sidx(c, t, n)], line[0][c * TP + t]);
      const int g = TL::gidx(qb + t, n);
      post_point<double, OP == OP_POST_T0>(w, ssb[e], ka + n, N, kb + 3 * t, out[g], out[N3 + g], out[2 * N3 + g]);
    }
  } else {
    // z axis: inverse transform, M per cell in FP64, forward transform
    static_assert(OP == OP_SANDWICH || OP == OP_SANDWICH_EPS, "z sandwich");
    const double* M = static_cast<const double*>(a.M);
    const uchar4* mid = static_cast<const uchar4*>(a.mid);
    uchar4* sid = reinterpret_cast<uchar4*>(mtab + 9 * a.n_mat);   // [TP * N]
    if (mid) {
      for (int w = threadIdx.x; w < TP * N; w += C::THREADS) {
        const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(&sid[w]));
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(&mid[(w / TP) * N2 + (qb + w % TP)])
                     : "memory");
      }
    }
    __syncthreads();   // twiddles, scales
    fft_fixed<N, 2, +1, 1, 0>(s, tw, line[0], in, nullptr, qb);
    cp_async_commit_wait_all();
    __syncthreads();
    for (int w = threadIdx.x; w < TP * N; w += C::THREADS) {   // pencils fastest
      const int t = w % TP, n = w / TP;
      D e[3];
#pragma unroll
      for (int c = 0; c < 3; ++c)   // with the transforms' 1 / N^3
        e[c] = line_value<-3 * ilog2(N)>(s[TL::sidx(c, t, n)], line[0][c * TP + t]);
      cell_point<double, N, OP == OP_SANDWICH_EPS>(e, mid ? &sid[w] : nullptr, mtab, M, n * N2 + (qb + t), 1.0);
#pragma unroll
      for (int c = 0; c < 3; ++c) sd[TL::sidx(c, t, n)] = e[c];
    }
    __syncthreads();
    fft_fixed<N, 2, -1, 2, 1>(s, tw, line[1], nullptr, out, qb);
  }
}

}  // namespace fixed
}  // namespace fftk
}  // namespace pcx
