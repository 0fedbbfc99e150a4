// Gram products G = A^H B (Sec. 4: the Rayleigh-Ritz matrices of LOBPCG) with
// A complex128 and B complex128 or complex64, by integer digits on the tensor
// cores (splitting a product into exact tensor-core products: Ozaki, Ogita,
// Oishi and Rump, Numer. Algorithms 59 (2012) 95; Mukunoki et al., ISC High
// Performance 2020).  The mixed product gives the rows X^H [P W] of the
// refinement, whose entries are far below the FP32 rounding of the products.
//
// In every chunk of KC = 32 rows a column gets an exponent E (|re|, |im| <
// 2^E in the chunk) and its entries become signed fixed-point integers of 49
// bits below 2^E, cut into five balanced digits of base 2^10.  A digit lies
// in [-512, 512] and is exact in half precision, so the product of two digit
// columns on mma.sync (FP16 operands, FP32 accumulators) is a sum of integers
// of at most 2^18.  Digit pairs (i, j) of one weight g = i + j share an
// accumulator; pairs beyond g = 4 are left out.  Over the rows of a chunk the
// sums of groups 0 and 1 are at most 2^24 and exact; those of later groups
// could pass 2^24 only where all digits are near their limit in every row,
// and round by units 2^-38 and less then.  The chunk sums join double-float
// sums (FP32 pairs) whose unit follows the columns' largest exponents so far.
//
// Accuracy.  The pairs left out and the rounding of the entries come to 2^-50
// 2^(Ea + Eb) rms in a product of two reals, so an entry of G is off by about
// 2^-47.5 sqrt(sum over rows of (M_c M'_c)^2), M_c the largest part of the
// column in the row's chunk, and each chunk's addition rounds 2^-49 of the
// running sum.  Exponents per chunk, and sums that float, keep columns that
// are graded against each other accurate (A falling and B rising, so that all
// rows weigh alike): only what falls inside 32 rows counts.  Largest error of
// G over ||A_i|| ||B_j||, 16 x 43 columns of 3 128^3 rows falling off with
// the mode as |p|^-power (powers of A, B), double-float sums / this kernel:
// (0, 0) 4.8e-16 / 2e-17, (1, 1) 2.6e-15 / 1.2e-16, (2, 2) 1.3e-13 / 5.8e-15,
// (4, 4) 1.1e-13 / 1.6e-14, (2, 0) 4.3e-16 / 2.8e-17; complex64 B (2, 2)
// 2.2e-12 / 4.9e-15.  Over sum |a||b| with opposite powers (2, -2) 6.1e-16 /
// 5e-17, (4, -4) 6.4e-16 / 2.4e-14, and one entry 1000 times all others in
// both columns 5e-15 / 8e-15 (1.4e-14 at 3 64^3).
//
// The complex product is a real one over stacked columns, D = [Ar Ai]^T
// [Br Bi]: Re G = D[i][j] + D[n+i][m+j], Im G = D[i][m+j] - D[n+i][j].  For
// A^H A, D is symmetric, one digit set serves both operands and only the
// tiles on and above the diagonal are formed.
//
// One CTA walks a range of rows in chunks of 32.  Half of its warps cut the
// next chunk into digits (integer and FP64 pipes: one FMA per real), the
// other half multiply the current one (tensor pipe; a warp owns up to MT
// 16 x 16 tiles of D); hardware named barriers hand two digit buffers over.
// Raw rows arrive by cp.async two chunks ahead, in slots private to the
// thread that cuts them.
//
// What bounds it at 48 x 48: issue slots and latency of 16 warps (counters at 3 64^3
// rows: tensor pipe 41%, no pipe above, SM throughput 58%; mma.sync peaks at 1,036
// multiply-adds per clock and SM, measured); beside the products the multiplying
// warps add the chunk sums, 20 FP32 operations each.  Narrow products wait for the
// cutting warps (16 x 16: tensor pipe 20%, FP64 pipe 45%).  Measured at 3 128^3 rows (GB300):
// complex128 48 x 48 30.4 ms in double-float on the FP32 pipes, 7.2 ms here;
// 16 x 16 3.46 and 1.58 ms; complex128 x complex64 16 x 32 4.93 and 2.21 ms.
// (64-bit integer sums of one unit per column, with one conversion per digit
// group, took 6.65, 1.51 and 2.10 ms, but were off by 2e-11 of sum |a||b| for
// powers (4, -4) and by 1.9e-13 beside one large entry.)
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>
#include <type_traits>

#include "cx.cuh"
#include "dfloat.cuh"
#include "pcx_internal.h"
#include "stream_scratch.h"

namespace pcx {
namespace {

constexpr int KC = 32;                 // rows per chunk
constexpr int MAXC = 48;               // columns of A or B per launch
constexpr int NS = 5;                  // digits
constexpr int DB = 10;                 // bits per digit
constexpr int MB = DB - 1 + DB * (NS - 1);   // magnitude bits of the fixed-point value
constexpr int UNIT_BITS = 2 * (DB - 1);   // a product of leading digits has the unit 2^(Ea + Eb - UNIT_BITS)
constexpr long long MAX_ROWS = 16000;  // rows per CTA: longer columns take more waves
constexpr int E_MIN = 128;             // smallest exponent of a complex128 column (biased): keeps 2^(MB - E) finite

template <typename T>
struct Entry;
template <>
struct Entry<double> {
  using C = double2;
  static constexpr int BIAS = 1022;   // a value of biased exponent e is below 2^(e - BIAS)
  static constexpr int BAD = 2047;    // exponent of Inf and NaN
};
template <>
struct Entry<float> {
  using C = float2;
  static constexpr int BIAS = 126;
  static constexpr int BAD = 255;
};

__device__ __forceinline__ int exp_bits(double a, double b) {
  const uint32_t x = (uint32_t)(__double_as_longlong(a) >> 32) & 0x7fffffffu;
  const uint32_t y = (uint32_t)(__double_as_longlong(b) >> 32) & 0x7fffffffu;
  return (int)(max(x, y) >> 20);
}
__device__ __forceinline__ int exp_bits(float a, float b) {
  return (int)(max(__float_as_uint(a) & 0x7fffffffu, __float_as_uint(b) & 0x7fffffffu) >> 23);
}

// The fixed-point value of an entry as digit fields of DB bits, field value =
// digit + 2^(DB - 1); a leading field can be 2^DB (digit + 2^(DB - 1)).
//
// complex128: one FMA against 1.5 2^52 rounds v 2^(MB - E) to an integer in
// the low mantissa bits; half a base added to every digit balances them.
struct Fields64 {
  template <int I>
  static __device__ __forceinline__ constexpr bool leading() { return I == 0; }
  uint32_t lo, hi;
  __device__ __forceinline__ Fields64(double v, double scale) {
    // 1.5 2^52 + sum_i 512 1024^i over all digits
    constexpr double magic =
        6755399441055744.0 + (double)((1ll << (DB - 1)) * (((1ll << (DB * NS)) - 1) / ((1 << DB) - 1)));
    const unsigned long long u = (unsigned long long)__double_as_longlong(fma(v, scale, magic));
    lo = (uint32_t)u;
    hi = (uint32_t)(u >> 32);
  }
  // field I (0: leading) in the low bits, other bits above it
  template <int I>
  __device__ __forceinline__ uint32_t field() const {
    constexpr int sh = DB * (NS - 1 - I);
    if constexpr (sh == 0) return lo;
    else if constexpr (sh + DB < 32) return lo >> sh;
    else if constexpr (sh < 32) return __funnelshift_r(lo, hi, sh);
    else return hi >> (sh - 32);
  }
};
// complex64: the leading two digits by an FMA against 1.5 2^23, then two
// digits at a time of the exact remainder
struct Fields32 {
  template <int I>
  static __device__ __forceinline__ constexpr bool leading() { return (I & 1) == 0; }
  uint32_t w[3];   // two digits each (the leading one at bit DB), the last word one
  static constexpr uint32_t HALF2 = (1u << (DB - 1)) * ((1u << DB) + 1);   // half a base in two digits
  __device__ __forceinline__ Fields32(float v, float2 scale) {
    constexpr float magic = 12582912.f;
    float r = v * scale.x * scale.y;   // |r| < 2^MB
    constexpr float unit0 = (float)(1ll << (DB * (NS - 2))), unit1 = (float)(1 << DB);   // units of the words
    const float t0 = fmaf(r, 1.f / unit0, magic);
    r = fmaf(t0 - magic, -unit0, r);
    w[0] = __float_as_uint(t0) + HALF2;
    const float t1 = fmaf(r, 1.f / unit1, magic);
    r = fmaf(t1 - magic, -unit1, r);
    w[1] = __float_as_uint(t1) + HALF2;
    w[2] = __float_as_uint(r + (magic + (float)(1 << (DB - 1))));
  }
  template <int I>
  __device__ __forceinline__ uint32_t field() const {
    if constexpr (I == NS - 1) return w[NS / 2];
    else return (I & 1) ? w[I / 2] : w[I / 2] >> DB;
  }
};
template <typename T>
using Fields = std::conditional_t<sizeof(T) == 8, Fields64, Fields32>;
// 2^(MB - (E - BIAS)); as two factors for complex64, where one could not
// reach far enough
__device__ __forceinline__ double scale_of(double, int E) {
  return __hiloint2double((1023 + MB + Entry<double>::BIAS - E) << 20, 0);
}
__device__ __forceinline__ float2 scale_of(float, int E) {
  const int sh = MB + Entry<float>::BIAS - E, s1 = sh < 100 ? sh : 100;
  return make_float2(__int_as_float((127 + s1) << 23), __int_as_float((127 + sh - s1) << 23));
}

__device__ __forceinline__ uint32_t sm_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// asynchronous copy of one complex entry (zero fill when !ok)
__device__ __forceinline__ void copy_entry(uint32_t dst, const double2* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(ok ? 16u : 0u) : "memory");
}
__device__ __forceinline__ void copy_entry(uint32_t dst, const float2* src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(dst), "l"(src), "r"(ok ? 8u : 0u) : "memory");
}

// byte offset of digit pair q (rows q and q + 16 of the chunk) of real
// column r: 64-byte rows whose 16-byte pieces are swizzled so that the eight
// rows of an ldmatrix hit distinct banks
__device__ __forceinline__ int digit_off(int r, int q) {
  return r * 64 + (((q >> 2) ^ ((r >> 1) & 3)) << 4) + (q & 3) * 4;
}

__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t r[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void mma16816(float c[4], const uint32_t a[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Hardware named barriers between the cutting and the multiplying warps
template <int N>
__device__ __forceinline__ void bar_wait(int id) { asm volatile("bar.sync %0, %1;\n" ::"r"(id), "n"(N) : "memory"); }
template <int N>
__device__ __forceinline__ void bar_arrive(int id) { asm volatile("bar.arrive %0, %1;\n" ::"r"(id), "n"(N) : "memory"); }
constexpr int BAR_FULL = 1, BAR_EMPTY = 3;   // + digit buffer

// v += sigma (g[0] + 2^-10 g[1] + ... + 2^-40 g[4]), the digit groups of a
// chunk.  The first three groups are added without error (their sums are
// integers of a few more than 24 bits; what a step rounds off the next one
// takes up), the last two round 2^-24 of what is left; sigma is a power of
// two.  So a chunk's sum carries 2^-48 of itself into the running TwoSum.
using dfloat::DF;
__device__ __forceinline__ void add_chunk(DF& v, const float g[NS], float sigma) {
  constexpr float U1 = 1.f / (1 << DB), U2 = U1 * U1, U3 = U2 * U1;
  const float p = fmaf(g[1], U1, g[0]);
  const float q = fmaf(g[2], U2, fmaf(g[1], U1, -__fsub_rn(p, g[0])));
  const float h = __fadd_rn(p, q);
  const float l = fmaf(fmaf(g[4], U1, g[3]), U3, __fsub_rn(q, __fsub_rn(h, p)));
  dfloat::add(v, __fmul_rn(h, sigma), __fmul_rn(l, sigma));
}

__device__ __forceinline__ void mma16816_zero(float c[4], const uint32_t a[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};\n"
      : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}

struct DigitArgs {
  const void* A;
  const void* B;
  int na, nb;          // complex columns, at most MAXC each
  int na8, nb8;        // the same rounded up to multiples of 8
  int sym;             // A^H A: one digit set, upper tiles only
  long long L, rows;   // column length, rows per CTA (a multiple of KC)
  double* partial;     // [CTA][2 na8][2 nb8]
};

// MW multiplying warps of up to MT tiles each, SW cutting warps, CTAS CTAs
// per SM.  REG > 0: the multiplying warps take REG registers and the cutting
// warps give them up (MW = SW = 8 at 128 each: REG + cut_regs = 256).

template <typename TA, typename TB, int MW, int SW, int MT, int CTAS, int REG>
__global__ void __launch_bounds__((MW + SW) * 32, CTAS) gram_digits_kernel(DigitArgs g) {
  static_assert(REG == 0 || (MW == 8 && SW == 8 && CTAS == 1 && REG % 8 == 0), "register split");
  using CA = typename Entry<TA>::C;
  using CB = typename Entry<TB>::C;
  constexpr int THREADS = (MW + SW) * 32;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ra = 2 * g.na8, rb = 2 * g.nb8;
  const int rtot = g.sym ? ra : ra + rb;            // real columns staged
  const int pa = (g.na + 1) / 2, pb = g.sym ? 0 : (g.nb + 1) / 2;   // column pairs
  extern __shared__ __align__(128) unsigned char sm[];
  const int slice_bytes = rtot * 64, buf_bytes = NS * slice_bytes;
  // raw rows [2][pair][row half][lane]: A's pairs, then B's
  const int rawa_bytes = pa * 64 * (int)sizeof(CA), raw_bytes = rawa_bytes + pb * 64 * (int)sizeof(CB);
  unsigned char* raw = sm + 2 * buf_bytes;
  int* expo = reinterpret_cast<int*>(raw + 2 * raw_bytes);           // [3][2 MAXC]
  int* changed = expo + 3 * 2 * MAXC;                                // [3]
  int* bad = changed + 4;                                            // [2 MAXC]
  float* ratio = reinterpret_cast<float*>(bad + 2 * MAXC);           // [2][2 MAXC]: 2^(chunk's exponent - running one)
  for (int i = tid; i < 2 * buf_bytes / 16; i += THREADS) reinterpret_cast<uint4*>(sm)[i] = make_uint4(0, 0, 0, 0);
  for (int i = tid; i < 3 * 2 * MAXC; i += THREADS) {
    const bool dbl = i % (2 * MAXC) < MAXC ? sizeof(TA) == 8 : sizeof(TB) == 8;
    expo[i] = dbl ? E_MIN : 1;
  }
  for (int i = tid; i < 2 * MAXC; i += THREADS) {
    bad[i] = 0;
    ratio[i] = ratio[2 * MAXC + i] = 0.f;
  }
  if (tid < 4) changed[tid] = 0;
  __syncthreads();

  const long long l0 = (long long)blockIdx.x * g.rows;
  const long long l1 = l0 + g.rows < g.L ? l0 + g.rows : g.L;
  const int nch = l1 > l0 ? (int)((l1 - l0 + KC - 1) / KC) : 0;

  if (warp >= MW) {
    // ---- cutting warps --------------------------------------------------
    if constexpr (REG > 0) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(256 - REG));
    const int sw = warp - MW, half = lane >> 4, q = lane & 15;
    auto fetch_cols = [&](auto* base, int ncol, int npair, unsigned char* dst0, long long r0) {
      using C = std::remove_const_t<std::remove_pointer_t<decltype(base)>>;
      for (int p = sw; p < npair; p += SW) {
        const int c = 2 * p + half;
        const C* src = base + (size_t)(c < ncol ? c : 0) * g.L;
        const uint32_t dst = sm_addr(dst0 + ((size_t)p * 64 + lane) * sizeof(C));
        const bool ok0 = c < ncol && r0 < l1, ok1 = c < ncol && r0 + 16 < l1;
        copy_entry(dst, src + (ok0 ? r0 : 0), ok0);
        copy_entry(dst + 32 * (uint32_t)sizeof(C), src + (ok1 ? r0 + 16 : 0), ok1);
      }
    };
    // rows q and q + 16 of chunk f of this thread's columns
    auto fetch = [&](int f) {
      if (f < nch) {
        unsigned char* dst = raw + (f & 1) * raw_bytes;
        const long long r0 = l0 + (long long)f * KC + q;
        fetch_cols(static_cast<const CA*>(g.A), g.na, pa, dst, r0);
        fetch_cols(static_cast<const CB*>(g.B), g.nb, pb, dst + rawa_bytes, r0);
      }
      asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    // digits of NB column pairs at a time: exponents, then the cut
    auto cut_cols = [&](auto* entries, int ncol, int npair, int f, int x0, int row0, int n8, unsigned char* buf) {
      using C = std::remove_const_t<std::remove_pointer_t<decltype(entries)>>;
      using T = decltype(C::x);
      using F = Fields<T>;
      constexpr int NB = 2, EMIN = sizeof(T) == 8 ? E_MIN : 1;
      float* rt = ratio + (f & 1) * 2 * MAXC + x0;
      const int* eold = expo + ((f + 2) % 3) * 2 * MAXC + x0;
      int* enew = expo + (f % 3) * 2 * MAXC + x0;
      for (int p0 = sw; p0 < npair; p0 += NB * SW) {
        C v[NB][2];
        int E[NB], old[NB];
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          const int p = p0 + b * SW < npair ? p0 + b * SW : p0;
          v[b][0] = entries[(size_t)p * 64 + lane];
          v[b][1] = entries[(size_t)p * 64 + 32 + lane];
          old[b] = eold[2 * p + half];
        }
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          const int eb = max(exp_bits(v[b][0].x, v[b][0].y), exp_bits(v[b][1].x, v[b][1].y));
          const int m0 = __reduce_max_sync(0xffffffffu, half ? 0 : eb), m1 = __reduce_max_sync(0xffffffffu, half ? eb : 0);
          E[b] = half ? m1 : m0;
        }
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          const int p = p0 + b * SW, c = 2 * p + half;
          if (p >= npair) break;
          const bool isbad = E[b] == Entry<T>::BAD;
          E[b] = max(E[b], EMIN);
          if (q == 0 && c < ncol) {
            const int top = max(E[b], old[b]);
            enew[c] = top;
            rt[c] = __int_as_float(max(127 + E[b] - top, 0) << 23);
            if (top != old[b]) changed[f % 3] = 1;
            if (isbad) bad[x0 + c] = 1;
          }
          const auto sc = scale_of((T)0, E[b]);
#pragma unroll
          for (int part = 0; part < 2; ++part) {
            const F f0(part ? v[b][0].y : v[b][0].x, sc), f1(part ? v[b][1].y : v[b][1].x, sc);
            unsigned char* o = buf + digit_off(row0 + part * n8 + c, q);
            uint32_t d[NS];
            auto put = [&](auto ic) {
              constexpr int I = decltype(ic)::value;
              // 1024 + field as two halves, minus 1024 + 512: the digits, exact in FP16
              // (a leading field of 1024 carries into the exponent: 2048)
              constexpr bool LEAD = F::template leading<I>();
              constexpr uint32_t MSK = LEAD ? 2 * (1u << DB) - 1 : (1u << DB) - 1;
              const uint32_t a0 = f0.template field<I>() & MSK, a1 = f1.template field<I>() & MSK;
              const uint32_t w = LEAD ? (a1 << 16) + a0 + 0x64006400u : ((a1 << 16) | (a0 | 0x64006400u));
              __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&w), __float2half2_rn(1536.f));
              d[I] = *reinterpret_cast<const uint32_t*>(&h);
            };
            static_for<NS>(put);
            if (c < ncol) {
#pragma unroll
              for (int i = 0; i < NS; ++i) *reinterpret_cast<uint32_t*>(o + i * slice_bytes) = d[i];
            }
          }
        }
      }
    };
    fetch(0);
    fetch(1);
    for (int f = 0; f < nch; ++f) {
      if (f >= 2) bar_wait<THREADS>(BAR_EMPTY + (f & 1));   // the multiplying warps are done with chunk f - 2
      asm volatile("cp.async.wait_group 1;\n" ::: "memory");
      unsigned char* buf = sm + (f & 1) * buf_bytes;
      const unsigned char* rf = raw + (f & 1) * raw_bytes;
      cut_cols(reinterpret_cast<const CA*>(rf), g.na, pa, f, 0, 0, g.na8, buf);
      cut_cols(reinterpret_cast<const CB*>(rf + rawa_bytes), g.nb, pb, f, MAXC, ra, g.nb8, buf);
      __syncwarp();   // the exponents just written by two lanes are read by the whole warp in the next chunk
      bar_arrive<THREADS>(BAR_FULL + (f & 1));
      fetch(f + 2);   // into the slots just read
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    return;
  }

  // ---- multiplying warps --------------------------------------------------
  if constexpr (REG > 0) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;\n" ::"n"(REG));
  const int tr_n = ra / 16, tc_n = rb / 16;
  const int items = g.sym ? tr_n * (tr_n + 1) / 2 : tr_n * tc_n;
  int tile[MT];   // row tile << 8 | column tile (-1: none)
  DF v[MT][8];    // sums in units of 2^(running exponents - UNIT_BITS)
#pragma unroll
  for (int k = 0; k < MT; ++k) {
    int it = warp + k * MW, r = 0;
    if (it >= items) {
      tile[k] = -1;
    } else {
      if (g.sym) {
        while (it >= tr_n - r) {
          it -= tr_n - r;
          ++r;
        }
        it += r;
      } else {
        r = it / tc_n;
        it = it % tc_n;
      }
      tile[k] = r << 8 | it;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) v[k][i] = DF{0.f, 0.f};
  }
  const int gid = lane >> 2, tg = lane & 3;
  // exponent slot of a real row of A / real column of B (padding: slot of column 0, their sums are 0)
  auto slot_a = [&](int r) { const int c = r < g.na8 ? r : r - g.na8; return c < g.na ? c : 0; };
  auto slot_b = [&](int r) { const int c = r < g.nb8 ? r : r - g.nb8; return (g.sym ? 0 : MAXC) + (c < g.nb ? c : 0); };

  for (int f = 0; f < nch; ++f) {
    bar_wait<THREADS>(BAR_FULL + (f & 1));
    if (tid == 0) changed[(f + 2) % 3] = 0;   // chunk f - 1's, read by all before this barrier
    const uint32_t base = sm_addr(sm + (f & 1) * buf_bytes);
    const bool rescale = changed[f % 3] != 0;
#pragma unroll
    for (int k = 0; k < MT; ++k) {
      if (tile[k] < 0) continue;
      const int tr = tile[k] >> 8, tc = tile[k] & 255;
      if (rescale) {
        const int* e1 = expo + (f % 3) * 2 * MAXC;
        const int* e0 = expo + ((f + 2) % 3) * 2 * MAXC;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int sa = slot_a(tr * 16 + gid + 8 * ((i >> 1) & 1));
          const int sb = slot_b(tc * 16 + 8 * (i >> 2) + 2 * tg + (i & 1));
          const int sh = (e1[sa] - e0[sa]) + (e1[sb] - e0[sb]);
          const float w = __int_as_float(max(127 - sh, 0) << 23);
          v[k][i].s *= w;
          v[k][i].c *= w;
        }
      }
      float acc[NS][8];
      const int ar = tr * 16 + (lane & 15), ap = lane >> 4;
      const int br = (g.sym ? 0 : ra) + tc * 16 + (lane & 7) + ((lane >> 4) << 3), bp = (lane >> 3) & 1;
#pragma unroll
      for (int ks = 0; ks < KC / 16; ++ks) {
        const uint32_t aa = base + ar * 64 + (((2 * ks + ap) ^ ((ar >> 1) & 3)) << 4);
        const uint32_t ba = base + br * 64 + (((2 * ks + bp) ^ ((br >> 1) & 3)) << 4);
        uint32_t b[NS][4];
#pragma unroll
        for (int j = 0; j < NS; ++j) ldsm4(ba + j * slice_bytes, b[j]);
#pragma unroll
        for (int i = 0; i < NS; ++i) {
          uint32_t a[4];
          ldsm4(aa + i * slice_bytes, a);
#pragma unroll
          for (int j = 0; j < NS - i; ++j) {
            if (ks == 0 && i == 0) {
              mma16816_zero(acc[j], a, b[j][0], b[j][1]);
              mma16816_zero(acc[j] + 4, a, b[j][2], b[j][3]);
            } else {
              mma16816(acc[i + j], a, b[j][0], b[j][1]);
              mma16816(acc[i + j] + 4, a, b[j][2], b[j][3]);
            }
          }
        }
      }
      // the chunk's sums join the running ones
      const float* rt = ratio + (f & 1) * 2 * MAXC;
      float ra2[2], rb4[4];
#pragma unroll
      for (int i = 0; i < 2; ++i) ra2[i] = rt[slot_a(tr * 16 + gid + 8 * i)];
#pragma unroll
      for (int i = 0; i < 4; ++i) rb4[i] = rt[slot_b(tc * 16 + 8 * (i >> 1) + 2 * tg + (i & 1))];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float g5[NS] = {acc[0][i], acc[1][i], acc[2][i], acc[3][i], acc[4][i]};
        add_chunk(v[k][i], g5, ra2[(i >> 1) & 1] * rb4[2 * (i >> 2) + (i & 1)]);
        if ((f & 3) == 3) dfloat::renorm(v[k][i]);
      }
    }
    if (f + 2 < nch) bar_arrive<THREADS>(BAR_EMPTY + (f & 1));
  }
  const int ef = nch > 0 ? ((nch - 1) % 3) * 2 * MAXC : 0;
  double* out = g.partial + (size_t)blockIdx.x * ra * rb;
#pragma unroll
  for (int k = 0; k < MT; ++k) {
    if (tile[k] < 0) continue;
    const int tr = tile[k] >> 8, tc = tile[k] & 255;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int r = tr * 16 + gid + 8 * ((i >> 1) & 1), c = tc * 16 + 8 * (i >> 2) + 2 * tg + (i & 1);
      const int sa = slot_a(r), sb = slot_b(c);
      double d = ldexp((double)v[k][i].s + (double)v[k][i].c,
                       expo[ef + sa] - Entry<TA>::BIAS + expo[ef + sb] - Entry<TB>::BIAS - UNIT_BITS);
      if (bad[sa] | bad[sb]) d = __longlong_as_double(0x7ff8000000000000LL);
      out[(size_t)r * rb + c] = d;
    }
  }
}

// G[i][j] from the CTAs' partial D, summed in FP64 in a fixed order: 32
// entries of a row per CTA (lanes) by 8 strides over the partials (warps).
constexpr int RWARPS = 8;
__global__ void __launch_bounds__(RWARPS * 32) gram_digits_sum_kernel(const double* __restrict__ partial, int nz, int na,
                                                                       int nb, int na8, int nb8, int sym,
                                                                       double* __restrict__ G, int ldg) {
  __shared__ double red[2][RWARPS][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int i = blockIdx.x, j = blockIdx.y * 32 + lane;
  const int rb = 2 * nb8;
  const size_t per = (size_t)2 * na8 * rb;
  const bool use = j < nb && (!sym || i <= j);
  double re = 0.0, im = 0.0;
  if (use) {
    const size_t o00 = (size_t)i * rb + j, o11 = (size_t)(na8 + i) * rb + nb8 + j, o01 = (size_t)i * rb + nb8 + j;
    // D[na8 + i][j]; the symmetric form keeps only the upper tiles
    const size_t o10 = sym ? (size_t)j * rb + nb8 + i : (size_t)(na8 + i) * rb + j;
    for (int z = w; z < nz; z += RWARPS) {
      const double* p = partial + (size_t)z * per;
      re += p[o00] + p[o11];
      im += p[o01] - p[o10];
    }
  }
  red[0][w][lane] = re;
  red[1][w][lane] = im;
  __syncthreads();
  if (w == 0 && use) {
    re = im = 0.0;
#pragma unroll
    for (int k = 0; k < RWARPS; ++k) {
      re += red[0][k][lane];
      im += red[1][k][lane];
    }
    double* o = G + 2 * ((size_t)i * ldg + j);
    o[0] = re;
    o[1] = im;
    if (sym && i != j) {
      o = G + 2 * ((size_t)j * ldg + i);
      o[0] = re;
      o[1] = -im;
    }
  }
}

// per-CTA partial D, one buffer per (device, stream)
StreamScratch& dscratch() {
  static StreamScratch s;
  return s;
}

template <typename TA, typename TB, int MW, int SW, int MT, int CTAS, int REG>
cudaError_t run_block(DigitArgs g, int sms, double* G, int ldg, cudaStream_t s) {
  auto kern = gram_digits_kernel<TA, TB, MW, SW, MT, CTAS, REG>;
  const int rtot = 2 * g.na8 + (g.sym ? 0 : 2 * g.nb8);
  const size_t smem = (size_t)2 * NS * rtot * 64 + (size_t)2 * ((g.na + 1) / 2) * 64 * sizeof(typename Entry<TA>::C) +
                      (g.sym ? 0 : (size_t)2 * ((g.nb + 1) / 2) * 64 * sizeof(typename Entry<TB>::C)) +
                      (3 * 2 * MAXC + 4 + 2 * MAXC) * sizeof(int) + 2 * 2 * MAXC * sizeof(float);
  cudaError_t e = raise_dyn_smem(reinterpret_cast<const void*>(kern), smem);
  if (e != cudaSuccess) return e;
  // whole waves of CTAs, at least 4 chunks and at most MAX_ROWS rows each
  const long long chunks = (g.L + KC - 1) / KC;
  const long long fill = (long long)CTAS * sms;
  long long waves = (g.L + fill * MAX_ROWS - 1) / (fill * MAX_ROWS);
  if (waves < 1) waves = 1;
  long long per = (chunks + fill * waves - 1) / (fill * waves);
  if (per < 4) per = 4;
  const long long nz = (chunks + per - 1) / per;
  g.rows = per * KC;
  void* buf = nullptr;
  if ((e = dscratch().get(s, (size_t)nz * 4 * g.na8 * g.nb8 * sizeof(double), &buf)) != cudaSuccess) return e;
  g.partial = static_cast<double*>(buf);
  kern<<<(unsigned)nz, (MW + SW) * 32, smem, s>>>(g);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  gram_digits_sum_kernel<<<dim3((unsigned)g.na, (unsigned)((g.nb + 31) / 32)), RWARPS * 32, 0, s>>>(
      g.partial, (int)nz, g.na, g.nb, g.na8, g.nb8, g.sym, G, ldg);
  return cudaGetLastError();
}

// Whether the kernels of the wide products may run: their register split hands
// out what the launch allocated, so the compiler must have given them exactly
// 128 registers a thread (it does, at the launch bounds' limit).
template <typename TA, typename TB>
cudaError_t wide_kernels(bool* ok) {
  static std::atomic<int> state{0};   // 1: yes, 2: no
  if (state.load() == 0) {
    bool all = true;
    for (auto kern : {gram_digits_kernel<TA, TB, 8, 8, 2, 1, 144>, gram_digits_kernel<TA, TB, 8, 8, 3, 1, 152>,
                      gram_digits_kernel<TA, TB, 8, 8, 5, 1, 184>}) {
      cudaFuncAttributes fa;
      const cudaError_t e = cudaFuncGetAttributes(&fa, kern);
      if (e != cudaSuccess) return e;
      all = all && fa.numRegs == 128;
    }
    state.store(all ? 1 : 2);
  }
  *ok = state.load() == 1;
  return cudaSuccess;
}

template <typename TA, typename TB>
cudaError_t run_digits(const void* A, int na, const void* B, int nb, size_t L, double* G, cudaStream_t s) {
  int dev = 0, sms = 0;
  bool wide = true;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = wide_kernels<TA, TB>(&wide);
  if (e != cudaSuccess) return e;
  // column blocks of at most MAXC, or of what the kernels without a register
  // split take (8 tiles)
  const int ca = wide ? MAXC : 16, cb = wide ? MAXC : 32;
  const int ba = (na + ca - 1) / ca, bb = (nb + cb - 1) / cb;
  const int sa = (na + ba - 1) / ba, sb = (nb + bb - 1) / bb;
  for (int i0 = 0; i0 < na; i0 += sa)
    for (int j0 = 0; j0 < nb; j0 += sb) {
      DigitArgs g{};
      g.A = static_cast<const char*>(A) + (size_t)i0 * L * sizeof(typename Entry<TA>::C);
      g.B = static_cast<const char*>(B) + (size_t)j0 * L * sizeof(typename Entry<TB>::C);
      g.na = na - i0 < sa ? na - i0 : sa;
      g.nb = nb - j0 < sb ? nb - j0 : sb;
      g.na8 = (g.na + 7) / 8 * 8;
      g.nb8 = (g.nb + 7) / 8 * 8;
      g.sym = sizeof(TA) == sizeof(TB) && g.A == g.B && g.na == g.nb;
      g.L = (long long)L;
      double* out = G + 2 * ((size_t)i0 * nb + j0);
      const int tr = 2 * g.na8 / 16, tc = 2 * g.nb8 / 16;
      const int items = g.sym ? tr * (tr + 1) / 2 : tr * tc;
      // tiles per multiplying warp
      if (items <= 4) e = run_block<TA, TB, 4, 4, 1, 2, 0>(g, sms, out, nb, s);
      else if (items <= 8) e = run_block<TA, TB, 4, 4, 2, 2, 0>(g, sms, out, nb, s);
      else if (items <= 16) e = run_block<TA, TB, 8, 8, 2, 1, 144>(g, sms, out, nb, s);
      else if (items <= 24) e = run_block<TA, TB, 8, 8, 3, 1, 152>(g, sms, out, nb, s);
      else e = run_block<TA, TB, 8, 8, 5, 1, 184>(g, sms, out, nb, s);
      if (e != cudaSuccess) return e;
    }
  return cudaSuccess;
}

}  // namespace

cudaError_t launch_gram_digits(const void* A, int na, const void* B, int prec_b, int nb, size_t L, double* G,
                               cudaStream_t s) {
  if (na < 1 || nb < 1 || !A || !B) return cudaErrorInvalidValue;
  if (L == 0) return cudaMemsetAsync(G, 0, sizeof(double) * 2 * (size_t)na * nb, s);
  return prec_b == PCX_FP64 ? run_digits<double, double>(A, na, B, nb, L, G, s)
                            : run_digits<double, float>(A, na, B, nb, L, G, s);
}

void gram_digits_release_stream(cudaStream_t s) { dscratch().release(s); }

}  // namespace pcx
