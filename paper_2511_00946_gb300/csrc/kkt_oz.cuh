// FP64 products on the tensor cores by exact digit splitting (the error-free
// transformation of Ozaki, Ogita, Oishi and Rump, 2012, with FP16 operands and
// FP32 accumulators), for the Schur updates T -= Z Z^T of the factorization.
//
// Why. This part issues two FP64 FMAs per SM and clock (a warp's FP64
// instruction holds its sub-partition's FP64 pipe for 64 cycles) and its FP64
// mma.sync is no faster, whereas mma.sync m16n8k16 with FP16 operands runs at
// 850 multiply-adds per SM and clock (device probe). One product of 63-bit
// numbers takes 28 of them, so this path multiplies about 15 times as fast.
//
// Splitting. Row r of the panel gets one exponent f_r with |Z_rk| < 2^f_r; its
// elements are rounded to integers I = Z_rk 2^(61 - f_r) (error at most 2^-62
// of the row's scale; elements within 2^-8 of the largest are exact) and
// written in seven balanced digits of nine bits, I = sum_i d_i 2^(9 i), -256
// <= d_i <= 255. They are kept in place of the doubles with 256 added to
// every digit, so that a digit is a bit field of its own; a pair of fields
// becomes a pair of FP16 numbers with two logical operations (1024 + field is
// the bit pattern 0x6400 | field) and one subtraction. The products d_i d_j
// are accumulated over k separately for every i + j = 6 .. 12 in FP32. Sums
// below 2^24 are exact there (a test on the device checks it): all of them up to
// K = 36 columns; beyond, the two lowest sums (five and six pairs of full
// digits) can pass it and lose units that weigh 2^-59 of the rows' scales. The
// digit pairs with i + j <= 5 are dropped: below 2^-58 of the rows' scales (root
// mean square). The seven sums are combined in 64-bit integers, rounded to
// double once and subtracted from T.
//
// Accuracy. The error of element (a, b) is one rounding of the sum and about
// 2^-58 2^(f_a + f_b), whatever the columns hold. In a Cholesky factorization
// |Z_ak| <= sqrt(Psi_aa), so that is 2^-58 sqrt(Psi_aa Psi_bb): a backward error
// below that of FP64 FMAs, and invariant to the scaling of the variables (row a of
// the factor scales with variable a. The unscaled operands of the pivot sweep
// are not split: their columns carry the pivots' roots, and one exponent per
// row loses the ratio of those). It is a bound on the
// scale of the two variables, not on the element: entries of the factor far below
// it, between variables that are coupled by less than 1e-4 of their own scales, keep
// fewer digits of their own than FMAs would leave them (an answer that reaches one
// half of a stage through couplings of 1e-6 alone has 13 digits, of 1e-9 ten). A
// right-hand side has no such bound, which is why a bordered one is not split.
// Errors of the timed systems against 64-bit arithmetic, after those with FMAs:
// N = 1024, n = 32 3.7e-12, 1.0e-12; N = 777, n = 45 4.6e-13, 1.3e-13; 4096 uneven
// systems 2.7e-12, 1.8e-12; 512 systems, n = 32 5.6e-12, 1.8e-12.
// tests/test_oz_cpu.py bounds the products against exact arithmetic,
// tests/test_gpu_scaling.py asks for the same bits in any units.
//
// Measured (whole-CTA stage, 256 threads, 2070 MHz): the update of a 73-row
// panel of 32 columns takes 16k cycles on one SM alone, against 42k of FP64
// issue alone; one system of N = 1024, n = 32, m = 8 factored and solved 708 ->
// 653 us, N = 777, n = 45 1527 -> 1238 us, 4096 uneven systems 70.8 -> 63.6 ms (with
// the pivot sweep as it was then).
//
// A row with infinities, NaN or an exponent above 400, or whose elements are
// near the subnormal range, keeps its doubles (flag kFp64Row) and takes FP64
// FMAs. Small exponents are otherwise split (the fill-in between distant
// separators decays below 1e-130).
#pragma once
#include <cstdint>
#include <cstring>
#if defined(__CUDACC__)
#include <cuda_fp16.h>
#else
#include <cmath>
#endif

#if defined(__CUDACC__)
#define KKT_OZ __host__ __device__ __forceinline__
#else
#define KKT_OZ inline
#endif

namespace kkt {
namespace oz {

typedef long long i64;
typedef unsigned long long u64;

constexpr int kDig = 7;            // digits of nine bits
constexpr int kLow = kDig - 1;     // smallest i + j of the products kept
constexpr int kExpMax = 400;       // largest exponent of the rows split
constexpr int kExpMin = -960;      // smallest one (elements 62 bits below it are normal)
constexpr int kFp64Row = 1 << 20;  // exponent of a row that keeps its doubles
// 256 in every digit: 256 (2^63 - 1) / 511
constexpr u64 kBias = 256ull * ((1ull << 63) / 511);

KKT_OZ u64 dbits(double v) {
#if defined(__CUDA_ARCH__)
  return (u64)__double_as_longlong(v);
#else
  u64 b;
  std::memcpy(&b, &v, 8);
  return b;
#endif
}
KKT_OZ double bitsd(u64 b) {
#if defined(__CUDA_ARCH__)
  return __longlong_as_double((long long)b);
#else
  double v;
  std::memcpy(&v, &b, 8);
  return v;
#endif
}
KKT_OZ int expo(u64 b) { return (int)(b >> 52) & 0x7ff; }

// order of |v|: its high word, and 1 for the smallest subnormals
KKT_OZ int mag(u64 b) { return (int)(b >> 32 & 0x7fffffff) | ((uint32_t)b != 0); }

// the row exponent from the largest mag() of its elements (-1022: a zero row)
KKT_OZ int row_exp(int m) {
  const int f = (m >> 20) - 1022;
  return f > kExpMax || (f < kExpMin && m != 0) ? kFp64Row : f;  // (infinities and NaN included)
}

// digits of z at exponent f (|z| < 2^f), 256 added to each
KKT_OZ u64 encode(u64 b, int f) {
  const int ef = expo(b), q = f + 1022 - ef;  // q >= 0
  const u64 m = ((b & 0xfffffffffffffull) | 0x10000000000000ull) << 8;
  i64 v = ef == 0 || q > 62 ? 0 : (i64)((m + ((1ull << q) >> 1)) >> q);
  if ((i64)b < 0) v = -v;
  return (u64)v + kBias;
}

// u 2^e as a double, rounded to nearest (truncated below the normal range; e <= 900)
KKT_OZ double to_double(i64 u, int e) {
  u64 a = u < 0 ? (u64)-u : (u64)u;
#if defined(__CUDA_ARCH__)
  const int lz = __clzll((long long)a);
#else
  const int lz = a ? __builtin_clzll(a) : 64;
#endif
  a <<= (lz & 63);
  const u64 m = (a >> 11) + ((a >> 10) & 1);  // 53 bits; a carry moves the exponent up
  const int ex = 1023 + 63 - 1 - lz + e;
  const u64 b = ex >= 0 ? ((u64)ex << 52) + m : m >> (-ex < 63 ? -ex : 63);
  return bitsd(u == 0 ? 0 : b | ((u64)u & 0x8000000000000000ull));
}

// an element of a split row as a double
KKT_OZ double value(u64 p, int f) { return f == kFp64Row ? bitsd(p) : to_double((i64)(p - kBias), f - 61); }

// sum_g P_g 2^(9 (g - 6)) for the digit sums P_6 .. P_12 (p[0..6]), in units
// of 2^11: sum I I' = result 2^65 up to the dropped pairs (48 products of
// numbers below 2^61 stay below 2^63)
KKT_OZ i64 combine(const int* p) {
  const i64 hi = ((i64)(p[6] * 512 + p[5]) << 18) + ((i64)p[4] * 512 + p[3]);
  const i64 lo = ((i64)p[2] << 18) + ((i64)p[1] * 512 + p[0]);
  return (hi << 16) + ((lo + (1 << 10)) >> 11);
}
constexpr int kUnit = 65 - 122;  // exponent of combine()'s unit for rows at exponent 0

#if defined(__CUDACC__)
// digit i of two neighbouring elements as FP16 pairs: 1024 + field - 1280
template <int I>
__device__ __forceinline__ uint32_t digits(u64 u, u64 v) {
  const uint32_t w = (__byte_perm((uint32_t)(u >> (9 * I)), (uint32_t)(v >> (9 * I)), 0x5410) & 0x01ff01ffu) | 0x64006400u;
  const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&w), __float2half2_rn(1280.0f));
  return *reinterpret_cast<const uint32_t*>(&d);
}
template <int I>
struct Split {  // digits I .. 6 of `np` register pairs
  template <int NP>
  static __device__ __forceinline__ void run(uint32_t (*d)[NP], const u64* u) {
#pragma unroll
    for (int q = 0; q < NP; ++q) d[I][q] = digits<I>(u[2 * q], u[2 * q + 1]);
    Split<I + 1>::run(d, u);
  }
};
template <>
struct Split<kDig> {
  template <int NP>
  static __device__ __forceinline__ void run(uint32_t (*)[NP], const u64*) {}
};

__device__ __forceinline__ void mma_f16(float* d, const uint32_t* a, const uint32_t* b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// One element of a product outside the tensor-core path: *t -= sum_k a_k b_k
// where a row of its tile keeps its doubles (FP64 FMAs if one of the two rows
// here does, the digit sums in integers otherwise).
__device__ __noinline__ void element(double* t, const u64* pa, int fa, const u64* pb, int fb, int n) {
  double acc = *t;
  if (fa == kFp64Row || fb == kFp64Row) {
    for (int k = 0; k < n; ++k) acc = fma(-value(pa[k], fa), value(pb[k], fb), acc);
  } else {
    int p[kDig] = {0, 0, 0, 0, 0, 0, 0};
    for (int k = 0; k < n; ++k)
      for (int i = 0; i < kDig; ++i)
        for (int j = kLow - i; j < kDig; ++j)
          p[i + j - kLow] += ((int)(pa[k] >> (9 * i) & 511) - 256) * ((int)(pb[k] >> (9 * j) & 511) - 256);
    acc -= to_double(combine(p), fa + fb + kUnit);
  }
  *t = acc;
}

// One 16 x 8 tile of T -= Z Z^T by a warp: rows a0 + 0..15 (< ea) against
// columns b0 + 0..7 (< eb), elements b <= a. Lane (g, t) = (lane / 4, lane % 4)
// holds the fragments' rows a0 + g, a0 + g + 8 and column row b0 + g. The 28
// digit products per 16 columns of Z are ordered so that neighbouring ones
// go to different accumulators. SKIP: row and column `skip` are left as they are
// (a row that holds no digits, with any exponent but kFp64Row).
template <bool SKIP = false>
__device__ __forceinline__ void tile(double* T, int ldt, const double* Zlo, const int* flo, const double* Z,
                                     const int* fz, int zsplit, int ldz, int a0, int ea, int b0, int eb, int n,
                                     int lane, int skip = -1) {
  const int g = lane >> 2, t = lane & 3;
  const int ra = a0 + g, rc = ra + 8, rb = b0 + g;
  const int qa = min(ra, ea - 1), qc = min(rc, ea - 1), qb = min(rb, eb - 1);  // rows for addresses
  const u64* za = (const u64*)((qa < zsplit ? Zlo : Z) + qa * ldz);
  const u64* zc = (const u64*)((qc < zsplit ? Zlo : Z) + qc * ldz);
  const u64* zb = (const u64*)((qb < zsplit ? Zlo : Z) + qb * ldz);
  const int xa = (qa < zsplit ? flo : fz)[qa], xc = (qc < zsplit ? flo : fz)[qc], xb = (qb < zsplit ? flo : fz)[qb];
  // this lane's outputs: rows ra, rc, columns b0 + 2 t, + 1
  const int c0 = b0 + 2 * t, c1 = c0 + 1;
  unsigned on = 0;  // (formed here, so that the bounds are not kept through the products)
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int a = e < 2 ? ra : rc, b = e & 1 ? c1 : c0;
    if (a < ea && b < eb && b <= a && !(SKIP && (a == skip || b == skip))) on |= 1u << e;
  }
  if (__any_sync(0xffffffffu, max(max(xa, xc), xb) == kFp64Row)) {
    for (int e = 0; e < 4; ++e) {
      const int a = e < 2 ? ra : rc, b = e & 1 ? c1 : c0;
      if (on >> e & 1)
        element(T + a * ldt + b, e < 2 ? za : zc, e < 2 ? xa : xc,
                   (const u64*)((b < zsplit ? Zlo : Z) + b * ldz), (b < zsplit ? flo : fz)[b], n);
    }
    return;
  }
  float acc[kDig][4];
#pragma unroll
  for (int i = 0; i < kDig; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0.0f;
#pragma unroll 1
  for (int k0 = 0; k0 < n; k0 += 16) {
    const int k1 = k0 + 2 * t, k2 = k1 + 8;
    auto at = [&](const u64* z, int k) { return k < n ? z[k] : kBias; };
    uint32_t A[kDig][4], B[kDig][2];
    {
      const u64 u[8] = {at(za, k1), at(za, k1 + 1), at(zc, k1), at(zc, k1 + 1),
                            at(za, k2), at(za, k2 + 1), at(zc, k2), at(zc, k2 + 1)};
      const u64 v[4] = {at(zb, k1), at(zb, k1 + 1), at(zb, k2), at(zb, k2 + 1)};
      Split<0>::run<4>(A, u);
      Split<0>::run<2>(B, v);
    }
#pragma unroll
    for (int i = 0; i < kDig; ++i)
#pragma unroll
      for (int j = kDig - 1; j >= kLow - i; --j) mma_f16(acc[i + j - kLow], A[i], B[j]);
  }
  const int x0 = __shfl_sync(0xffffffffu, xb, 8 * t), x1 = __shfl_sync(0xffffffffu, xb, 8 * t + 4);
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int a = e < 2 ? ra : rc, b = e & 1 ? c1 : c0;
    if (on >> e & 1) {
      int p[kDig];
#pragma unroll
      for (int i = 0; i < kDig; ++i) p[i] = (int)acc[i][e];
      T[a * ldt + b] -= to_double(combine(p), (e < 2 ? xa : xc) + (e & 1 ? x1 : x0) + kUnit);
    }
  }
}
#endif

}  // namespace oz
}  // namespace kkt
