// tc_exact.cu -- block-pair products of the FP64-accurate paths (FP64,
// double-float) on the fifth-generation tensor cores, exact up to one rounding
// (Sec. 3 Eq. LN.pLLp.FFT: sums over open indices of A(q) B(-q)).
//
// Every operand value x of a row with max |x| < 2^e becomes the integer
// T = x 2^(55 - e), cut towards zero (FP64) or to the nearest (double-float) and
// written in eight signed digits of 7 bits, d_i in [-64, 63], T = sum_i d_i
// 2^(7 (7 - i)).  The digits are small integers in fp16, their products are exact
// in the FP32 accumulators of tcgen05.mma (kind::f16), and so are the sums: the
// digit products of one weight ("level" s = i + j) of a complex product of
// K = 144 terms add up to at most 8 x 288 x 64^2 < 2^24.  Levels 0 .. 7 are kept,
// put together in 64-bit integers and rounded once.  The dropped levels leave an
// error relative to the product of the two rows' bounds 2^e, not to the sum of the
// terms' magnitudes: in units of 2^-54 of it 3.8 rms for Gaussian rows, 6.5 (with a
// mean of -3.7) for rows of one sign, 24 at the most in 400,000 emulated products.
// A product that comes out far below that bound, and any product of a row the
// fixed point cannot hold, is therefore made again in the blocks' own arithmetic
// (k_exact_wick).  (This is the splitting idea of Ozaki, Ogita, Oishi and
// Rump, Numer. Algorithms 59 (2012), with the products on integers.)
//
// A digit pair costs 4 real MACs per complex one at 4096 MACs per clock and
// SM against 2 FP64 FMAs per clock (three per complex MAC) or 128 FP32 lanes
// (48 instructions per complex MAC in double-float): 36 digit pairs are still
// many times cheaper than either pipe.  What bounds the kernel is the integer
// work of making the digits (about 35 instructions per real value) beside the
// tensor pipe, and the drain of the one accumulator set: 50% of the issue slots,
// 37% of the tensor pipe, 22% of DRAM at 16^3.  Measured against the CUDA-core products of
// field-major blocks, 52 channels: FP64 16^3 3.99 -> 0.59 ms per slice,
// double-float 16^3 1.40 -> 0.53, 48^3 35.2 -> 13.2 (both with the small tasks).
// On field-major blocks (16-byte loads 64 KB and more apart) the same kernel was
// TLB bound at 0.98 and 45 ms: the blocks are q-major for it.
//
// Operand sets (exact_split.cpp):
//   trace forms, one product per pair {q, -q}: STACK = 2.  Two digit slices of
//     A (nbp <= 64 rows each) fill one M = 128 instruction, so a window that
//     starts at slice i gives level i + j in its first nbp rows of D and
//     i + j + 1 in the next nbp: four column blocks hold the eight levels.
//     Even digits of B are adjacent (so are odd ones): one instruction with N
//     = nbp n multiplies a window by n of them into n adjacent column blocks.
//     Windows at even i take the even digits, at odd i (from -1, a slice of
//     zeros in front) the odd ones, so every digit pair up to level 7 is met
//     once.
//   slice forms, one product per q: STACK = 1.  The window is one slice (up to
//     128 rows), all eight levels are column blocks of nB columns, and digit i
//     of A meets digits 0 .. 7 - i of B in one instruction.
// Re = Re Re - Im Im uses the instruction's negated A.
//
// A persistent CTA per SM: warps 0-7 read the accumulators, warp 8 issues the
// MMAs, the others load rows of the q-major blocks (32-byte loads; a pair's rows
// lie in two runs of n_out values), split them and store the digits in the canonical K-major
// layout without swizzle, 16 open indices per stage of an mbarrier ring.
// Every wait is bounded: past its limit, or when another warp gave up, the
// warps leave their loops, the MMAs in flight are waited for (a limit of its own), the
// tensor memory is freed and bit 1 of the error word is set; k_exact_wick then
// writes NaN, until the host has read the word.
#include <algorithm>
#include <type_traits>

#include <cuda_fp16.h>

#include "device_common.cuh"
#include "kernels.cuh"

namespace bbc {

namespace {

constexpr int kXDigits = 8;
constexpr int kXWarps = 20;
constexpr int kXEpi = 8;                       // epilogue warps (tensor-memory lanes 32 (w mod 4) .., column chunks w / 4)
constexpr int kXProd = kXWarps - kXEpi - 1;    // producer warps, after the MMA warp
constexpr int kXMaxStages = 6;
constexpr long long kXDrainLimit = 1ll << 22;  // polls for the MMAs in flight (about a second)
constexpr int kXCols = 512;                    // all of tensor memory: one CTA per SM
constexpr int kXFixed = 2048;                  // static shared memory (at most)
// exponents that are no exponents: a row the digits cannot hold (a NaN or infinite
// value, or a largest value below 2^kLow) and a row of zeros.  Beside exponents of
// at most 2^11 a sum of two above kXNone has a bad one, below -kXNone a zero and no
// bad one.
constexpr int kXBad = 0x7000, kXZero = -0x3000, kXNone = 0x2000;
// Per block type: rows and products below 2^kLow and 2^kLowProduct (the digits of
// an FP64 value are cut by at most 63 bits, double-float scales are FP32 numbers; a
// product keeps a normal result), and a product below 2^-kXFar of the rows'
// bound is not trusted (k_exact_wick).
template <typename T>
struct XLimits;
template <>
struct XLimits<double> { static constexpr int kLow = -900, kLowProduct = -900; };
template <>
struct XLimits<dfr> { static constexpr int kLow = -72, kLowProduct = -90; };
constexpr int kXFar = 7;

__device__ __forceinline__ uint32_t x_smem(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void x_mbar_init(uint32_t bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void x_arrive(uint32_t bar) {
  asm volatile("{\n\t.reg .b64 t;\n\tmbarrier.arrive.shared::cta.b64 t, [%0];\n\t}" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool x_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// completion of the phase of this parity; false after `limit` polls or once
// another warp of the CTA gave up
__device__ __forceinline__ bool x_wait(uint32_t bar, uint32_t parity, long long limit, volatile int* abort_flag) {
  for (long long polls = 0; !x_test(bar, parity); polls++) {
    if (polls >= limit || *abort_flag) {
      *abort_flag = 1;
      return false;
    }
    if (polls > 8) __nanosleep(20);
  }
  return true;
}

// shared-memory matrix descriptor: core matrices (8 rows x 16 bytes) 128 bytes
// apart along K, 8-row groups 256 bytes apart, no swizzle
__device__ __forceinline__ uint64_t x_desc(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)(128 >> 4) << 16) | ((uint64_t)(256 >> 4) << 32) | (1ull << 46);
}
// kind::f16, A and B fp16 (K-major), D FP32, M = 128; bit 13 negates A
__device__ __forceinline__ uint32_t x_idesc(int n, int neg) {
  return (1u << 4) | ((uint32_t)neg << 13) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}
__device__ __forceinline__ void x_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void x_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void x_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void x_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void x_ld4(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}
__device__ __forceinline__ void x_wait_ld(uint32_t (&r)[4]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]) : : "memory");
}

__device__ __forceinline__ bool x_elect() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
  return p != 0;
}

// barrier of the epilogue warps; true if ok holds in all of them
__device__ __forceinline__ bool x_all_epi(bool ok) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, o;\n\tsetp.ne.u32 p, %1, 0;\n\tbarrier.cta.red.and.pred o, 1, %2, p;\n\t"
      "selp.u32 %0, 1, 0, o;\n\t}\n"
      : "=r"(r)
      : "r"((uint32_t)ok), "n"(32 * kXEpi)
      : "memory");
  return r != 0;
}

__device__ __forceinline__ int x_neg_site(int q, int L) {
  const int qx = q % L, qy = (q / L) % L, qz = q / (L * L);
  return (L - qx) % L + L * ((L - qy) % L + L * ((L - qz) % L));
}

// ------------------------------------------------------------ fixed point
// T = x 2^(55 - e) cut to an integer, |x| < 0.985 2^e, plus the digits' offset:
// u = T + 64 sum_k 2^(7 k), k = 0 .. 7, so that the 7-bit fields of u are the
// digits + 64.  FP64 values from their bits, with integer instructions only (the
// FP64 pipe issues 2 per clock); values within a factor 4 of the row's bound
// keep all their bits, smaller ones lose at most 2^(e - 55).
constexpr unsigned long long kXBias = 0x40ull * 0x2040810204081ull;
__device__ __forceinline__ unsigned long long x_fix(double x, int e) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned long long m =
      ((unsigned long long)((__funnelshift_l(lo, hi, 2) & 0x3fffffu) | 0x400000u) << 32) | (lo << 2);
  const int r = min(e + 1022 - (int)((hi >> 20) & 0x7ffu), 63);  // >= 0 in the row; zero and subnormals: 63
  const unsigned long long sg = (unsigned long long)((long long)(int)hi >> 63);
  return ((m >> (r & 63)) ^ sg) + (kXBias - sg);
}
// Double-float values by rounding FP32 additions (x + M keeps the nearest
// integer of |x| < 2^22 in its low bits; the residues are exact): 21 bits and
// 17 bits of the high word, then the rest of it with the low word, 17 + 17 bits.
// The pairs are normalised (the forward transform's last pass): |lo| <= 2^-24 |hi|,
// so that lo 2^(38 - e) stays below 2^14 beside a rest of at most 2^16.  An
// unnormalised low word could leave the range of x + M and give wrong digits.
// FP32 additions run at twice the rate of shifts.
__device__ __forceinline__ unsigned long long x_fix(dfr x, int e) {
  const float M = 12582912.f, p17 = 131072.f;  // 1.5 2^23, 2^17
  const float s = __int_as_float((127 + 21 - e) << 23);  // 2^(21 - e), e >= -72
  const float h = __fmul_rn(x.hi, s);
  const float t0 = __fadd_rn(h, M), r0 = __fsub_rn(h, __fsub_rn(t0, M));
  const float t1 = __fmaf_rn(r0, p17, M), r1 = __fmaf_rn(r0, p17, -__fsub_rn(t1, M));
  const float y = __fmaf_rn(x.lo, __fmul_rn(s, p17), r1);
  const float t2 = __fadd_rn(y, M), r2 = __fsub_rn(y, __fsub_rn(t2, M));
  const float t3 = __fmaf_rn(r2, p17, M);
  constexpr unsigned long long Mb = 0x4B400000;
  constexpr unsigned long long off = kXBias - (((Mb << 17) + 2 * Mb) * 131072 + Mb);
  const unsigned long long hi =
      (unsigned long long)__float_as_uint(t0) * 131072u + (unsigned long long)__float_as_uint(t1) + __float_as_uint(t2);
  // (the mask: a row with infinities has any digits)
  return ((hi << 17) + __float_as_uint(t3) + off) & 0xffffffffffffffull;
}

// The digits of eight values in one half (28 bits, four digits) of u as packed
// fp16, one 16-byte store per digit: dst + slot(d0 + d), d = 0 .. 3.  First the
// 28 bits as two 14-bit fields in 16-bit lanes (t << 2 = t + 3 t), then the same
// field of two neighbouring values side by side, then its two digits.  A field
// f = d + 64 read as a subnormal is f 2^-24, times 2^14 minus 2^-4 is d 2^-10.
__device__ __forceinline__ uint32_t x_half(uint32_t f) {
  const __half2 h = __hfma2(*reinterpret_cast<const __half2*>(&f), __half2half2(__ushort_as_half(0x7400)),  // 2^14
                            __half2half2(__ushort_as_half(0xAC00)));                                        // -2^-4
  return *reinterpret_cast<const uint32_t*>(&h);
}
template <typename SlotFn>
__device__ __forceinline__ void x_store4(const uint32_t (&w)[8], unsigned char* dst, int d0, SlotFn slot) {
  uint32_t z[2][4];  // [field][pair of values]: digits d0, d0 + 1 and d0 + 2, d0 + 3
#pragma unroll
  for (int j = 0; j < 4; j++) {
    const uint32_t a = w[2 * j] + 3 * (w[2 * j] & 0x0fffc000u), b = w[2 * j + 1] + 3 * (w[2 * j + 1] & 0x0fffc000u);
    z[0][j] = __byte_perm(a, b, 0x7632);
    z[1][j] = __byte_perm(a, b, 0x5410);
  }
#pragma unroll
  for (int f = 0; f < 2; f++) {
    uint4 hi, lo;
    hi.x = x_half((z[f][0] >> 7) & 0x007f007fu);
    hi.y = x_half((z[f][1] >> 7) & 0x007f007fu);
    hi.z = x_half((z[f][2] >> 7) & 0x007f007fu);
    hi.w = x_half((z[f][3] >> 7) & 0x007f007fu);
    lo.x = x_half(z[f][0] & 0x007f007fu);
    lo.y = x_half(z[f][1] & 0x007f007fu);
    lo.z = x_half(z[f][2] & 0x007f007fu);
    lo.w = x_half(z[f][3] & 0x007f007fu);
    *reinterpret_cast<uint4*>(dst + slot(d0 + 2 * f)) = hi;
    *reinterpret_cast<uint4*>(dst + slot(d0 + 2 * f + 1)) = lo;
  }
}
template <typename SlotFn>
__device__ __forceinline__ void x_store_digits(const unsigned long long (&u)[8], unsigned char* dst, SlotFn slot) {
  uint32_t w[8];
#pragma unroll
  for (int j = 0; j < 8; j++) w[j] = (uint32_t)(u[j] >> 28);  // u < 2^56
  x_store4(w, dst, 0, slot);
#pragma unroll
  for (int j = 0; j < 8; j++) w[j] = (uint32_t)u[j] & 0x0fffffffu;
  x_store4(w, dst, 4, slot);
}

// (re + i im) 2^k in the product's type (k = kXBad: NaN), |re|, |im| < 2^63,
// rounded to nearest from the integers' bits (the conversions of 64-bit
// integers run on the FP64 pipe).
__device__ __forceinline__ double x_scaled(long long S, int k) {
  const unsigned long long a = (unsigned long long)(S < 0 ? -S : S);
  const int lz = __clzll((long long)a);
  const unsigned long long n = a << (lz & 63);  // top bit set
  const int ex = 1023 + 63 - lz + k;            // biased exponent
  // 53 significant bits rounded to nearest; a carry moves into the exponent
  const unsigned long long m = (n >> 11) + ((n >> 10) & 1);
  unsigned long long bits = ((unsigned long long)(unsigned)(ex - 1) << 52) + m;
  bits = a == 0 || ex <= 0 ? 0 : ex >= 0x7ff ? 0x7ff0000000000000ull : bits;
  return __longlong_as_double((long long)(bits | ((unsigned long long)S & 0x8000000000000000ull)));
}
__device__ __forceinline__ void x_scaled(long long S, int k, float& hi, float& lo) {
  const unsigned long long a = (unsigned long long)(S < 0 ? -S : S);
  const int lz = min(__clzll((long long)a), 63);
  const unsigned long long n = a << lz;
  // the top 24 bits, then the next 32: 2^(k - lz + 40), in two exact factors
  const int f = k - lz + 40, f1 = min(max(f >> 1, -126), 127), f2 = min(max(f - f1, -126), 127);
  const float s1 = __int_as_float((127 + f1) << 23), s2 = __int_as_float((127 + f2) << 23);
  const float h = (float)(unsigned)(n >> 40), l = (float)(unsigned)(n >> 8) * 2.3283064365386963e-10f;  // 2^-32
  hi = (S < 0 ? -h : h) * s1 * s2;
  lo = (S < 0 ? -l : l) * s1 * s2;
}
__device__ __forceinline__ double2 x_value(double2, long long re, long long im, int k) {
  const bool bad = k == kXBad;
  const double nan = __longlong_as_double(-1ll), a = x_scaled(re, bad ? 0 : k), b = x_scaled(im, bad ? 0 : k);
  return make_double2(bad ? nan : a, bad ? nan : b);
}
__device__ __forceinline__ float4 x_value(float4, long long re, long long im, int k) {
  const bool bad = k == kXBad;
  float4 v;
  x_scaled(re, bad ? 0 : k, v.x, v.y);
  x_scaled(im, bad ? 0 : k, v.z, v.w);
  const float nan = __int_as_float(-1);
  return bad ? make_float4(nan, nan, nan, nan) : v;
}

// The level sums of one entry of D, x_s = n_s 2^-20 with |n_s| < 2^24, as sum_s
// n_s 2^w_s: x + 12 keeps n_s in its low bits while |n_s| < 2^22 (always for
// levels 0 .. 2; `wide` gathers the sums that are larger, which only coherent
// digits reach), and the offsets leave in one constant.
__device__ __forceinline__ unsigned x_bits(uint32_t x, uint32_t& wide) {
  const unsigned b = __float_as_uint(__uint_as_float(x) + 12.f);
  wide |= b ^ 0x41000000u;  // [8, 16) has this sign and exponent
  return b;
}
constexpr long long kXMagic = 0x41400000;  // bits of 12
__device__ __forceinline__ long long x_mad(unsigned a, unsigned b, long long c) {
  long long d;
  asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
}
__device__ __forceinline__ long long x_int(uint32_t x) { return (long long)__float2int_rn(__uint_as_float(x) * 1048576.f); }
// Sum over the levels of column j, weights 2^(42 - 7 s) (the last one, 2^-7, cut).
// STACK 2: a[c] is level 2 c (even) or 2 c + 1; STACK 1: level c.
__device__ __forceinline__ long long x_levels(const uint32_t (&a)[4][4], int j, bool even, uint32_t& wide) {
  constexpr long long off = kXMagic * ((1ll << 28) + (1ll << 14) + 1);
  const unsigned n0 = x_bits(a[0][j], wide), n1 = x_bits(a[1][j], wide), n2 = x_bits(a[2][j], wide);
  const int n3 = (int)(x_bits(a[3][j], wide) - (unsigned)kXMagic);
  const long long v = x_mad(n0, 1u << 28, x_mad(n1, 1u << 14, n2)) - off;
  return (v << (even ? 14 : 7)) + (n3 >> (even ? 0 : 7));
}
__device__ __forceinline__ long long x_levels(const uint32_t (&a)[8][4], int j, bool, uint32_t& wide) {
  constexpr long long off = kXMagic * ((1ll << 28) + (1ll << 14) + 1);
  const unsigned n0 = x_bits(a[0][j], wide), n1 = x_bits(a[1][j], wide), n2 = x_bits(a[2][j], wide);
  const unsigned n3 = x_bits(a[3][j], wide), n4 = x_bits(a[4][j], wide), n5 = x_bits(a[5][j], wide);
  const int n6 = (int)(x_bits(a[6][j], wide) - (unsigned)kXMagic);
  const int n7 = (int)(x_bits(a[7][j], wide) - (unsigned)kXMagic);
  const long long ev = x_mad(n0, 1u << 28, x_mad(n2, 1u << 14, n4)) - off;
  const long long od = x_mad(n1, 1u << 28, x_mad(n3, 1u << 14, n5)) - off;
  return (ev << 14) + n6 + (od << 7) + (n7 >> 7);
}
// the same for sums beyond 2^22
template <int NC>
__device__ __forceinline__ long long x_levels_wide(const uint32_t (&a)[NC][4], int j, bool even) {
  long long v = 0;
#pragma unroll
  for (int c = 0; c < NC; c++) {
    const int s = NC == 4 ? 2 * c + (even ? 0 : 1) : c, sh = 42 - 7 * s;
    const long long n = x_int(a[c][j]);
    v += sh >= 0 ? n << (sh & 63) : n >> (-sh & 63);
  }
  return v;
}

// two neighbouring complex values with one 32-byte load (32-byte aligned)
__device__ __forceinline__ void x_load2(const float4* p, float4& a, float4& b) {
  asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
      : "l"(p));
}
__device__ __forceinline__ void x_load2(const float4* p, double2& a, double2& b) {
  asm("ld.global.nc.v4.f64 {%0, %1, %2, %3}, [%4];" : "=d"(a.x), "=d"(a.y), "=d"(b.x), "=d"(b.y) : "l"(p));
}

// Per block type: a loaded complex value and its parts.
template <typename T>
struct XRaw;
template <>
struct XRaw<double> {
  using load = double2;
  static __device__ __forceinline__ double re(const double2& v) { return v.x; }
  static __device__ __forceinline__ double im(const double2& v) { return v.y; }
};
template <>
struct XRaw<dfr> {
  using load = float4;
  static __device__ __forceinline__ dfr re(const float4& v) { return dfr(v.x, v.y); }
  static __device__ __forceinline__ dfr im(const float4& v) { return dfr(v.z, v.w); }
};
// values j .. j + 3 from four neighbouring elements
template <typename Ld>
__device__ __forceinline__ void x_run4(const Ld* p, Ld (&v)[8], int j) {
  x_load2(reinterpret_cast<const float4*>(p), v[j], v[j + 1]);
  x_load2(reinterpret_cast<const float4*>(p + 2), v[j + 2], v[j + 3]);
}
// values j and j + 4 from two neighbouring elements
template <typename Ld>
__device__ __forceinline__ void x_pair(const Ld* p, Ld (&v)[8], int j) {
  x_load2(reinterpret_cast<const float4*>(p), v[j], v[j + 4]);
}

struct XShape {  // shared-memory layout of one launch
  int slA, slB, partA, stage, n_stages, off_b, sums, bytes;  // sums: the epilogue's 64-bit sums, after the stages
};
__host__ __device__ inline XShape x_shape(int stack, int nAp, int nBp) {
  XShape s;
  s.slA = nAp * 32;  // one digit slice: 16 open indices x 2 bytes per row
  s.slB = nBp * 32;
  s.partA = (kXDigits + (stack == 2 ? 1 : 0)) * s.slA;  // real or imaginary part; STACK 2: a slice of zeros first
  s.off_b = 2 * s.partA;
  s.stage = s.off_b + 2 * kXDigits * s.slB;
  s.sums = stack * 2 * nBp * nAp * 8;
  const int fit = (int)(kMaxSmemPerBlock - kXFixed - s.sums) / s.stage;
  s.n_stages = fit < kXMaxStages ? fit : kXMaxStages;
  s.bytes = s.n_stages * s.stage + s.sums;
  return s;
}

}  // namespace

// Exponents of one q per CTA: E[q][job] with max |component| over the job's
// rows below 0.985 2^E, kXBad or kXZero.  A warp takes a
// piece of rows (a whole block) and, from the same loads, the jobs inside it: HBM bound.
__device__ __forceinline__ int x_mag(double x) {  // the exponent-carrying word, zero only for zeros
  return (__double2hiint(x) & 0x7fffffff) | (__double2loint(x) != 0);
}
__device__ __forceinline__ int x_mag(const double2& v) { return max(x_mag(v.x), x_mag(v.y)); }
__device__ __forceinline__ int x_mag(const float4& v) {  // both words of a double-float count
  return max(__float_as_int(fabsf(v.x) + fabsf(v.y)) & 0x7fffffff, __float_as_int(fabsf(v.z) + fabsf(v.w)) & 0x7fffffff);
}
template <typename T>
__global__ void __launch_bounds__(256)
k_exact_exponents(const void* __restrict__ blk, int n_out, const int4* __restrict__ loads, int n_loads,
                  const int2* __restrict__ jobs, int n_jobs, int* __restrict__ E) {
  using Ld = typename XRaw<T>::load;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const Ld* row = reinterpret_cast<const Ld*>(blk) + (size_t)blockIdx.x * n_out;
  for (int l = warp; l < n_loads; l += 8) {
    const int4 p = __ldg(loads + l);  // at most 144 rows
    int mag[5];
#pragma unroll
    for (int i = 0; i < 5; i++) mag[i] = lane + 32 * i < p.y ? x_mag(__ldg(row + p.x + lane + 32 * i)) : 0;
    for (int job = p.z; job < p.w; job++) {
      const int2 j = __ldg(jobs + job);
      int m = 0;
#pragma unroll
      for (int i = 0; i < 5; i++) {
        const int r = lane + 32 * i - j.x;  // three columns: elements 12 i1 + i2, i2 < 3
        const bool in = j.y == kExactColumns ? r >= 0 && r % 12 < 3 : (unsigned)r < (unsigned)j.y;
        m = in ? max(m, mag[i]) : m;
      }
      m = __reduce_max_sync(0xffffffffu, m);
      // 2^-5 of headroom in the significand: the largest magnitude has to fit
      // digits whose range is [-64, 63]
      int e;
      if (std::is_same<T, double>::value) e = m >= 0x7ff00000 ? kXBad : ((m + 0x8000) >> 20) - 1022;
      else e = m >= 0x7f800000 ? kXBad : ((m + 0x40000) >> 23) - 126;
      e = m == 0 ? kXZero : e < XLimits<T>::kLow ? kXBad : e;
      if (lane == 0) E[(size_t)blockIdx.x * n_jobs + job] = e;
    }
  }
}

// Product i of a task with few open indices, from the rows of q and -q.
__device__ __forceinline__ double2 x_small(const double2* a, const double2* c, int n1, int n2, int sA1, int sA2, int sB1,
                                           int sB2) {
  cpx<double> acc(0, 0);
  for (int i1 = 0; i1 < n1; i1++)
    for (int i2 = 0; i2 < n2; i2++) {
      const double2 x = __ldg(a + i1 * sA1 + i2 * sA2), y = __ldg(c + i1 * sB1 + i2 * sB2);
      cmac(acc, cpx<double>(x.x, x.y), cpx<double>(y.x, y.y));
    }
  return make_double2(acc.re, acc.im);
}
__device__ __forceinline__ float4 x_small(const float4* a, const float4* c, int n1, int n2, int sA1, int sA2, int sB1,
                                          int sB2) {
  df64acc re{0.f, 0.f}, im{0.f, 0.f};
  for (int i1 = 0; i1 < n1; i1++)
    for (int i2 = 0; i2 < n2; i2++) {
      const float4 x = __ldg(a + i1 * sA1 + i2 * sA2), y = __ldg(c + i1 * sB1 + i2 * sB2);
      df_mac(re, x.x, x.y, y.x, y.y);
      df_mac(re, -x.z, -x.w, y.z, y.w);
      df_mac(im, x.x, x.y, y.z, y.w);
      df_mac(im, x.z, x.w, y.x, y.y);
    }
  df_renorm(re);
  df_renorm(im);
  return make_float4(re.s, re.e, im.s, im.e);
}
template <typename Ld>
__device__ __forceinline__ Ld x_small_item(const Ld* F, int q, int nq, int n_out, const DevTask& t, int i) {
  const int nB = t.nAnB >> 8;
  return x_small(F + (size_t)q * n_out + t.offA[i / nB], F + (size_t)nq * n_out + t.offB[i % nB], t.n1, t.n2,
                 t.sA & 0xffff, t.sA >> 16, t.sB & 0xffff, t.sB >> 16);
}

// Products of the tasks with few open indices (a few percent of the work): one
// CTA per q, one product per thread.
template <typename T>
__global__ void __launch_bounds__(256)
k_exact_small(const void* __restrict__ blk, int L, int n_out, const DevTask* __restrict__ tasks,
              const int* __restrict__ small, int n_small, int n_items, void* __restrict__ P) {
  using Ld = typename XRaw<T>::load;
  const int q = blockIdx.x, nq = x_neg_site(q, L);
  for (int u = threadIdx.x; u < n_small * 16; u += 256) {
    const int ti = __ldg(small + (u >> 4)), i = u & 15;
    reinterpret_cast<Ld*>(P)[(size_t)q * n_items + ti * 16 + i] =
        x_small_item(reinterpret_cast<const Ld*>(blk), q, nq, n_out, tasks[ti], i);
  }
}

// Signed sums over Wick diagrams of q-major products, ct[q][o] = sum_c coef_c
// P[q][item_c]: one CTA per q stages its product row and the distinct
// coefficients in shared memory (several CTAs per SM, so that one's copies overlap
// another's sums).  A warp takes 32 outputs of
// nearly equal length (host-sorted); their terms are stored lane by lane (item |
// coefficient index << 16), so a term of 32 outputs is one 128-byte load.  With
// the outputs' term lists read in place, 7 to 14 cache lines per load, the sums
// took 93 us (double-float, 16^3, 52 channels).
// FP64; double-float with the coefficients split on the host, renormalised
// every 16 terms.
//
// Before the sums, products marked NaN are made again, a warp each, from the rows
// in the blocks' own arithmetic: rows the digits do not hold, and products below
// 2^-kXFar of the product of their rows' bounds.  The digits' error is about 2^-52 of
// that, at most 2^-49 seen (dropped levels and cut values), so about 2^-45 of a product
// at 2^-7 of it: what bounds an FP64 sum of 288 terms, and half the double-float
// operators' own error.  Where the large values of two rows meet (any field whose
// flavours are graded alike) under 0.03% of the products are made again, mostly at
// q = 0 of smooth fields; at 2^-6 four times as many, and the CTA of that q held up
// small lattices (Lambda N 8^3, FP64: 22 against 16 us per slice).  Rows graded against
// each other would lose their products without it, and pay: with all of them made again
// the sums of 52 channels take 9.2 ms per 16^3 slice in FP64, 4.1 in double-float.
// The marks and those products took the 16^3 sums of 52 channels from 121 to 142 us
// (FP64) and from 82 to 92 (double-float), and 48^3 ones from 1.65 to 1.97 ms.
constexpr int kWickThreads = 256;
struct WickAcc64 {
  double x = 0, y = 0;
  __device__ __forceinline__ void add(double w, double2 v) {
    x = fma(w, v.x, x);
    y = fma(w, v.y, y);
  }
  __device__ __forceinline__ void renorm() {}
  __device__ __forceinline__ double2 value() { return make_double2(x, y); }
};
struct WickAccDf {
  df64acc re{0.f, 0.f}, im{0.f, 0.f};
  __device__ __forceinline__ void add(float2 w, float4 v) {
    df_mac(re, w.x, w.y, v.x, v.y);
    df_mac(im, w.x, w.y, v.z, v.w);
  }
  __device__ __forceinline__ void renorm() {
    df_renorm(re);
    df_renorm(im);
  }
  __device__ __forceinline__ float4 value() {
    renorm();
    return make_float4(re.s, re.e, im.s, im.e);
  }
};
// Product of the rows a and c of a task by one warp (the result in every lane),
// kTerms per lane on their way together (as the registers of five CTAs per SM allow).
struct WarpSum64 {
  static constexpr int kTerms = 3;
  cpx<double> acc = cpx<double>(0, 0);
  __device__ __forceinline__ void mac(double2 x, double2 y) { cmac(acc, cpx<double>(x.x, x.y), cpx<double>(y.x, y.y)); }
  __device__ __forceinline__ void join(int d) {
    acc.re += __shfl_xor_sync(0xffffffffu, acc.re, d);
    acc.im += __shfl_xor_sync(0xffffffffu, acc.im, d);
  }
  __device__ __forceinline__ double2 value() { return make_double2(acc.re, acc.im); }
};
struct WarpSumDf {
  static constexpr int kTerms = 2;
  df64acc re{0.f, 0.f}, im{0.f, 0.f};
  __device__ __forceinline__ void mac(float4 x, float4 y) {
    df_mac(re, x.x, x.y, y.x, y.y);
    df_mac(re, -x.z, -x.w, y.z, y.w);
    df_mac(im, x.x, x.y, y.z, y.w);
    df_mac(im, x.z, x.w, y.x, y.y);
  }
  __device__ __forceinline__ void join(df64acc& v, int d) {
    const float s = __shfl_xor_sync(0xffffffffu, v.s, d), e = __shfl_xor_sync(0xffffffffu, v.e, d);
    float t;
    two_sum(v.s, s, v.s, t);
    v.e = __fadd_rn(__fadd_rn(v.e, e), t);
  }
  __device__ __forceinline__ void join(int d) {
    join(re, d);
    join(im, d);
  }
  __device__ __forceinline__ float4 value() {
    df_renorm(re);
    df_renorm(im);
    return make_float4(re.s, re.e, im.s, im.e);
  }
};
template <typename Sum, typename Ld>
__device__ __forceinline__ Ld x_again(const Ld* rq, const Ld* rn, const DevTask* task, int i) {
  static_assert(sizeof(DevTask) == 21 * sizeof(int), "fields by position");
  const int lane = threadIdx.x & 31;
  const int f = lane < 21 ? __ldg(reinterpret_cast<const int*>(task) + lane) : 0;  // the task in one load
  auto field = [&](int at) { return __shfl_sync(0xffffffffu, f, at); };
  const int nB = field(16) >> 8, n2 = field(18), K = field(17) * n2, sA = field(19), sB = field(20);
  const Ld *a = rq + field(i / nB), *c = rn + field(8 + i % nB);
  Sum sum;
  constexpr int n = Sum::kTerms;
  for (int k0 = lane; k0 < K; k0 += 32 * n) {
    Ld x[n], y[n];
#pragma unroll
    for (int j = 0; j < n; j++) {
      const int k = min(k0 + 32 * j, K - 1), i1 = k / n2, i2 = k - i1 * n2;
      x[j] = __ldg(a + i1 * (sA & 0xffff) + i2 * (sA >> 16));
      y[j] = __ldg(c + i1 * (sB & 0xffff) + i2 * (sB >> 16));
    }
#pragma unroll
    for (int j = 0; j < n; j++)
      if (k0 + 32 * j < K) sum.mac(x[j], y[j]);
  }
#pragma unroll
  for (int d = 16; d; d >>= 1) sum.join(d);
  return sum.value();
}
template <typename T, typename C, typename Acc, typename Sum>
__global__ void __launch_bounds__(kWickThreads, 5)
k_exact_wick(const void* __restrict__ P, int n_items, const WickDev W, const C* __restrict__ coefs, int n_outputs,
             const void* __restrict__ blk, int L, int n_out, const DevTask* __restrict__ tasks,
             const int* __restrict__ err, void* __restrict__ ct) {
  using Ld = typename XRaw<T>::load;
  extern __shared__ __align__(128) unsigned char smem[];
  Ld* s_p = reinterpret_cast<Ld*>(smem);                                // [n_items]
  C* s_c = reinterpret_cast<C*>(smem + (size_t)n_items * sizeof(Ld));  // [n_coefs]
  uint32_t* s_again = reinterpret_cast<uint32_t*>(s_c + W.n_coefs);     // a bit per item
  const int q = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  {
    const Ld* src = reinterpret_cast<const Ld*>(P) + (size_t)q * n_items;
    for (int i = threadIdx.x; i < n_items; i += kWickThreads) cp_async16(s_p + i, src + i);
    for (int i = threadIdx.x; i < W.n_coefs; i += kWickThreads) s_c[i] = __ldg(coefs + i);
    cp_async_wait_all();
  }
  const bool lost = __ldg(err) & 2;  // a wait of the products gave up: they are not valid
  bool any = false;
  for (int i0 = 32 * warp; i0 < n_items; i0 += kWickThreads) {  // (each thread's own copies)
    const int i = i0 + lane;
    const uint32_t bits = __ballot_sync(0xffffffffu, i < n_items && s_p[i].x != s_p[i].x);
    if (lane == 0) s_again[i0 >> 5] = bits;
    any |= bits != 0;
  }
  if (__syncthreads_or(any)) {
    const Ld* F = reinterpret_cast<const Ld*>(blk);
    const Ld *rq = F + (size_t)q * n_out, *rn = F + (size_t)x_neg_site(q, L) * n_out;
    // a warp takes every eighth marked product (they come in runs and patterns)
    const int words = (n_items + 31) / 32;
    int n = 0;
    for (int w0 = 0; w0 < words; w0 += 32) {
      const uint32_t word = w0 + lane < words ? s_again[w0 + lane] : 0;
      for (uint32_t live = __ballot_sync(0xffffffffu, word != 0); live; live &= live - 1) {
        const int l = __ffs((int)live) - 1;
        for (uint32_t bits = __shfl_sync(0xffffffffu, word, l); bits; bits &= bits - 1)
          if (n++ % (kWickThreads / 32) == warp) {
            const int item = 32 * (w0 + l) + __ffs((int)bits) - 1;
            const Ld v = x_again<Sum>(rq, rn, tasks + (item >> 4), item & 15);
            if (lane == 0) s_p[item] = v;
          }
      }
    }
    __syncthreads();
  }
  for (int c = warp; c < W.n_chunks; c += kWickThreads / 32) {
    const Ld* p = s_p;
    const int2 ch = __ldg(W.chunks + c);  // offset, terms of the longest output
    const int2 out = __ldg(W.outputs + 32 * c + lane);  // output (-1: none), its terms
    const uint32_t* ep = W.ell + ch.x + lane;
    Acc acc;
    for (int j0 = 0; j0 < ch.y; j0 += 4) {  // four terms and their products on their way together
      uint32_t e[4];
      Ld v[4];
#pragma unroll
      for (int j = 0; j < 4; j++) e[j] = __ldg(ep + 32 * min(j0 + j, ch.y - 1));
#pragma unroll
      for (int j = 0; j < 4; j++) v[j] = p[e[j] & 0xffffu];
#pragma unroll
      for (int j = 0; j < 4; j++)
        if (j0 + j < out.y) acc.add(s_c[e[j] >> 16], v[j]);
      if ((j0 & 12) == 12) acc.renorm();  // every 16 terms
    }
    if (out.x >= 0) reinterpret_cast<Ld*>(ct)[(size_t)q * n_outputs + out.x] = lost ? x_value(Ld(), 0, 0, kXBad) : acc.value();
  }
}

struct XShared {
  uint64_t bars[kExactSets][2 * kXMaxStages + 5];  // one group per operand set
  uint32_t tmem;
  int abort;
  short ex[2][kExactMaxSliceA], ey[2][kExactMaxBlocks];  // exponents of the product's operand rows, by parity
};
static_assert(sizeof(XShared) <= kXFixed && kExactMaxBlocks >= kExactMaxSliceB && kExactMaxSliceA >= kExactMaxBlocks,
              "exponents of either set");

// One operand set: the products of qlist[n_q] (nullptr: q = 0 .. n_q - 1).
template <typename T, int FORM>
__device__ __forceinline__ void exact_set(unsigned char* smem, XShared& xs, const void* __restrict__ blk, int L,
                                          int n_out, const ExactDev& S, const int* __restrict__ E, int n_jobs,
                                          const int* __restrict__ qlist, int n_q, void* __restrict__ P,
                                          int n_items, long long spin_limit) {
  constexpr int STACK = FORM < kExactSlice ? 2 : 1;
  using Raw = XRaw<T>;
  using Ld = typename Raw::load;
  constexpr int ND = kXDigits;
  const Ld* F = reinterpret_cast<const Ld*>(blk);
  uint64_t* bars = xs.bars[FORM];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const XShape sh = x_shape(STACK, S.nAp, S.nBp);
  const int NS = sh.n_stages, NB = S.nBp, nC = (S.K + 15) / 16;
  const int TA = S.nAp / 16, TT = TA + NB / 16;  // warp tasks per stage: 16 rows x 2 k-groups each
  const int n_mine = (n_q - 1 - (int)blockIdx.x) / (int)gridDim.x + 1;
  const int bufW = (STACK == 2 ? ND : 2 * ND) * NB, n_buf = 2 * bufW <= kXCols ? 2 : 1;
  const uint32_t bar_full = x_smem(bars), bar_empty = bar_full + 8 * kXMaxStages;
  const uint32_t bar_acc = bar_empty + 8 * kXMaxStages, bar_free = bar_acc + 16, bar_drain = bar_free + 16;
  if (tid == 0) {
    for (int i = 0; i < NS; i++) {
      x_mbar_init(bar_full + 8 * i, TT);
      x_mbar_init(bar_empty + 8 * i, 1);
    }
    for (int i = 0; i < 2; i++) {
      x_mbar_init(bar_acc + 8 * i, 1);
      x_mbar_init(bar_free + 8 * i, kXEpi);
    }
    x_mbar_init(bar_drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (STACK == 2) {  // the slices of zeros
    for (int i = tid; i < NS * 2 * (sh.slA / 16); i += kXWarps * 32) {
      const int st = i / (2 * (sh.slA / 16)), r = i % (2 * (sh.slA / 16));
      const int part = r / (sh.slA / 16), o = r % (sh.slA / 16);
      reinterpret_cast<uint4*>(smem + (size_t)st * sh.stage + part * sh.partA)[o] = make_uint4(0, 0, 0, 0);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncthreads();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(&xs.tmem);
  volatile int* abort_flag = &xs.abort;
  auto q_of = [&](int i) {
    const int p = blockIdx.x + i * (int)gridDim.x;
    return qlist ? __ldg(qlist + p) : p;
  };

  if (warp > kXEpi) {
    // ------------------------------------------------------- producers
    // Warp tasks in order: product i, chunk c of 16 open indices, then 16 operand
    // rows (A's, then B's) x 2 groups of 8 indices; warp pw takes every kXProd-th.
    struct Cursor {
      int i, c, w, st, n, q, nq;  // n: earlier uses of stage st
    };
    const int pw = warp - kXEpi - 1;
    const int r8 = lane & 7, kg = (lane >> 3) & 1, rg = lane >> 4;
    auto start = [&](Cursor& t) {
      t.i = t.c = t.st = t.n = 0;
      t.w = pw;
      t.q = q_of(0);
      t.nq = x_neg_site(t.q, L);
    };
    auto settle = [&](Cursor& t) {  // w back below TT; false past the last product
      while (t.w >= TT) {
        t.w -= TT;
        if (++t.st == NS) {
          t.st = 0;
          t.n++;
        }
        if (++t.c == nC) {
          t.c = 0;
          if (++t.i >= n_mine) return false;
          t.q = q_of(t.i);
          t.nq = x_neg_site(t.q, L);
        }
      }
      return true;
    };
    Ld v[8];
    int e = 0;
    auto load = [&](const Cursor& t) {
      const bool sideB = t.w >= TA;
      const int row = 16 * (sideB ? t.w - TA : t.w) + 8 * rg + r8;
      const int q = sideB ? t.nq : t.q;
      e = 0;
#pragma unroll
      for (int j = 0; j < 8; j++) v[j] = Ld();
      if (row < (sideB ? S.nB : S.nA)) {
        const Ld* p = F + (size_t)q * n_out + __ldg((sideB ? S.rowB : S.rowA) + row);
        e = __ldg(E + (size_t)q * n_jobs + __ldg((sideB ? S.expB : S.expA) + row));
        e = abs(e) > kXNone ? 0 : e;  // any digits, or zeros
        if (STACK == 2) {
          // chunk c is the 4 x 4 tile (u, v) = (4 tu .., 4 tv ..) of the open
          // indices, k-group kg its u = 4 tu + 2 kg + (0, 1): values j = 4 du + dv
          // are element 12 u + v of A's block and of B's, or 12 v + u of B's (transposed)
          const int tu = t.c / 3, tv = t.c - 3 * tu;
          if (FORM == kExactTrace && sideB) {
            p += 48 * tv + 4 * tu + 2 * kg;
#pragma unroll
            for (int dv = 0; dv < 4; dv++) x_pair(p + 12 * dv, v, dv);
          } else {
            p += 48 * tu + 24 * kg + 4 * tv;
            x_run4(p, v, 0);
            x_run4(p + 12, v, 4);
          }
        } else {
          const int k0 = 16 * t.c + 8 * kg;
          if (FORM == kExactSliceT && !sideB) {  // k = 12 i2 + i1 is element 12 i1 + i2
#pragma unroll
            for (int j = 0; j < 8; j++) {
              const int k = k0 + j, i2 = k / 12;
              if (k < S.K) v[j] = __ldg(p + 12 * (k - 12 * i2) + i2);
            }
          } else {
            if (k0 < S.K) x_run4(p + k0, v, 0);  // K is a multiple of 4
            if (k0 + 4 < S.K) x_run4(p + k0 + 4, v, 4);
          }
        }
      }
    };
    Cursor t;
    start(t);
    bool more = settle(t);
    if (more) load(t);
    while (more) {
      const Cursor now = t;
      unsigned long long u[2][8];
#pragma unroll
      for (int j = 0; j < 8; j++) {
        u[0][j] = x_fix(Raw::re(v[j]), e);
        u[1][j] = x_fix(Raw::im(v[j]), e);
      }
      t.w += kXProd;
      more = settle(t);
      if (more) load(t);  // the next rows fly while these are stored
      if (now.n > 0) {
        const bool ok = x_wait(bar_empty + 8 * now.st, (uint32_t)((now.n - 1) & 1), spin_limit, abort_flag);
        if (!__all_sync(0xffffffffu, ok)) break;
      }
      const bool sideB = now.w >= TA;
      const int row0 = 16 * (sideB ? now.w - TA : now.w) + 8 * rg;
      unsigned char* dst = smem + (size_t)now.st * sh.stage + (row0 >> 3) * 256 + kg * 128 + r8 * 16;
#pragma unroll
      for (int part = 0; part < 2; part++) {
        if (sideB) {
          // STACK 2: even digits, then odd digits
          x_store_digits(u[part], dst + sh.off_b + part * ND * sh.slB, [&](int d) {
            return (STACK == 2 ? (d & 1) * (ND / 2) + (d >> 1) : d) * sh.slB;
          });
        } else {
          x_store_digits(u[part], dst + part * sh.partA + (STACK == 2 ? sh.slA : 0), [&](int d) { return d * sh.slA; });
        }
      }
      __syncwarp();
      if (lane == 0) x_arrive(bar_full + 8 * now.st);  // (release; the MMA thread orders the proxies)
    }
  } else if (warp == kXEpi) {
    // ------------------------------------------------------- MMA issue
    // The warp runs the loop together, so that descriptors stay in uniform
    // registers; one elected thread issues.  Per window: offsets of its first A
    // and B slice in descriptor units, its first accumulator column, its
    // instructions' descriptors.
    uint32_t wa[ND], wb[ND], wn[ND];
    int wc[ND];
#pragma unroll
    for (int w = 0; w < ND; w++) {
      // STACK 2: slices of A count from the zeros (digit i is slice i + 1);
      // windows at even digits, then at odd ones from the zeros
      const int col = STACK == 2 ? w % (ND / 2) : w;
      const bool odd = STACK == 2 && w >= ND / 2;
      wa[w] = (uint32_t)((STACK == 2 ? (odd ? 2 * col : 2 * col + 1) : w) * sh.slA) >> 4;
      wb[w] = (uint32_t)((odd ? ND / 2 : 0) * sh.slB) >> 4;
      wc[w] = col * NB;
      wn[w] = x_idesc(NB * ((STACK == 2 ? ND / 2 : ND) - col), 0);
    }
    const uint64_t desc0 = x_desc(x_smem(smem));
    const uint32_t d_im_part = (uint32_t)sh.partA >> 4, b_im_part = (uint32_t)(ND * sh.slB) >> 4;
    const bool leader = x_elect();
    int st = 0;
    uint32_t ph = 0;
    for (int i = 0; i < n_mine; i++) {
      const int buf = n_buf == 2 ? i & 1 : 0, m = n_buf == 2 ? i >> 1 : i;
      bool ok = m == 0 || x_wait(bar_free + 8 * buf, (uint32_t)((m - 1) & 1), spin_limit, abort_flag);
      if (!__all_sync(0xffffffffu, ok)) break;
      x_fence_after();
      const uint32_t d_re = tmem + buf * bufW, d_im = d_re + bufW / 2;
      for (int c = 0; c < nC; c++) {
        ok = __all_sync(0xffffffffu, x_wait(bar_full + 8 * st, ph, spin_limit, abort_flag));
        if (!ok) break;
        // the producers' stores, acquired through the barrier, before the
        // tensor core's reads of the same bytes (a fence in each producer
        // would also wait for the row loads it has in flight)
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        x_fence_after();
        const uint64_t da = desc0 + (uint32_t)(st * (sh.stage >> 4)), db = da + (uint32_t)(sh.off_b >> 4);
        const uint32_t first = c == 0 ? 0u : 1u;  // the first window covers every column
        if (leader) {
#pragma unroll
          for (int w = 0; w < ND; w++) {
            const uint64_t are = da + wa[w], aim = are + d_im_part, bre = db + wb[w], bim = bre + b_im_part;
            x_mma(d_re + wc[w], are, bre, wn[w], w == 0 ? first : 1u);
            x_mma(d_im + wc[w], are, bim, wn[w], w == 0 ? first : 1u);
            x_mma(d_re + wc[w], aim, bim, wn[w] | (1u << 13), 1u);
            x_mma(d_im + wc[w], aim, bre, wn[w], 1u);
          }
          x_commit(bar_empty + 8 * st);
          if (c == nC - 1) x_commit(bar_acc + 8 * buf);
        }
        __syncwarp();
        if (++st == NS) {
          st = 0;
          ph ^= 1;
        }
      }
      if (!ok) break;
    }
    // every MMA issued has finished before the tensor memory is freed, also when a
    // wait above gave up early; this wait has its own, long limit
    if (leader) {
      x_commit(bar_drain);
      long long polls = 0;
      for (; !x_test(bar_drain, 0) && polls < kXDrainLimit; polls++) __nanosleep(20);
      if (polls == kXDrainLimit) *abort_flag = 1;
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------- epilogue
    // First every sum of levels leaves the accumulator as a 64-bit integer into
    // shared memory, so that the next product may overwrite it; then the entries
    // that some task reads are scaled, rounded and stored, spread over all threads.
    long long* sums = reinterpret_cast<long long*>(smem + (size_t)NS * sh.stage);  // [STACK][2 nB][nAp]
    const int half = warp >> 2;            // which groups of 4 columns (even, odd)
    const int r = 32 * (warp & 3) + lane;  // row of D
    const bool has = 32 * (warp & 3) < STACK * S.nAp;  // (warp) rows of D that are read
    const bool top = r < S.nAp, mine = r < STACK * S.nAp;
    long long* dst = sums + (top ? r : r - S.nAp + 2 * NB * S.nAp);  // STACK 2: even levels first, then the odd ones
    const uint32_t tw = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
    // the entries of this thread are the same in every product: the first ones stay
    // in registers (row | column << 16, item at q | item at -q << 16)
    constexpr int kHeld = STACK == 2 ? 6 : 4;
    int2 held[kHeld];
#pragma unroll
    for (int j = 0; j < kHeld; j++) {
      const int t = tid + j * 32 * kXEpi;
      held[j] = t < S.n_ent ? __ldg(S.entries + t) : make_int2(0, -1);  // -1: no items
    }
    // exponents are read one product ahead
    const int jx = tid < S.nA ? __ldg(S.expA + tid) : 0, jy = tid < S.nB ? __ldg(S.expB + tid) : 0;
    int q = q_of(0), nq = x_neg_site(q, L);
    int ex_next = __ldg(E + (size_t)q * n_jobs + jx), ey_next = __ldg(E + (size_t)nq * n_jobs + jy);
    for (int i = 0; i < n_mine; i++) {
      const int buf = n_buf == 2 ? i & 1 : 0, m = n_buf == 2 ? i >> 1 : i;
      short* s_ex = xs.ex[i & 1];
      short* s_ey = xs.ey[i & 1];
      if (tid < S.nA) s_ex[tid] = (short)ex_next;
      if (tid < S.nB) s_ey[tid] = (short)ey_next;
      Ld* pq = reinterpret_cast<Ld*>(P) + (size_t)q * n_items;
      Ld* pn = reinterpret_cast<Ld*>(P) + (size_t)nq * n_items;
      const bool self = STACK == 2 && nq == q;  // q = -q has its products from the items at q
      if (i + 1 < n_mine) {
        q = q_of(i + 1);
        nq = x_neg_site(q, L);
        ex_next = __ldg(E + (size_t)q * n_jobs + jx);
        ey_next = __ldg(E + (size_t)nq * n_jobs + jy);
      }
      const bool ok = x_wait(bar_acc + 8 * buf, (uint32_t)(m & 1), spin_limit, abort_flag);
      if (!x_all_epi(ok)) break;  // one verdict for all of them; the sums of the last product are read
      x_fence_after();
      const uint32_t d_re = tw + buf * bufW, d_im = d_re + bufW / 2;
      for (int j0 = 4 * half; has && j0 < S.nB; j0 += 8) {
        // a group's level sums: STACK 2, level 2 c of the first rows of D and 2 c + 1
        // of the next at column block c; STACK 1, level c at column block c
        constexpr int NC = STACK == 2 ? ND / 2 : ND;
#pragma unroll
        for (int part = 0; part < 2; part++) {
          uint32_t a[NC][4], wide = 0;
#pragma unroll
          for (int c = 0; c < NC; c++) x_ld4((part ? d_im : d_re) + c * NB + j0, a[c]);
#pragma unroll
          for (int c = 0; c < NC; c++) x_wait_ld(a[c]);
          long long v[4];
#pragma unroll
          for (int j = 0; j < 4; j++) v[j] = x_levels(a, j, top, wide);
          if (wide & 0xff800000u) {
#pragma unroll
            for (int j = 0; j < 4; j++) v[j] = x_levels_wide(a, j, top);
          }
          __syncwarp();
          if (mine) {
#pragma unroll
            for (int j = 0; j < 4; j++) dst[(part * NB + j0 + j) * S.nAp] = v[j];
          }
        }
      }
      x_fence_before();
      __syncwarp();
      if (lane == 0) x_arrive(bar_free + 8 * buf);
      asm volatile("bar.sync 1, %0;" ::"n"(32 * kXEpi) : "memory");  // the sums are in place
      auto entry = [&](int2 en) {
        const int row = en.x & 0xffff, col = en.x >> 16;
        const long long* p = sums + col * S.nAp + row;
        long long re = p[0], im = p[NB * S.nAp];
        if (STACK == 2) {
          re += p[2 * NB * S.nAp];
          im += p[3 * NB * S.nAp];
        }
        // the sum is (sum of T_A T_B) 2^-56, T = x 2^(55 - e): 2^54 stands for the
        // product of the rows' bounds.  NaN marks what k_exact_wick makes again.
        const int e = s_ex[row] + s_ey[col], hr = (int)(re >> 32), hi = (int)(im >> 32);
        const bool far = max(hr ^ (hr >> 31), hi ^ (hi >> 31)) < (1 << (22 - kXFar));
        const bool again = e > kXNone || (e >= -kXNone && (far || e < XLimits<T>::kLowProduct));
        const Ld v = x_value(Ld(), re, im, again ? kXBad : e - 54);
        const int item_q = (int)(short)en.y, item_n = en.y >> 16;
        if (item_q >= 0) pq[item_q] = v;
        if (item_n >= 0 && !self) pn[item_n] = v;
      };
#pragma unroll
      for (int j = 0; j < kHeld; j++) entry(held[j]);
      for (int t = tid + kHeld * 32 * kXEpi; t < S.n_ent; t += 32 * kXEpi) entry(__ldg(S.entries + t));
    }
  }
  // every warp has left its loop: accumulators read, stages free
  x_fence_before();
  __syncthreads();
  x_fence_after();
}

template <typename T, int FORM>
__device__ __forceinline__ void exact_form(unsigned char* smem, XShared& xs, const void* blk, int L, int n_out,
                                           const ExactArgs& A, const int* E, const int* qlist, int n_q, void* P,
                                           long long spin_limit) {
  if (A.set[FORM].nAp && (int)blockIdx.x < n_q && !*(volatile int*)&xs.abort)
    exact_set<T, FORM>(smem, xs, blk, L, n_out, A.set[FORM], E, A.n_jobs, qlist, n_q, P, A.n_items, spin_limit);
}

// blk: q-major blocks [V][n_out]; P[V][n_items]; the trace sets run over the
// pairs qlist[n_pairs], the slice sets over every q.  err: bit 1 is set when a
// wait gave up.
template <typename T>
__global__ void __launch_bounds__(kXWarps * 32, 1)
k_contract_exact(const void* __restrict__ blk, int L, int n_out, const ExactArgs A, const int* __restrict__ E,
                 const int* __restrict__ qlist, int n_pairs, void* __restrict__ P, int* __restrict__ err,
                 long long spin_limit) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ XShared xs;
  const int tid = threadIdx.x, warp = tid >> 5, V = L * L * L;
  if (tid == 0) xs.abort = 0;
  if (warp == kXEpi) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(x_smem(&xs.tmem)),
                 "r"(kXCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  x_fence_before();
  __syncthreads();
  x_fence_after();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(&xs.tmem);
  exact_form<T, kExactTrace>(smem, xs, blk, L, n_out, A, E, qlist, n_pairs, P, spin_limit);
  exact_form<T, kExactSame>(smem, xs, blk, L, n_out, A, E, qlist, n_pairs, P, spin_limit);
  exact_form<T, kExactSlice>(smem, xs, blk, L, n_out, A, E, nullptr, V, P, spin_limit);
  exact_form<T, kExactSliceT>(smem, xs, blk, L, n_out, A, E, nullptr, V, P, spin_limit);
  if (tid == 0 && *(volatile int*)&xs.abort) atomicOr(err, 2);
  if (warp == kXEpi)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kXCols) : "memory");
}

static bool exact_set_ok(const ExactDev& S, int form) {
  if (S.nAp == 0) return true;
  const int stack = form < kExactSlice ? 2 : 1;
  // a window of 128 rows that starts at the last slices reads past them into
  // the B digits: that stays inside the stage
  return S.nAp % 16 == 0 && S.nBp % 16 == 0 && S.nA <= S.nAp && S.nB <= S.nBp &&
         (stack == 2 ? S.nAp <= kExactMaxBlocks && S.nAp == S.nBp && S.K == 144
                     : S.nAp <= kExactMaxSliceA && S.nBp <= kExactMaxSliceB && S.K <= 144 && S.K % 4 == 0) &&
         x_shape(stack, S.nAp, S.nBp).n_stages >= 2;
}

cudaError_t launch_exact_exponents(const void* blk, bool df, long long n_q, int n_out, const ExactArgs& a, int* E,
                                   cudaStream_t st) {
  if (n_q <= 0 || a.n_jobs <= 0) return cudaErrorInvalidValue;
  if (df)
    k_exact_exponents<dfr><<<(unsigned)n_q, 256, 0, st>>>(blk, n_out, a.loads, a.n_loads, a.jobs, a.n_jobs, E);
  else
    k_exact_exponents<double><<<(unsigned)n_q, 256, 0, st>>>(blk, n_out, a.loads, a.n_loads, a.jobs, a.n_jobs, E);
  return cudaGetLastError();
}

template <typename T>
static cudaError_t launch_exact_t(const void* blk, int L, int n_out, const ExactArgs& a, const int* E,
                                  const int* qlist, int n_pairs, void* P, int* err, long long spin_limit, int n_sm,
                                  cudaStream_t st) {
  const int V = L * L * L;
  if (a.n_small > 0) {
    k_exact_small<T><<<V, 256, 0, st>>>(blk, L, n_out, a.tasks, a.small, a.n_small, a.n_items, P);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  size_t sm = 0;
  int n_q = n_pairs;
  for (int form = 0; form < kExactSets; form++) {
    const ExactDev& S = a.set[form];
    if (!S.nAp) continue;
    if (!exact_set_ok(S, form)) return cudaErrorInvalidValue;
    sm = std::max(sm, (size_t)x_shape(form < kExactSlice ? 2 : 1, S.nAp, S.nBp).bytes);
    if (form >= kExactSlice) n_q = V;
  }
  if (!sm) return cudaErrorInvalidValue;
  static int granted[64] = {0};
  const cudaError_t e = ensure_smem(k_contract_exact<T>, sm, granted);
  if (e != cudaSuccess) return e;
  k_contract_exact<T><<<std::min(n_q, n_sm), kXWarps * 32, sm, st>>>(blk, L, n_out, a, E, qlist, n_pairs, P, err,
                                                                     spin_limit);
  return cudaGetLastError();
}

cudaError_t launch_contract_exact(const void* blk, int L, int n_out, bool df, const ExactArgs& a, const int* E,
                                  const int* qlist, int n_pairs, void* P, int* err, long long spin_limit,
                                  cudaStream_t st) {
  // 32-byte loads: rows and row length even (exact_split.cpp takes no other plan)
  if ((n_out & 1) || (((uintptr_t)blk) & 31) || !err) return cudaErrorInvalidValue;
  static int n_sm[64] = {0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!n_sm[dev]) {
    e = cudaDeviceGetAttribute(&n_sm[dev], cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
  }
  return df ? launch_exact_t<dfr>(blk, L, n_out, a, E, qlist, n_pairs, P, err, spin_limit, n_sm[dev], st)
            : launch_exact_t<double>(blk, L, n_out, a, E, qlist, n_pairs, P, err, spin_limit, n_sm[dev], st);
}

static size_t wick_smem(int n_items, int n_coefs) {
  return 16 * (size_t)n_items + 8 * (size_t)n_coefs + 4 * (((size_t)n_items + 31) / 32);
}
bool exact_wick_fits(int n_items, int n_coefs) { return wick_smem(n_items, n_coefs) <= kMaxSmemPerBlock; }

template <typename T, typename C, typename Acc, typename Sum>
static cudaError_t launch_wick_t(const void* P, int L, const ExactArgs& a, const C* coefs, int n_outputs,
                                 const void* blk, int n_out, const int* err, void* ct, cudaStream_t st) {
  const size_t sm = wick_smem(a.n_items, a.wick.n_coefs);
  if (sm > kMaxSmemPerBlock) return cudaErrorInvalidValue;
  static int granted[64] = {0};
  const cudaError_t e = ensure_smem(k_exact_wick<T, C, Acc, Sum>, sm, granted);
  if (e != cudaSuccess) return e;
  k_exact_wick<T, C, Acc, Sum><<<(unsigned)(L * L * L), kWickThreads, sm, st>>>(P, a.n_items, a.wick, coefs, n_outputs, blk,
                                                                           L, n_out, a.tasks, err, ct);
  return cudaGetLastError();
}

cudaError_t launch_exact_wick(const void* P, int L, const ExactArgs& a, bool df, int n_outputs, const void* blk,
                              int n_out, const int* err, void* ct, cudaStream_t st) {
  return df ? launch_wick_t<dfr, float2, WickAccDf, WarpSumDf>(P, L, a, a.wick.coefs_df, n_outputs, blk, n_out, err, ct, st)
            : launch_wick_t<double, double, WickAcc64, WarpSum64>(P, L, a, a.wick.coefs, n_outputs, blk, n_out, err, ct, st);
}

}  // namespace bbc
