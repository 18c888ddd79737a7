// tc_exact.cu -- block-pair products of the FP64-accurate paths (FP64,
// double-float) on the fifth-generation tensor cores, exact up to one rounding
// (Sec. 3 Eq. LN.pLLp.FFT: sums over open indices of A(q) B(-q)).
//
// Every operand value x of a row with max |x| < 2^e becomes the integer
// T = round(x 2^(55 - e)), written in eight signed digits of 7 bits, d_i in
// [-64, 63], T = sum_i d_i 2^(7 (7 - i)).  The digits are small integers in
// fp16, their products are exact in the FP32 accumulators of tcgen05.mma
// (kind::f16), and so are the sums: the digit products of one weight ("level"
// s = i + j) of a complex product of K = 144 terms add up to at most
// 8 x 288 x 64^2 < 2^24.  Levels 0 .. 7 are kept, an absolute error of
// about 2^-54 of (row maximum)^2 per product, below the rounding errors of
// the FP64 sums this replaces; the levels are put together in 64-bit integers
// and rounded once.  (This is the splitting idea of Ozaki, Ogita, Oishi and
// Rump, Numer. Algorithms 59 (2012), with the products on integers.)
//
// A digit pair costs 4 real MACs per complex one at 4096 MACs per clock and
// SM against 2 FP64 FMAs per clock (three per complex MAC) or 128 FP32 lanes
// (48 instructions per complex MAC in double-float): 36 digit pairs are still
// many times cheaper than either pipe.  What bounds the kernel is the tensor
// pipe together with the integer work of making the digits (about 35
// instructions per real value).  Measured against the CUDA-core products of
// field-major blocks, 52 channels: FP64 16^3 3.99 -> 0.57 ms per slice,
// double-float 16^3 1.40 -> 0.52, 48^3 35.2 -> 13.0 (both with the small tasks).
// On field-major blocks (16-byte loads 64 KB and more apart) the same kernel was
// TLB bound at 0.98 and 45 ms: the blocks are q-major for it.
//
// Two operand sets (exact_split.cpp):
//   trace form, one product per pair {q, -q}: STACK = 2.  Two digit slices of
//     A (nbp <= 64 rows each) fill one M = 128 instruction, so a window that
//     starts at slice i gives level i + j in its first nbp rows of D and
//     i + j + 1 in the next nbp: four column blocks hold the eight levels.
//     Even digits of B are adjacent (so are odd ones): one instruction with N
//     = nbp n multiplies a window by n of them into n adjacent column blocks.
//     Windows at even i take the even digits, at odd i (from -1, a slice of
//     zeros in front) the odd ones, so every digit pair up to level 7 is met
//     once.
//   slice form, one product per q: STACK = 1.  The window is one slice (up to
//     128 rows), all eight levels are column blocks of nB columns, and digit i
//     of A meets digits 0 .. 7 - i of B in one instruction.
// Re = Re Re - Im Im uses the instruction's negated A.
//
// A persistent CTA per SM: warps 0-7 read the accumulators, warp 8 issues the
// MMAs, the others load rows of the q-major blocks (32-byte loads; a pair's rows
// lie in two runs of n_out values), split them and store the digits in the canonical K-major
// layout without swizzle, 16 open indices per stage of an mbarrier ring.
// Every wait is bounded: past its limit, or when another warp gave up, the
// warps leave their loops, the MMAs in flight are waited for (bounded), the
// tensor memory is freed and bit 1 of the error word is set.
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
constexpr int kXMaxStages = 8;
constexpr int kXCols = 512;                    // all of tensor memory: one CTA per SM
constexpr int kXFixed = 2048;                  // static shared memory (at most)
constexpr int kXBad = 0x7fffffff;              // exponent of a row with a NaN or infinite value

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
// 17 bits of the high word, then the rest of it with the low word (the low word
// is a few units of the high word's last place, so their sum loses nothing that
// T holds), 17 + 17 bits.  FP32 additions run at twice the rate of shifts.
__device__ __forceinline__ unsigned long long x_fix(dfr x, int e) {
  const float M = 12582912.f, p17 = 131072.f;  // 1.5 2^23, 2^17
  const float s = __int_as_float((127 + 21 - e) << 23);  // 2^(21 - e), e >= -72
  const float h = __fmul_rn(x.hi, s);
  const float t0 = __fadd_rn(h, M), r0 = __fsub_rn(h, __fsub_rn(t0, M));
  const float t1 = __fmaf_rn(r0, p17, M), r1 = __fmaf_rn(r0, p17, -__fsub_rn(t1, M));
  const float y = __fmaf_rn(x.lo, __fmul_rn(s, p17), r1);
  const float t2 = __fadd_rn(y, M), r2 = __fsub_rn(y, __fsub_rn(t2, M));
  const float t3 = __fmaf_rn(r2, p17, M);
  constexpr long long Mb = 0x4B400000;
  constexpr unsigned long long off = kXBias - (unsigned long long)(((Mb << 17) + 2 * Mb) * 131072 + Mb);
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
// weights 2^42, 2^28, 2^14, 1 (shift 0: the even levels) or 2^35, 2^21, 2^7, 2^-7 (the odd ones)
__device__ __forceinline__ long long x_sum4(long long n0, long long n1, long long n2, long long n3, bool even) {
  const long long e = (n0 << 28) + (n1 << 14) + n2;
  return even ? (e << 14) + n3 : (e << 7) + (n3 >> 7);
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

template <typename T>
struct XRaw;  // a loaded complex value: re, im
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
// rows below 0.985 2^E (kXBad: a NaN or infinite value among them); a warp per
// job, one pass over the operand rows: HBM bound.
template <typename T>
__global__ void __launch_bounds__(256)
k_exact_exponents(const float4* __restrict__ F, int n_out, const int* __restrict__ jobs, int n_jobs,
                  int* __restrict__ E) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float4* row = F + (size_t)blockIdx.x * n_out;
  for (int job = warp; job < n_jobs; job += 8) {
    const int first = __ldg(jobs + 2 * job), rows = __ldg(jobs + 2 * job + 1);
    int m = 0;
#pragma unroll 5
    for (int r = lane; r < rows; r += 32) {
      const float4 v = __ldg(row + first + r);
      // the exponent-carrying words of re and im; double-float: both words count
      const float x = std::is_same<T, double>::value ? v.y : fabsf(v.x) + fabsf(v.y);
      const float y = std::is_same<T, double>::value ? v.w : fabsf(v.z) + fabsf(v.w);
      m = max(m, max(__float_as_int(x) & 0x7fffffff, __float_as_int(y) & 0x7fffffff));
    }
    m = __reduce_max_sync(0xffffffffu, m);
    // 2^-5 of headroom in the significand: the largest magnitude has to fit
    // eight digits whose range is [-64, 63]; a row of zeros or subnormals counts as zero
    int e;
    if (std::is_same<T, double>::value) e = m >= 0x7ff00000 ? kXBad : m < 0x100000 ? 0 : ((m + 0x8000) >> 20) - 1022;
    else e = m >= 0x7f800000 ? kXBad : max(((m + 0x40000) >> 23) - 126, -72);
    if (lane == 0) E[(size_t)blockIdx.x * n_jobs + job] = e;
  }
}

// Products of the tasks with few open indices (a few percent of the work): one
// CTA per q, one product per thread.
template <typename T>
__global__ void __launch_bounds__(256)
k_exact_small(const float4* __restrict__ F, int L, int n_out, const DevTask* __restrict__ tasks,
              const int* __restrict__ small, int n_small, int n_items, float4* __restrict__ P) {
  const int q = blockIdx.x, nq = x_neg_site(q, L);
  for (int u = threadIdx.x; u < n_small * 16; u += 256) {
    const int ti = __ldg(small + (u >> 4)), i = u & 15;
    const DevTask& t = tasks[ti];
    const int nB = t.nAnB >> 8;
    const float4* a = F + (size_t)q * n_out + t.offA[i / nB];
    const float4* c = F + (size_t)nq * n_out + t.offB[i % nB];
    const int sA1 = t.sA & 0xffff, sA2 = t.sA >> 16, sB1 = t.sB & 0xffff, sB2 = t.sB >> 16;
    float4* out = P + (size_t)q * n_items + ti * 16 + i;
    if constexpr (std::is_same<T, double>::value) {
      cpx<double> acc(0, 0);
      for (int i1 = 0; i1 < t.n1; i1++)
        for (int i2 = 0; i2 < t.n2; i2++) {
          const double2 x = __ldg((const double2*)(a + i1 * sA1 + i2 * sA2));
          const double2 y = __ldg((const double2*)(c + i1 * sB1 + i2 * sB2));
          cmac(acc, cpx<double>(x.x, x.y), cpx<double>(y.x, y.y));
        }
      *(double2*)out = make_double2(acc.re, acc.im);
    } else {
      df64acc re{0.f, 0.f}, im{0.f, 0.f};
      for (int i1 = 0; i1 < t.n1; i1++)
        for (int i2 = 0; i2 < t.n2; i2++) {
          const float4 x = __ldg(a + i1 * sA1 + i2 * sA2);
          const float4 y = __ldg(c + i1 * sB1 + i2 * sB2);
          df_mac(re, x.x, x.y, y.x, y.y);
          df_mac(re, -x.z, -x.w, y.z, y.w);
          df_mac(im, x.x, x.y, y.z, y.w);
          df_mac(im, x.z, x.w, y.x, y.y);
        }
      df_renorm(re);
      df_renorm(im);
      *out = make_float4(re.s, re.e, im.s, im.e);
    }
  }
}

// Signed sums over Wick diagrams of q-major products, ct[q][o] = sum_c coef_c
// P[q][item_c]: one CTA per kWickQ values of q stages their product rows in
// shared memory, so that every product is read once and the term lists once
// per kWickQ.  FP64, or double-float with the coefficients split on the host,
// renormalised every 16 terms.
constexpr int kWickQ = 2, kWickThreads = 512;
template <typename T, typename C>
__global__ void __launch_bounds__(kWickThreads)
k_exact_wick(const float4* __restrict__ P, int V, int n_items, const int* __restrict__ cptr,
             const int* __restrict__ citem, const C* __restrict__ ccoef, int n_outputs, float4* __restrict__ ct) {
  extern __shared__ __align__(16) unsigned char smem[];
  float4* s_p = reinterpret_cast<float4*>(smem);  // [kWickQ][n_items]
  const int q0 = blockIdx.x * kWickQ, nq = min(kWickQ, V - q0);
  for (int i = threadIdx.x; i < nq * n_items; i += kWickThreads) cp_async16(s_p + i, P + (size_t)q0 * n_items + i);
  cp_async_wait_all();
  __syncthreads();
  for (int u = threadIdx.x; u < nq * n_outputs; u += kWickThreads) {
    const int k = u / n_outputs, o = u - k * n_outputs;
    const float4* p = s_p + (size_t)k * n_items;
    const int c0 = __ldg(cptr + o), c1 = __ldg(cptr + o + 1);
    float4* out = ct + (size_t)(q0 + k) * n_outputs + o;
    if constexpr (std::is_same<T, double>::value) {
      double2 s = make_double2(0.0, 0.0);
      for (int c = c0; c < c1; c += 4) {  // four terms' coefficients and products on their way together
        C w[4];
        float4 v[4];
#pragma unroll
        for (int j = 0; j < 4; j++) {
          const int cj = min(c + j, c1 - 1);
          w[j] = __ldg(ccoef + cj);
          v[j] = p[__ldg(citem + cj)];
        }
#pragma unroll
        for (int j = 0; j < 4; j++)
          if (c + j < c1) {
            const double2 x = *reinterpret_cast<const double2*>(&v[j]);
            s.x = fma(w[j], x.x, s.x);
            s.y = fma(w[j], x.y, s.y);
          }
      }
      *reinterpret_cast<double2*>(out) = s;
    } else {
      df64acc re{0.f, 0.f}, im{0.f, 0.f};
      for (int c = c0; c < c1; c += 4) {
        C w[4];
        float4 v[4];
#pragma unroll
        for (int j = 0; j < 4; j++) {
          const int cj = min(c + j, c1 - 1);
          w[j] = __ldg(ccoef + cj);
          v[j] = p[__ldg(citem + cj)];
        }
#pragma unroll
        for (int j = 0; j < 4; j++)
          if (c + j < c1) {
            df_mac(re, w[j].x, w[j].y, v[j].x, v[j].y);
            df_mac(im, w[j].x, w[j].y, v[j].z, v[j].w);
          }
        if (((c - c0) & 12) == 12) {  // every 16 terms
          df_renorm(re);
          df_renorm(im);
        }
      }
      df_renorm(re);
      df_renorm(im);
      *out = make_float4(re.s, re.e, im.s, im.e);
    }
  }
}

struct XShared {
  uint64_t bars[2][2 * kXMaxStages + 5];  // one set per operand set
  uint32_t tmem;
  int abort;
  int ex[2][kExactMaxSliceA], ey[2][kExactMaxBlocks];  // exponents of the product's operand rows, by parity
};
static_assert(sizeof(XShared) <= kXFixed && kExactMaxBlocks >= kExactMaxSliceB && kExactMaxSliceA >= kExactMaxBlocks,
              "exponents of either set");

// One operand set: the products of qlist[n_q] (nullptr: q = 0 .. n_q - 1).
template <typename T, int STACK>
__device__ __forceinline__ void exact_set(unsigned char* smem, XShared& xs, const float4* __restrict__ F, int L,
                                          int n_out, const ExactDev& S, const int* __restrict__ E, int n_jobs,
                                          const int* __restrict__ qlist, int n_q, float4* __restrict__ P,
                                          int n_items, long long spin_limit) {
  uint64_t* bars = xs.bars[STACK - 1];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const XShape sh = x_shape(STACK, S.nAp, S.nBp);
  const int NS = sh.n_stages, NB = S.nBp, nC = (S.K + 15) / 16;
  const int TA = S.nAp / 16, TT = TA + NB / 16;  // warp tasks per stage: 16 rows x 2 k-groups each
  const int n_mine = (n_q - 1 - (int)blockIdx.x) / (int)gridDim.x + 1;
  const int bufW = (STACK == 2 ? 8 : 16) * NB, n_buf = 2 * bufW <= kXCols ? 2 : 1;
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
    using Raw = XRaw<T>;
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
    typename Raw::load v[8];
    int e = 0;
    auto load = [&](const Cursor& t) {
      const bool sideB = t.w >= TA;
      const int row = 16 * (sideB ? t.w - TA : t.w) + 8 * rg + r8;
      const int q = sideB ? t.nq : t.q;
      e = 0;
#pragma unroll
      for (int j = 0; j < 8; j++) v[j] = typename Raw::load();
      if (row < (sideB ? S.nB : S.nA)) {
        const float4* p = F + (size_t)q * n_out + __ldg((sideB ? S.rowB : S.rowA) + row);
        e = __ldg(E + (size_t)q * n_jobs + __ldg((sideB ? S.expB : S.expA) + row));
        e = e == kXBad ? 0 : e;  // any digits: the epilogue writes NaN
        if (STACK == 2) {
          // chunk c is the 4 x 4 tile (u, v) = (4 tu .., 4 tv ..) of the open
          // indices, k-group kg its u = 4 tu + 2 kg + (0, 1): values j = 4 du + dv
          // are element 12 u + v of A's block and element 12 v + u of B's
          const int tu = t.c / 3, tv = t.c - 3 * tu;
          if (sideB) {
            p += 48 * tv + 4 * tu + 2 * kg;
#pragma unroll
            for (int dv = 0; dv < 4; dv++) x_load2(p + 12 * dv, v[dv], v[4 + dv]);
          } else {
            p += 48 * tu + 24 * kg + 4 * tv;
#pragma unroll
            for (int du = 0; du < 2; du++) {
              x_load2(p + 12 * du, v[4 * du], v[4 * du + 1]);
              x_load2(p + 12 * du + 2, v[4 * du + 2], v[4 * du + 3]);
            }
          }
        } else {
          const int k0 = 16 * t.c + 8 * kg;
#pragma unroll
          for (int j = 0; j < 8; j += 2)
            if (k0 + j < S.K) x_load2(p + k0 + j, v[j], v[j + 1]);  // K is even
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
          x_store_digits(u[part], dst + sh.off_b + part * kXDigits * sh.slB, [&](int d) {
            return (STACK == 2 ? (d & 1) * (kXDigits / 2) + (d >> 1) : d) * sh.slB;
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
    uint32_t wa[8], wb[8], wn[8];
    int wc[8];
#pragma unroll
    for (int w = 0; w < 8; w++) {
      // STACK 2: slices of A count from the zeros (digit i is slice i + 1);
      // windows at even digits, then at odd ones from the zeros
      const int col = STACK == 2 ? w & 3 : w;
      const bool odd = STACK == 2 && w >= 4;
      wa[w] = (uint32_t)((STACK == 2 ? (odd ? 2 * col : 2 * col + 1) : w) * sh.slA) >> 4;
      wb[w] = (uint32_t)((odd ? kXDigits / 2 : 0) * sh.slB) >> 4;
      wc[w] = col * NB;
      wn[w] = x_idesc(NB * ((STACK == 2 ? 4 : 8) - col), 0);
    }
    const uint64_t desc0 = x_desc(x_smem(smem));
    const uint32_t d_im_part = (uint32_t)sh.partA >> 4, b_im_part = (uint32_t)(kXDigits * sh.slB) >> 4;
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
          for (int w = 0; w < 8; w++) {
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
    // every MMA issued has finished before the tensor memory is freed
    if (leader) {
      x_commit(bar_drain);
      for (long long polls = 0; !x_test(bar_drain, 0) && polls < spin_limit; polls++) __nanosleep(20);
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
    for (int i = 0; i < n_mine; i++) {
      const int buf = n_buf == 2 ? i & 1 : 0, m = n_buf == 2 ? i >> 1 : i;
      const int q = q_of(i), nq = x_neg_site(q, L);
      int* s_ex = xs.ex[i & 1];
      int* s_ey = xs.ey[i & 1];
      if (tid < S.nA) s_ex[tid] = __ldg(E + (size_t)q * n_jobs + __ldg(S.expA + tid));
      if (tid < S.nB) s_ey[tid] = __ldg(E + (size_t)nq * n_jobs + __ldg(S.expB + tid));
      const bool ok = x_wait(bar_acc + 8 * buf, (uint32_t)(m & 1), spin_limit, abort_flag);
      if (!x_all_epi(ok)) break;  // one verdict for all of them; the sums of the last product are read
      x_fence_after();
      const uint32_t d_re = tw + buf * bufW, d_im = d_re + bufW / 2;
      for (int j0 = 4 * half; has && j0 < S.nB; j0 += 8) {
        if (STACK == 2) {
          // level 2 c in the first rows of D, 2 c + 1 in the next
          uint32_t a[4][4], b[4][4], wide = 0;
          constexpr long long off = kXMagic * ((1ll << 28) + (1ll << 14) + 1);
#pragma unroll
          for (int c = 0; c < 4; c++) {
            x_ld4(d_re + c * NB + j0, a[c]);
            x_ld4(d_im + c * NB + j0, b[c]);
          }
#pragma unroll
          for (int c = 0; c < 4; c++) {
            x_wait_ld(a[c]);
            x_wait_ld(b[c]);
          }
          const int s1 = top ? 14 : 7, s2 = top ? 0 : 7;
          long long sr[4], si[4];
#pragma unroll
          for (int j = 0; j < 4; j++) {
            const unsigned r0 = x_bits(a[0][j], wide), r1 = x_bits(a[1][j], wide), r2 = x_bits(a[2][j], wide);
            const unsigned i0 = x_bits(b[0][j], wide), i1 = x_bits(b[1][j], wide), i2 = x_bits(b[2][j], wide);
            const int r3 = (int)(x_bits(a[3][j], wide) - (unsigned)kXMagic);
            const int i3 = (int)(x_bits(b[3][j], wide) - (unsigned)kXMagic);
            sr[j] = ((x_mad(r0, 1u << 28, x_mad(r1, 1u << 14, r2)) - off) << s1) + (r3 >> s2);
            si[j] = ((x_mad(i0, 1u << 28, x_mad(i1, 1u << 14, i2)) - off) << s1) + (i3 >> s2);
          }
          if (wide & 0xff800000u) {
#pragma unroll
            for (int j = 0; j < 4; j++) {
              sr[j] = x_sum4(x_int(a[0][j]), x_int(a[1][j]), x_int(a[2][j]), x_int(a[3][j]), top);
              si[j] = x_sum4(x_int(b[0][j]), x_int(b[1][j]), x_int(b[2][j]), x_int(b[3][j]), top);
            }
          }
          __syncwarp();
          if (mine) {
#pragma unroll
            for (int j = 0; j < 4; j++) {
              dst[(j0 + j) * S.nAp] = sr[j];
              dst[(NB + j0 + j) * S.nAp] = si[j];
            }
          }
        } else {
#pragma unroll
          for (int part = 0; part < 2; part++) {
            uint32_t a[8][4], wide = 0;
            constexpr long long off = kXMagic * ((1ll << 28) + (1ll << 14) + 1);
#pragma unroll
            for (int s = 0; s < 8; s++) x_ld4((part ? d_im : d_re) + s * NB + j0, a[s]);
#pragma unroll
            for (int s = 0; s < 8; s++) x_wait_ld(a[s]);
            long long v[4];
#pragma unroll
            for (int j = 0; j < 4; j++) {
              const unsigned n0 = x_bits(a[0][j], wide), n1 = x_bits(a[1][j], wide), n2 = x_bits(a[2][j], wide);
              const unsigned n3 = x_bits(a[3][j], wide), n4 = x_bits(a[4][j], wide), n5 = x_bits(a[5][j], wide);
              const int n6 = (int)(x_bits(a[6][j], wide) - (unsigned)kXMagic);
              const int n7 = (int)(x_bits(a[7][j], wide) - (unsigned)kXMagic);
              const long long ev = x_mad(n0, 1u << 28, x_mad(n2, 1u << 14, n4)) - off;
              const long long od = x_mad(n1, 1u << 28, x_mad(n3, 1u << 14, n5)) - off;
              v[j] = (ev << 14) + n6 + (od << 7) + (n7 >> 7);
            }
            if (wide & 0xff800000u) {
#pragma unroll
              for (int j = 0; j < 4; j++)
                v[j] = x_sum4(x_int(a[0][j]), x_int(a[2][j]), x_int(a[4][j]), x_int(a[6][j]), true) +
                       x_sum4(x_int(a[1][j]), x_int(a[3][j]), x_int(a[5][j]), x_int(a[7][j]), false);
            }
            __syncwarp();
            if (mine) {
#pragma unroll
              for (int j = 0; j < 4; j++) dst[(part * NB + j0 + j) * S.nAp] = v[j];
            }
          }
        }
      }
      x_fence_before();
      __syncwarp();
      if (lane == 0) x_arrive(bar_free + 8 * buf);
      asm volatile("bar.sync 1, %0;" ::"n"(32 * kXEpi) : "memory");  // the sums are in place
      using Out = typename XRaw<T>::load;
      Out* pq = reinterpret_cast<Out*>(P + (size_t)q * n_items);
      Out* pn = reinterpret_cast<Out*>(P + (size_t)nq * n_items);
      for (int t = tid; t < S.n_ent; t += 32 * kXEpi) {
        const int2 en = __ldg(S.entries + t);  // row | column << 16; item at q | item at -q << 16
        const int row = en.x & 0xffff, col = en.x >> 16;
        const long long* p = sums + col * S.nAp + row;
        long long re = p[0], im = p[NB * S.nAp];
        if (STACK == 2) {
          re += p[2 * NB * S.nAp];
          im += p[3 * NB * S.nAp];
        }
        // the sum is (sum of T_A T_B) 2^-56, T = x 2^(55 - e)
        const int ex = s_ex[row], ey = s_ey[col];
        const Out v = x_value(Out(), re, im, ex == kXBad || ey == kXBad ? kXBad : ex + ey - 54);
        const int item_q = (int)(short)en.y, item_n = en.y >> 16;
        if (item_q >= 0) pq[item_q] = v;
        // STACK 2: q = -q has its products from the items at q already
        if (item_n >= 0 && !(STACK == 2 && nq == q)) pn[item_n] = v;
      }
    }
  }
  // every warp has left its loop: accumulators read, stages free
  x_fence_before();
  __syncthreads();
  x_fence_after();
}

// F: q-major blocks [V][n_out] (16 bytes per complex value); P[V][n_items]; the
// trace set runs over the pairs qlist[n_pairs], the slice set over every q.
// err: bit 1 is set when a wait gave up.
template <typename T>
__global__ void __launch_bounds__(kXWarps * 32, 1)
k_contract_exact(const float4* __restrict__ F, int L, int n_out, const ExactDev trace, const ExactDev slice,
                 const int* __restrict__ E, int n_jobs, const int* __restrict__ qlist, int n_pairs,
                 float4* __restrict__ P, int n_items, int* __restrict__ err, long long spin_limit) {
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
  if (trace.nAp && (int)blockIdx.x < n_pairs)
    exact_set<T, 2>(smem, xs, F, L, n_out, trace, E, n_jobs, qlist, n_pairs, P, n_items, spin_limit);
  if (slice.nAp && (int)blockIdx.x < V && !*(volatile int*)&xs.abort)
    exact_set<T, 1>(smem, xs, F, L, n_out, slice, E, n_jobs, nullptr, V, P, n_items, spin_limit);
  if (tid == 0 && *(volatile int*)&xs.abort) atomicOr(err, 2);
  if (warp == kXEpi)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kXCols) : "memory");
}

static bool exact_set_ok(const ExactDev& S, int stack) {
  if (S.nAp == 0) return true;
  // a window of 128 rows that starts at the last slices reads past them into
  // the B digits: that stays inside the stage
  return S.nAp % 16 == 0 && S.nBp % 16 == 0 && S.nA <= S.nAp && S.nB <= S.nBp &&
         (stack == 2 ? S.nAp <= kExactMaxBlocks && S.nAp == S.nBp && S.K == 144
                     : S.nAp <= kExactMaxSliceA && S.nBp <= kExactMaxSliceB && S.K <= 144 && S.K % 2 == 0) &&
         x_shape(stack, S.nAp, S.nBp).n_stages >= 2;
}

cudaError_t launch_exact_exponents(const void* blk, bool df, long long n_q, int n_out, const int* jobs, int n_jobs,
                                   int* E, cudaStream_t st) {
  if (n_q <= 0 || n_jobs <= 0) return cudaSuccess;
  if (df) k_exact_exponents<dfr><<<(unsigned)n_q, 256, 0, st>>>((const float4*)blk, n_out, jobs, n_jobs, E);
  else k_exact_exponents<double><<<(unsigned)n_q, 256, 0, st>>>((const float4*)blk, n_out, jobs, n_jobs, E);
  return cudaGetLastError();
}

template <typename T>
static cudaError_t launch_exact_t(const float4* F, int L, int n_out, const ExactArgs& a, const int* E,
                                  const int* qlist, int n_pairs, float4* P, int* err, long long spin_limit, int n_sm,
                                  cudaStream_t st) {
  const int V = L * L * L;
  if (a.n_small > 0) {
    k_exact_small<T><<<V, 256, 0, st>>>(F, L, n_out, a.tasks, a.small, a.n_small, a.n_items, P);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  size_t sm = 0;
  if (a.trace.nAp) sm = (size_t)x_shape(2, a.trace.nAp, a.trace.nBp).bytes;
  if (a.slice.nAp) sm = std::max(sm, (size_t)x_shape(1, a.slice.nAp, a.slice.nBp).bytes);
  static int granted[64] = {0};
  const cudaError_t e = ensure_smem(k_contract_exact<T>, sm, granted);
  if (e != cudaSuccess) return e;
  const int n_q = a.slice.nAp ? V : n_pairs;
  k_contract_exact<T><<<std::min(n_q, n_sm), kXWarps * 32, sm, st>>>(F, L, n_out, a.trace, a.slice, E, a.n_jobs, qlist,
                                                                     n_pairs, P, a.n_items, err, spin_limit);
  return cudaGetLastError();
}

cudaError_t launch_contract_exact(const void* blk, int L, int n_out, bool df, const ExactArgs& a, const int* E,
                                  const int* qlist, int n_pairs, void* P, int* err, long long spin_limit,
                                  cudaStream_t st) {
  if (!a.trace.nAp && !a.slice.nAp) return cudaErrorInvalidValue;
  // 32-byte loads: rows and row length even (exact_split.cpp takes no other plan)
  if (!exact_set_ok(a.trace, 2) || !exact_set_ok(a.slice, 1) || (n_out & 1) || (((uintptr_t)blk) & 31) || !err)
    return cudaErrorInvalidValue;
  static int n_sm[64] = {0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!n_sm[dev]) {
    e = cudaDeviceGetAttribute(&n_sm[dev], cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
  }
  const float4* F = (const float4*)blk;
  return df ? launch_exact_t<dfr>(F, L, n_out, a, E, qlist, n_pairs, (float4*)P, err, spin_limit, n_sm[dev], st)
            : launch_exact_t<double>(F, L, n_out, a, E, qlist, n_pairs, (float4*)P, err, spin_limit, n_sm[dev], st);
}

size_t exact_wick_smem(int n_items) { return (size_t)kWickQ * n_items * 16; }

cudaError_t launch_exact_wick(const void* P, int V, int n_items, const int* cptr, const int* citem,
                              const double* ccoef, const float2* ccoef_df, int n_outputs, void* ct, bool df,
                              cudaStream_t st) {
  const size_t sm = exact_wick_smem(n_items);
  if (sm > kMaxSmemPerBlock) return cudaErrorInvalidValue;
  static int granted_d[64] = {0}, granted_f[64] = {0};
  cudaError_t e = df ? ensure_smem(k_exact_wick<dfr, float2>, sm, granted_f)
                     : ensure_smem(k_exact_wick<double, double>, sm, granted_d);
  if (e != cudaSuccess) return e;
  const unsigned grid = (unsigned)((V + kWickQ - 1) / kWickQ);
  if (df)
    k_exact_wick<dfr, float2><<<grid, kWickThreads, sm, st>>>((const float4*)P, V, n_items, cptr, citem, ccoef_df, n_outputs,
                                                     (float4*)ct);
  else
    k_exact_wick<double, double><<<grid, kWickThreads, sm, st>>>((const float4*)P, V, n_items, cptr, citem, ccoef, n_outputs,
                                                        (float4*)ct);
  return cudaGetLastError();
}

}  // namespace bbc
