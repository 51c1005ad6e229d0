// Complex arithmetic policies for the state-vector kernels.
//
// A kernel is written once over a policy A:
//   A::store_t  element as it sits in HBM (float2 for complex64, double2 for complex128)
//   A::reg_t    element as the kernel computes on it (registers and shared memory)
//   A::mat_t    gate-matrix entry in the policy's own format
//
// AF32  complex64 storage, FP32 arithmetic.
// AF64  complex128 storage, native FP64 arithmetic (reference policy; on GB300 the FP64
//       pipe issues about 2 DFMA per clock per SM, 1/64 of FP32, so this policy is
//       ALU-bound by a wide margin).
// ADF   complex128 storage, "double-float" arithmetic on the FP32 pipe: each real number is
//       an unevaluated sum hi + lo of two floats (Dekker 1971 TwoProduct via FMA; Knuth
//       TwoSum; Shewchuk 1997 renormalisation).  About 47-48 significant bits, relative
//       error ~1e-14 per operation.  The FP64 <-> (hi, lo) conversions are done with
//       integer bit manipulation so that no instruction touches the FP64 pipe; the real
//       and imaginary lanes run through packed f32x2 instructions.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

namespace qs {

// ------------------------------------------------------------------------------------------
// complex64, FP32
// ------------------------------------------------------------------------------------------
struct AF32 {
  using store_t = float2;
  using reg_t = float2;
  using mat_t = float2;
  static constexpr int kStoreBytes = 8;
  static constexpr bool kFrame = false;
  static constexpr bool kConst = false;
  static __device__ __forceinline__ mat_t ld(const mat_t* p) { return *p; }
  static __device__ __forceinline__ reg_t from_store(store_t v) { return v; }
  static __device__ __forceinline__ store_t to_store(reg_t v) { return v; }
  static __device__ __forceinline__ reg_t from_store_f(store_t v, bool) { return v; }
  static __device__ __forceinline__ store_t to_store_f(reg_t v, bool) { return v; }
  static __device__ __forceinline__ reg_t zero() { return make_float2(0.f, 0.f); }
  // u*a + v*b
  static __device__ __forceinline__ reg_t mac2(mat_t u, reg_t a, mat_t v, reg_t b) {
    float re = u.x * a.x;
    re = fmaf(-u.y, a.y, re);
    re = fmaf(v.x, b.x, re);
    re = fmaf(-v.y, b.y, re);
    float im = u.x * a.y;
    im = fmaf(u.y, a.x, im);
    im = fmaf(v.x, b.y, im);
    im = fmaf(v.y, b.x, im);
    return make_float2(re, im);
  }
  // acc + u*a
  static __device__ __forceinline__ reg_t mac(reg_t acc, mat_t u, reg_t a) {
    float re = fmaf(u.x, a.x, acc.x);
    re = fmaf(-u.y, a.y, re);
    float im = fmaf(u.x, a.y, acc.y);
    im = fmaf(u.y, a.x, im);
    return make_float2(re, im);
  }
  static __device__ __forceinline__ reg_t mul(mat_t u, reg_t a) {
    return make_float2(fmaf(u.x, a.x, -u.y * a.y), fmaf(u.x, a.y, u.y * a.x));
  }
  // (c*a.re + s*b.im, c*a.im - s*b.re): the RX-type update c*a - i*s*b
  static __device__ __forceinline__ reg_t rx(mat_t cs, reg_t a, reg_t b) {
    return make_float2(fmaf(cs.x, a.x, cs.y * b.y), fmaf(cs.x, a.y, -cs.y * b.x));
  }
  // u + t v with the real t in t.x (tangent-form RX), and -i b
  static __device__ __forceinline__ reg_t axpy(mat_t t, reg_t v, reg_t u) {
    return make_float2(fmaf(t.x, v.x, u.x), fmaf(t.x, v.y, u.y));
  }
  static __device__ __forceinline__ reg_t mul_mi(reg_t b) { return make_float2(b.y, -b.x); }
  static __device__ __forceinline__ reg_t neg(reg_t a) { return make_float2(-a.x, -a.y); }
  static __device__ __forceinline__ double norm2(reg_t a) {
    return (double)a.x * (double)a.x + (double)a.y * (double)a.y;
  }
};

// ------------------------------------------------------------------------------------------
// complex128, native FP64
// ------------------------------------------------------------------------------------------
struct AF64 {
  using store_t = double2;
  using reg_t = double2;
  using mat_t = double2;
  static constexpr int kStoreBytes = 16;
  static constexpr bool kFrame = false;
  static constexpr bool kConst = false;
  static __device__ __forceinline__ mat_t ld(const mat_t* p) { return *p; }
  static __device__ __forceinline__ reg_t from_store(store_t v) { return v; }
  static __device__ __forceinline__ store_t to_store(reg_t v) { return v; }
  static __device__ __forceinline__ reg_t from_store_f(store_t v, bool) { return v; }
  static __device__ __forceinline__ store_t to_store_f(reg_t v, bool) { return v; }
  static __device__ __forceinline__ reg_t zero() { return make_double2(0.0, 0.0); }
  static __device__ __forceinline__ reg_t mac2(mat_t u, reg_t a, mat_t v, reg_t b) {
    double re = u.x * a.x;
    re = fma(-u.y, a.y, re);
    re = fma(v.x, b.x, re);
    re = fma(-v.y, b.y, re);
    double im = u.x * a.y;
    im = fma(u.y, a.x, im);
    im = fma(v.x, b.y, im);
    im = fma(v.y, b.x, im);
    return make_double2(re, im);
  }
  static __device__ __forceinline__ reg_t mac(reg_t acc, mat_t u, reg_t a) {
    double re = fma(u.x, a.x, acc.x);
    re = fma(-u.y, a.y, re);
    double im = fma(u.x, a.y, acc.y);
    im = fma(u.y, a.x, im);
    return make_double2(re, im);
  }
  static __device__ __forceinline__ reg_t mul(mat_t u, reg_t a) {
    return make_double2(fma(u.x, a.x, -u.y * a.y), fma(u.x, a.y, u.y * a.x));
  }
  static __device__ __forceinline__ reg_t rx(mat_t cs, reg_t a, reg_t b) {
    return make_double2(fma(cs.x, a.x, cs.y * b.y), fma(cs.x, a.y, -cs.y * b.x));
  }
  static __device__ __forceinline__ reg_t axpy(mat_t t, reg_t v, reg_t u) {
    return make_double2(fma(t.x, v.x, u.x), fma(t.x, v.y, u.y));
  }
  static __device__ __forceinline__ reg_t mul_mi(reg_t b) { return make_double2(b.y, -b.x); }
  static __device__ __forceinline__ reg_t neg(reg_t a) { return make_double2(-a.x, -a.y); }
  static __device__ __forceinline__ double norm2(reg_t a) { return a.x * a.x + a.y * a.y; }
};

// ------------------------------------------------------------------------------------------
// double-float building blocks (all explicitly rounded: no contraction changes them).
// They are host-callable as well, so that the formulas can be checked on a CPU against
// binary64; on the host the float operations are plain IEEE binary32 with
// round-to-nearest (build with contraction off).
// ------------------------------------------------------------------------------------------
#define QS_HD __host__ __device__ __forceinline__

QS_HD float f_add(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fadd_rn(a, b);
#else
  return a + b;
#endif
}
QS_HD float f_sub(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fsub_rn(a, b);
#else
  return a - b;
#endif
}
QS_HD float f_mul(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fmul_rn(a, b);
#else
  return a * b;
#endif
}
QS_HD float f_fma(float a, float b, float c) {
#ifdef __CUDA_ARCH__
  return __fmaf_rn(a, b, c);
#else
  return fmaf(a, b, c);
#endif
}
QS_HD unsigned int f_bits(float x) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(x);
#else
  unsigned int u;
  memcpy(&u, &x, 4);
  return u;
#endif
}
QS_HD float f_from_bits(unsigned int u) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(u);
#else
  float x;
  memcpy(&x, &u, 4);
  return x;
#endif
}
QS_HD unsigned long long d_bits(double x) {
#ifdef __CUDA_ARCH__
  return (unsigned long long)__double_as_longlong(x);
#else
  unsigned long long u;
  memcpy(&u, &x, 8);
  return u;
#endif
}
QS_HD double d_from_bits(unsigned long long u) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)u);
#else
  double x;
  memcpy(&x, &u, 8);
  return x;
#endif
}
QS_HD float u32_to_f_rn(unsigned int r) {
#ifdef __CUDA_ARCH__
  return __uint2float_rn(r);
#else
  return (float)r;
#endif
}
QS_HD int f_to_i_rn(float x) {
#ifdef __CUDA_ARCH__
  return __float2int_rn(x);
#else
  return (int)lrintf(x);
#endif
}

// Packed lane pairs: one f32x2 instruction (FADD2 / FMUL2 / FFMA2 on sm_100 and later)
// does the same operation on both floats of a 64-bit register pair.
QS_HD float2 add2(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
  return __fadd2_rn(a, b);
#else
  return make_float2(a.x + b.x, a.y + b.y);
#endif
}
QS_HD float2 sub2(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rd;\n\t"
      "mov.b64 ra, {%2, %3};\n\t"
      "mov.b64 rb, {%4, %5};\n\t"
      "sub.rn.f32x2 rd, ra, rb;\n\t"
      "mov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
#else
  return make_float2(a.x - b.x, a.y - b.y);
#endif
}
QS_HD float2 mul2(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
  return __fmul2_rn(a, b);
#else
  return make_float2(a.x * b.x, a.y * b.y);
#endif
}
QS_HD float2 fma2(float2 a, float2 b, float2 c) {
#ifdef __CUDA_ARCH__
  return __ffma2_rn(a, b, c);
#else
  return make_float2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y));
#endif
}

struct dfl { float hi, lo; };

// s + e == a + b exactly (Knuth TwoSum, 6 flops)
QS_HD dfl two_sum(float a, float b) {
  float s = f_add(a, b);
  float bb = f_sub(s, a);
  float e = f_add(f_sub(a, f_sub(s, bb)), f_sub(b, bb));
  return {s, e};
}
// p + e == a * b exactly (TwoProduct with FMA)
QS_HD dfl two_prod(float a, float b) {
  float p = f_mul(a, b);
  float e = f_fma(a, b, -p);
  return {p, e};
}
// lane-wise TwoSum: s + e == a + b exactly in each lane
QS_HD void two_sum2(float2 a, float2 b, float2& s, float2& e) {
  s = add2(a, b);
  const float2 bb = sub2(s, a);
  e = add2(sub2(a, sub2(s, bb)), sub2(b, bb));
}
// sign flip of both lanes (integer operations, not the FMA pipe)
QS_HD float2 neg2(float2 a) {
  return make_float2(f_from_bits(f_bits(a.x) ^ 0x80000000u), f_from_bits(f_bits(a.y) ^ 0x80000000u));
}
// Lane-wise s + d + c = a + U v to about 2^-48 |s|: TwoSum of a and p = RN(U v) in which the
// FMA d = U v - (what p added to s) replaces TwoSum's last difference and the product's own
// rounding error: 6 instructions where TwoProduct and TwoSum take 8.  s is the sum of two
// floats and not one FMA of the exact product: under cancellation the FMA's result has bits
// below ulp(a), and the differences with a would no longer be exact (errors of 2^-25).  The
// product is therefore an FMA with 0: the assembler contracts a packed multiply whose only
// use is a packed add, explicit .rn or not, and it leaves an FMA alone.
QS_HD void add_prod2(float2 a, float2 U, float2 v, float2& s, float2& d, float2& c) {
  s = add2(a, fma2(U, v, make_float2(0.f, 0.f)));
  const float2 nb = sub2(a, s);       // -(what the product added)
  d = fma2(U, v, nb);
  c = sub2(a, add2(s, nb));
}

// Split a binary64 value into hi + lo floats without FP64 instructions.
// hi keeps the leading 24 significant bits (truncated), lo = x - hi (its 29 bits rounded
// to 24): |x - (hi + lo)| <= 2^-47 |x|.  |x| < 2^-126 flushes to 0 (absolute error
// below 1.2e-38); the lo part flushes when it would leave the normal float range
// (|x| below about 2^-98; absolute error below 2^-120).
QS_HD dfl split_double(double x) {
  const unsigned long long b = d_bits(x);
  const unsigned int w1 = (unsigned int)(b >> 32);
  const unsigned int w0 = (unsigned int)b;
  const unsigned int sign = w1 & 0x80000000u;
  const int e = (int)((w1 >> 20) & 0x7FFu);
  const int ef = e - 896;                                   // float biased exponent
  const unsigned int m23 = ((w1 & 0xFFFFFu) << 3) | (w0 >> 29);
  float hi = f_from_bits(sign | ((unsigned int)ef << 23) | m23);
  hi = (ef > 0) ? hi : 0.0f;
  const unsigned int r = w0 & 0x1FFFFFFFu;                   // low 29 mantissa bits
  // lo = r * 2^(e - 1075): convert r exactly-rounded, then move its exponent field
  const unsigned int rb = f_bits(u32_to_f_rn(r));
  const int el = (int)(rb >> 23) + (e - 1075);               // biased exponent of lo
  float lo = f_from_bits(sign | ((unsigned int)el << 23) | (rb & 0x7FFFFFu));
  lo = (r != 0u && el > 0 && ef > 0) ? lo : 0.0f;
  return {hi, lo};
}

// Join hi + lo (|lo| <= ulp(hi)/2, as produced by the arithmetic below) into a binary64
// with integer operations only: the binary64 pattern of hi plus lo counted in binary64 ulps
// (IEEE patterns are monotonic in magnitude for a fixed sign, so adding k to the pattern
// moves the value by k ulps, across a binade boundary included).
QS_HD double join_double(float hi, float lo) {
  const unsigned int hb = f_bits(hi);
  const unsigned int sign = hb & 0x80000000u;
  const int ef = (int)((hb >> 23) & 0xFFu);
  if (ef == 0) return 0.0;
  unsigned long long db = ((unsigned long long)(sign | ((unsigned int)(ef + 896) << 20) |
                                                ((hb & 0x7FFFFFu) >> 3)) << 32) |
                          ((unsigned long long)(hb & 7u) << 29);
  const unsigned int lb = f_bits(lo);
  const int el = (int)((lb >> 23) & 0xFFu);
  // lo is counted in binary64 ulps of hi's binade, 2^(ef-179); when hi is a power of two and
  // lo points down, the result lies in the binade below, whose ulp is half as large
  const bool down = ((lb ^ hb) & 0x80000000u) && ((hb & 0x7FFFFFu) == 0u);
  const int ne = el + (down ? 180 : 179) - ef;             // exponent of lo / ulp
  int k = 0;
  if (el != 0 && ne > 0) {
    float ls = f_from_bits((lb & 0x807FFFFFu) | ((unsigned int)ne << 23));
    k = f_to_i_rn(ls);
  }
  long long delta = sign ? -(long long)k : (long long)k;
  db = (unsigned long long)((long long)db + delta);
  return d_from_bits(db);
}

QS_HD unsigned int funnel_l(unsigned int lo, unsigned int hi, int n) {   // high word of (hi:lo) << n
#ifdef __CUDA_ARCH__
  return __funnelshift_l(lo, hi, n);
#else
  return (hi << n) | (lo >> (32 - n));
#endif
}

// The same two conversions in fewer instructions, for the per-gate kernels, which convert every
// amplitude both ways around one update: same bits, about 14 and 20 instead of 22 and 25 instructions
// (26-qubit 2x2 gate 491 -> 463 us, 4x4 gate 622 -> 584 us).  The tile kernel keeps the forms above: with
// these it came out 2 to 4 % slower, converting only in a plan's first and last passes.
// Exponents are moved inside the shifted word: after a shift by 3 the 11-bit exponent's low nine bits
// stand above the float's 23 mantissa bits, where e - 896 and e - 1075 are additions modulo 2^32.
QS_HD dfl split_double_gate(double x) {
  const unsigned long long b = d_bits(x);
  const unsigned int w1 = (unsigned int)(b >> 32);
  const unsigned int w0 = (unsigned int)b;
  const unsigned int sign = w1 & 0x80000000u;
  const unsigned int fs = funnel_l(w0, w1, 3);
  const bool ok = (w1 & 0x7FFFFFFFu) >= (897u << 20);        // float biased exponent e - 896 >= 1
  const unsigned int hb = ((fs + 0x40000000u) & 0x7FFFFFFFu) | sign;   // - 896 << 23
  // lo = r * 2^(e - 1075): convert r, the low 29 mantissa bits, exactly-rounded, then move its exponent
  const unsigned int r = w0 & 0x1FFFFFFFu;
  const unsigned int lb = f_bits(u32_to_f_rn(r)) + (fs & 0xFF800000u) - 0x19800000u;   // - 1075 << 23
  const bool lok = ok && r != 0u && (int)lb >= 0x00800000;
  return {f_from_bits(ok ? hb : 0u), f_from_bits(lok ? (lb | sign) : 0u)};
}

QS_HD double join_double_gate(float hi, float lo) {
  const unsigned int hb = f_bits(hi), lb = f_bits(lo);
  const unsigned int hm = hb & 0x7FFFFFFFu, lm = lb & 0x7FFFFFFFu, flip = (lb ^ hb) & 0x80000000u;
  const unsigned int w1 = ((hm >> 3) + (896u << 20)) | (hb & 0x80000000u);
  const unsigned int w0 = hb << 29;
  // lo is counted in binary64 ulps of hi's binade, 2^(ef-179); when hi is a power of two and
  // lo points down, the result lies in the binade below, whose ulp is half as large
  int t = (int)(lm + (179u << 23) - (hm & 0x7F800000u));
  if (flip != 0u && (hb & 0x7FFFFFu) == 0u) t += 0x00800000;
  const bool some = lm >= 0x00800000u && t >= 0x00800000;
  const int k = f_to_i_rn(f_from_bits(some ? ((unsigned int)t | flip) : 0u));   // along hi's magnitude
  const unsigned long long db = (((unsigned long long)w1 << 32) | w0) + (unsigned long long)(long long)k;
  return d_from_bits(hm >= 0x00800000u ? db : 0ull);
}

// ------------------------------------------------------------------------------------------
// complex128 storage, double-float arithmetic, two lanes per instruction
//
// reg_t = (re.hi, im.hi, re.lo, im.lo): the (re, im) lanes of the high parts and of the
// low parts are each one 64-bit register pair, so each step of the complex arithmetic is
// one packed f32x2 instruction instead of two scalar ones.  Register values are kept
// unnormalised between operations (hi need not be the rounded value of hi + lo);
// to_store normalises once with TwoSum before the exact integer join.
//
// mat_t (32 bytes, prepared on the host) holds a complex u = ur + i ui as lane patterns:
//   h = ( ur.hi,  ur.hi, -ui.hi,  ui.hi)     ur on both lanes; (-ui, ui): i ui acting on a swapped (im, re)
//   l = (-ur.lo, -ur.lo, -ui.lo,  ui.lo)     low parts, that of ur negated
// so that u a = ur (.) a + (-ui, ui) (.) swap(a) lane-wise; the other sign of ur is two integer
// operations away.  An entry is read by every lane of a warp, and such a load returns its bytes 32 times
// over: with both signs stored (48 bytes, three 16-byte loads) the phase tables were bound by
// those returns (table time at 26 qubits 12.5 ms of 48.4 against 9.6 of arithmetic).
//
// Instruction counts per amplitude (packed, two lanes each): u + t v 10, a complex product 14,
// acc + u a 22.  Each sum of a value and a product is one add_prod2; with a TwoProduct and a
// TwoSum the three took 12, 16 and 24.
//
// Tile passes run in a phase frame: amplitude i of a tile is held as (-i)^popcount(i)
// times its value (S^dagger on every tile bit).  Diagonal gates are unchanged, RX becomes
// the real rotation [[c, s], [-s, c]] (no lane swaps at all), X becomes [[0, i], [-i, 0]],
// and the host transforms the matrices of general gates (entry (r, c) times
// (-i)^(popcount r - popcount c)).  The per-gate kernels use the plain frame.
// ------------------------------------------------------------------------------------------
struct alignas(16) dfm {
  float4 h, l;
};
// a real double-float factor t as the lane pairs the products need: high and low part on both
// lanes, and their negations
struct dfr {
  float2 h, nh, l, nl;
};

struct ADF {
  using store_t = double2;
  using reg_t = float4;
  using mat_t = dfm;
  static constexpr int kStoreBytes = 16;
  static constexpr bool kFrame = true;
  static constexpr bool kConst = false;

  static QS_HD float2 hi(reg_t v) { return make_float2(v.x, v.y); }
  static QS_HD float2 lo(reg_t v) { return make_float2(v.z, v.w); }
  static QS_HD float2 swp(float2 v) { return make_float2(v.y, v.x); }
  static QS_HD reg_t mk(float2 h, float2 l) { return make_float4(h.x, h.y, l.x, l.y); }

  // An entry loaded where it is used: the loads are volatile so that the compiler
  // cannot hoist the entries of a whole matrix out of a loop (8 registers each).
  static QS_HD mat_t ld(const mat_t* p) {
#ifdef __CUDA_ARCH__
    mat_t m;
    asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(m.h.x), "=f"(m.h.y), "=f"(m.h.z), "=f"(m.h.w) : "l"(p));
    asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4+16];"
                 : "=f"(m.l.x), "=f"(m.l.y), "=f"(m.l.z), "=f"(m.l.w) : "l"(p));
    return m;
#else
    return *p;
#endif
  }
  // the real part of an entry (t, 0)
  static QS_HD dfr ld_real(const mat_t* p) {
#ifdef __CUDA_ARCH__
    float2 h, nl;
    asm volatile("ld.global.nc.v2.f32 {%0, %1}, [%2];" : "=f"(h.x), "=f"(h.y) : "l"(p));
    asm volatile("ld.global.nc.v2.f32 {%0, %1}, [%2+16];" : "=f"(nl.x), "=f"(nl.y) : "l"(p));
    return dfr{h, neg2(h), neg2(nl), nl};
#else
    return real_of(*p);
#endif
  }
  static QS_HD dfr real_of(const mat_t& m) { return dfr{mA(m), mnA(m), mAl(m), mnAl(m)}; }
  // an entry as an amplitude and back (its own lane patterns of a value that is not normalised)
  static QS_HD reg_t from_mat(const mat_t& m) { return make_float4(m.h.x, m.h.w, -m.l.x, m.l.w); }
  static QS_HD mat_t to_mat(reg_t v) {
    mat_t m;
    m.h = make_float4(v.x, v.x, -v.y, v.y);
    m.l = make_float4(-v.z, -v.z, -v.w, v.w);
    return m;
  }
  // the lane patterns of an entry
  static QS_HD float2 mA(const mat_t& m) { return make_float2(m.h.x, m.h.y); }     // ( ur,  ur)
  static QS_HD float2 mnA(const mat_t& m) { return neg2(mA(m)); }                  // (-ur, -ur)
  static QS_HD float2 mB(const mat_t& m) { return make_float2(m.h.z, m.h.w); }     // (-ui,  ui)
  static QS_HD float2 mnAl(const mat_t& m) { return make_float2(m.l.x, m.l.y); }   // low parts
  static QS_HD float2 mAl(const mat_t& m) { return neg2(mnAl(m)); }
  static QS_HD float2 mBl(const mat_t& m) { return make_float2(m.l.z, m.l.w); }
  static QS_HD reg_t from_store(store_t v) {
    const dfl r = split_double(v.x), i = split_double(v.y);
    return make_float4(r.hi, i.hi, r.lo, i.lo);
  }
  static QS_HD store_t to_store(reg_t v) {
    const dfl r = two_sum(v.x, v.z), i = two_sum(v.y, v.w);
    return make_double2(join_double(r.hi, r.lo), join_double(i.hi, i.lo));
  }
  // the same value with hi the rounded value of hi + lo
  static QS_HD reg_t normalised(reg_t v) {
    float2 s, e;
    two_sum2(hi(v), lo(v), s, e);
    return mk(s, e);
  }
  // The double-float storage form a plan keeps between consecutive tile passes: the four
  // floats of a normalised register value in the 16 bytes of an element (no binary64
  // split or join).  It exists only inside one plan execution; the state holds binary64
  // before and after.
  static QS_HD reg_t from_df(store_t v) {
    const unsigned long long a = d_bits(v.x), b = d_bits(v.y);
    return make_float4(f_from_bits((unsigned int)a), f_from_bits((unsigned int)(a >> 32)),
                       f_from_bits((unsigned int)b), f_from_bits((unsigned int)(b >> 32)));
  }
  static QS_HD store_t to_df(reg_t v) {
    float2 s, e;
    two_sum2(hi(v), lo(v), s, e);
    return make_double2(d_from_bits(((unsigned long long)f_bits(s.y) << 32) | f_bits(s.x)),
                        d_from_bits(((unsigned long long)f_bits(e.y) << 32) | f_bits(e.x)));
  }
  static QS_HD reg_t from_store_f(store_t v, bool df) { return df ? from_df(v) : from_store(v); }
  static QS_HD store_t to_store_f(reg_t v, bool df) { return df ? to_df(v) : to_store(v); }
  static QS_HD reg_t zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }

  // U x + V y lane-wise for double-float patterns, U given by its high part and the negated
  // parts, V by its parts; the two products' low-order terms run in two chains, smallest first
  static QS_HD reg_t dot2(float2 Uh, float2 nUh, float2 nUl, float2 xh, float2 xl, float2 Vh, float2 Vl, float2 yh,
                          float2 yl) {
    const float2 p = mul2(Uh, xh);
    float2 n = fma2(nUh, xh, p);             // -(rounding error of p), exact
    n = fma2(nUl, xh, n);
    n = fma2(nUh, xl, n);
    float2 s, d, c;
    add_prod2(p, Vh, yh, s, d, c);
    d = add2(c, d);
    d = fma2(Vl, yh, d);
    d = fma2(Vh, yl, d);
    return mk(s, sub2(d, n));
  }
  // u a
  static QS_HD reg_t mul(const mat_t& u, reg_t a) {
    return dot2(mA(u), mnA(u), mnAl(u), hi(a), lo(a), mB(u), mBl(u), swp(hi(a)), swp(lo(a)));
  }
  static QS_HD reg_t add(reg_t x, reg_t y) {
    float2 s, e;
    two_sum2(hi(x), hi(y), s, e);
    return mk(s, add2(e, add2(lo(x), lo(y))));
  }
  // acc + u a
  static QS_HD reg_t mac(reg_t acc, const mat_t& u, reg_t a) { return add(acc, mul(u, a)); }
  // u a + v b
  static QS_HD reg_t mac2(const mat_t& u, reg_t a, const mat_t& v, reg_t b) { return add(mul(u, a), mul(v, b)); }
  // c a - i s b for cs = (c, s), plain frame: c (.) a + (s, -s) (.) swap(b), and (s, -s) is
  // the negated (-ui, ui) pattern of the entry
  static QS_HD reg_t rx(const mat_t& cs, reg_t a, reg_t b) {
    return dot2(mA(cs), mnA(cs), mnAl(cs), hi(a), lo(a), neg2(mB(cs)), neg2(mBl(cs)), swp(hi(b)), swp(lo(b)));
  }

  // ---- phase-frame updates with a real double-float factor t
  // u + (th + tl) v
  static QS_HD reg_t add_prod(float2 th, float2 tl, reg_t v, float2 uh, float2 ul) {
    float2 s, d, c;
    add_prod2(uh, th, hi(v), s, d, c);
    d = add2(c, d);
    d = fma2(tl, hi(v), d);
    d = fma2(th, lo(v), d);
    return mk(s, add2(ul, d));
  }
  // u + t v
  static QS_HD reg_t axpy_r(const dfr& t, reg_t v, reg_t u) { return add_prod(t.h, t.l, v, hi(u), lo(u)); }
  // u - t v
  static QS_HD reg_t axmy_r(const dfr& t, reg_t v, reg_t u) { return add_prod(t.nh, t.nl, v, hi(u), lo(u)); }
  // t v - u
  static QS_HD reg_t ymx_r(const dfr& t, reg_t v, reg_t u) {
    return add_prod(t.h, t.l, v, neg2(hi(u)), neg2(lo(u)));
  }
  // (a, b) -> (c a + s b, c b - s a) with real c and s
  static QS_HD void rot_r(const dfr& c, const dfr& sn, reg_t a, reg_t b, reg_t& a2, reg_t& b2) {
    const reg_t ra = dot2(c.h, c.nh, c.nl, hi(a), lo(a), sn.h, sn.l, hi(b), lo(b));
    b2 = dot2(c.h, c.nh, c.nl, hi(b), lo(b), sn.nh, sn.nl, hi(a), lo(a));
    a2 = ra;
  }
  // v (-i)^q, exact (a lane swap and sign flips); q in 0..3
  static QS_HD reg_t rot_q(reg_t v, unsigned int q) {
    const bool sw = (q & 1u) != 0u;
    const float r0 = sw ? v.y : v.x, r1 = sw ? v.x : v.y, l0 = sw ? v.w : v.z, l1 = sw ? v.z : v.w;
    const unsigned int n0 = (q >> 1) << 31, n1 = ((q ^ (q >> 1)) & 1u) << 31;
    return make_float4(f_from_bits(f_bits(r0) ^ n0), f_from_bits(f_bits(r1) ^ n1), f_from_bits(f_bits(l0) ^ n0),
                       f_from_bits(f_bits(l1) ^ n1));
  }
  static QS_HD reg_t neg(reg_t a) { return make_float4(-a.x, -a.y, -a.z, -a.w); }
  static QS_HD double norm2(reg_t a) {
    double r = (double)a.x + (double)a.z, i = (double)a.y + (double)a.w;
    return r * r + i * i;
  }
};

// The per-gate kernels' double-float policy.
struct ADFG : ADF {
  static QS_HD reg_t from_store(store_t v) {
    const dfl r = split_double_gate(v.x), i = split_double_gate(v.y);
    return make_float4(r.hi, i.hi, r.lo, i.lo);
  }
  static QS_HD store_t to_store(reg_t v) {
    float2 s, e;
    two_sum2(hi(v), lo(v), s, e);
    return make_double2(join_double_gate(s.x, e.x), join_double_gate(s.y, e.y));
  }
};

// Policies of the tile kernel whose program sits in the constant bank (kernel parameters): the ops'
// fields stay uniform, and in ADFC the matrix entries are plain loads, uniform too.
struct AF32C : AF32 {
  static constexpr bool kConst = true;
};
struct ADFC : ADF {
  static constexpr bool kConst = true;
  static __device__ __forceinline__ mat_t ld(const mat_t* p) { return *p; }
  static __device__ __forceinline__ dfr ld_real(const mat_t* p) { return real_of(*p); }
};

// one host matrix entry, (re, im) in double, in a policy's format (df_entry: gates.cpp)
void df_entry(const double* z, float* e);
inline void host_entry(const double* z, float2* m) { *m = make_float2((float)z[0], (float)z[1]); }
inline void host_entry(const double* z, double2* m) { *m = make_double2(z[0], z[1]); }
inline void host_entry(const double* z, dfm* m) { df_entry(z, (float*)m); }

}  // namespace qs
