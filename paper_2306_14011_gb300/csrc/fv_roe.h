// The Roe flux on the integer pipes: 64-bit block-floating-point arithmetic.
//
// A warp-wide FP64 instruction holds a sub-partition's FP64 unit for ~64
// cycles; an integer instruction issues every cycle or two.  The flux needs
// some thirty additions and as many products per face, and its operands are a
// face's few velocities, pressures and enthalpies, whose sizes are related.
// So each quantity is kept as a 64-bit integer significand with one exponent
// (per side, or shared by both sides of the face): a product is three
// 32x32-bit multiply-adds without unpacking, rounding or normalising, a sum is
// two adds after one shift, and nothing is rounded to 53 bits before the flux
// itself.  Significands carry 56 to 63 bits, so the flux is closer to the exact
// one than its FP64 evaluation (checked on the CPU against extended precision).
//
// The flux is the one of roe_F_fp64 (fv_device.cuh): the upwind side's
// physical flux plus the one acoustic wave that crosses from downwind,
//   F = F(Q_up) + g r_s,   g = k alpha_s,   k = min(|u~_n| - c~, 0).
// Faces this arithmetic does not take -- a density or energy that is not a
// positive number between 2^-300 and 2^300, an infinite or NaN momentum, a pressure or
// c~^2 that is not positive, sides so far apart that a shared exponent would
// lose digits -- are reported, and the caller evaluates them in FP64.
//
// Host and device: the same integer steps, so the CPU checks what the GPU runs.
#pragma once
#include <cmath>
#include <cstdint>

#ifdef __CUDACC__
#define FV_HD __host__ __device__ __forceinline__
#else
#define FV_HD inline
#endif

namespace fvk {

// ---------------------------------------------------------------- 64-bit pieces
FV_HD uint32_t fx_hi(uint64_t a) { return (uint32_t)(a >> 32); }
FV_HD uint32_t fx_lo(uint64_t a) { return (uint32_t)a; }
FV_HD uint64_t fx_pack(uint32_t hi, uint32_t lo) { return ((uint64_t)hi << 32) | lo; }

FV_HD uint32_t fx_umulhi32(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
  return __umulhi(a, b);
#else
  return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}
FV_HD int32_t fx_smulhi32(int32_t a, int32_t b) {
#ifdef __CUDA_ARCH__
  return __mulhi(a, b);
#else
  return (int32_t)(((int64_t)a * b) >> 32);
#endif
}
FV_HD int fx_min(int a, int b) { return a < b ? a : b; }
FV_HD int fx_max(int a, int b) { return a > b ? a : b; }

// a * b / 2^64 without the product of the low words: at most 2 units below.
// Written as a carry chain, which compiles to three wide multiply-adds and one
// carry (5 instructions and 14 cycles of a sub-partition per warp; from 64-bit
// C++ products, or __umul64hi, 8 and 18).
FV_HD uint64_t fx_mulhi(uint64_t a, uint64_t b) {
  const uint32_t ah = fx_hi(a), al = fx_lo(a), bh = fx_hi(b), bl = fx_lo(b);
#ifdef __CUDA_ARCH__
  uint32_t lo, hi;
  asm("{\n\t.reg .u32 p0, p1, q0, q1, c;\n\t"
      "mul.lo.u32 p0, %3, %4;\n\tmul.hi.u32 p1, %3, %4;\n\t"
      "mad.lo.cc.u32 q0, %2, %5, p0;\n\tmadc.hi.cc.u32 q1, %2, %5, p1;\n\taddc.u32 c, 0, 0;\n\t"
      "mad.lo.cc.u32 %0, %2, %4, q1;\n\tmadc.hi.u32 %1, %2, %4, c;\n\t}"
      : "=r"(lo), "=r"(hi)
      : "r"(ah), "r"(al), "r"(bh), "r"(bl));
  return fx_pack(hi, lo);
#else
  const uint64_t p = (uint64_t)al * bh, q = (uint64_t)ah * bl + p;
  return (uint64_t)ah * bh + ((q >> 32) | ((uint64_t)(q < p) << 32));
#endif
}
FV_HD uint64_t fx_sqrhi(uint64_t a) {
  const uint32_t ah = fx_hi(a), al = fx_lo(a);
  const uint64_t p = (uint64_t)ah * al;
  return (uint64_t)ah * ah + (p >> 31);
}

// a >> s for any s >= 0: from 64 on nothing is left (of a negative a: its sign).  A
// negative s, which is reported apart, counts as a large one.  The instruction
// takes such counts itself; C++ does not.
FV_HD uint64_t fx_shr(uint64_t a, int s) {
#ifdef __CUDA_ARCH__
  uint64_t r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(a), "r"(s));
  return r;
#else
  return (uint32_t)s < 64u ? a >> s : 0;
#endif
}
FV_HD int64_t fx_sar(int64_t a, int s) {
#ifdef __CUDA_ARCH__
  int64_t r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(a), "r"(s));
  return r;
#else
  return a >> ((uint32_t)s < 64u ? s : 63);
#endif
}

FV_HD int fx_clz32(uint32_t a) {
#ifdef __CUDA_ARCH__
  return __clz((int)a);
#else
  return a ? __builtin_clz(a) : 32;
#endif
}
FV_HD int fx_clz(uint64_t a) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)a);
#else
  return a ? __builtin_clzll(a) : 64;
#endif
}

// (a ^ m) - m: -a for m = -1, a for m = 0.
FV_HD int64_t fx_negate_if(uint64_t a, int32_t m) {
  const uint64_t w = (uint64_t)(int64_t)m;
  return (int64_t)((a ^ w) - w);
}
FV_HD uint64_t fx_abs(int64_t a) { return (uint64_t)fx_negate_if((uint64_t)a, (int32_t)(a >> 63)); }

FV_HD uint64_t fx_bits(double x) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(x);
#else
  uint64_t b;
  __builtin_memcpy(&b, &x, 8);
  return b;
#endif
}
FV_HD double fx_double(uint64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double x;
  __builtin_memcpy(&x, &b, 8);
  return x;
#endif
}
FV_HD uint32_t fx_float_bits(float f) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(f);
#else
  uint32_t b;
  __builtin_memcpy(&b, &f, 4);
  return b;
#endif
}
FV_HD float fx_float(uint32_t b) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  float f;
  __builtin_memcpy(&f, &b, 4);
  return f;
#endif
}
// FP32 seeds of 1/sqrt(x) and 1/x (special-function unit).
FV_HD float fx_rsqrt32(float x) {
#ifdef __CUDA_ARCH__
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
#else
  return (float)(1.0 / std::sqrt((double)x));
#endif
}
FV_HD float fx_rcp32(float x) {
#ifdef __CUDA_ARCH__
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
#else
  return (float)(1.0 / (double)x);
#endif
}
FV_HD float fx_u2f(uint32_t a) {
#ifdef __CUDA_ARCH__
  return __uint2float_rz(a);
#else
  return (float)(a & 0xffffff80u);
#endif
}

// ---------------------------------------------------------------- 1/sqrt and 1/x
// t 2^64 for t = 1/sqrt(x), x in [1, 4), X = x 2^61, from an FP32 seed y.
// With Y = y 2^22 (an integer) and e = 1 - x y^2, |e| < 2^-20, the binomial
// series gives t = y (1 + e/2 + 3 e^2/8) to 2^-62.  X Y^2 = (1 - e) 2^105:
// words 1 and 2 of the product are -e 2^73 modulo 2^64, so neither its top nor
// its bottom word is formed.  t = 1 (x = 1) saturates to 2^64 - 1.
FV_HD uint64_t fx_rsqrt(uint64_t X, float y) {
  const uint32_t Y = fx_float_bits(y + 2.0f) - 0x40000000u;
  const uint64_t Y2 = (uint64_t)Y * Y;  // y^2 2^44
  const uint32_t xh = fx_hi(X), xl = fx_lo(X), yh = fx_hi(Y2), yl = fx_lo(Y2);
  uint64_t S = (uint64_t)xl * yh + fx_umulhi32(xl, yl);
  S += (uint64_t)xh * yl;
  S += (uint64_t)(xh * yh) << 32;
  const int64_t e = (int64_t)(0ull - S);                 // e 2^73
  const int32_t es = (int32_t)(e >> 24);         // e 2^49
  const uint32_t c2 = (uint32_t)fx_smulhi32(es, es);  // e^2 2^66
  const int64_t w = e + (int64_t)((uint64_t)c2 * 96u);  // (e/2 + 3 e^2/8) 2^74
  uint64_t t = (uint64_t)((int64_t)(int32_t)Y * (int64_t)(int32_t)(w >> 32)) + fx_umulhi32(Y, fx_lo((uint64_t)w));
  t += (uint64_t)(Y << 10) << 32;
  const uint32_t sat = ~(uint32_t)((int32_t)fx_hi(t) >> 31);  // all ones when t passed 2^64
  return t | fx_pack(sat, sat);
}

// 2^60 / z for z in [1/2, 1), Z = z 2^64, from an FP32 seed a = 1/(2 z): with
// Y = 2 a 2^30 and e = 1 - z y, 1/z = y (1 + e + e^2) to 2^-60.  Z Y =
// (1 - e) 2^94, of which words 1 and 2 give e 2^62.
FV_HD uint64_t fx_rcp60(uint64_t Z, float a) {
  uint32_t Y = (fx_float_bits(a + 1.0f) - 0x3f800000u) << 8;
  Y = Y < 0x7fffffffu ? Y : 0x7fffffffu;
  const uint64_t S = (uint64_t)fx_hi(Z) * Y + fx_umulhi32(fx_lo(Z), Y);
  const int64_t e = (int64_t)((1ull << 62) - S);  // e 2^62
  const int32_t es = (int32_t)(e >> 14);          // e 2^48
  const uint32_t c2 = (uint32_t)fx_smulhi32(es, es);  // e^2 2^64
  const int64_t w = e + (int64_t)(uint64_t)(c2 >> 2);  // (e + e^2) 2^62
  uint64_t r = (uint64_t)((int64_t)(int32_t)Y * (int64_t)(int32_t)(w >> 32)) + fx_umulhi32(Y, fx_lo((uint64_t)w));
  return r + ((uint64_t)Y << 30);
}

// The double nearest to (-1)^neg n 2^-63 2^(field - 1023) for n with its top
// bit set, or zero; below the normal range: zero.  (The operands' range keeps
// results away from the other end.)
FV_HD double fx_round_normal(uint64_t n, int field, uint32_t neg) {
  const uint64_t m = (n >> 11) + ((n >> 10) & 1u);  // 53 bits, rounded (a carry moves into the exponent)
  const uint32_t hi = fx_hi(m) + ((uint32_t)(field - 1) << 20);
  const bool some = field >= 1 && (int32_t)fx_hi(n) < 0;
  return fx_double(some ? fx_pack(hi | (neg & 0x80000000u), fx_lo(m)) : 0ull);
}
// The same of any v < 2^63, in 2^-63 2^(x - 1023).
FV_HD double fx_round(uint64_t v, int x, uint32_t neg) {
  const int lz = fx_clz(v);
  const uint64_t n = (v << ((lz - 1) & 63)) + 0x200u;  // bit 62 set (v > 0), and half a unit of the 53 bits
  const int field = x - lz;
  const uint32_t hi = fx_hi(n >> 10) + ((uint32_t)(field - 1) << 20);
  const bool some = field >= 1 && fx_hi(n) >= 0x40000000u;
  return fx_double(some ? fx_pack(hi | (neg & 0x80000000u), fx_lo(n >> 10)) : 0ull);
}

// ---------------------------------------------------------------- single operations on doubles
// a * b rounded to 53 bits from its leading 62 or more (within 0.51 units in the
// last place); subnormal operands and results count as zero.  Results beyond
// the double's range, infinities and NaN set bad's sign bit.  25 integer
// instructions and no FP64 one.
FV_HD double fx_mul(double a, double b, int &bad) {
  const uint64_t ba = fx_bits(a), bb = fx_bits(b);
  const uint32_t ha = fx_hi(ba), hb = fx_hi(bb);
  const int ea = (int)((ha >> 20) & 0x7ffu), eb = (int)((hb >> 20) & 0x7ffu);
  const uint64_t p = fx_mulhi((ba << 11) | 0x8000000000000000ull, ((bb & 0xfffffffffffffull) | 0x10000000000000ull) << 10);
  const int t = (int)(fx_hi(p) >> 30);  // p in [2^61, 2^63): 1 when the product of the significands is 2 or more
  const uint64_t n = (p << (1 - t)) + 0x200u;
  const int field = ea + eb + t - 1023;
  const uint32_t hi = fx_hi(n >> 10) + ((uint32_t)(field - 1) << 20);
  const bool some = field >= 1 && fx_min(ea, eb) > 0;
  bad |= (2046 - fx_max(ea, eb)) | (2045 - field);
  return fx_double(some ? fx_pack(hi | ((ha ^ hb) & 0x80000000u), fx_lo(n >> 10)) : 0ull);
}
// 1/sqrt(x) for positive normal x and 1/x for x in [2^-1021, 2^1022) (else bad's
// sign bit), within 0.51 units in the last place.
FV_HD double fx_rsqrt64(double x, int &bad) {
  const uint64_t b = fx_bits(x);
  const int e = (int)(fx_hi(b) >> 20);
  bad |= (e - 1) | (2046 - e);
  const int odd = (e + 1) & 1, q = (e - 1023 - odd) >> 1;
  const uint64_t X = (((b & 0xfffffffffffffull) | 0x10000000000000ull) << 9) << odd;
  const float x32 = fx_float(0x3f800000u + ((uint32_t)odd << 23) + (uint32_t)((b >> 29) & 0x7fffffu));
  return fx_round_normal(fx_rsqrt(X, fx_rsqrt32(x32)), 1022 - q, 0u);
}
FV_HD double fx_rcp64(double x, int &bad) {
  const uint64_t b = fx_bits(x);
  const int e = (int)(fx_hi(b) >> 20);
  bad |= (e - 2) | (2044 - e);
  const uint64_t Z = (b << 11) | 0x8000000000000000ull;  // x = Z 2^-63 2^(e - 1023)
  const uint64_t r = fx_rcp60(Z, fx_rcp32(fx_float(0x3f800000u | (uint32_t)((b >> 29) & 0x7fffffu))));
  return fx_round(r, 2048 - e, 0u);  // 1/x = r 2^-61 2^(1023 - e)
}

// 2ab / s for a and b of one sign and s = a + b as FP64 rounds it, rounded once from
// 58 bits or more (so that with s's own rounding the result is closer to exact than
// the FP64 operations').  Operands and sums near the ends of the range, infinities
// and NaN set bad's sign bit; the result lies between the smaller operand and twice
// it, so nothing leaves the range in between.
FV_HD double fx_vanleer(double a, double b, double s, int &bad) {
  const uint64_t ba = fx_bits(a), bb = fx_bits(b), bs = fx_bits(s);
  const int ea = (int)((fx_hi(ba) >> 20) & 0x7ffu), eb = (int)((fx_hi(bb) >> 20) & 0x7ffu);
  const int es = (int)((fx_hi(bs) >> 20) & 0x7ffu);
  bad |= (fx_min(ea, eb) - 2) | (2044 - es);
  // |ab| = p 2^-61 2^(ea + eb - 2046), 1/|s| = r 2^-61 2^(1023 - es)
  const uint64_t p = fx_mulhi((ba << 11) | 0x8000000000000000ull, ((bb & 0xfffffffffffffull) | 0x10000000000000ull) << 10);
  const uint64_t r = fx_rcp60((bs << 11) | 0x8000000000000000ull,
                              fx_rcp32(fx_float(0x3f800000u | (uint32_t)((bs >> 29) & 0x7fffffu))));
  return fx_round(fx_mulhi(p << 1, r << 2), ea + eb - es + 3, fx_hi(ba));
}

// Constants of a scheme, formed once on the host.
struct RoeConst {
  uint64_t G;      // gamma - 1 = G 2^(j - 64), G in [2^63, 2^64)
  int j, je;       // je = max(j, 0): total enthalpies are kept in units of 2^je
  int jh;          // half of je rounded up: LARGE_GAMMA's H~ - c~ |u~_n| in units of 2^jh
  uint64_t efix;   // efix 2^64 (efix < 1)
};

inline RoeConst roe_const(double g1, double efix) {
  RoeConst c;
  const double g = std::frexp(g1, &c.j);  // [1/2, 1)
  c.je = c.j > 0 ? c.j : 0;
  c.jh = (c.je + 1) / 2;
  c.G = (uint64_t)(g * 18446744073709551616.0);
  c.efix = (uint64_t)(efix * 18446744073709551616.0);
  return c;
}

// ---------------------------------------------------------------- the flux
// States normal-first: q = (rho, m_n, m_t[0..NT-1], E).  Returns false (G is
// then meaningless) for a face that this arithmetic does not take.  From gamma = 3
// on H~ - c~ |u~_n| can be negative and c~ beyond the unit that bounds |u~|: such
// faces, and every one from gamma = 9 on, need LARGE_GAMMA.
template <int NT, bool LARGE_GAMMA = false>
FV_HD bool roe_fixed(const double (&QL)[NT + 3], const double (&QR)[NT + 3], const RoeConst &rc,
                     double (&G)[NT + 3]) {
  constexpr int NC = NT + 1, E = NT + 2;  // velocity components, index of the energy
  // gamma - 1 from 2^-41 to 8 or 256; the sign bit collects everything that is not taken
  int bad = ((LARGE_GAMMA ? 8 : 3) - rc.j) | (rc.j + 40);

  // ---- each side in its own scale
  uint64_t T[2], S[2], U[2][NC], K[2], Pe[2], En[2], M[2][NC];
  uint32_t sg[2][NC];  // sign words of the momenta
  int q[2], xm[2][NC], xu[2][NC], xE[2], xk[2];
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const double(&Q)[NT + 3] = s == 0 ? QL : QR;
    // rho = x 4^q, x in [1, 4)
    const uint64_t br = fx_bits(Q[0]);
    const uint32_t hr = fx_hi(br);
    const int er = (int)(hr >> 20);                  // the sign included
    bad |= (er - 723) | (1323 - er);                 // 2^-300 .. 2^300: no product leaves the double's range
    const int odd = (er + 1) & 1;
    q[s] = (er - 1023 - odd) >> 1;
    const uint64_t X = (((br & 0xfffffffffffffull) | 0x10000000000000ull) << 9) << odd;  // x 2^61
    const float x32 = fx_float(0x3f800000u + ((uint32_t)odd << 23) + (uint32_t)((br >> 29) & 0x7fffffu));
    T[s] = fx_rsqrt(X, fx_rsqrt32(x32));             // 1/sqrt(rho) = T 2^-64 2^-q
    const uint64_t R = fx_sqrhi(T[s]);               // 1/rho = R 2^-64 4^-q
    S[s] = fx_mulhi(X, T[s]);                        // sqrt(rho) = S 2^-61 2^q, S in [2^61, 2^62)
    // E = 2^-59 2^(xE - 1023) units: the significand's 53 bits shifted by 7
    const uint64_t be = fx_bits(Q[E]);
    xE[s] = (int)(fx_hi(be) >> 20);
    bad |= (xE[s] - 723) | (1323 - xE[s]);
    const uint64_t E59 = ((be & 0xfffffffffffffull) | 0x10000000000000ull) << 7;
    // velocities |u| = U 2^-63 2^(xu - 1023) and E - rho |u|^2 / 2
    uint64_t pe = E59;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const uint64_t bm = fx_bits(Q[1 + c]);
      sg[s][c] = fx_hi(bm);
      const int em = (int)((sg[s][c] >> 20) & 0x7ffu);
      const uint64_t f = bm << 11;
      M[s][c] = em != 0 ? (f | 0x8000000000000000ull) : 0ull;  // |m| = M 2^-63 2^(em - 1023); below 2^-1022: 0
      xm[s][c] = em;
      U[s][c] = fx_mulhi(M[s][c], R);
      xu[s][c] = em - 2 * q[s];
      const uint64_t k = fx_mulhi(M[s][c], U[s][c]);  // m u / 2 = k 2^-63 2^(em + xu - 2046)
      const int sh = xE[s] + 1027 - em - xu[s][c];  // negative: kinetic energy far beyond E, infinite, NaN
      const uint64_t ks = fx_shr(k, sh);
      pe -= ks;
      // p > 0, term by term: a term reaches 2^64 (32 E), and two or three of them
      // can wrap pe round to a positive number
      bad |= sh | (int)fx_hi(ks) | (int)fx_hi(pe);
      if (c == 0) {
        K[s] = k;
        xk[s] = em + xu[s][0];
      }
    }
    bad |= (int)fx_hi(pe - 1ull);                    // p > 0: not zero either
    // p / 2^j and the total enthalpy rho h_t / 2^je in the energy's units
    Pe[s] = fx_mulhi(pe, rc.G);
    En[s] = (E59 >> rc.je) + (Pe[s] >> (rc.je - rc.j));
  }

  // ---- Roe weights
  const int dq = q[0] - q[1];
  bad |= (16 - dq) | (16 + dq);
  const int qm = fx_max(q[0], q[1]);
  const uint64_t SL = fx_shr(S[0], qm - q[0]), SR = fx_shr(S[1], qm - q[1]);
  const uint64_t sum = SL + SR;                      // [2^61, 2^63)
  const int n = 2 - (int)(fx_hi(sum) >> 30);
  const uint64_t Z = sum << n;                       // [2^63, 2^64)
  const uint64_t inv = fx_rcp60(Z, fx_rcp32(fx_float(0x3f800000u | ((fx_hi(Z) >> 8) & 0x7fffffu)))) << 2;  // 2^62 / z
  const uint64_t wl = fx_mulhi(SL << n, inv) << 2;   // sL / (sL + sR) in 2^-64

  // ---- velocities in a scale shared by both sides: u = w 2^-61 2^(xw - 1023)
  int64_t W[NC], dU0 = 0;
  int xw[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    xw[c] = fx_max(xu[0][c], xu[1][c]);
    const int64_t a = fx_negate_if(fx_shr(U[0][c], xw[c] + 2 - xu[0][c]), (int32_t)sg[0][c] >> 31);
    const int64_t b = fx_negate_if(fx_shr(U[1][c], xw[c] + 2 - xu[1][c]), (int32_t)sg[1][c] >> 31);
    const int64_t d = (int64_t)((uint64_t)b - (uint64_t)a);
    // b - wl d (the unsigned product, corrected for a negative d)
    uint64_t p = fx_mulhi((uint64_t)d, wl);
    p -= wl & (uint64_t)(d >> 63);
    W[c] = (int64_t)((uint64_t)b - p);
    if (c == 0) dU0 = d;
  }

  // ---- enthalpy H~ and c~
  const int h0 = xE[0] - q[0], h1 = xE[1] - q[1], hm = fx_max(h0, h1);
  const uint64_t HT = fx_shr(fx_mulhi(En[0], T[0]), hm - h0) + fx_shr(fx_mulhi(En[1], T[1]), hm - h1);
  const uint64_t HH = fx_mulhi(HT << 2, inv);        // H~ = HH 2^-62 2^xH
  const int xH = hm - 1023 - qm + rc.je + n;
  const int o = xH & 1, xe = xH + o;                 // even exponent
  const uint64_t Hh = HH >> (1 + o);                 // H~ = Hh 2^-61 2^xe
  const int bv = (xe + 2) >> 1;                      // |u~| <= 2^bv
  uint64_t Cq = Hh, v0 = 0;
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    const int sv = bv + 1025 - xw[c];
    bad |= sv;
    const uint64_t v = fx_shr(fx_abs(W[c]), sv) << 4;  // |u~| = v 2^-63 2^bv
    if (c == 0) v0 = v;
    Cq -= fx_sqrhi(v);                               // u~^2 / 2 in H~'s units
  }
  // c~^2 > 0.  (No wrap here: with both pressures positive u~^2 / 2 is below H~, so
  // Cq is negative by a few units of rounding at most.)
  bad |= (int)fx_hi(Cq - 1ull);
  const uint64_t Pc = fx_mulhi(Cq, rc.G);            // c~^2 = Pc 2^-61 2^(xe + j)
  const int lz = fx_clz32(fx_hi(Pc));
  bad |= 31 - lz;                                    // c~^2 keeps 32 bits at least, or FP64 decides
  const int sh = ((lz - 1 - rc.j) & ~1) + rc.j;
  const uint64_t Xc = Pc << (sh & 63);               // [2^61, 2^63)
  const uint64_t Tc = fx_rsqrt(Xc, fx_rsqrt32(fx_u2f(fx_hi(Xc)) * 0x1p-29f));
  const int qc = (xe + rc.j - sh) >> 1;              // 1/c~ = Tc 2^-64 2^-qc
  const uint64_t Cs = fx_mulhi(Xc, Tc) << 2;         // c~ = Cs 2^-63 2^qc, Cs in [2^63, 2^64)

  // ---- x = |u~_n| - c~ = X1 2^-61 2^xv, and |k| = max(-x, 0), entropy-fixed
  const int xun = xw[0] - 1023;
  const uint64_t aw = fx_abs(W[0]);
  const int xv = fx_max(xun, qc);
  const uint64_t cb = fx_shr(Cs, xv - qc + 2);
  const int64_t X1 = (int64_t)(fx_shr(aw, xv - xun) - cb);
  const uint64_t ax = fx_abs(X1);
  uint64_t Kk = X1 < 0 ? ax : 0ull;
  // 32-bit words say which faces may need the fix (never missing one: the high word
  // of efix c~ is at most 2 above the product of the high words), 64-bit ones which do
  if (fx_hi(ax) <= fx_umulhi32(fx_hi(cb), fx_hi(rc.efix)) + 2u) {
    const uint64_t d = fx_mulhi(cb, rc.efix);
    if (ax < d) {  // |k| = (delta - x)^2 / (4 delta)
      const double delta = (double)d, D = delta - (double)X1;
      Kk = (uint64_t)(D * D * (0.25 / delta));
    }
  }

  // ---- num = dp -+ rho~ c~ du_n (upper sign: u~_n >= 0) = N 2^-58 2^xn
  const int em = fx_max(xE[0], xE[1]);
  const int64_t dp = (int64_t)(fx_shr(Pe[1], em - xE[1]) - fx_shr(Pe[0], em - xE[0]));
  const uint64_t RS = fx_mulhi(S[0] << 2, S[1] << 2);  // rho~ = RS 2^-62 2^(qL + qR)
  const uint64_t RC = fx_mulhi(RS, Cs);                // rho~ c~ = RC 2^-61 2^(qL + qR + qc)
  const uint64_t ND = fx_mulhi(RC, fx_abs(dU0));       // rho~ c~ |du_n| = ND 2^-58 2^xd
  const int xd = q[0] + q[1] + qc + xun, xp = em - 1024 + rc.j;
  const int xn = fx_max(xd, xp) + 1;
  const int32_t right = (int32_t)(W[0] >> 63);         // -1: the upwind side is the right one
  const int32_t minus = ~((int32_t)(dU0 >> 63) ^ right);  // -1: +-du_n > 0 is subtracted
  const int64_t N = fx_sar(dp, xn - xp) + fx_negate_if(fx_shr(ND, xn - xd), minus);

  // ---- g = -|k| num / (2 c~^2) = (-1)^(N >= 0) g 2^-58 2^xg
  const uint64_t an = fx_abs(N);
  const int ln = fx_clz32(fx_hi(an));                  // (32: what is left below costs num nothing)
  const uint64_t A = fx_mulhi(an << ln, fx_sqrhi(Tc));
  const uint64_t gu = fx_mulhi(A, Kk << 2);
  const int lg = fx_clz(gu);                           // normalised, so that a small g costs F(Q_up) no digits
  const uint64_t g = gu << (lg & 63);
  const int xg = xn - 2 * qc + xv - ln - lg;
  const uint32_t gneg = ~fx_hi((uint64_t)N);           // sign word of g (N >= 0: negative)

  // ---- F(Q_up) + g r_s
  const bool up = right != 0;                          // the right side is upwind
  const uint64_t Mu = up ? M[1][0] : M[0][0], Uu = up ? U[1][0] : U[0][0];
  const uint32_t su = up ? sg[1][0] : sg[0][0];
  const int xmu = up ? xm[1][0] : xm[0][0], xuu = up ? xu[1][0] : xu[0][0];
  const int xEu = up ? xE[1] : xE[0];
  // mass
  G[0] = (up ? QR[1] : QL[1]) + fx_round_normal(g, xg + 5 + 1023, gneg);
  {  // m_n u_n + p + g (+-x)
    const uint64_t k = up ? K[1] : K[0], p = up ? Pe[1] : Pe[0];
    const int y1 = (up ? xk[1] : xk[0]) - 2046, y2 = xEu - 1020 + rc.j;  // 2^-62 2^y
    const uint64_t gx = fx_mulhi(g, ax);
    const int y3 = xg + xv + 7;
    const int y = fx_max(fx_max(y1, y2 - 2), y3) + 2;
    // g x carries the sign of g, flipped when x < 0, flipped again on the right
    const int32_t neg = (int32_t)(gneg ^ fx_hi((uint64_t)X1)) >> 31;
    const uint64_t v = fx_shr(k, y - y1) + fx_shr(p, y - y2) + (uint64_t)fx_negate_if(fx_shr(gx, y - y3), neg ^ right);
    const int lz = fx_clz32(fx_hi(v));
    bad |= (lz - 1) | (31 - lz);  // a positive sum with 32 bits at least, or FP64
    const uint64_t m = (v << ((lz - 1) & 31)) + 0x200u;
    G[1] = fx_double(fx_pack(fx_hi(m >> 10) + ((uint32_t)(y + 1023 - lz) << 20), fx_lo(m >> 10)));
  }
#pragma unroll
  for (int t = 0; t < NT; ++t) {  // m_n u_t + g u~_t
    const uint64_t a = fx_mulhi(Mu, up ? U[1][1 + t] : U[0][1 + t]);
    const int y1 = xmu + (up ? xu[1][1 + t] : xu[0][1 + t]) - 2046;
    const uint64_t b = fx_mulhi(g, fx_abs(W[1 + t]));
    const int y2 = xg + xw[1 + t] - 1023 + 7;
    const int y = fx_max(y1 + 1, y2) + 1;
    const uint32_t n1 = su ^ (up ? sg[1][1 + t] : sg[0][1 + t]);
    const int32_t opposite = (int32_t)(n1 ^ gneg ^ fx_hi((uint64_t)W[1 + t])) >> 31;
    const int64_t v = (int64_t)(fx_shr(a, y - y1) + (uint64_t)fx_negate_if(fx_shr(b, y - y2), opposite));
    G[2 + t] = fx_round(fx_abs(v), y + 1 + 1023, fx_hi((uint64_t)v) ^ n1);
  }
  {  // u_n rho h_t + g (H~ - c~ |u~_n|)
    const uint64_t a = fx_mulhi(Uu, up ? En[1] : En[0]);
    const int y1 = xuu + xEu - 2046 + rc.je + 3;        // 2^-61 2^y
    const int jh = LARGE_GAMMA ? rc.jh : 0, sc = bv - 1 - qc + jh;
    bad |= sc;
    uint64_t hr = (Hh >> jh) - fx_shr(fx_mulhi(Cs, v0), sc);
    const uint32_t hneg = LARGE_GAMMA ? fx_hi(hr) : 0u;
    if (LARGE_GAMMA)
      hr = fx_abs((int64_t)hr);
    else
      bad |= (int)fx_hi(hr);
    const uint64_t b = fx_mulhi(g, hr);
    const int y2 = xg + xe + 6 + jh;
    const int y = fx_max(y1, y2) + 1;
    const int64_t v = (int64_t)(fx_shr(a, y - y1) + (uint64_t)fx_negate_if(fx_shr(b, y - y2), (int32_t)(su ^ gneg ^ hneg) >> 31));
    G[E] = fx_round(fx_abs(v), y + 2 + 1023, fx_hi((uint64_t)v) ^ su);
  }
  return bad >= 0;
}

}  // namespace fvk
