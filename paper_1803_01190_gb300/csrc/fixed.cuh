// Pair arithmetic of the binary64 mode in 64-bit fixed point, on the integer
// pipes: GB300 issues one FP64 instruction in the time of 32 integer ones, so
// a pair of Eq. 2 costs less in integers than the 9 FP64 instructions of the
// binary64 body, and no precision is lost on the way.
//
// For one j-tile against one i-block a unit u = 2^L is chosen such that every
// coordinate difference (and eps) is below 2^61 u.  Coordinates become
// integers X = x / u modulo 2^64 (to nearest; exact when the last bit of x is
// worth at least u), so D = X_j - X_i is the exact difference of the rounded
// coordinates whatever their magnitude.  Per pair:
//   r2 = Dx^2 + Dy^2 + Dz^2 + eps^2 as a 96-bit integer (error below 2^-53 r2
//        at the closest pairs taken, falling as 1/r),
//   x  = r2 normalised by an even shift 2h to [1/4, 1) with 64 bits,
//   y  = 1/sqrt(x): SFU seed S0 (24 bits), exact integer residual
//        e = 1 - x S0^2, y = S0 (1 + e/2 + 3 e^2/8); R = y 2^62, error < 2^-59,
//   Q  = y^2 2^61,  Y = m y,  F = Y y^2 (top 64 bits of the products with the
//        63-bit mass; error of F < 2^-56),
//   force sums += D F, potential sum += Y, aligned by h, in 96-bit integers,
// converted to binary64 once per tile.  A pair with |d| below 2^51 u, where the
// rounding of the coordinates (1/2 u each) and the last place of the sums
// approach the rounding of a binary64 pair term, is left to the binary64 body by
// the caller.  At that limit d is off by up to 2^-51 of itself and its term cut
// off below 2^-52, both falling as 1/|d|; a binary64 difference may be off by
// 2^-53 at any distance.  The limit is one of |d| and not of the softened r:
// where eps is far above the separations, r says nothing of what the unit
// leaves of them (two clumps 1e-6 eps across and 512 eps apart, the force in
// the one at the origin, by host emulation: 1.1e-10 with a limit of r, 3e-16
// with this one; a system of 1e-4 eps 1.1e-14 and 6e-16).
//
// What bounds it: the FMA-heavy pipe, where a 32 x 32 -> 64 multiply takes 4
// cycles per warp (an addition on the ALU pipe takes 2).  So the products that
// only reach the last bits are 16-bit ones (2 cycles): the squares and cross
// terms of the low words.  Measured in a loop of the pair body alone
// (cycles per warp and pair): 345 with 41 wide products and y^3 formed apart
// from m y, 317 with F = Y y^2, 297 with the 16-bit products as well.
#pragma once

#include <stdint.h>

namespace nb {

constexpr int FX_BITS = 61;        // differences and eps below 2^61 units
// Masses over at most 2^FX_MASS_NARROW share one exponent (F keeps 53 bits for
// the smallest); over at most 2^FX_MASS_RANGE each has its own, added to the
// shifts of its terms (WIDE below).  Beyond it the binary64 body is taken: the
// terms of the light ones are cut off at a place set by the heaviest, and where
// its own term is missing (it is the particle itself) or vanishes (both at one
// place, softened) nothing covers what they lose.  Host emulation of such sums
// (127 equal masses on a sphere around one 2^R to 2^(R+1) times as heavy, error
// over the sum of the terms' magnitudes): R = 8 1.0e-16, 9 2.1e-16, 10 4.1e-16,
// 20 4e-13, against 1.3e-16 for binary64 terms.
constexpr int FX_MASS_NARROW = 4, FX_MASS_RANGE = 8;

// 96-bit two's complement accumulator
struct fx96 {
  uint32_t w0, w1;
  int32_t w2;
};

#ifdef __CUDA_ARCH__
#define FX_HD __device__ __forceinline__
#else
#define FX_HD inline
#endif

FX_HD uint32_t fx_shl(uint32_t lo, uint32_t hi, int s) {  // high word of (hi:lo) << s, s < 32
#ifdef __CUDA_ARCH__
  return __funnelshift_l(lo, hi, s);
#else
  return (uint32_t)(((((uint64_t)hi << 32) | lo) << s) >> 32);
#endif
}
FX_HD uint32_t fx_shr(uint32_t lo, uint32_t hi, int s) {  // low word of (hi:lo) >> s, s < 32
#ifdef __CUDA_ARCH__
  return __funnelshift_r(lo, hi, s);
#else
  return (uint32_t)((((uint64_t)hi << 32) | lo) >> s);
#endif
}
FX_HD uint32_t fx_umulhi(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
  return __umulhi(a, b);
#else
  return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}
FX_HD int32_t fx_mulhi(int32_t a, int32_t b) {
#ifdef __CUDA_ARCH__
  return __mulhi(a, b);
#else
  return (int32_t)(((int64_t)a * b) >> 32);
#endif
}
FX_HD int64_t fx_mads(int32_t a, int32_t b, int64_t c) { return (int64_t)a * b + c; }
FX_HD uint64_t fx_madu(uint32_t a, uint32_t b, uint64_t c) { return (uint64_t)a * b + c; }
// a * b + c for a 32-bit c (the signed one: c_hi is 0 or c's sign).  ALU: the
// product and two additions on the ALU pipe instead of the 64-bit addend that
// a fused multiply-add takes, whose moves go to the busier multiply pipe.  The
// each-pair-once kernel is faster with it (N = 65536, equal / unequal masses:
// 219 / 152 Gint/s against 215 / 147), the one-sided one without (133 / 123
// against 127 / 118).
template <bool ALU>
FX_HD uint64_t fx_madw(uint32_t a, uint32_t b, uint32_t c) {
#ifdef __CUDA_ARCH__
  if (ALU) {
    uint64_t d;
    asm("{\n\t.reg .u32 l, h;\n\t.reg .u64 t;\n\t"
        "mul.wide.u32 t, %1, %2;\n\t"
        "mov.b64 {l, h}, t;\n\t"
        "add.cc.u32 l, l, %3;\n\t"
        "addc.u32 h, h, 0;\n\t"
        "mov.b64 %0, {l, h};\n\t}"
        : "=l"(d)
        : "r"(a), "r"(b), "r"(c));
    return d;
  }
#endif
  return (uint64_t)a * b + c;
}
template <bool ALU>
FX_HD int64_t fx_madws(int32_t a, int32_t b, int32_t c, int32_t c_hi) {
#ifdef __CUDA_ARCH__
  if (ALU) {
    int64_t d;
    asm("{\n\t.reg .u32 l, h;\n\t.reg .u64 t;\n\t"
        "mul.wide.s32 t, %1, %2;\n\t"
        "mov.b64 {l, h}, t;\n\t"
        "add.cc.u32 l, l, %3;\n\t"
        "addc.u32 h, h, %4;\n\t"
        "mov.b64 %0, {l, h};\n\t}"
        : "=l"(d)
        : "r"(a), "r"(b), "r"(c), "r"(c_hi));
    return d;
  }
#endif
  return (int64_t)a * b + (int64_t)(((uint64_t)(uint32_t)c_hi << 32) | (uint32_t)c);
}

FX_HD void fx_add(fx96 &a, uint32_t w0, uint32_t w1, uint32_t w2) {
#ifdef __CUDA_ARCH__
  asm("add.cc.u32 %0, %0, %3;\n\t"
      "addc.cc.u32 %1, %1, %4;\n\t"
      "addc.u32 %2, %2, %5;"
      : "+r"(a.w0), "+r"(a.w1), "+r"(a.w2)
      : "r"(w0), "r"(w1), "r"(w2));
#else
  const uint64_t s0 = (uint64_t)a.w0 + w0, s1 = (uint64_t)a.w1 + w1 + (s0 >> 32);
  a.w0 = (uint32_t)s0;
  a.w1 = (uint32_t)s1;
  a.w2 = (int32_t)((uint32_t)a.w2 + w2 + (uint32_t)(s1 >> 32));
#endif
}

// x (halves hi, lo of a finite binary64) in units of 2^L, modulo 2^64, to nearest.
FX_HD uint64_t fx_coord(uint32_t hi, uint32_t lo, int L) {
  const int ex = (int)((hi >> 20) & 0x7FF);
  if (ex == 0) return 0;  // zero or subnormal: far below a unit
  const uint64_t sig = ((uint64_t)((hi & 0xFFFFF) | 0x100000) << 32) | lo;
  const int sh = ex - 1075 - L;
  uint64_t v;
  if (sh >= 0)
    v = sh < 64 ? sig << sh : 0;
  else
    v = sh > -64 ? (sig + ((uint64_t)1 << (-sh - 1))) >> -sh : 0;
  return (hi >> 31) ? 0 - v : v;
}

// Mass m as M 2^(em - 62 - dm), em the exponent of the tile's largest mass:
// dm = 0 (masses down to 2^-10 of it exact) or, WIDE, M in [2^62, 2^63).
struct FxMass {
  uint32_t h, l;
  int dm;
};
template <bool WIDE>
FX_HD FxMass fx_mass(uint32_t hi, uint32_t lo, int em) {
  const int ex = (int)(hi >> 20);
  if (ex == 0) return FxMass{0, 0, 0};
  const uint64_t sig = ((uint64_t)((hi & 0xFFFFF) | 0x100000) << 32) | lo;
  const int dm = em + 1023 - ex;
  const uint64_t M = WIDE ? sig << 10 : sig << (10 - dm);
  return FxMass{(uint32_t)(M >> 32), (uint32_t)M, WIDE ? dm : 0};
}

// eps^2 / u^2 split for the accumulation of r2: e.hi * 2^64 + e.mid * 2^33.
struct FxEps {
  uint64_t hi;
  int64_t mid;
};
FX_HD FxEps fx_eps2(double eps2, int L) {
  FxEps e{0, 0};
#ifdef __CUDA_ARCH__
  const uint64_t b = (uint64_t)__double_as_longlong(eps2);
#else
  uint64_t b;
  __builtin_memcpy(&b, &eps2, 8);
#endif
  const int ex = (int)(b >> 52);
  if (ex == 0) return e;
  const uint64_t sig = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  const int sh = ex - 1075 - 2 * L - 33;  // in units of 2^33 u^2
  // value = sig 2^sh: hi = its part above 2^31, mid the 31 bits below
  if (sh >= 31) {
    e.hi = sig << (sh - 31);
  } else if (sh > -64) {
    const uint64_t lo = sh >= 0 ? (sh < 12 ? sig << sh : 0) : sig >> -sh;
    if (sh >= 12) {
      e.hi = sig >> (31 - sh);
      e.mid = (int64_t)((sig << sh) & 0x7FFFFFFFull);
    } else {
      e.hi = lo >> 31;
      e.mid = (int64_t)(lo & 0x7FFFFFFFull);
    }
  }
  return e;
}

// The geometry of one pair, shared by its two sides.
struct FxPair {
  int32_t dh[3], dl[3];  // D = dh 2^32 + dl, both signed
  uint32_t Rh, Rl;       // 1/sqrt(x) 2^62
  uint32_t Qh, Ql;       // 1/x 2^61
  int s, sp;             // right shifts of the force and potential terms
};

// false: |d| is below 2^51 units (EARLY: nothing else is set;
// otherwise 1/r and 1/r^2 are 0, so that its terms add nothing, and no branch
// keeps the pairs of several calls from being interleaved).
template <bool ALU, bool EARLY = true, class RSQRT>
FX_HD bool fx_geometry(const uint64_t (&Xj)[3], const uint64_t (&Xi)[3], const FxEps &e2,
                       RSQRT rsqrt, FxPair &p) {
  uint64_t S2 = e2.hi;
  int64_t S1 = e2.mid;
  uint32_t q = 0;  // sum of the squares of the low words, in units of 2^32
#pragma unroll
  for (int c = 0; c < 3; c++) {
    const uint64_t D = Xj[c] - Xi[c];
    const uint32_t lo = (uint32_t)D;
    p.dl[c] = (int32_t)lo;
    p.dh[c] = (int32_t)((uint32_t)(D >> 32) + (lo >> 31));
    S2 = (uint64_t)fx_mads(p.dh[c], p.dh[c], (int64_t)S2);
    S1 = fx_mads(p.dh[c], p.dl[c], S1);
    q += (uint32_t)((p.dl[c] >> 16) * (p.dl[c] >> 16));
  }
  // r2 = S2 2^64 + Mid 2^33
  const int64_t Mid = S1 + (int64_t)(q >> 1);
  const uint64_t T = S2 + (uint64_t)(Mid >> 31);
  const uint32_t th = (uint32_t)(T >> 32), tl = (uint32_t)T, t0 = (uint32_t)Mid << 1;
  // |d| >= 2^51 units, from the upper words alone: the limit lies between
  // sqrt(63/64) 2^51 and 2^51, by what eps^2 carries over from the word below
  const bool far = th - (uint32_t)(e2.hi >> 32) >= 64u;
  if (EARLY && !far) return false;
#ifdef __CUDA_ARCH__
  const int h = __clz(th) >> 1;
#else
  const int h = __builtin_clz(th | 1) >> 1;
#endif
  const uint32_t xh = fx_shl(tl, th, 2 * h), xl = fx_shl(t0, tl, 2 * h);
  const uint32_t S0 = rsqrt(xh) - 0x37000000u;  // 2^23 / sqrt(x), an integer
  const uint64_t SS = (uint64_t)S0 * S0;
  const uint32_t ss1 = (uint32_t)(SS >> 32), ss0 = (uint32_t)SS;
  // E = -e 2^78: bits 32..95 of x S0^2 2^64 (2^110 vanishes modulo 2^96)
  uint64_t Eu = fx_madw<ALU>(xl, ss1, fx_umulhi(xl, ss0));
  Eu = fx_madu(xh, ss0, Eu);
  Eu += (uint64_t)(xh * ss1) << 32;
  const int64_t E = (int64_t)Eu;
  const int32_t E27 = (int32_t)(E >> 27);
  const int64_t E1 = fx_mads(fx_mulhi(E27, E27), -192, E);  // -(e + 3 e^2/4) 2^78
  const int64_t V =
      fx_madws<ALU>((int32_t)S0, (int32_t)(E1 >> 32), (int32_t)fx_umulhi(S0, (uint32_t)E1), 0);
  uint64_t R = ((uint64_t)(S0 << 7) << 32) - (uint64_t)(V >> 8);
  if (!EARLY && !far) R = 0;
  const uint32_t Rh = (uint32_t)(R >> 32), Rl = (uint32_t)R;
  p.Rh = Rh;
  p.Rl = Rl;
  // R^2: twice the cross product over 2^32 is its shift by 31 (R <= 2^63)
  const uint64_t m1 = fx_madu(Rl, Rh, 0);
  const uint64_t R2 =
      fx_madw<ALU>(Rh, Rh, (uint32_t)(ALU ? m1 >> 31 : fx_madu(Rl, Rh, m1) >> 32));
  p.Qh = (uint32_t)(R2 >> 31);
  p.Ql = (uint32_t)R2 << 1;
  p.s = 36 - 3 * h;
  p.sp = 23 - h;
  return far;
}

// a += w >> s for the 96-bit w (WIDE: s < 64, else s < 32)
template <bool WIDE>
FX_HD void fx_add_shifted(fx96 &a, uint32_t w0, uint32_t w1, int32_t w2, int s) {
  if (WIDE) {
    if (s >= 32) {
      w0 = w1;
      w1 = (uint32_t)w2;
      w2 >>= 31;
    }
    s &= 31;
  }
  fx_add(a, fx_shr(w0, w1, s), fx_shr(w1, (uint32_t)w2, s), (uint32_t)(w2 >> s));
}

// The terms of one side, aligned for the 96-bit sums: potential (Y aligned by
// p.sp, three words) and force components (of D: the side at j takes the sum
// with its sign changed).
struct FxTerm {
  uint32_t w0, w1;
  int32_t w2;
};
FX_HD FxTerm fx_align(uint32_t w0, uint32_t w1, int32_t w2, int s) {
  return FxTerm{fx_shr(w0, w1, s), fx_shr(w1, (uint32_t)w2, s), w2 >> s};
}
// R, unsigned: 2^63 where x = 1/4 (r^2 a power of four)
FX_HD FxTerm fx_align_r(const FxPair &p) {
  return FxTerm{fx_shr(0, p.Rl, p.sp), fx_shr(p.Rl, p.Rh, p.sp), (int32_t)(p.Rh >> p.sp)};
}
// D_c F, unaligned
template <bool ALU>
FX_HD FxTerm fx_force(const FxPair &p, int c, int32_t fh, int32_t fl) {
  int64_t mid = fx_mads(p.dl[c], fh, (int64_t)((p.dl[c] >> 16) * (fl >> 16)));
  mid = fx_mads(p.dh[c], fl, mid);
  const int32_t mh = (int32_t)(mid >> 32);
  const int64_t hh =
      ALU ? fx_madws<ALU>(p.dh[c], fh, mh, mh >> 31) : fx_mads(p.dh[c], fh, 0) + (mid >> 32);
  return FxTerm{(uint32_t)mid, (uint32_t)hh, (int32_t)(hh >> 32)};
}
template <bool ALU>
FX_HD uint64_t fx_mulhi64(uint32_t ah, uint32_t al, uint32_t bh, uint32_t bl) {
  const uint64_t m = fx_madu(al, bh, fx_madu(ah, bl, 0xC0000000u));
  return fx_madw<ALU>(ah, bh, (uint32_t)(m >> 32));
}

// The sums of one side for the mass at the other end.
template <bool ALU, bool WIDE>
FX_HD void fx_side(const FxPair &p, const FxMass &M, fx96 (&f)[3], fx96 &pot) {
  const uint64_t Y = fx_mulhi64<ALU>(M.h, M.l, p.Rh, p.Rl);
  const uint32_t yh = (uint32_t)(Y >> 32), yl = (uint32_t)Y;
  fx_add_shifted<WIDE>(pot, 0, yl, (int32_t)yh, p.sp + M.dm);
  const uint64_t F = fx_mulhi64<ALU>(yh, yl, p.Qh, p.Ql);
  const int32_t fl = (int32_t)(uint32_t)F;
  const int32_t fh = (int32_t)((uint32_t)(F >> 32) + ((uint32_t)F >> 31));
#pragma unroll
  for (int c = 0; c < 3; c++) {
    const FxTerm t = fx_force<ALU>(p, c, fh, fl);
    fx_add_shifted<WIDE>(f[c], t.w0, t.w1, t.w2, p.s + M.dm);
  }
}

// Equal masses on each side: the terms without the mass (y and y^3), the same
// for both sides; the sums are multiplied by the masses when they are
// converted, with FX_EQ_EM for em.
constexpr int FX_EQ_EM = -2;
template <bool ALU>
FX_HD void fx_both(const FxPair &p, fx96 (&f)[3], fx96 &pot, fx96 (*g)[3], fx96 *gpot) {
  const FxTerm y = fx_align_r(p);
  fx_add(pot, y.w0, y.w1, (uint32_t)y.w2);
  if (gpot) fx_add(*gpot, y.w0, y.w1, (uint32_t)y.w2);
  const uint64_t F = fx_mulhi64<ALU>(p.Rh, p.Rl, p.Qh, p.Ql);
  const int32_t fl = (int32_t)(uint32_t)F;
  const int32_t fh = (int32_t)((uint32_t)(F >> 32) + ((uint32_t)F >> 31));
#pragma unroll
  for (int c = 0; c < 3; c++) {
    const FxTerm w = fx_force<ALU>(p, c, fh, fl), t = fx_align(w.w0, w.w1, w.w2, p.s);
    fx_add(f[c], t.w0, t.w1, (uint32_t)t.w2);
    if (g) fx_add((*g)[c], t.w0, t.w1, (uint32_t)t.w2);
  }
}

// Binary exponents of the converted sums: force = acc 2^fx_force_exp, potential
// sum = acc 2^fx_pot_exp.
FX_HD int fx_force_exp(int L, int em) { return em - 181 - 2 * L; }
FX_HD int fx_pot_exp(int L, int em) { return em - 133 - L; }

}  // namespace nb
