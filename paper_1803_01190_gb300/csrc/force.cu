// Force kernels: Eq. 1-2 of the paper (section 1), the O(N^2) sum over all
// pairs of softened gravitational accelerations
//     a_i = G sum_{j != i} m_j (r_j - r_i) / (|r_j - r_i|^2 + eps^2)^{3/2}
// and potentials pot_i = -G sum_{j != i} m_j / (|r_j - r_i|^2 + eps^2)^{1/2}.
//
// One thread block owns BT*R i-particles (R per thread, in registers) and one
// j-segment; it walks the segment in tiles of T j-particles staged through
// shared memory (the paper's GFC kernel stages i and j data in shared memory,
// section 2; here only j is staged: i stays in registers).  Every thread reads
// the same tile entry at the same time, a shared-memory broadcast.  The self
// pair j == i is excluded by a select in the few tiles that overlap the
// block's own i-range; all other tiles run without a predicate.
//
// The kernels write raw sums (no G, positive potential sum) per j-segment;
// the epilogue kernels in update.cu sum the segments in a fixed order, apply
// G and the update of the integrator.
//
// Four arithmetics:
//   f64   binary64.  GB300 issues binary64 at about 1/72 of the binary32
//         rate, one FP64 instruction in the time of 32 integer ones, so the
//         one-sided kernel sums softened pairs in 64-bit fixed point on the
//         integer pipes (fixed.cuh), with less rounding than binary64 pair
//         terms have.  Where that does not apply (eps = 0; masses of one tile
//         over more than 2^8, negative or subnormal ones; single pairs too
//         close for their tile's unit) it takes the binary64 body, bound by the
//         FP64 pipe with 9 FP64 instructions per pair (3 DADD for d, 3 DFMA for
//         |d|^2 + eps^2, 3 DFMA for the acceleration sums); the rest of that
//         body runs on the integer and FP32 pipes: 1/r and 1/r^2 within 0.52 ulp
//         (SFU seed, exact integer residual), the products m/r and (m/r)/r^2 by a
//         correctly rounded integer binary64 multiply, and the potential sum by a
//         correctly rounded integer binary64 add.  At large N the FP64 path
//         evaluates each pair once for both particles: softened ones in the same
//         fixed point (k_force_fx_sym), eps = 0 in binary64 (k_force_f64_sym: 12
//         FP64 instructions per pair, 6 per interaction).
//   mixed binary32 pair arithmetic (packed: two j per instruction, SFU
//         reciprocal square root) on coordinates re-centred on an anchor (the
//         per-coordinate median) per j-tile, with the i coordinates held as
//         float-float pairs so that the per-tile shift costs three binary32
//         operations per coordinate and no FP64 instruction; per-tile binary32
//         partial sums are folded into float-float (compensated, TwoSum)
//         accumulators, returned as binary64.
//   f64e  binary64-class accuracy on the binary32 pipes: float-float (about 48
//         significant bits) pair arithmetic on coordinates re-centred per
//         j-tile, float-float tile partials folded into binary64 per tile.
//         About 136 to 148 binary32 operations per pair (86 to 98 per
//         interaction when each pair is evaluated once), but on pipes 64 times
//         faster than GB300's FP64 pipe.  From 64 blocks of 256 particles it
//         evaluates each pair once for both particles (k_force_f64e_sym).
//   f32   binary32 throughout (packed pairs, SFU reciprocal square root) with
//         plain binary32 accumulation: the paper's SP.  The two halves of a
//         thread's packed accumulators (even and odd j) are added at the end.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>

#include "fixed.cuh"
#include "nbody_internal.cuh"

namespace nb {

__device__ __forceinline__ float rsqrt_approx(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// 1/sqrt(x) and 1/x in binary64 (each within about 0.52 ulp) for x in
// [2^-60, 2^60), without any FP64 instruction: GB300's FP64 pipe is the
// bottleneck of the FP64 force kernel, while its FP32 and integer pipes are
// idle there.  Inputs are the two halves of x; outputs are the 53-bit
// significands (in [2^52, 2^53)) and biased binary64 exponents.
//  1. x = xh + xl in binary32: xh = the top 24 significant bits of x moved
//     into a float by integer operations (exponent 1023 -> 127), xl = the
//     next 29 bits converted and scaled (relative error 2^-47 of x).
//  2. Seed y0 = SFU rsqrt(xh) (relative error below 2^-21), improved on the
//     FP32 pipe: e0 = 1 - x y0^2 from exact products (TwoProd by FMA);
//     g = e0 (1/2 + 3 e0/8), the second-order correction.
//  3. s = y0 (1 + g) as an integer significand S in [2^30, 2^31) with a
//     binary64 exponent E: s = S 2^(E - 1053), |x s^2 - 1| < 2^-29.
//  4. Exact residual in integers: with X the 53-bit significand of x,
//     P = X S^2 is within 2^(K-29) of 2^K, K = 3181 - Ex - 2E; the low 96 bits
//     of P (three 32x32 products and the high half of the fourth) give
//     T = (P - 2^K) / 2^32 exactly as a signed 64-bit integer, and
//     e = 1 - x s^2 = -T 2^(32-K).
//  5. 1/sqrt(x) = s (1 + e/2 + 3e^2/8 + ...) and 1/x = s^2 (1 + e + e^2 ...);
//     e^2 < 2^-58 is below the rounding, so the significands are
//     S 2^22 - S T 2^(53-K) and S^2 / 2^sh - (S^2 / 2^32) T 2^(64-K-sh), formed
//     with 8 fraction bits, renormalised by one bit if they left [2^52, 2^53)
//     and rounded to nearest.
__device__ __forceinline__ void rsqrt_recip_sig(unsigned hi, unsigned lo, uint64_t &R, int &ER,
                                                uint64_t &Q, int &EQ) {
  // 1-2: binary32 seed and second-order correction
  const float xh = __uint_as_float(__funnelshift_l(lo, hi - 0x38000000u, 3));
  const float scale = __uint_as_float(((hi >> 20) - 948u) << 23);  // 2^(Ex - 1075)
  const float xl = __uint2float_rn(lo & 0x1FFFFFFFu) * scale;
  const float y0 = rsqrt_approx(xh);
  const float th = y0 * y0, tl = fmaf(y0, y0, -th);
  const float u = xh * th, ue = fmaf(xh, th, -u);
  const float e0 = __fsub_rn(__fsub_rn(__fsub_rn(1.0f, u), ue), fmaf(xh, tl, xl * th));
  const float g = e0 * fmaf(e0, 0.375f, 0.5f);
  // 3: S = y0's significand at a 2^30 scale plus y0 g rounded at that scale
  const unsigned yb = __float_as_uint(y0);
  const float y0m = __uint_as_float((yb & 0x7FFFFFu) | 0x3F800000u);  // y0's significand in [1, 2)
  const int ci = __float2int_rn(y0m * (g * 1073741824.0f));
  unsigned S = (((yb & 0x7FFFFFu) | 0x800000u) << 7) + (unsigned)ci;
  int E = (int)((yb >> 23) & 0xFFu) + 896;
  if (S >= 0x80000000u) {
    S >>= 1;
    E += 1;
  } else if (S < 0x40000000u) {
    S <<= 1;
    E -= 1;
  }
  // 4: T = (X S^2 - 2^K) / 2^32 from the low 96 bits of the product
  const int Ex = (int)(hi >> 20);
  const unsigned a1 = (hi & 0xFFFFFu) | 0x100000u;
  const uint64_t S2 = (uint64_t)S * S;
  const unsigned b1 = (unsigned)(S2 >> 32), b0 = (unsigned)S2;
  uint64_t Tu = (uint64_t)a1 * b0 + __umulhi(lo, b0);
  Tu += (uint64_t)lo * b1;
  Tu += (uint64_t)(a1 * b1) << 32;
  const int Th = (int)(Tu >> 32);
  const unsigned Tl = (unsigned)Tu;
  // 5a: 1/sqrt(x)
  const int64_t ST = (int64_t)(int)S * Th + (int64_t)__umulhi(S, Tl);  // S T / 2^32
  const int64_t Rf = (int64_t)((uint64_t)S << 30) - (ST >> (3088 - Ex - 2 * E));
  const int sR = 8 + (Rf >= (int64_t)1 << 61) - (Rf < (int64_t)1 << 60);
  R = (uint64_t)(Rf + ((int64_t)1 << (sR - 1))) >> sR;
  ER = E + sR - 8;
  // 5b: 1/x
  const int sh = 8 + (b1 >= 0x20000000u);
  const int64_t BT = (int64_t)b1 * Th + (int64_t)__umulhi(b1, Tl);  // (S^2 / 2^32) T / 2^32
  const int64_t Qf = (int64_t)(S2 >> (sh - 8)) - (BT >> (3077 - Ex - 2 * E + sh));
  const int sQ = 8 + (Qf >= (int64_t)1 << 61) - (Qf < (int64_t)1 << 60);
  Q = (uint64_t)(Qf + ((int64_t)1 << (sQ - 1))) >> sQ;
  EQ = sh + 2 * E - 1031 + sQ - 8;
}

// Binary64 multiplication on the integer pipes, correctly rounded (to nearest,
// ties to even): significands A in [2^52, 2^53] and B in [2^52, 2^53) with
// biased exponents ea, eb; the caller guarantees a normal result.  The 106-bit
// product comes from four 32x32 products; U = its top 64 bits (in [2^62, 2^64)),
// the bits below form the sticky bit.  Returns the significand (2^53 after a
// rounding carry, which the packing below absorbs into the exponent) and the
// biased exponent.
__device__ __forceinline__ uint64_t mul_sig(uint64_t A, int ea, uint64_t B, int eb, int &e) {
  const unsigned a1 = (unsigned)(A >> 32), a0 = (unsigned)A;
  const unsigned b1 = (unsigned)(B >> 32), b0 = (unsigned)B;
  const uint64_t lo = (uint64_t)a0 * b0;
  uint64_t V = (uint64_t)a1 * b0 + (lo >> 32);
  V += (uint64_t)a0 * b1;
  const uint64_t U = (((uint64_t)a1 * b1) << 22) + (V >> 10);
  const int n = (int)(U >> 63);
  const int sft = 10 + n;
  const uint64_t sig = U >> sft;
  const uint64_t rb = (U >> (sft - 1)) & 1u;
  const bool st = ((U & (((uint64_t)1 << (sft - 1)) - 1u)) | (V & 0x3FFu) | (unsigned)lo) != 0;
  e = ea + eb - 1023 + n;
  return sig + (rb & (uint64_t)(st | (bool)(sig & 1u)));
}
__device__ __forceinline__ double pack_f64(uint64_t sig, int e) {
  return __longlong_as_double((long long)((((uint64_t)(e - 1)) << 52) + sig));
}

// Binary64 addition of two non-negative numbers on the integer pipes (the
// potential sum of the one-sided kernel), correctly rounded to nearest even and
// bit-identical to DADD: significands at bit 62 of a 64-bit word, the smaller
// one shifted right by the exponent difference with a sticky bit, at most a
// one-bit normalisation after a carry, rounded at bit 10.  ok = false for a
// subnormal or overflowing result or a negative operand, where the caller adds
// in binary64 out of line.  It costs about 40 ALU-pipe instructions, less ALU
// time than the FP64 pipe time of one DADD (one FP64 instruction takes the
// pipe as long as 32 ALU instructions): +12 % measured in the one-sided
// kernel, and in the each-pair-once kernel, for both of its potential sums,
// +22 % together with the block shape that makes room for the registers.
__device__ __forceinline__ uint64_t add_pos_bits(uint64_t a, uint64_t b, bool &ok) {
  const uint64_t M52 = 0xFFFFFFFFFFFFFull;
  const bool sw = b > a;
  const uint64_t X = sw ? b : a, Y = sw ? a : b;
  const int eX = (int)(X >> 52), eY = (int)(Y >> 52);
  const uint64_t MX = ((X & M52) | ((uint64_t)1 << 52)) << 10;
  const uint64_t MY0 = ((Y & M52) | ((uint64_t)(eY != 0) << 52)) << 10;
  const int dc = min(eX - eY, 63);
  const uint64_t st = (MY0 & (((uint64_t)1 << dc) - 1u)) != 0;
  const uint64_t S = (MX + (MY0 >> dc)) | st;
  const int c = (int)(S >> 63);
  const uint64_t N = (S >> c) | (S & (uint64_t)c);
  uint64_t sig = N >> 10;
  sig += ((N >> 9) & 1u) & (uint64_t)(((N & 0x1FFu) != 0) | (bool)(sig & 1u));
  const int E = eX + c;
  ok = (E <= 2046 && !(eY == 0 && Y != 0) && eX != 0 && ((a | b) >> 63) == 0) || X == 0;
  return X == 0 ? 0 : ((uint64_t)(E - 1) << 52) + sig;
}
__device__ __noinline__ uint64_t add_pos_slow(uint64_t a, uint64_t b) {
  return (uint64_t)__double_as_longlong(__longlong_as_double((long long)a) +
                                        __longlong_as_double((long long)b));
}
// acc += v for the bit pattern acc of a non-negative binary64 sum
__device__ __forceinline__ void acc_pos(uint64_t &acc, double v) {
  bool ok;
  const uint64_t vb = (uint64_t)__double_as_longlong(v);
  const uint64_t r = add_pos_bits(acc, vb, ok);
  if (ok)
    acc = r;
  else
    acc = add_pos_slow(acc, vb);
}

// The same quantities in binary64 arithmetic, out of line: for r^2 outside
// [2^-60, 2^60) (and zero or non-finite) and for masses outside
// [2^-895, 2^897) (and zero), where the integer path's ranges do not hold.
__device__ __noinline__ double2 pair_scale_f64_slow(double r2, double m) {
  const double my = m * (1.0 / sqrt(r2));
  return make_double2(my, my * (1.0 / r2));
}

// float-float accumulation a += b (Knuth's TwoSum; exact error term).
__device__ __forceinline__ void two_sum_acc(float &hi, float &lo, float b) {
  const float s = __fadd_rn(hi, b);
  const float bb = __fsub_rn(s, hi);
  const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  hi = s;
  lo = __fadd_rn(lo, err);
}

// a += s m, the product with its rounding error (m = 1: exactly a += s).
__device__ __forceinline__ void fold_tile(float &hi, float &lo, float s, float m) {
  const float p = __fmul_rn(s, m);
  two_sum_acc(hi, lo, p);
  lo = __fadd_rn(lo, __fmaf_rn(s, m, -p));
}

// ---------------------------------------------------------------- work descriptors
// A kernel runs units k = first(), first() + stride(), ... < count().
// Dense: one system of n particles; block (x, y) = i-block x of the rows
// [i_base, i_base + rows) against j-segment y of all n; the row sums go to
// part[y * rows + (i - i_base)] (all rows: i_base = 0, rows = n).  i-blocks
// start at multiples of per_block whatever i_base is: how a tile is summed
// depends on the whole i-block (the unit of the fixed-point sums; whether the
// tile holds some of the block's own particles), so a row's sum is the same,
// bit for bit, whichever rows are asked for.  Only the rows asked for are
// written.
struct DenseWork {
  int64_t n, seg, i_base, rows;
  double eps2;
  int per_block, tile;
  __device__ __forceinline__ int64_t first() const { return 0; }
  __device__ __forceinline__ int64_t stride() const { return 1; }
  __device__ __forceinline__ int64_t count() const { return 1; }
  __device__ __forceinline__ Unit get(int64_t) const {
    Unit u;
    const int64_t r0 = (int64_t)blockIdx.x * per_block - i_base % per_block;
    u.i0 = i_base + r0;
    u.ni = (int)min((int64_t)per_block, n - i_base - r0);
    u.w0 = (int)max((int64_t)0, -r0);
    u.w1 = (int)min((int64_t)u.ni, rows - r0);
    u.j0 = (int64_t)blockIdx.y * seg;
    u.nj = (int)min(seg, n - u.j0);
    u.out = (int64_t)blockIdx.y * rows + r0;
    u.anchor = u.j0 / tile;
    u.eps2 = eps2;
    return u;
  }
};
// Table: block x runs units[x], units[x + gridDim.x], ... (many systems of
// uneven size in one launch; a grid smaller than the table makes the launch
// persistent, which caps how many of its blocks sit on an SM at once).
struct TableWork {
  const Unit *units;
  int64_t n;
  __device__ __forceinline__ int64_t first() const { return blockIdx.x; }
  __device__ __forceinline__ int64_t stride() const { return gridDim.x; }
  __device__ __forceinline__ int64_t count() const { return n; }
  __device__ __forceinline__ Unit get(int64_t k) const { return units[k]; }
};

// Writes the sums v of i-particle li of the unit u.  IW > 1: the IW threads that share
// it (thread `it` of IT, share jw) add theirs in order first.
template <int IW, class V>
__device__ __forceinline__ void store_shares(V *part, const Unit &u, int li, V v, V *red, int it,
                                             int IT, int jw) {
  if (IW > 1) {
    __syncthreads();
    red[threadIdx.x] = v;
    __syncthreads();
    if (jw != 0) return;
#pragma unroll
    for (int w = 1; w < IW; w++) {
      const V o = red[w * IT + it];
      v.x += o.x;
      v.y += o.y;
      v.z += o.z;
      v.w += o.w;
    }
  }
  if (li >= u.w0 && li < min(u.ni, u.w1)) part[u.out + li] = v;
}

// ---------------------------------------------------------------- binary64
template <bool MASK>
__device__ __forceinline__ void body_f64(const d4 &pj, double xi, double yi, double zi,
                                         double eps2, double &ax, double &ay, double &az,
                                         uint64_t &pt, bool self) {
  const double dx = pj.x - xi, dy = pj.y - yi, dz = pj.z - zi;
  double r2 = fma(dx, dx, fma(dy, dy, fma(dz, dz, eps2)));
  double m = pj.w;
  if (MASK && self) {
    r2 = 1.0;
    m = 0.0;
  }
  // my = m / r and f = my / r^2, both binary64 products correctly rounded
  const unsigned hi = (unsigned)__double2hiint(r2);
  const unsigned mh = (unsigned)__double2hiint(m);
  double my, f;
  if (hi - 0x3C300000u < 0x43B00000u - 0x3C300000u && (mh >> 20) - 128u < 1793u) {
    uint64_t R, Q;
    int ER, EQ, emy, ef;
    rsqrt_recip_sig(hi, (unsigned)__double2loint(r2), R, ER, Q, EQ);
    const uint64_t Am = ((uint64_t)((mh & 0xFFFFFu) | 0x100000u) << 32) | (unsigned)__double2loint(m);
    const uint64_t smy = mul_sig(Am, (int)(mh >> 20), R, ER, emy);
    const uint64_t sf = mul_sig(smy, emy, Q, EQ, ef);
    my = pack_f64(smy, emy);
    f = pack_f64(sf, ef);
  } else {
    const double2 v = pair_scale_f64_slow(r2, m);
    my = v.x;
    f = v.y;
  }
  ax = fma(dx, f, ax);
  ay = fma(dy, f, ay);
  az = fma(dz, f, az);
  acc_pos(pt, my);  // the potential sum: integer pipes
}

// One pair of the binary64 body, out of line: (d_x, d_y, d_z) m / r^3 and m / r.
__device__ __noinline__ d4 pair_f64(double dx, double dy, double dz, double m, double eps2) {
  double ax = 0.0, ay = 0.0, az = 0.0;
  uint64_t pt = 0;
  body_f64<false>(d4{dx, dy, dz, m}, 0.0, 0.0, 0.0, eps2, ax, ay, az, pt, false);
  return d4{ax, ay, az, __longlong_as_double((long long)pt)};
}

// ---------------------------------------------------------------- fixed point: tile scale
// Enclosing box of a set of particles from the high words of their coordinates
// (order-preserving signed keys), their largest mass and smallest positive
// mass (high words); mmin = -1 marks a non-finite value or a negative or
// subnormal mass.
struct FxBox {
  int lo[3], hi[3], mmax, mmin;
};
__device__ __forceinline__ void fx_box_init(FxBox &b) {
#pragma unroll
  for (int c = 0; c < 3; c++) {
    b.lo[c] = 0x7FFFFFFF;
    b.hi[c] = (int)0x80000000;
  }
  b.mmax = 0;
  b.mmin = 0x7FFFFFFF;
}
__device__ __forceinline__ void fx_box_add(FxBox &b, const d4 &p) {
  const int h[4] = {__double2hiint(p.x), __double2hiint(p.y), __double2hiint(p.z),
                    __double2hiint(p.w)};
#pragma unroll
  for (int c = 0; c < 3; c++) {
    b.lo[c] = min(b.lo[c], fx_key(h[c]));
    b.hi[c] = max(b.hi[c], fx_key(h[c]));
  }
  bool bad = h[3] < 0 || (h[3] < 0x00100000 && (h[3] | __double2loint(p.w)) != 0);
#pragma unroll
  for (int c = 0; c < 4; c++) bad |= (h[c] & 0x7FF00000) == 0x7FF00000;
  b.mmax = max(b.mmax, h[3]);
  b.mmin = min(b.mmin, bad ? -1 : p.w > 0.0 ? h[3] : 0x7FFFFFFF);
}
__device__ __forceinline__ void fx_box_warp(FxBox &b) {
#pragma unroll
  for (int c = 0; c < 3; c++) {
    b.lo[c] = __reduce_min_sync(0xFFFFFFFFu, b.lo[c]);
    b.hi[c] = __reduce_max_sync(0xFFFFFFFFu, b.hi[c]);
  }
  b.mmax = __reduce_max_sync(0xFFFFFFFFu, b.mmax);
  b.mmin = __reduce_min_sync(0xFFFFFFFFu, b.mmin);
}
__device__ __forceinline__ void fx_box_join(FxBox &b, const FxBox &o) {
#pragma unroll
  for (int c = 0; c < 3; c++) {
    b.lo[c] = min(b.lo[c], o.lo[c]);
    b.hi[c] = max(b.hi[c], o.hi[c]);
  }
  b.mmax = max(b.mmax, o.mmax);
  b.mmin = min(b.mmin, o.mmin);
}

// Unit exponent L and mass exponent em for the i's of box bi against the j's
// of box bj; ok = false: the fixed-point form does not apply (non-finite
// values, negative masses, masses over too wide a range, extreme exponents, or
// eps = 0).  eps = 0 stays in binary64: there every pair term is specified to
// the ulp of the binary64 operations.  range: exponents that the j's positive
// masses span.  Box: largest extent below 2^box.
struct FxScale {
  int L, em, range, box;
  bool ok;
};
// em and range of a box's masses; false: outside the rule whatever their range
__device__ __forceinline__ bool fx_mass_scale(const FxBox &b, int &em, int &range) {
  const int ex = b.mmax >> 20;
  em = b.mmax == 0 ? 0 : ex - 1023;
  range = b.mmax == 0 ? 0 : ex - (b.mmin >> 20);
  return b.mmin >= 0 && (b.mmax == 0 || (ex > 623 && ex < 1423));
}
__device__ __forceinline__ int fx_eps_exp(double eps2) {  // eps < 2^it
  return ((__double2hiint(eps2) >> 20) - 1021) >> 1;
}
__device__ __forceinline__ FxScale fx_scale(const FxBox &bi, const FxBox &bj, double eps2) {
  FxScale f;
  f.box = -1023;
#pragma unroll
  for (int c = 0; c < 3; c++) {
    // bounds of the coordinate: the low words of the keys are unknown
    const int l = fx_key(min(bi.lo[c], bj.lo[c])), h = fx_key(max(bi.hi[c], bj.hi[c]));
    const double lo = __hiloint2double(l, l < 0 ? -1 : 0), hi = __hiloint2double(h, h < 0 ? 0 : -1);
    f.box = max(f.box, (__double2hiint(hi - lo) >> 20) - 1022);
  }
  const int top = max(f.box, fx_eps_exp(eps2));
  f.L = top - FX_BITS;
  f.ok = fx_mass_scale(bj, f.em, f.range) && eps2 > 0.0 && bi.mmin >= 0 && top > -200 && top < 200;
  return f;
}
// Do masses over `range` exponents keep their digits in this tile?  Light ones lose
// some to the heaviest, and all lose some where eps, not the extent, sets the unit
// (the gap): both count towards FX_MASS_RANGE.  With eps at 2^6 times the system's
// size a force on the heaviest of masses over 2^8 was off by 1.3e-14 of its terms'
// magnitudes without the gap.  It is an upper bound; where the upper words of the
// coordinates do not tell the box's size (far from the origin) it rules unequal
// masses out.  Equal ones lose nothing by it that the pairs too close for the unit
// do not cover.
__device__ __forceinline__ bool fx_masses_fit(int range, const FxScale &f, const FxBox &bi,
                                              const FxBox &bj, double eps2) {
  if (range == 0) return true;
  int far = 0;
#pragma unroll
  for (int c = 0; c < 3; c++)
    far = max(far, max(fx_key(min(bi.lo[c], bj.lo[c])) & 0x7FFFFFFF,
                       fx_key(max(bi.hi[c], bj.hi[c])) & 0x7FFFFFFF));
  // an upper word is worth less than 2^(far's exponent - 1042)
  const int gap =
      f.box > (far >> 20) - 1040 ? max(fx_eps_exp(eps2) - f.box + 1, 0) : FX_MASS_RANGE;
  return range + gap <= FX_MASS_RANGE;
}
__device__ __forceinline__ double fx_exp2(int e) { return __hiloint2double((e + 1023) << 20, 0); }
// acc + a 2^e, a the accumulator, scale = 2^(e + 32)
__device__ __forceinline__ double fx_fold(double acc, const fx96 &a, double scale) {
  const double v = fma((double)a.w0, 0x1p-32, fma((double)a.w2, 0x1p32, (double)a.w1));
  return fma(v, scale, acc);
}
__device__ __forceinline__ void fx_coords(const d4 &p, int L, uint64_t (&X)[3]) {
  X[0] = fx_coord((uint32_t)__double2hiint(p.x), (uint32_t)__double2loint(p.x), L);
  X[1] = fx_coord((uint32_t)__double2hiint(p.y), (uint32_t)__double2loint(p.y), L);
  X[2] = fx_coord((uint32_t)__double2hiint(p.z), (uint32_t)__double2loint(p.z), L);
}
// Too many of a tile's pairs too close for its unit?  One far particle makes all pairs
// within 2^-10 of the distance to it such pairs; each costs its fixed-point geometry
// and then a call for all lanes of the warp, so that from a small share of them on the
// binary64 body is the cheaper one for the whole tile.  The share is estimated from
// one pair a thread: its first i-particle against the tile entry 16 lanes off (never
// itself: blocks and tiles start at multiples of 32), differences taken from the
// upper words; FX_NEAR of a block's 128 such pairs send the tile to binary64.
// Measured (Gint/s, N = 65536, Plummer sphere of unit core, every 128th particle put
// at 200, 400, 1000; one-sided): never 107, 78, 56; at 1 89, 71, 71; 2 100, 72, 71; 4 106,
// 76, 71; 8 105, 84, 71; 16 104, 85, 71; each pair once (never: with every pair of a tile
// out of line) 99, 50, 41; 1 105, 93, 93; 4 115, 93, 93; 8 118, 91, 93; 16 118, 90, 93.
// The estimate costs a sphere without far particles nothing that shows (one-sided
// 132.1 -> 132.5, each pair once 228.1 -> 228.7).
constexpr int FX_NEAR = 8;
__device__ __forceinline__ bool fx_near(const uint64_t (&Xj)[3], const uint64_t (&Xi)[3]) {
  bool near = true;
#pragma unroll
  for (int c = 0; c < 3; c++) {
    const unsigned j = __shfl_xor_sync(0xFFFFFFFFu, (unsigned)(Xj[c] >> 32), 16);
    near &= j - (unsigned)(Xi[c] >> 32) + 0x80000u < 0x100000u;
  }
  return near;
}
struct FxRsqrt {
  __device__ __forceinline__ uint32_t operator()(uint32_t x) const {
    return __float_as_uint(rsqrt_approx(__uint2float_rn(x)));
  }
};

// How the masses of a tile enter (fixed.cuh): all equal, one exponent, or an
// exponent each.  FX_SELF is FX_NARROW for a tile that may hold the block's own
// particles (FX_WIDE looks for them too).
enum FxMode { FX_EQUAL, FX_NARROW, FX_SELF, FX_WIDE };
struct FxEarly {
  static constexpr bool value = true;
};
struct FxLate {
  static constexpr bool value = false;
};

// The fixed-point sum of RI i-particles against the tile entries [k0, k1).
// self(r, k): the pair of particle r with itself (looked at in FX_SELF and
// FX_WIDE);
// close(r, k): adds a pair too close for the tile's unit in binary64.
// U tile entries are taken at a time, interleaved (U = 2 in the split shape, for
// the few warps of a small system, whose time is the latency of a pair: N =
// 1000 21.3 us against 23.2, 4096 139 against 149; U = 4 21.1 and 145).
template <int RI, int U, FxMode MODE, class Self, class Close>
__device__ __forceinline__ void fx_tile(const uint4 *txy, const uint4 *tzm, const int *tdm, int k0,
                                        int k1, const FxEps &e2, const uint64_t (&Xi)[RI][3],
                                        fx96 (&f)[RI][3], fx96 (&pt)[RI], Self self, Close close) {
  auto pair = [&](int k, int r, auto early) {
    const uint4 a = txy[k], b = tzm[k];
    const uint64_t Xj[3] = {((uint64_t)a.y << 32) | a.x, ((uint64_t)a.w << 32) | a.z,
                            ((uint64_t)b.y << 32) | b.x};
    const int dm = MODE == FX_WIDE ? tdm[k] : 0;
    const bool s = (MODE == FX_WIDE || MODE == FX_SELF) && self(r, k);
    FxPair p;
    const bool far = fx_geometry<false, decltype(early)::value>(Xj, Xi[r], e2, FxRsqrt(), p);
    if (!decltype(early)::value || far) {
      if (MODE == FX_EQUAL)
        fx_both<false>(p, f[r], pt[r], nullptr, nullptr);
      else
        fx_side<false, MODE == FX_WIDE>(p, FxMass{s ? 0u : b.w, s ? 0u : b.z, dm}, f[r], pt[r]);
    }
    return far || s;
  };
  int k = k0;
  if (U > 1) {
#pragma unroll 1
    for (; k + U <= k1; k += U) {
      bool done[U][RI], all = true;
#pragma unroll
      for (int u = 0; u < U; u++)
#pragma unroll
        for (int r = 0; r < RI; r++) {
          done[u][r] = pair(k + u, r, FxLate());
          all &= done[u][r];
        }
      if (!all)
#pragma unroll
        for (int u = 0; u < U; u++)
#pragma unroll
          for (int r = 0; r < RI; r++)
            if (!done[u][r]) close(r, k + u);
    }
  }
#pragma unroll 1
  for (; k < k1; k++)
#pragma unroll
    for (int r = 0; r < RI; r++)
      if (!pair(k, r, FxEarly())) close(r, k);
}

// The binary64 force sum, bound by the FMA-heavy pipe (the wide integer
// multiplies of fixed.cuh; 89 % busy by ncu at N = 16384), not by the FP64
// pipe.  Measured on GB300 (N = 65536, equal masses): 132 Gint/s at R = 1 (123
// for unequal masses), 127 at R = 2, against 63 for the binary64 body with its 9 FP64 instructions; the relative
// error of the accelerations against binary64 terms with pairwise sums falls
// from 4.5e-16 to 1.9e-16 (it is the rounding of the tile sums).  R above 2
// runs in groups of two.
//
// IW warps of a block share the same i-particles and split each j-tile (IW =
// 1: BT * R i-particles per block; IW = 4, for small n: BT / 4 * R, four times
// as many blocks and a quarter of the sequential pairs per thread).  Each tile
// is summed in fixed point where fx_scale allows it and few of its pairs are
// too close for its unit (FX_NEAR), and in binary64 otherwise; single pairs too
// close for the unit go through pair_f64.  i-particles are
// taken two at a time (RI), whatever R is.
template <int BT, int R, int T, int IW, class W>
__global__ void __launch_bounds__(BT) k_force_f64(const d4 *__restrict__ posm, W work,
                                                  d4 *__restrict__ part) {
  chain_begin();
  static_assert(T == BT, "one j per thread");
  constexpr int NW = BT / 32, RI = R < 2 ? R : 2, NG = R / RI, IT = BT / IW;
  __shared__ d4 tile[T];
  __shared__ uint4 txy[T], tzm[T];
  __shared__ int tdm[T];
  __shared__ FxBox sbox[NW];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // i-thread, share of the j-tile
  const int it = IW == 1 ? tid : tid % IT, jw = IW == 1 ? 0 : tid / IT;
  for (int64_t uk = work.first(); uk < work.count(); uk += work.stride()) {
    const Unit u = work.get(uk);
    const int64_t j1 = u.j0 + u.nj;
    const double eps2 = u.eps2;
    d4 acc[NG][RI];
    FxBox bi;
    fx_box_init(bi);
    for (int g = 0; g < NG; g++)
#pragma unroll
      for (int r = 0; r < RI; r++) {
        const int li = (g * RI + r) * IT + it;
        fx_box_add(bi, posm[u.i0 + (li < u.ni ? li : 0)]);
        acc[g][r] = d4{0.0, 0.0, 0.0, 0.0};
      }
    fx_box_warp(bi);
    __syncthreads();
    if (lane == 0) sbox[warp] = bi;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < NW; w++) fx_box_join(bi, sbox[w]);
    for (int64_t jt = u.j0; jt < j1; jt += T) {
      const int cnt = (int)min((int64_t)T, j1 - jt);
      __syncthreads();
      d4 pj = d4{0.0, 0.0, 0.0, 0.0};
      FxBox bj;
      fx_box_init(bj);
      if (tid < cnt) {
        pj = posm[jt + tid];
        tile[tid] = pj;
        fx_box_add(bj, pj);
      }
      fx_box_warp(bj);
      if (lane == 0) sbox[warp] = bj;
      __syncthreads();
#pragma unroll
      for (int w = 0; w < NW; w++) fx_box_join(bj, sbox[w]);
      const FxScale sc = fx_scale(bi, bj, eps2);
      const int k0 = cnt * jw / IW, k1 = cnt * (jw + 1) / IW;
      const bool diag = (jt < u.i0 + u.ni) && (jt + cnt > u.i0);
      const bool wide = sc.range > FX_MASS_NARROW;  // the masses need exponents of their own
      bool fixed = sc.ok && fx_masses_fit(sc.range, sc, bi, bj, eps2), equal = false;
      const double m0 = tile[0].w;
      uint64_t Xi[RI][3];
      auto load_i = [&](int g) {
#pragma unroll
        for (int r = 0; r < RI; r++) {
          const int li = (g * RI + r) * IT + it;
          fx_coords(posm[u.i0 + (li < u.ni ? li : 0)], sc.L, Xi[r]);
        }
      };
      if (fixed) {
        uint64_t X[3];
        fx_coords(pj, sc.L, X);
        load_i(0);
        const bool near = fx_near(X, Xi[0]) && (tid ^ 16) < cnt;
        const uint32_t mh = (uint32_t)__double2hiint(pj.w), ml = (uint32_t)__double2loint(pj.w);
        const FxMass M = wide ? fx_mass<true>(mh, ml, sc.em) : fx_mass<false>(mh, ml, sc.em);
        txy[tid] = make_uint4((uint32_t)X[0], (uint32_t)(X[0] >> 32), (uint32_t)X[1],
                              (uint32_t)(X[1] >> 32));
        tzm[tid] = make_uint4((uint32_t)X[2], (uint32_t)(X[2] >> 32), M.l, M.h);
        tdm[tid] = M.dm;
        equal = __syncthreads_and(__double_as_longlong(pj.w) == __double_as_longlong(m0) ||
                                  tid >= cnt);
        fixed = __syncthreads_count(near) < FX_NEAR;
      }
      if (fixed) {
        // FX_SELF in the split shape alone, where such tiles are a large share
        // (N = 4096: 139 us against 147); elsewhere one more form of the loop
        // made the others slower (N = 20011: 3.54 ms against 3.35)
        const FxMode mode = wide || (diag && IW == 1) ? FX_WIDE
                            : diag                    ? FX_SELF
                            : equal                   ? FX_EQUAL
                                                      : FX_NARROW;
        const int em = mode == FX_EQUAL ? FX_EQ_EM : sc.em;
        const FxEps e2 = fx_eps2(eps2, sc.L);
        double fs = fx_exp2(fx_force_exp(sc.L, em) + 32), ps = fx_exp2(fx_pot_exp(sc.L, em) + 32);
        if (mode == FX_EQUAL) {
          fs *= m0;
          ps *= m0;
        }
        for (int g = 0; g < NG; g++) {
          fx96 f[RI][3] = {}, pt[RI] = {};
          if (g > 0) load_i(g);
          const int ii = (int)(u.i0 - jt) + g * RI * IT + it;  // tile entry of particle 0
          auto self = [&](int r, int k) { return diag && k == ii + r * IT; };
          auto close = [&](int r, int k) {
            const int li = (g * RI + r) * IT + it;
            const d4 pi = posm[u.i0 + (li < u.ni ? li : 0)], q = tile[k];
            const d4 v = pair_f64(q.x - pi.x, q.y - pi.y, q.z - pi.z, q.w, eps2);
            acc[g][r].x += v.x;
            acc[g][r].y += v.y;
            acc[g][r].z += v.z;
            acc[g][r].w += v.w;
          };
          if (mode == FX_WIDE)
            fx_tile<RI, IW == 1 ? 1 : 2, FX_WIDE>(txy, tzm, tdm, k0, k1, e2, Xi, f, pt, self, close);
          else if (IW > 1 && mode == FX_SELF)
            fx_tile<RI, IW == 1 ? 1 : 2, FX_SELF>(txy, tzm, tdm, k0, k1, e2, Xi, f, pt, self, close);
          else if (mode == FX_EQUAL)
            fx_tile<RI, IW == 1 ? 1 : 2, FX_EQUAL>(txy, tzm, tdm, k0, k1, e2, Xi, f, pt, self, close);
          else
            fx_tile<RI, IW == 1 ? 1 : 2, FX_NARROW>(txy, tzm, tdm, k0, k1, e2, Xi, f, pt, self, close);
#pragma unroll
          for (int r = 0; r < RI; r++) {
            acc[g][r].x = fx_fold(acc[g][r].x, f[r][0], fs);
            acc[g][r].y = fx_fold(acc[g][r].y, f[r][1], fs);
            acc[g][r].z = fx_fold(acc[g][r].z, f[r][2], fs);
            acc[g][r].w = fx_fold(acc[g][r].w, pt[r], ps);
          }
        }
      } else {
        for (int g = 0; g < NG; g++) {
          d4 pi[RI];
          uint64_t pt[RI];  // bit patterns of the potential sums
#pragma unroll
          for (int r = 0; r < RI; r++) {
            const int li = (g * RI + r) * IT + it;
            pi[r] = posm[u.i0 + (li < u.ni ? li : 0)];
            pt[r] = (uint64_t)__double_as_longlong(acc[g][r].w);
          }
          if (!diag) {
#pragma unroll 2
            for (int k = k0; k < k1; k++) {
              const d4 q = tile[k];
#pragma unroll
              for (int r = 0; r < RI; r++)
                body_f64<false>(q, pi[r].x, pi[r].y, pi[r].z, eps2, acc[g][r].x, acc[g][r].y,
                                acc[g][r].z, pt[r], false);
            }
          } else {
            for (int k = k0; k < k1; k++) {
              const d4 q = tile[k];
#pragma unroll
              for (int r = 0; r < RI; r++)
                body_f64<true>(q, pi[r].x, pi[r].y, pi[r].z, eps2, acc[g][r].x, acc[g][r].y,
                               acc[g][r].z, pt[r], jt + k == u.i0 + (g * RI + r) * IT + it);
            }
          }
#pragma unroll
          for (int r = 0; r < RI; r++) acc[g][r].w = __longlong_as_double((long long)pt[r]);
        }
      }
    }
    const int w1 = min(u.ni, u.w1);
    if (IW == 1) {
      for (int g = 0; g < NG; g++)
#pragma unroll
        for (int r = 0; r < RI; r++) {
          const int li = (g * RI + r) * IT + it;
          if (li >= u.w0 && li < w1) part[u.out + li] = acc[g][r];
        }
    } else {  // the shares of the j-tiles, added in order
      for (int g = 0; g < NG; g++)
#pragma unroll
        for (int r = 0; r < RI; r++) {
          __syncthreads();
          tile[tid] = acc[g][r];
          __syncthreads();
          const int li = (g * RI + r) * IT + it;
          if (jw == 0 && li >= u.w0 && li < w1) {
            d4 s = tile[it];
#pragma unroll
            for (int w = 1; w < IW; w++) {
              const d4 v = tile[w * IT + it];
              s.x += v.x;
              s.y += v.y;
              s.z += v.z;
              s.w += v.w;
            }
            part[u.out + li] = s;
          }
        }
    }
  }
}

// ---------------------------------------------------------------- binary64, each pair once
// Newton's third law: the pair (i, j) contributes m_j d / w to a_i and
// -m_i d / w to a_j with the same d = r_j - r_i and w = (|d|^2 + eps^2)^{3/2},
// so one evaluation of d, |d|^2 + eps^2, 1/r and 1/r^2 serves both: 12 FP64
// instructions for two interactions instead of 18 (the one-sided kernel's 9 twice).
//
// Particles are cut into M blocks of B = BT*R.  A work item (d, I), d >= 1,
// pairs i-block I with j-block J = (I + d) mod M; d = 1 .. floor(M/2) covers
// every unordered pair of distinct blocks once (for d = M/2 with M even, only
// I < M/2 computes; the other items write zeros).  For a fixed d every block
// is the row block of one item and the column block of one item, so the
// item's row sums (block I) and column sums (block J) each own a slice of the
// per-diagonal buffers rows[dl], cols[dl] without any atomic or race; the
// slices are added in diagonal order afterwards (deterministic).  Pairs
// inside a block (d = 0) run through the one-sided kernel.
//
// Column sums: i stays in registers (R per thread); a j-tile of T particles
// is in shared memory and is walked in chunks of 32.  At step k of a chunk,
// lane l works on j = (l + k) mod 32 with its R i-particles and then hands the
// running sum of that j to lane l - 1, so after 32 steps lane l holds the sum
// over the warp's i-particles of j = l.  The warps' sums are then added in a
// fixed order in shared memory.
__device__ __noinline__ double2 rq_f64_slow(double r2) {
  return make_double2(1.0 / sqrt(r2), 1.0 / r2);
}

struct MassSig {
  uint64_t A;  // 53-bit significand
  int e;       // biased exponent
  bool fast;   // in [2^-895, 2^897): the integer multiply applies
};
__device__ __forceinline__ MassSig mass_sig(double m) {
  const unsigned mh = (unsigned)__double2hiint(m);
  MassSig s;
  s.A = ((uint64_t)((mh & 0xFFFFFu) | 0x100000u) << 32) | (unsigned)__double2loint(m);
  s.e = (int)(mh >> 20);
  s.fast = (mh >> 20) - 128u < 1793u;
  return s;
}

// m/r and (m/r)/r^2 from the integer 1/r, 1/r^2 (or, for masses outside the
// integer range, binary64 products of their packed values)
__device__ __forceinline__ void scale_pair(double m, const MassSig &ms, uint64_t R, int ER,
                                           uint64_t Q, int EQ, double &my, double &f) {
  if (ms.fast) {
    int emy, ef;
    const uint64_t smy = mul_sig(ms.A, ms.e, R, ER, emy);
    const uint64_t sf = mul_sig(smy, emy, Q, EQ, ef);
    my = pack_f64(smy, emy);
    f = pack_f64(sf, ef);
  } else {
    my = m * pack_f64(R, ER);
    f = my * pack_f64(Q, EQ);
  }
}

// Both potential sums, pt (row) and gp (column), are bit patterns added on the
// integer pipes (acc_pos, bit-identical to DADD): 12 FP64 instructions per
// pair, 6 per interaction.
__device__ __forceinline__ void body_f64_sym(const d4 &pj, const MassSig &mj, double xi,
                                             double yi, double zi, double mi,
                                             const MassSig &msi, double eps2, double &ax,
                                             double &ay, double &az, uint64_t &pt, double &gx,
                                             double &gy, double &gz, uint64_t &gp) {
  const double dx = pj.x - xi, dy = pj.y - yi, dz = pj.z - zi;
  const double r2 = fma(dx, dx, fma(dy, dy, fma(dz, dz, eps2)));
  const unsigned hi = (unsigned)__double2hiint(r2);
  double my, f, myj, fj;
  if (hi - 0x3C300000u < 0x43B00000u - 0x3C300000u) {
    uint64_t R, Q;
    int ER, EQ;
    rsqrt_recip_sig(hi, (unsigned)__double2loint(r2), R, ER, Q, EQ);
    scale_pair(pj.w, mj, R, ER, Q, EQ, my, f);
    scale_pair(mi, msi, R, ER, Q, EQ, myj, fj);
  } else {
    const double2 v = rq_f64_slow(r2);
    my = pj.w * v.x;
    f = my * v.y;
    myj = mi * v.x;
    fj = myj * v.y;
  }
  ax = fma(dx, f, ax);
  ay = fma(dy, f, ay);
  az = fma(dz, f, az);
  acc_pos(pt, my);
  gx = fma(-dx, fj, gx);
  gy = fma(-dy, fj, gy);
  gz = fma(-dz, fj, gz);
  acc_pos(gp, myj);
}

// Padding beyond n: massless and far away (finite r^2, zero contribution).
__device__ __forceinline__ d4 pad_or_load(const d4 *posm, int64_t k, int64_t n) {
  return k < n ? posm[k] : d4{1e30, 1e30, 1e30, 0.0};
}

// One column tile (the first cnt entries, in chunks of 32) against R i-particles of
// each thread: row sums into acc, the warp's column sums into colw (ADD: onto it).
template <int R, int T, bool ADD>
__device__ __forceinline__ void f64_sym_tile(const d4 *tile, int cnt, const d4 (&p)[R],
                                             const MassSig (&ms)[R], double eps2, d4 (&acc)[R],
                                             d4 *colw) {
  const int lane = threadIdx.x & 31;
  uint64_t pt[R];
#pragma unroll
  for (int r = 0; r < R; r++) pt[r] = (uint64_t)__double_as_longlong(acc[r].w);
#pragma unroll 1
  for (int c = 0; c < T; c += 32) {
    if (c >= cnt) break;
    double gx = 0.0, gy = 0.0, gz = 0.0;
    uint64_t gp = 0;  // bit pattern of the column potential sum, as pt
    // not unrolled: measured on GB300 at N = 2^18, unroll 2 ran 4 % slower
#pragma unroll 1
    for (int k = 0; k < 32; k++) {
      const d4 pj = tile[c + ((lane + k) & 31)];
      const MassSig mj = mass_sig(pj.w);
#pragma unroll
      for (int r = 0; r < R; r++)
        body_f64_sym(pj, mj, p[r].x, p[r].y, p[r].z, p[r].w, ms[r], eps2, acc[r].x, acc[r].y,
                     acc[r].z, pt[r], gx, gy, gz, gp);
      const int src = (lane + 1) & 31;
      gx = __shfl_sync(0xFFFFFFFFu, gx, src);
      gy = __shfl_sync(0xFFFFFFFFu, gy, src);
      gz = __shfl_sync(0xFFFFFFFFu, gz, src);
      gp = __shfl_sync(0xFFFFFFFFu, gp, src);
    }
    d4 g = d4{gx, gy, gz, __longlong_as_double((long long)gp)};
    if (ADD) {
      const d4 s = colw[c + lane];
      g.x += s.x;
      g.y += s.y;
      g.z += s.z;
      g.w += s.w;
    }
    colw[c + lane] = g;
  }
#pragma unroll
  for (int r = 0; r < R; r++) acc[r].w = __longlong_as_double((long long)pt[r]);
}

template <int BT, int R, int T>
__global__ void __launch_bounds__(BT) k_force_f64_sym(const d4 *__restrict__ posm, int64_t n,
                                                      double eps2, int M, int d0,
                                                      d4 *__restrict__ rows,
                                                      d4 *__restrict__ cols) {
  constexpr int B = BT * R, NW = BT / 32;
  static_assert(T == BT && B % T == 0, "one column sum per thread per tile");
  __shared__ d4 tile[T];
  __shared__ d4 colw[NW][T];
  const int tid = threadIdx.x, warp = tid >> 5;
  const int dl = blockIdx.x / M, I = blockIdx.x % M, d = d0 + dl;
  const int J = (I + d) % M;
  const int64_t i0 = (int64_t)I * B, j0 = (int64_t)J * B;
  d4 *rowo = rows + (int64_t)dl * n;
  d4 *colo = cols + (int64_t)dl * n;
  if (2 * d == M && I >= M / 2) {  // the pair of blocks is the item (I - M/2, I)
    for (int k = tid; k < B; k += BT) {
      if (i0 + k < n) rowo[i0 + k] = d4{0.0, 0.0, 0.0, 0.0};
      if (j0 + k < n) colo[j0 + k] = d4{0.0, 0.0, 0.0, 0.0};
    }
    return;
  }
  d4 p[R], acc[R];
  MassSig ms[R];
#pragma unroll
  for (int r = 0; r < R; r++) {
    p[r] = pad_or_load(posm, i0 + r * BT + tid, n);
    ms[r] = mass_sig(p[r].w);
    acc[r] = d4{0.0, 0.0, 0.0, 0.0};
  }
  for (int t0 = 0; t0 < B; t0 += T) {
    const int64_t jt = j0 + t0;
    __syncthreads();
    for (int k = tid; k < T; k += BT) tile[k] = pad_or_load(posm, jt + k, n);
    __syncthreads();
    f64_sym_tile<R, T, false>(tile, T, p, ms, eps2, acc, colw[warp]);
    __syncthreads();
    {
      d4 s = colw[0][tid];
#pragma unroll
      for (int w = 1; w < NW; w++) {
        const d4 v = colw[w][tid];
        s.x += v.x;
        s.y += v.y;
        s.z += v.z;
        s.w += v.w;
      }
      if (jt + tid < n) colo[jt + tid] = s;
    }
  }
#pragma unroll
  for (int r = 0; r < R; r++) {
    const int64_t i = i0 + r * BT + tid;
    if (i < n) rowo[i] = acc[r];
  }
}

// One pair out of line: what it adds to i's sums and to j's.
struct F64Both {
  d4 i, j;
};
__device__ __noinline__ F64Both pair_f64_both(double dx, double dy, double dz, double mj,
                                              double mi, double eps2) {
  F64Both v = {};
  uint64_t pi = 0, pj = 0;
  body_f64_sym(d4{dx, dy, dz, mj}, mass_sig(mj), 0.0, 0.0, 0.0, mi, mass_sig(mi), eps2, v.i.x,
               v.i.y, v.i.z, pi, v.j.x, v.j.y, v.j.z, pj);
  v.i.w = __longlong_as_double((long long)pi);
  v.j.w = __longlong_as_double((long long)pj);
  return v;
}

// ---------------------------------------------------------------- fixed point, each pair once
// The work items, row and column slices of k_force_f64_sym with the pair
// arithmetic of fixed.cuh: the geometry of a pair (d, 1/r, 1/r^2: 20 of the 38
// wide multiplies of one side) serves both particles.  Sums of a tile are
// 96-bit integers in registers; the column sums of a chunk of 32 j travel
// around the lanes (12 words per step).  Single pairs too close for the unit
// are evaluated in binary64 out of line and added in binary64 (rows in
// registers, columns in the warp's slots of colw, where a lane owns its j at
// each step); tiles that fx_scale does not take, or with many such pairs
// (FX_NEAR), go through the tile loop of k_force_f64_sym.  Measured
// (whole force evaluation, N = 65536): 229 Gint/s for equal masses, where
// the two sides share their terms, 155 for lognormal masses, against 92 for
// k_force_f64_sym; relative error of the accelerations 1.6e-16 against 2.6e-16.
// Four blocks of 128 per SM (128 registers, R = 2): 202 at 166 registers and
// three blocks, 214 at R = 1, 175 at R = 3.
template <int BT, int R, int T, FxMode MODE>
__device__ __forceinline__ void fx_sym_tile(const d4 *__restrict__ posm, int64_t n, int64_t i0,
                                            double eps2, const FxEps &e2,
                                            const d4 *tile, const uint4 *txy, const uint4 *tzm,
                                            const int *tdm, int cnt, const uint64_t (&Xi)[R][3],
                                            const FxMass (&Mi)[R], d4 (&acc)[R], double fs,
                                            double ps, double gs, double qs, d4 *colw) {
  const int tid = threadIdx.x, lane = tid & 31;
  fx96 f[R][3] = {}, pt[R] = {};
#pragma unroll 1
  for (int c = 0; c < T; c += 32) {
    if (c >= cnt) break;
    fx96 g[3] = {}, gp = {};
#pragma unroll 1
    for (int k = 0; k < 32; k++) {
      const int jj = c + ((lane + k) & 31);
      const uint4 a = txy[jj], b = tzm[jj];
      const uint64_t Xj[3] = {((uint64_t)a.y << 32) | a.x, ((uint64_t)a.w << 32) | a.z,
                              ((uint64_t)b.y << 32) | b.x};
      const FxMass Mj{b.w, b.z, MODE == FX_WIDE ? tdm[jj] : 0};
#pragma unroll
      for (int r = 0; r < R; r++) {
        FxPair p;
        if (fx_geometry<true>(Xj, Xi[r], e2, FxRsqrt(), p)) {
          if (MODE == FX_EQUAL) {
            fx_both<true>(p, f[r], pt[r], &g, &gp);
          } else {
            fx_side<true, MODE == FX_WIDE>(p, Mj, f[r], pt[r]);
            fx_side<true, MODE == FX_WIDE>(p, Mi[r], g, gp);
          }
        } else {
          const int64_t i = i0 + r * BT + tid;
          if (jj < cnt && i < n) {
            const d4 pi = posm[i], q = tile[jj];
            const F64Both v =
                pair_f64_both(q.x - pi.x, q.y - pi.y, q.z - pi.z, q.w, pi.w, eps2);
            acc[r].x += v.i.x;
            acc[r].y += v.i.y;
            acc[r].z += v.i.z;
            acc[r].w += v.i.w;
            colw[jj].x += v.j.x;
            colw[jj].y += v.j.y;
            colw[jj].z += v.j.z;
            colw[jj].w += v.j.w;
          }
        }
      }
      __syncwarp();  // the slots of colw change hands
      const int src = (lane + 1) & 31;
#pragma unroll
      for (int q = 0; q < 3; q++) {
        g[q].w0 = __shfl_sync(0xFFFFFFFFu, g[q].w0, src);
        g[q].w1 = __shfl_sync(0xFFFFFFFFu, g[q].w1, src);
        g[q].w2 = __shfl_sync(0xFFFFFFFFu, g[q].w2, src);
      }
      gp.w0 = __shfl_sync(0xFFFFFFFFu, gp.w0, src);
      gp.w1 = __shfl_sync(0xFFFFFFFFu, gp.w1, src);
      gp.w2 = __shfl_sync(0xFFFFFFFFu, gp.w2, src);
    }
    d4 s = colw[c + lane];
    s.x = fx_fold(s.x, g[0], -gs);
    s.y = fx_fold(s.y, g[1], -gs);
    s.z = fx_fold(s.z, g[2], -gs);
    s.w = fx_fold(s.w, gp, qs);
    colw[c + lane] = s;
  }
#pragma unroll
  for (int r = 0; r < R; r++) {
    acc[r].x = fx_fold(acc[r].x, f[r][0], fs);
    acc[r].y = fx_fold(acc[r].y, f[r][1], fs);
    acc[r].z = fx_fold(acc[r].z, f[r][2], fs);
    acc[r].w = fx_fold(acc[r].w, pt[r], ps);
  }
}

template <int BT, int R, int T>
__global__ void __launch_bounds__(BT, 4) k_force_fx_sym(const d4 *__restrict__ posm, int64_t n,
                                                     double eps2, int M, int d0,
                                                     d4 *__restrict__ rows,
                                                     d4 *__restrict__ cols) {
  constexpr int B = BT * R, NW = BT / 32;
  static_assert(T == BT && B % T == 0, "one column sum per thread per tile");
  __shared__ d4 tile[T];
  __shared__ uint4 txy[T], tzm[T];
  __shared__ int tdm[T], snear[NW];
  __shared__ d4 colw[NW][T];
  __shared__ FxBox sbox[NW];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int dl = blockIdx.x / M, I = blockIdx.x % M, d = d0 + dl;
  const int J = (I + d) % M;
  const int64_t i0 = (int64_t)I * B, j0 = (int64_t)J * B;
  d4 *rowo = rows + (int64_t)dl * n;
  d4 *colo = cols + (int64_t)dl * n;
  if (2 * d == M && I >= M / 2) {  // the pair of blocks is the item (I - M/2, I)
    for (int k = tid; k < B; k += BT) {
      if (i0 + k < n) rowo[i0 + k] = d4{0.0, 0.0, 0.0, 0.0};
      if (j0 + k < n) colo[j0 + k] = d4{0.0, 0.0, 0.0, 0.0};
    }
    return;
  }
  // particles beyond n stand at the block's first one, without mass
  d4 acc[R];
  FxBox bi;
  fx_box_init(bi);
#pragma unroll
  for (int r = 0; r < R; r++) {
    const int64_t i = i0 + r * BT + tid;
    fx_box_add(bi, posm[i < n ? i : i0]);
    acc[r] = d4{0.0, 0.0, 0.0, 0.0};
  }
  fx_box_warp(bi);
  if (lane == 0) sbox[warp] = bi;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < NW; w++) fx_box_join(bi, sbox[w]);
  int emi;
  int rangei;
  const bool oki = fx_mass_scale(bi, emi, rangei);
  const double mi0 = posm[i0].w;
  bool equali = i0 + B <= n;
#pragma unroll
  for (int r = 0; r < R; r++) {
    const int64_t i = i0 + r * BT + tid;
    equali = equali && __double_as_longlong(posm[i < n ? i : i0].w) == __double_as_longlong(mi0);
  }
  for (int t0 = 0; t0 < B && j0 + t0 < n; t0 += T) {
    const int64_t jt = j0 + t0;
    const int cnt = (int)min((int64_t)T, n - jt);
    __syncthreads();
    d4 pj = posm[jt + (tid < cnt ? tid : 0)];
    FxBox bj;
    fx_box_init(bj);
    fx_box_add(bj, pj);
    if (tid >= cnt) pj.w = 0.0;
    tile[tid] = pj;
    fx_box_warp(bj);
    if (lane == 0) sbox[warp] = bj;
#pragma unroll
    for (int w = 0; w < NW; w++) colw[w][tid] = d4{0.0, 0.0, 0.0, 0.0};
    __syncthreads();
#pragma unroll
    for (int w = 0; w < NW; w++) fx_box_join(bj, sbox[w]);
    const FxScale sc = fx_scale(bi, bj, eps2);
    const double mj0 = tile[0].w;
    const int range = max(sc.range, rangei);
    const bool wide = range > FX_MASS_NARROW;
    bool fixed = sc.ok && oki && fx_masses_fit(range, sc, bi, bj, eps2), equal = false;
    uint64_t Xi[R][3];
    FxMass Mi[R];
    if (fixed) {
      uint64_t X[3];
      fx_coords(pj, sc.L, X);
      const uint32_t mh = (uint32_t)__double2hiint(pj.w), ml = (uint32_t)__double2loint(pj.w);
      const FxMass m = wide ? fx_mass<true>(mh, ml, sc.em) : fx_mass<false>(mh, ml, sc.em);
      txy[tid] = make_uint4((uint32_t)X[0], (uint32_t)(X[0] >> 32), (uint32_t)X[1],
                            (uint32_t)(X[1] >> 32));
      tzm[tid] = make_uint4((uint32_t)X[2], (uint32_t)(X[2] >> 32), m.l, m.h);
      tdm[tid] = m.dm;
#pragma unroll
      for (int r = 0; r < R; r++) {
        const int64_t i = i0 + r * BT + tid;
        const d4 p = posm[i < n ? i : i0];
        fx_coords(p, sc.L, Xi[r]);
        const double mi = i < n ? p.w : 0.0;
        const uint32_t ih = (uint32_t)__double2hiint(mi), il = (uint32_t)__double2loint(mi);
        Mi[r] = wide ? fx_mass<true>(ih, il, emi) : fx_mass<false>(ih, il, emi);
      }
      const unsigned near = __ballot_sync(0xFFFFFFFFu, fx_near(X, Xi[0]) && (tid ^ 16) < cnt);
      if (lane == 0) snear[warp] = __popc(near);
      equal = __syncthreads_and(equali && tid < cnt &&
                                __double_as_longlong(pj.w) == __double_as_longlong(mj0));
      int n_near = 0;
#pragma unroll
      for (int w = 0; w < NW; w++) n_near += snear[w];
      fixed = n_near < FX_NEAR;
    }
    if (fixed) {
      const FxMode mode = wide ? FX_WIDE : equal ? FX_EQUAL : FX_NARROW;
      const FxEps e2 = fx_eps2(eps2, sc.L);
      const int er = mode == FX_EQUAL ? FX_EQ_EM : sc.em, ec = mode == FX_EQUAL ? FX_EQ_EM : emi;
      double fs = fx_exp2(fx_force_exp(sc.L, er) + 32), ps = fx_exp2(fx_pot_exp(sc.L, er) + 32);
      double gs = fx_exp2(fx_force_exp(sc.L, ec) + 32), qs = fx_exp2(fx_pot_exp(sc.L, ec) + 32);
      if (mode == FX_EQUAL) {
        fs *= mj0;
        ps *= mj0;
        gs *= mi0;
        qs *= mi0;
      }
      if (mode == FX_WIDE)
        fx_sym_tile<BT, R, T, FX_WIDE>(posm, n, i0, eps2, e2, tile, txy, tzm, tdm, cnt, Xi, Mi, acc,
                                       fs, ps, gs, qs, colw[warp]);
      else if (mode == FX_EQUAL)
        fx_sym_tile<BT, R, T, FX_EQUAL>(posm, n, i0, eps2, e2, tile, txy, tzm, tdm, cnt, Xi, Mi, acc,
                                        fs, ps, gs, qs, colw[warp]);
      else
        fx_sym_tile<BT, R, T, FX_NARROW>(posm, n, i0, eps2, e2, tile, txy, tzm, tdm, cnt, Xi, Mi,
                                         acc, fs, ps, gs, qs, colw[warp]);
    } else {  // one i-particle at a time: 92 Gint/s against 85 for both at once (N = 65536)
#pragma unroll
      for (int r = 0; r < R; r++) {
        const int64_t i = i0 + r * BT + tid;
        d4 p[1] = {posm[i < n ? i : i0]}, a[1] = {acc[r]};
        if (i >= n) p[0].w = 0.0;
        const MassSig ms[1] = {mass_sig(p[0].w)};
        f64_sym_tile<1, T, true>(tile, cnt, p, ms, eps2, a, colw[warp]);
        acc[r] = a[0];
      }
    }
    __syncthreads();
    {
      d4 s = colw[0][tid];
#pragma unroll
      for (int w = 1; w < NW; w++) {
        const d4 v = colw[w][tid];
        s.x += v.x;
        s.y += v.y;
        s.z += v.z;
        s.w += v.w;
      }
      if (jt + tid < n) colo[jt + tid] = s;
    }
  }
#pragma unroll
  for (int r = 0; r < R; r++) {
    const int64_t i = i0 + r * BT + tid;
    if (i < n) rowo[i] = acc[r];
  }
}

// acc_rows[i] (+)= rows[0][i] + ... + rows[D-1][i], the same for the columns,
// in diagonal order, in groups of eight (one after another the roundings of a
// sum over hundreds of diagonals would exceed those of the pair sums).
__global__ void k_sym_combine(const d4 *__restrict__ rows, const d4 *__restrict__ cols, int D,
                              int64_t n, d4 *__restrict__ acc_rows, d4 *__restrict__ acc_cols,
                              int first) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    d4 a = first ? d4{0.0, 0.0, 0.0, 0.0} : acc_rows[i];
    d4 b = first ? d4{0.0, 0.0, 0.0, 0.0} : acc_cols[i];
    for (int k0 = 0; k0 < D; k0 += 8) {
      d4 c = {0.0, 0.0, 0.0, 0.0}, e = {0.0, 0.0, 0.0, 0.0};
      for (int k = k0; k < min(k0 + 8, D); k++) {
        const d4 u = rows[(int64_t)k * n + i], v = cols[(int64_t)k * n + i];
        c.x += u.x;
        c.y += u.y;
        c.z += u.z;
        c.w += u.w;
        e.x += v.x;
        e.y += v.y;
        e.z += v.z;
        e.w += v.w;
      }
      a.x += c.x;
      a.y += c.y;
      a.z += c.z;
      a.w += c.w;
      b.x += e.x;
      b.y += e.y;
      b.z += e.z;
      b.w += e.w;
    }
    acc_rows[i] = a;
    acc_cols[i] = b;
  }
}

// ---------------------------------------------------------------- packed binary32 pairs
// Two j-particles per instruction with the packed FP32 instructions of sm_100+
// (one issue slot drives two lanes of FMA-pipe work).  Shared-memory tile
// entry k holds j = 2k and 2k+1 as A = (x0, x1, y0, y1), B = (z0, z1, m0, m1).
// (nx, ny, nz) are the negated i coordinates in both halves.  An odd tail is
// padded with a massless particle at 1e18 (finite r^2, zero contribution).
__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }

// REFINE adds one Newton step to the SFU reciprocal square root (4 more FMA-pipe
// operations).  Both packed kernels run without it: measured against the oracle
// on the disk + halo and uniform-sphere workloads, the step changed the RMS force
// error of the mixed kernel by less than 0.2 % (coordinate rounding and
// accumulation dominate) while costing 26 % of its throughput.
// EQUAL leaves the mass out: the sums are those of 1/r^3 and 1/r, multiplied by
// the tile's one mass when they are folded: 12 lane operations instead of 13.
// Measured at N = 131072: MIXED 2735 Gint/s against 2545, FP32 (R = 2) 2731
// against 2620 (there for masses that are powers of two, in the binary32 kernel).
// Masses up to 1 alone, so that no term is smaller than with the mass, and from
// eps = 2^-40, so that 1/r^3 is finite: systems in other units (masses in kg at
// distances in m) keep the mass in the body, where it brings 1/r^3 into range.
__device__ __forceinline__ bool leave_mass_out(float eps2) { return eps2 >= 0x1p-80f; }
template <bool MASK, bool REFINE, bool EQUAL = false>
__device__ __forceinline__ void body_pair(const float4 &A, const float4 &B, float2 nx, float2 ny,
                                          float2 nz, float2 e2, float2 &ax, float2 &ay,
                                          float2 &az, float2 &pt, bool self0, bool self1) {
  const float2 dx = __fadd2_rn(f2(A.x, A.y), nx);
  const float2 dy = __fadd2_rn(f2(A.z, A.w), ny);
  const float2 dz = __fadd2_rn(f2(B.x, B.y), nz);
  float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __ffma2_rn(dz, dz, e2)));
  float2 m = f2(B.z, B.w);
  if (MASK) {
    if (self0) {
      r2.x = 1.0f;
      m.x = 0.0f;
    }
    if (self1) {
      r2.y = 1.0f;
      m.y = 0.0f;
    }
  }
  float2 y = f2(rsqrt_approx(r2.x), rsqrt_approx(r2.y));
  if (REFINE) {  // y += y (1 - r2 y^2) / 2, as (-y/2) (r2 y^2 - 1) + y
    const float2 e = __ffma2_rn(__fmul2_rn(r2, y), y, f2(-1.0f, -1.0f));
    y = __ffma2_rn(__fmul2_rn(y, f2(-0.5f, -0.5f)), e, y);
  }
  const float2 my = EQUAL ? y : __fmul2_rn(m, y);
  const float2 f = __fmul2_rn(my, __fmul2_rn(y, y));
  ax = __ffma2_rn(dx, f, ax);
  ay = __ffma2_rn(dy, f, ay);
  az = __ffma2_rn(dz, f, az);
  pt = __fadd2_rn(pt, my);
}

// Stage j-particles [jt, jt+cnt) of `src` (float4 x, y, z, m) as pairs.
template <int BT, int T>
__device__ __forceinline__ void load_pairs(const float4 *__restrict__ src, int64_t jt, int cnt,
                                           float4 *tA, float4 *tB) {
  const float4 dummy = make_float4(1e18f, 1e18f, 1e18f, 0.0f);
  for (int k = threadIdx.x; 2 * k < cnt; k += BT) {
    const float4 a = src[jt + 2 * k];
    const float4 b = 2 * k + 1 < cnt ? src[jt + 2 * k + 1] : dummy;
    tA[k] = make_float4(a.x, b.x, a.y, b.y);
    tB[k] = make_float4(a.z, b.z, a.w, b.w);
  }
}

// ---------------------------------------------------------------- float-float (F64E)
// Binary64-class arithmetic on the binary32 pipes: every quantity is an
// unevaluated sum hi + lo of two floats (about 48 significant bits), built
// from the error-free transformations TwoSum (Knuth), Fast2Sum (Dekker,
// |a| >= |b|) and TwoProd via FMA; two j-particles per packed instruction.
__device__ __forceinline__ float2 fsub2(float2 a, float2 b) {
  unsigned long long A, B, D;
  memcpy(&A, &a, 8);
  memcpy(&B, &b, 8);
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(D) : "l"(A), "l"(B));
  float2 d;
  memcpy(&d, &D, 8);
  return d;
}
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }

__device__ __forceinline__ void two_sum2(float2 a, float2 b, float2 &s, float2 &e) {
  s = __fadd2_rn(a, b);
  const float2 bb = fsub2(s, a);
  e = __fadd2_rn(fsub2(a, fsub2(s, bb)), fsub2(b, bb));
}
__device__ __forceinline__ void fast_two_sum2(float2 a, float2 b, float2 &s, float2 &e) {
  s = __fadd2_rn(a, b);
  e = fsub2(b, fsub2(s, a));
}
__device__ __forceinline__ void two_prod2(float2 a, float2 b, float2 &p, float2 &e) {
  p = __fmul2_rn(a, b);
  e = __ffma2_rn(a, b, neg2(p));
}
__device__ __forceinline__ void two_sum1(float a, float b, float &s, float &e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// Exact binary32 -> binary64 by integer moves, for finite values (subnormal ones
// are brought up by 2^24 first: the sums of small masses at large distances are
// made of them).
__device__ __forceinline__ double f2d_exact(float f) {
  const bool sub = fabsf(f) < 0x1p-126f;
  const unsigned b = __float_as_uint(sub ? __fmul_rn(f, 0x1p24f) : f);
  const unsigned mag = b & 0x7fffffffu;
  if (mag == 0) return 0.0;
  const unsigned shift = sub ? 0x38000000u - 0x01800000u : 0x38000000u;
  return __hiloint2double((int)((b & 0x80000000u) | ((mag >> 3) + shift)), (int)(b << 29));
}

// x = h + l in floats: h to nearest, l = the rest rounded to 24 bits.  The
// conversions run on the FP64 pipe (64 cycles a warp each: the three
// coordinates of an i-particle cost as much as 22 mixed pairs), so they are
// integer moves in the range where both halves are normal floats.
__device__ __forceinline__ void split_ff(double x, float &h, float &l) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned ex = (hi >> 20) & 0x7FFu;
  if (ex - 960u < 180u) {  // 2^-63 <= |x| < 2^117
    const unsigned mag = (hi & 0x7FFFFFFFu) - 0x38000000u;
    const unsigned rlo = lo + 0x10000000u;  // round the upper 24 bits to nearest
    const unsigned rhi = mag + (rlo < lo);
    const unsigned sign = hi & 0x80000000u;
    h = __uint_as_float(__funnelshift_l(rlo, rhi, 3) | sign);
    const int rest = (int)(lo << 3) >> 3;  // signed 29 bits below them
    const float scale = __uint_as_float(((ex - 948u) << 23) | sign);  // 2^(ex - 1075)
    l = __int2float_rn(rest) * scale;
  } else {
    h = __double2float_rn(x);
    l = __double2float_rn(x - (double)h);
  }
}
// h + l in binary64 (non-finite halves by conversion, which keeps them so)
__device__ __forceinline__ double join_ff(float h, float l) {
  const bool finite = fabsf(h) < INFINITY && fabsf(l) < INFINITY;
  return finite ? f2d_exact(h) + f2d_exact(l) : (double)h + (double)l;
}

// -(x - c) of an i-particle against a tile's anchor c, exact but for the split:
// the difference is taken in binary64, as the j side's is by the prep kernel, so
// both are off by 2^-49 of their distance from the anchor.  From float-floats of
// x and c each it would be off by 2^-49 of |x|, which is what bounded the
// accelerations: their relative error at N = 65539 (disk and halo) 9.4e-15 so,
// 5.1e-15 here, at the same time (32.5 ms for three evaluations: the FP64 pipe
// is idle otherwise).
__device__ __forceinline__ void ff_shift(const double (&x)[3], const double (&c)[3],
                                         float2 (&nh)[3], float2 (&nl)[3]) {
#pragma unroll
  for (int k = 0; k < 3; k++) {
    float h, l;
    split_ff(c[k] - x[k], h, l);
    nh[k] = f2(h, h);
    nl[k] = f2(l, l);
  }
}

// A pair's geometry: d, y = 1/r and q = 1/r^2 as float-float, for one tile entry
// (j = 2k, 2k+1 as H = (xh0, xh1, yh0, yh1), H2 = (zh0, zh1, mh0, mh1), L, L2 the
// matching low parts) and the negated float-float i coordinates (nxh, ...) in
// both halves.
//   d = (jh - ih) + (jl - il): TwoSum of the high parts, then Fast2Sum with the
//     low ones.  Fast2Sum(s, t) is exact here although |t| may exceed |s| after
//     cancellation: s is then a multiple of the smaller ulp of jh and ih, t is
//     below two of it, so s is a multiple of ulp(t), which is all it needs.
//   y = r2^{-1/2}: SFU seed y0, residual e = 1 - r2 y0^2 in float-float,
//     y = y0 (1 + e/2 + 3 e^2 / 8) = y0 + y0 e (1/2 + 3e/8).
struct FfPair {
  float2 dh[3], dl[3], y0, yl, q, ql, r2h, r2l;
};
template <bool MASK>
__device__ __forceinline__ void ff_geometry(const float4 &H, const float4 &H2, const float4 &L,
                                            const float4 &L2, const float2 (&nh)[3],
                                            const float2 (&nl)[3], float2 e2h, float2 e2l,
                                            bool self0, bool self1, FfPair &g) {
  const float2 jh[3] = {f2(H.x, H.y), f2(H.z, H.w), f2(H2.x, H2.y)};
  const float2 jl[3] = {f2(L.x, L.y), f2(L.z, L.w), f2(L2.x, L2.y)};
  float2 p[3], pe[3], cross;
#pragma unroll
  for (int c = 0; c < 3; c++) {
    float2 s, e;
    two_sum2(jh[c], nh[c], s, e);
    const float2 t = __fadd2_rn(__fadd2_rn(jl[c], nl[c]), e);
    fast_two_sum2(s, t, g.dh[c], g.dl[c]);
    two_prod2(g.dh[c], g.dh[c], p[c], pe[c]);
    cross = c == 0 ? __fmul2_rn(g.dh[c], g.dl[c]) : __ffma2_rn(g.dh[c], g.dl[c], cross);
  }
  // r2 = |d|^2 + eps^2
  float2 s1, e1, s2, e2, s3, e3;
  two_sum2(p[0], p[1], s1, e1);
  two_sum2(s1, p[2], s2, e2);
  two_sum2(s2, e2h, s3, e3);
  const float2 lo =
      __ffma2_rn(cross, f2(2.0f, 2.0f),
                 __fadd2_rn(__fadd2_rn(__fadd2_rn(pe[0], pe[1]), __fadd2_rn(pe[2], e2l)),
                            __fadd2_rn(__fadd2_rn(e1, e2), e3)));
  float2 r2h, r2l;
  fast_two_sum2(s3, lo, r2h, r2l);
  if (MASK) {
    if (self0) r2h.x = 1.0f, r2l.x = 0.0f;
    if (self1) r2h.y = 1.0f, r2l.y = 0.0f;
  }
  const float2 y0 = f2(rsqrt_approx(r2h.x), rsqrt_approx(r2h.y));
  float2 th, tl, u, ue;
  two_prod2(y0, y0, th, tl);
  two_prod2(r2h, th, u, ue);
  const float2 e = fsub2(fsub2(f2(1.0f, 1.0f), u), __ffma2_rn(r2h, tl, __ffma2_rn(r2l, th, ue)));
  g.y0 = y0;
  g.yl = __fmul2_rn(__fmul2_rn(y0, e), __ffma2_rn(e, f2(0.375f, 0.375f), f2(0.5f, 0.5f)));
  g.q = th;
  g.ql = __ffma2_rn(__fadd2_rn(y0, y0), g.yl, tl);
}

// The four terms of one side, d b (three components) and a, with a = m y and
// b = a q; EQUAL: without the mass, the same for both sides.
struct FfTerms {
  float2 h[4], l[4];
};
template <bool EQUAL>
__device__ __forceinline__ void ff_terms(const FfPair &g, float2 mh, float2 ml, FfTerms &t) {
  float2 a = g.y0, al = g.yl, ae, b, be;
  if (!EQUAL) {
    two_prod2(mh, g.y0, a, ae);
    al = __ffma2_rn(mh, g.yl, __ffma2_rn(ml, g.y0, ae));
  }
  two_prod2(a, g.q, b, be);
  const float2 bl = __ffma2_rn(a, g.ql, __ffma2_rn(al, g.q, be));
#pragma unroll
  for (int c = 0; c < 3; c++) {
    float2 ce;
    two_prod2(g.dh[c], b, t.h[c], ce);
    t.l[c] = __ffma2_rn(g.dh[c], bl, __ffma2_rn(g.dl[c], b, ce));
  }
  t.h[3] = a;
  t.l[3] = al;
}

// (h, l) += t: the high parts by TwoSum, the rest into the low part.  The
// potentials, whose error is that of the sum, are renormalised with every term;
// the accelerations, whose error is that of the coordinates, every FF_STEPS steps
// (ff_renorm), which saves 3 of 11 operations a term: their low part grows to a few
// ulps of the high one.  Measured each pair once (48 systems of 1500 to 65539
// particles; largest RMS error over that with every sum renormalised with every
// term): accelerations 1.08, potentials 1.00; potentials every second step 1.08, for
// an FR4 step of 65539 in 32.3 ms against 32.9.  Every sum with every term takes 9 %
// longer than every fourth step.
__device__ __forceinline__ void ff_add(const FfTerms &t, float2 (&h)[4], float2 (&l)[4]) {
#pragma unroll
  for (int c = 0; c < 4; c++) {
    float2 s, es;
    two_sum2(h[c], t.h[c], s, es);
    const float2 lo = __fadd2_rn(l[c], __fadd2_rn(es, t.l[c]));
    if (c < 3) {
      h[c] = s;
      l[c] = lo;
    } else {
      fast_two_sum2(s, lo, h[c], l[c]);
    }
  }
}
__device__ __forceinline__ void ff_renorm(float2 (&h)[4], float2 (&l)[4]) {
#pragma unroll
  for (int c = 0; c < 3; c++) {
    float2 s, e;
    fast_two_sum2(h[c], l[c], s, e);
    h[c] = s;
    l[c] = e;
  }
}

// Stage j-particles [jt, jt+cnt) of `src` (two float4 per particle: hi
// (x, y, z, m), lo (x, y, z, m)) as pairs; odd tail padded as in load_pairs.
template <int BT, int T>
__device__ __forceinline__ void load_pairs_ff(const float4 *__restrict__ src, int64_t jt, int cnt,
                                              float4 *tH, float4 *tH2, float4 *tL, float4 *tL2) {
  const float4 dh = make_float4(1e18f, 1e18f, 1e18f, 0.0f), dl = make_float4(0, 0, 0, 0);
  for (int k = threadIdx.x; 2 * k < cnt; k += BT) {
    const float4 ah = src[2 * (jt + 2 * k)], alo = src[2 * (jt + 2 * k) + 1];
    const bool hb = 2 * k + 1 < cnt;
    const float4 bh = hb ? src[2 * (jt + 2 * k + 1)] : dh;
    const float4 blo = hb ? src[2 * (jt + 2 * k + 1) + 1] : dl;
    tH[k] = make_float4(ah.x, bh.x, ah.y, bh.y);
    tH2[k] = make_float4(ah.z, bh.z, ah.w, bh.w);
    tL[k] = make_float4(alo.x, blo.x, alo.y, blo.y);
    tL2[k] = make_float4(alo.z, blo.z, alo.w, blo.w);
  }
}

// Steps between renormalisations of the acceleration sums.
constexpr int FF_STEPS = 4;

template <int R, bool EQUAL>
__device__ __forceinline__ void ff_tile(const float4 *tH, const float4 *tH2, const float4 *tL,
                                        const float4 *tL2, int k0, int k1,
                                        const float2 (&nh)[R][3], const float2 (&nl)[R][3],
                                        float2 e2h, float2 e2l, float2 (&ah)[R][4],
                                        float2 (&al)[R][4]) {
#pragma unroll 1
  for (int k = k0; k < k1; k += FF_STEPS) {
#pragma unroll
    for (int q = 0; q < FF_STEPS; q++) {
      const float4 H = tH[k + q], H2 = tH2[k + q], L = tL[k + q], L2 = tL2[k + q];
#pragma unroll
      for (int r = 0; r < R; r++) {
        FfPair g;
        FfTerms t;
        ff_geometry<false>(H, H2, L, L2, nh[r], nl[r], e2h, e2l, false, false, g);
        ff_terms<EQUAL>(g, f2(H2.z, H2.w), f2(L2.z, L2.w), t);
        ff_add(t, ah[r], al[r]);
        if (q == FF_STEPS - 1) ff_renorm(ah[r], al[r]);
      }
    }
  }
}

// F64E force: i coordinates re-centred on each j-tile's anchor in float-float
// (from the particle's own float-float and the anchor's), pair terms and
// per-tile partial sums in float-float, folded into binary64 once per tile.
template <int BT, int R, int T, int IW, class W>
__global__ void __launch_bounds__(BT) k_force_f64e(const d4 *__restrict__ posm,
                                                   const float4 *__restrict__ jff,
                                                   const float4 *__restrict__ anchor, W work,
                                                   d4 *__restrict__ part) {
  chain_begin();
  constexpr int IT = BT / IW;
  __shared__ float4 tH[T / 2], tH2[T / 2], tL[T / 2], tL2[T / 2];
  __shared__ d4 red[IW > 1 ? BT : 1];
  for (int64_t uk = work.first(); uk < work.count(); uk += work.stride()) {
    const Unit u = work.get(uk);
    const int tid = threadIdx.x;
    // i-thread, share of the j-tile
    const int it = IW == 1 ? tid : tid % IT, jw = IW == 1 ? 0 : tid / IT;
    const int64_t j1 = u.j0 + u.nj;
    const float e2hs = (float)u.eps2;
    const float e2ls = (float)(u.eps2 - (double)e2hs);
    const float2 e2h = f2(e2hs, e2hs), e2l = f2(e2ls, e2ls);
    const bool no_mass = leave_mass_out(e2hs);
    double x[R][3], acc[R][4];
#pragma unroll
    for (int r = 0; r < R; r++) {
      const int li = r * IT + it;
      const d4 p = posm[u.i0 + (li < u.ni ? li : 0)];
      x[r][0] = p.x;
      x[r][1] = p.y;
      x[r][2] = p.z;
#pragma unroll
      for (int c = 0; c < 4; c++) acc[r][c] = 0.0;
    }
    for (int64_t jt = u.j0; jt < j1; jt += T) {
      const int cnt = (int)min((int64_t)T, j1 - jt);
      __syncthreads();
      load_pairs_ff<BT, T>(jff, jt, cnt, tH, tH2, tL, tL2);
      __syncthreads();
      const int64_t tt = u.anchor + (jt - u.j0) / T;
      const float4 ch = anchor[2 * tt], cl = anchor[2 * tt + 1];
      const double ct[3] = {join_ff(ch.x, cl.x), join_ff(ch.y, cl.y), join_ff(ch.z, cl.z)};
      float2 nh[R][3], nl[R][3], ah[R][4], al[R][4];
#pragma unroll
      for (int r = 0; r < R; r++) {
        ff_shift(x[r], ct, nh[r], nl[r]);
#pragma unroll
        for (int c = 0; c < 4; c++) ah[r][c] = al[r][c] = f2(0.0f, 0.0f);
      }
      const int np = (cnt + 1) / 2;
      const int k0 = np * jw / IW, k1 = np * (jw + 1) / IW;
      const bool diag = (jt < u.i0 + u.ni) && (jt + cnt > u.i0);
      const bool full = cnt == T && !diag;
      const bool equal = full && ch.w != 0.0f && no_mass;
      if (full) {  // k1 - k0 is a multiple of FF_STEPS
        if (equal)
          ff_tile<R, true>(tH, tH2, tL, tL2, k0, k1, nh, nl, e2h, e2l, ah, al);
        else
          ff_tile<R, false>(tH, tH2, tL, tL2, k0, k1, nh, nl, e2h, e2l, ah, al);
      } else {
        for (int k = k0; k < k1; k++) {
          const float4 H = tH[k], H2 = tH2[k], L = tL[k], L2 = tL2[k];
          const int64_t j = jt + 2 * k;
#pragma unroll
          for (int r = 0; r < R; r++) {
            const int64_t i = u.i0 + r * IT + it;
            const bool self0 = diag && j == i, self1 = diag && j + 1 == i;
            FfPair g;
            FfTerms t;
            ff_geometry<true>(H, H2, L, L2, nh[r], nl[r], e2h, e2l, self0, self1, g);
            ff_terms<false>(g, f2(self0 ? 0.0f : H2.z, self1 ? 0.0f : H2.w),
                            f2(self0 ? 0.0f : L2.z, self1 ? 0.0f : L2.w), t);
            ff_add(t, ah[r], al[r]);
            ff_renorm(ah[r], al[r]);
          }
        }
      }
      const double m = equal ? posm[jt].w : 1.0;
      // fold the tile: even + odd lanes in float-float, then into binary64
#pragma unroll
      for (int r = 0; r < R; r++)
#pragma unroll
        for (int c = 0; c < 4; c++) {
          float s, e;
          two_sum1(ah[r][c].x, ah[r][c].y, s, e);
          const float l = __fadd_rn(__fadd_rn(al[r][c].x, al[r][c].y), e);
          acc[r][c] = fma(f2d_exact(s) + f2d_exact(l), m, acc[r][c]);
        }
    }
#pragma unroll
    for (int r = 0; r < R; r++) {
      const int li = r * IT + it;
      const d4 v = {acc[r][0], acc[r][1], acc[r][2], acc[r][3]};
      store_shares<IW>(part, work.get(uk), li, v, red, it, IT, jw);
    }
  }
}

// ---------------------------------------------------------------- float-float, each pair once
// The F64E pair evaluated once for both particles (Newton's third law): the
// geometry (d, |d|^2 + eps^2, 1/r, 1/r^2) is shared; the i side gets the terms
// with m_j, the j side those with m_i and -d (the sign is applied to the column
// sums at the end).  Equal masses in both blocks share the terms as well.  Two
// j-particles per packed instruction (one tile entry).
__device__ __forceinline__ float2 shfl2(float2 v, int src) {
  return f2(__shfl_sync(0xFFFFFFFFu, v.x, src), __shfl_sync(0xFFFFFFFFu, v.y, src));
}

// The column block's NE entries against the R i-particles of each thread: row
// sums in (ah, al), the warp's column sums into colw (binary64).
template <int R, int NE, int T, bool EQUAL>
__device__ __forceinline__ void ff_sym_tile(const float4 *tH, const float4 *tH2, const float4 *tL,
                                            const float4 *tL2, const float2 (&nh)[R][3],
                                            const float2 (&nl)[R][3], const float2 (&mh)[R],
                                            const float2 (&ml)[R], float2 e2h, float2 e2l,
                                            float2 (&ah)[R][4], float2 (&al)[R][4],
                                            double (*colw)[T]) {
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  for (int c0 = 0; c0 < NE; c0 += 32) {
    float2 gh[4], gl[4];
#pragma unroll
    for (int c = 0; c < 4; c++) gh[c] = gl[c] = f2(0.0f, 0.0f);
#pragma unroll 1
    for (int k = 0; k < 32; k += FF_STEPS) {
#pragma unroll
      for (int s = 0; s < FF_STEPS; s++) {
        const int ent = c0 + ((lane + k + s) & 31);
        const float4 H = tH[ent], H2 = tH2[ent], L = tL[ent], L2 = tL2[ent];
#pragma unroll
        for (int r = 0; r < R; r++) {
          FfPair g;
          FfTerms t;
          ff_geometry<false>(H, H2, L, L2, nh[r], nl[r], e2h, e2l, false, false, g);
          ff_terms<EQUAL>(g, f2(H2.z, H2.w), f2(L2.z, L2.w), t);
          ff_add(t, ah[r], al[r]);
          if (!EQUAL) ff_terms<false>(g, mh[r], ml[r], t);
          ff_add(t, gh, gl);
        }
        if (s == FF_STEPS - 1) {
          ff_renorm(gh, gl);
#pragma unroll
          for (int r = 0; r < R; r++) ff_renorm(ah[r], al[r]);
        }
        const int src = (lane + 1) & 31;
#pragma unroll
        for (int c = 0; c < 4; c++) {
          gh[c] = shfl2(gh[c], src);
          gl[c] = shfl2(gl[c], src);
        }
      }
    }
    // lane holds entry c0 + lane (j = 2 (c0 + lane) and 2 (c0 + lane) + 1)
#pragma unroll
    for (int c = 0; c < 4; c++) {
      colw[c][2 * (c0 + lane)] = f2d_exact(gh[c].x) + f2d_exact(gl[c].x);
      colw[c][2 * (c0 + lane) + 1] = f2d_exact(gh[c].y) + f2d_exact(gl[c].y);
    }
  }
}

// Work item (d, I) of the block-diagonal schedule of k_force_f64_sym with
// blocks of B = BT*R = T particles: one F64E tile (one anchor) per column
// block.  Row sums into rows[dl], column sums into cols[dl], binary64.
template <int BT, int R, int T>
__global__ void __launch_bounds__(BT) k_force_f64e_sym(const d4 *__restrict__ posm,
                                                       const float4 *__restrict__ jff,
                                                       const float4 *__restrict__ anchor,
                                                       int64_t n, double eps2, int M, int d0,
                                                       d4 *__restrict__ rows,
                                                       d4 *__restrict__ cols) {
  constexpr int B = BT * R, NW = BT / 32, NE = T / 2;  // NE tile entries of 2 j
  static_assert(B == T && NE == BT, "one tile per block, one column entry per thread");
  __shared__ float4 tH[NE], tH2[NE], tL[NE], tL2[NE];
  __shared__ double colw[NW][4][T];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int dl = blockIdx.x / M, I = blockIdx.x % M, d = d0 + dl;
  const int J = (I + d) % M;
  const int64_t i0 = (int64_t)I * B, j0 = (int64_t)J * B;
  d4 *rowo = rows + (int64_t)dl * n;
  d4 *colo = cols + (int64_t)dl * n;
  if (2 * d == M && I >= M / 2) {
    for (int k = tid; k < B; k += BT) {
      if (i0 + k < n) rowo[i0 + k] = d4{0.0, 0.0, 0.0, 0.0};
      if (j0 + k < n) colo[j0 + k] = d4{0.0, 0.0, 0.0, 0.0};
    }
    return;
  }
  const float e2hs = (float)eps2;
  const float e2ls = (float)(eps2 - (double)e2hs);
  const float2 e2h = f2(e2hs, e2hs), e2l = f2(e2ls, e2ls);
  {  // entry tid = j0 + 2 tid, j0 + 2 tid + 1; beyond n massless at 1e18 from the anchor
    const int64_t ja = j0 + 2 * tid, jb = ja + 1;
    const float4 dh = make_float4(1e18f, 1e18f, 1e18f, 0.0f), dz = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    const float4 ah_ = ja < n ? jff[2 * ja] : dh, alo = ja < n ? jff[2 * ja + 1] : dz;
    const float4 bh_ = jb < n ? jff[2 * jb] : dh, blo = jb < n ? jff[2 * jb + 1] : dz;
    tH[tid] = make_float4(ah_.x, bh_.x, ah_.y, bh_.y);
    tH2[tid] = make_float4(ah_.z, bh_.z, ah_.w, bh_.w);
    tL[tid] = make_float4(alo.x, blo.x, alo.y, blo.y);
    tL2[tid] = make_float4(alo.z, blo.z, alo.w, blo.w);
  }
  const float4 ch = anchor[2 * J], cl = anchor[2 * J + 1];
  const double ct[3] = {join_ff(ch.x, cl.x), join_ff(ch.y, cl.y), join_ff(ch.z, cl.z)};
  float2 nh[R][3], nl[R][3], ah[R][4], al[R][4], mh[R], ml[R];
#pragma unroll
  for (int r = 0; r < R; r++) {
    const int64_t i = i0 + r * BT + tid;
    // beyond n: massless, 1e18 from the anchor (finite r^2, zero contribution)
    const d4 pi = i < n ? posm[i] : d4{0.0, 0.0, 0.0, 0.0};
    const double x[3] = {pi.x, pi.y, pi.z};
    ff_shift(x, ct, nh[r], nl[r]);
    if (i >= n)
#pragma unroll
      for (int c = 0; c < 3; c++) nh[r][c] = f2(-1e18f, -1e18f), nl[r][c] = f2(0.0f, 0.0f);
    float m_h, m_l;
    split_ff(pi.w, m_h, m_l);
    mh[r] = f2(m_h, m_h);
    ml[r] = f2(m_l, m_l);
#pragma unroll
    for (int c = 0; c < 4; c++) ah[r][c] = al[r][c] = f2(0.0f, 0.0f);
  }
  __syncthreads();
  const bool equal = ch.w != 0.0f && anchor[2 * I].w != 0.0f && leave_mass_out(e2hs);
  if (equal)
    ff_sym_tile<R, NE, T, true>(tH, tH2, tL, tL2, nh, nl, mh, ml, e2h, e2l, ah, al, colw[warp]);
  else
    ff_sym_tile<R, NE, T, false>(tH, tH2, tL, tL2, nh, nl, mh, ml, e2h, e2l, ah, al, colw[warp]);
  __syncthreads();
  const double mj = equal ? posm[j0].w : 1.0, mi = equal ? posm[i0].w : 1.0;
  for (int k = tid; k < T; k += BT) {
    double v[4];
#pragma unroll
    for (int c = 0; c < 4; c++) {
      v[c] = colw[0][c][k];
#pragma unroll
      for (int w = 1; w < NW; w++) v[c] += colw[w][c][k];
    }
    if (j0 + k < n) colo[j0 + k] = d4{-v[0] * mi, -v[1] * mi, -v[2] * mi, v[3] * mi};
  }
  // rows: fold even + odd lanes in float-float, then into binary64
#pragma unroll
  for (int r = 0; r < R; r++) {
    const int64_t i = i0 + r * BT + tid;
    double v[4];
#pragma unroll
    for (int c = 0; c < 4; c++) {
      float s, e;
      two_sum1(ah[r][c].x, ah[r][c].y, s, e);
      const float l = __fadd_rn(__fadd_rn(al[r][c].x, al[r][c].y), e);
      v[c] = (f2d_exact(s) + f2d_exact(l)) * mj;
    }
    if (i < n) rowo[i] = d4{v[0], v[1], v[2], v[3]};
  }
}

// ---------------------------------------------------------------- mixed
// fpos[j] = (x_j - c_t, y_j - c_t, z_j - c_t, m_j) in binary32, c_t the anchor of
// j's tile; anchor[2t] = float hi part of c_t, anchor[2t+1] = float lo part;
// anchor[2t].w = the mass of a full tile of equal masses up to 1, or 0.
template <int BT, int R, int T, class W>
__global__ void __launch_bounds__(BT) k_force_mixed(const d4 *__restrict__ posm,
                                                    const float4 *__restrict__ fpos,
                                                    const float4 *__restrict__ anchor, W work,
                                                    d4 *__restrict__ part) {
  chain_begin();
  __shared__ float4 tA[T / 2], tB[T / 2];
  for (int64_t uk = work.first(); uk < work.count(); uk += work.stride()) {
    const Unit u = work.get(uk);
    const int tid = threadIdx.x;
    const int64_t j1 = u.j0 + u.nj;
    const float2 e2 = f2((float)u.eps2, (float)u.eps2);
    const bool no_mass = leave_mass_out(e2.x);
    float xh[R], yh[R], zh[R], xl[R], yl[R], zl[R];
    float axh[R], axl[R], ayh[R], ayl[R], azh[R], azl[R], pth[R], ptl[R];
#pragma unroll
    for (int r = 0; r < R; r++) {
      const int li = r * BT + tid;
      const d4 p = posm[u.i0 + (li < u.ni ? li : 0)];
      split_ff(p.x, xh[r], xl[r]);
      split_ff(p.y, yh[r], yl[r]);
      split_ff(p.z, zh[r], zl[r]);
      axh[r] = axl[r] = ayh[r] = ayl[r] = azh[r] = azl[r] = pth[r] = ptl[r] = 0.0f;
    }
    for (int64_t jt = u.j0; jt < j1; jt += T) {
      const int cnt = (int)min((int64_t)T, j1 - jt);
      __syncthreads();
      load_pairs<BT, T>(fpos, jt, cnt, tA, tB);
      __syncthreads();
      const int64_t tt = u.anchor + (jt - u.j0) / T;
      const float4 ch = anchor[2 * tt], cl = anchor[2 * tt + 1];
      float2 nx[R], ny[R], nz[R], sx[R], sy[R], sz[R], sp[R];
#pragma unroll
      for (int r = 0; r < R; r++) {
        // x_i - c_t rounded once: TwoSum of the high parts, then the low parts
        float x, y, z, s, e;
        two_sum1(xh[r], -ch.x, s, e);
        x = __fadd_rn(s, __fadd_rn(__fsub_rn(xl[r], cl.x), e));
        two_sum1(yh[r], -ch.y, s, e);
        y = __fadd_rn(s, __fadd_rn(__fsub_rn(yl[r], cl.y), e));
        two_sum1(zh[r], -ch.z, s, e);
        z = __fadd_rn(s, __fadd_rn(__fsub_rn(zl[r], cl.z), e));
        nx[r] = f2(-x, -x);
        ny[r] = f2(-y, -y);
        nz[r] = f2(-z, -z);
        sx[r] = sy[r] = sz[r] = sp[r] = f2(0.0f, 0.0f);
      }
      const int np = (cnt + 1) / 2;
      const bool diag = (jt < u.i0 + u.ni) && (jt + cnt > u.i0);
      const bool equal = ch.w != 0.0f && no_mass;
      // R = 1 is the small-N shape, of few warps per SM: eight pair steps in flight.
      // A KDK step at unroll 2, 4, 8 (us): N = 2048 28.2, 27.9, 26.3; 16387 153.0,
      // 152.6, 143.9; 32768 471, 471, 463.  R = 2 at unroll 2, 4: 2500, 2517 Gint/s
      // at N = 131072.
      if (cnt == T && !diag && equal) {
#pragma unroll(R == 1 ? 8 : 4)
        for (int k = 0; k < T / 2; k++) {
          const float4 A = tA[k], B = tB[k];
#pragma unroll
          for (int r = 0; r < R; r++)
            body_pair<false, false, true>(A, B, nx[r], ny[r], nz[r], e2, sx[r], sy[r], sz[r],
                                         sp[r], false, false);
        }
      } else if (cnt == T && !diag) {
#pragma unroll(R == 1 ? 8 : 4)
        for (int k = 0; k < T / 2; k++) {
          const float4 A = tA[k], B = tB[k];
#pragma unroll
          for (int r = 0; r < R; r++)
            body_pair<false, false>(A, B, nx[r], ny[r], nz[r], e2, sx[r], sy[r], sz[r], sp[r],
                                   false, false);
        }
      } else {
#pragma unroll(R == 1 ? 8 : 1)
        for (int k = 0; k < np; k++) {
          const float4 A = tA[k], B = tB[k];
          const int64_t j = jt + 2 * k;
#pragma unroll
          for (int r = 0; r < R; r++) {
            const int64_t i = u.i0 + r * BT + tid;
            body_pair<true, false>(A, B, nx[r], ny[r], nz[r], e2, sx[r], sy[r], sz[r], sp[r],
                                  j == i, j + 1 == i);
          }
        }
      }
      const float m = cnt == T && !diag && equal ? ch.w : 1.0f;
#pragma unroll
      for (int r = 0; r < R; r++) {
        fold_tile(axh[r], axl[r], __fadd_rn(sx[r].x, sx[r].y), m);
        fold_tile(ayh[r], ayl[r], __fadd_rn(sy[r].x, sy[r].y), m);
        fold_tile(azh[r], azl[r], __fadd_rn(sz[r].x, sz[r].y), m);
        fold_tile(pth[r], ptl[r], __fadd_rn(sp[r].x, sp[r].y), m);
      }
    }
#pragma unroll
    for (int r = 0; r < R; r++) {
      const int li = r * BT + tid;
      const Unit w = work.get(uk);  // again: not kept in registers over the pair loop
      if (li >= w.w0 && li < min(w.ni, w.w1))
        part[w.out + li] = d4{join_ff(axh[r], axl[r]), join_ff(ayh[r], ayl[r]),
                              join_ff(azh[r], azl[r]), join_ff(pth[r], ptl[r])};
    }
  }
}

// One block per j-tile: anchor c = the per-coordinate median of the tile's
// positions (binary64), fpos[j] = float(r_j - c), float(m_j); anchor[2t],
// anchor[2t+1] = float-float c.  The median follows the bulk of the tile: for
// a spatially compact tile it lies inside it, and for an unsorted tile it
// stays near the centre of the particle distribution even when a few members
// sit far out in a halo (a bounding-box centre would be pulled out there and
// cost every coordinate relative to it several digits).  It is found with a
// bitonic sort of the high words as integers, the three coordinates together
// (tile = block = 256; lane shuffles below strides of 32), and a count among
// the members that share the median's high word.  6.5 us at N = 2048; sorting
// the binary64 values in shared memory, one coordinate after the other, took
// about 15: its comparisons ran on the FP64 pipe and every stage had a barrier.
struct DensePrep {
  int64_t n;
  int tile;
  __device__ __forceinline__ PrepUnit get() const {
    PrepUnit u;
    u.anchor = blockIdx.x;
    u.j0 = (int64_t)blockIdx.x * tile;
    u.cnt = (int)min((int64_t)tile, n - u.j0);
    u.pad = 0;
    return u;
  }
};
struct TablePrep {
  const PrepUnit *units;
  __device__ __forceinline__ PrepUnit get() const { return units[blockIdx.x]; }
};

// FF = true (F64E): the re-centred coordinates and the mass are written as
// float-float, two float4 per particle (hi x, y, z, m; lo x, y, z, m).
template <int BT, class W, bool FF>
__global__ void __launch_bounds__(BT) k_mixed_prep(const d4 *__restrict__ posm, W work,
                                                   float4 *__restrict__ fpos,
                                                   float4 *__restrict__ anchor) {
  chain_begin();
  static_assert((BT & (BT - 1)) == 0, "bitonic sort needs a power-of-two block");
  __shared__ int v[2][3][BT];
  __shared__ int mid[3], first[3], same[3];
  __shared__ unsigned low[3][BT];
  __shared__ double med[3];
  const PrepUnit pu = work.get();
  const int64_t t = pu.anchor;
  const int64_t j0 = pu.j0;
  const int cnt = pu.cnt;
  const int tid = threadIdx.x;
  d4 p = {0, 0, 0, 0};
  if (tid < cnt) p = posm[j0 + tid];
  int key[3] = {0x7FFFFFFF, 0x7FFFFFFF, 0x7FFFFFFF};
  if (tid < cnt) {
    key[0] = fx_key(__double2hiint(p.x));
    key[1] = fx_key(__double2hiint(p.y));
    key[2] = fx_key(__double2hiint(p.z));
  }
  int buf = 0;
  for (int k = 2; k <= BT; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      const bool low = ((tid & j) == 0) == ((tid & k) == 0);  // keeps the smaller one
      if (j >= 32) {
#pragma unroll
        for (int q = 0; q < 3; q++) v[buf][q][tid] = key[q];
        __syncthreads();
      }
#pragma unroll
      for (int q = 0; q < 3; q++) {
        const int o = j >= 32 ? v[buf][q][tid ^ j] : __shfl_xor_sync(0xFFFFFFFFu, key[q], j);
        key[q] = low ? min(key[q], o) : max(key[q], o);
      }
      if (j >= 32) buf ^= 1;  // the next exchange writes the other buffer
    }
  }
  // key[q] is now the tid-th smallest high word; of the members with the
  // median's, in any order, the one of rank (cnt - 1) / 2 - first is the median
  const int rank = (cnt - 1) / 2;
  if (tid == rank) {
#pragma unroll
    for (int q = 0; q < 3; q++) {
      mid[q] = key[q];
      first[q] = rank;
      same[q] = 0;
    }
  }
  __syncthreads();
  const double x[3] = {p.x, p.y, p.z};
  bool member[3];
  unsigned lo[3];
#pragma unroll
  for (int q = 0; q < 3; q++) {
    if (tid < rank && key[q] == mid[q]) atomicMin(&first[q], tid);
    member[q] = tid < cnt && fx_key(__double2hiint(x[q])) == mid[q];
    // the low words ordered as the values (reversed below zero)
    lo[q] = (unsigned)__double2loint(x[q]) ^ (mid[q] < 0 ? 0xFFFFFFFFu : 0u);
    if (member[q]) low[q][atomicAdd(&same[q], 1)] = lo[q];
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 3; q++) {
    if (member[q]) {  // almost always one member
      const int want = rank - first[q];
      int below = 0, equal = 0;
      for (int o = 0; o < same[q]; o++) {
        below += low[q][o] < lo[q];
        equal += low[q][o] == lo[q];
      }
      if (below <= want && want < below + equal) med[q] = x[q];  // equal values write alike
    }
  }
  __syncthreads();
  double c[3] = {med[0], med[1], med[2]};
  if (FF)  // as the force kernels will read it back, to the last bit
#pragma unroll
    for (int q = 0; q < 3; q++) {
      float h, l;
      split_ff(c[q], h, l);
      c[q] = join_ff(h, l);
    }
  if (tid < cnt) {
    const double dx = p.x - c[0], dy = p.y - c[1], dz = p.z - c[2];
    const float hx = __double2float_rn(dx), hy = __double2float_rn(dy), hz = __double2float_rn(dz),
                hm = __double2float_rn(p.w);
    if (FF) {
      fpos[2 * (j0 + tid)] = make_float4(hx, hy, hz, hm);
      fpos[2 * (j0 + tid) + 1] =
          make_float4(__double2float_rn(dx - (double)hx), __double2float_rn(dy - (double)hy),
                      __double2float_rn(dz - (double)hz), __double2float_rn(p.w - (double)hm));
    } else {
      fpos[j0 + tid] = make_float4(hx, hy, hz, hm);
    }
  }
  const bool equal = __syncthreads_and(
      tid < cnt && __double_as_longlong(p.w) == __double_as_longlong(posm[j0].w));
  if (tid == 0) {
    const float hx = __double2float_rn(c[0]), hy = __double2float_rn(c[1]),
                hz = __double2float_rn(c[2]);
    anchor[2 * t] = make_float4(hx, hy, hz, equal && p.w <= 1.0 ? __double2float_rn(p.w) : 0.0f);
    anchor[2 * t + 1] = make_float4(__double2float_rn(c[0] - (double)hx),
                                    __double2float_rn(c[1] - (double)hy),
                                    __double2float_rn(c[2] - (double)hz), 0.0f);
  }
}

// ---------------------------------------------------------------- binary32 (paper's SP)
// Tiles of equal masses run without the mass when it is a power of two (masses
// 1 / 2^k, as of equal-mass systems of 2^k particles): the sums are then held in
// units of it, which changes no bit of them.  Other masses keep the product in
// the body: sums in another rounding would move single precision positions, and
// with them close pairs at a small softening, by as much as its whole error.
// The range of masses and the softening keep the terms in units of the mass
// finite (1/r <= 2^20) and not smaller than with it (m <= 1).  The sums so far,
// which tiles of other masses may have made large, are taken into those units
// only where that leaves every one of the warp's below 2^100; a tile's own terms
// add less than 2^50.  Otherwise the tile keeps its mass in the body, which gives
// the same bits.  R = 1, the shape of small systems, keeps it in every tile: there
// the operation saved does not show (N = 8192: 69 us either way) and the code
// around it costs 2 to 4 %.
__device__ __forceinline__ bool f32_unit_mass(float m, float eps2) {
  return (__float_as_uint(m) & 0x807FFFFFu) == 0 && m <= 1.0f && m >= 0x1p-40f && eps2 >= 0x1p-40f;
}
template <int BT, int R, int T, class W>
__global__ void __launch_bounds__(BT) k_force_f32(const float4 *__restrict__ posm, W work,
                                                  float4 *__restrict__ part) {
  chain_begin();
  constexpr bool UNITS = R > 1;
  __shared__ float4 tA[T / 2], tB[T / 2];
  for (int64_t uk = work.first(); uk < work.count(); uk += work.stride()) {
    const Unit u = work.get(uk);
    const int tid = threadIdx.x;
    const int64_t j1 = u.j0 + u.nj;
    const float2 e2 = f2((float)u.eps2, (float)u.eps2);
    float2 nx[R], ny[R], nz[R], ax[R], ay[R], az[R], pt[R];
    float unit = 1.0f;  // of the sums, the same for a warp
    auto fit_units_of = [&](float m) {
      if (m >= unit) return true;
      float top = 0.0f;
#pragma unroll
      for (int r = 0; r < R; r++) {
        const float2 v[4] = {ax[r], ay[r], az[r], pt[r]};
#pragma unroll
        for (int c = 0; c < 4; c++) top = fmaxf(top, fmaxf(fabsf(v[c].x), fabsf(v[c].y)));
      }
      return __all_sync(0xFFFFFFFFu, top * (unit / m) < 0x1p100f) != 0;
    };
    auto in_units_of = [&](float m) {
      if (m == unit) return;
      const float f = unit / m;  // of powers of two: exact
      const float2 f_2 = f2(f, f);
#pragma unroll
      for (int r = 0; r < R; r++) {
        ax[r] = __fmul2_rn(ax[r], f_2);
        ay[r] = __fmul2_rn(ay[r], f_2);
        az[r] = __fmul2_rn(az[r], f_2);
        pt[r] = __fmul2_rn(pt[r], f_2);
      }
      unit = m;
    };
#pragma unroll
    for (int r = 0; r < R; r++) {
      const int li = r * BT + tid;
      const float4 p = posm[u.i0 + (li < u.ni ? li : 0)];
      nx[r] = f2(-p.x, -p.x);
      ny[r] = f2(-p.y, -p.y);
      nz[r] = f2(-p.z, -p.z);
      ax[r] = ay[r] = az[r] = pt[r] = f2(0.0f, 0.0f);
    }
    for (int64_t jt = u.j0; jt < j1; jt += T) {
      const int cnt = (int)min((int64_t)T, j1 - jt);
      __syncthreads();
      load_pairs<BT, T>(posm, jt, cnt, tA, tB);
      float m = 0.0f;
      bool equal = false;
      if (UNITS) {
        m = posm[jt].w;
        equal = __syncthreads_and(tid < cnt && posm[jt + min(tid, cnt - 1)].w == m) &&
                f32_unit_mass(m, e2.x);
      } else {
        __syncthreads();
      }
      const int np = (cnt + 1) / 2;
      const bool diag = (jt < u.i0 + u.ni) && (jt + cnt > u.i0);
      if (UNITS && cnt == T && !diag && equal && fit_units_of(m)) {
        in_units_of(m);
#pragma unroll 2
        for (int k = 0; k < T / 2; k++) {
          const float4 A = tA[k], B = tB[k];
#pragma unroll
          for (int r = 0; r < R; r++)
            body_pair<false, false, true>(A, B, nx[r], ny[r], nz[r], e2, ax[r], ay[r], az[r],
                                         pt[r], false, false);
        }
        continue;
      }
      in_units_of(1.0f);
      if (cnt == T && !diag) {
#pragma unroll 2
        for (int k = 0; k < T / 2; k++) {
          const float4 A = tA[k], B = tB[k];
#pragma unroll
          for (int r = 0; r < R; r++)
            body_pair<false, false>(A, B, nx[r], ny[r], nz[r], e2, ax[r], ay[r], az[r], pt[r],
                                    false, false);
        }
      } else {
        for (int k = 0; k < np; k++) {
          const float4 A = tA[k], B = tB[k];
          const int64_t j = jt + 2 * k;
#pragma unroll
          for (int r = 0; r < R; r++) {
            const int64_t i = u.i0 + r * BT + tid;
            body_pair<true, false>(A, B, nx[r], ny[r], nz[r], e2, ax[r], ay[r], az[r], pt[r],
                                   j == i, j + 1 == i);
          }
        }
      }
    }
    in_units_of(1.0f);
#pragma unroll
    for (int r = 0; r < R; r++) {
      const int li = r * BT + tid;
      const Unit w = work.get(uk);  // again: not kept in registers over the pair loop
      if (li >= w.w0 && li < min(w.ni, w.w1))
        part[w.out + li] = make_float4(__fadd_rn(ax[r].x, ax[r].y), __fadd_rn(ay[r].x, ay[r].y),
                                       __fadd_rn(az[r].x, az[r].y), __fadd_rn(pt[r].x, pt[r].y));
    }
  }
}

// ---------------------------------------------------------------- dispatch
// Fixed block and tile sizes per arithmetic; R is chosen at run time.
constexpr int BT_F64 = 128, T_F64 = 128;
constexpr int BT_F32 = 256, T_F32 = 256;
constexpr int BT_FF = 128, T_FF = 256;

int force_block_threads(int mode) {
  return mode == NBODY_FP64 ? BT_F64 : mode == NBODY_F64E ? BT_FF : BT_F32;
}
// Warps of a block that share i-particles at small n: all of them.
constexpr int IW_F64 = BT_F64 / 32, IW_FF = BT_FF / 32;
int force_split(int mode) {
  return mode == NBODY_FP64 ? IW_F64 : mode == NBODY_F64E ? IW_FF : 1;
}
// Measured on GB300 (force kernel, split against one i-particle per thread, us):
// FP64 N = 1000 23 / 57, 3000 88 / 111, 4096 147 / 162, 6000 299 / 308; F64E 1000
// 14 / 35, 4096 88 / 100, 6000 174 / 187.  MIXED is not split: a pair costs it so
// little that what a thread does once per i-particle weighs more (4096: 39 / 18);
// FP32 neither: its sums keep their order (see above).
int64_t force_split_max_n(int mode) {
  return mode == NBODY_FP64 || mode == NBODY_F64E ? 8192 : 0;
}
int force_tile(int mode) { return mode == NBODY_FP64 ? T_F64 : mode == NBODY_F64E ? T_FF : T_F32; }

bool shape_supported(int mode, const Shape &sh) {
  if (sh.r != 1 && sh.r != 2 && sh.r != 4 && sh.r != 8) return false;
  if (mode == NBODY_F64E && sh.r == 8) return false;
  if (sh.s < 1 || sh.s > 65535) return false;
  if (sh.iw != 1 && (sh.iw != force_split(mode) || sh.r != 1)) return false;
  return sh.bt == force_block_threads(mode) && sh.t == force_tile(mode);
}

template <int R>
static const void *kernel_for(int mode) {
  switch (mode) {
    case NBODY_FP64: return (const void *)k_force_f64<BT_F64, R, T_F64, 1, DenseWork>;
    case NBODY_MIXED: return (const void *)k_force_mixed<BT_F32, R, T_F32, DenseWork>;
    case NBODY_F64E: return (const void *)k_force_f64e<BT_FF, (R < 4 ? R : 4), T_FF, 1, DenseWork>;
    default: return (const void *)k_force_f32<BT_F32, R, T_F32, DenseWork>;
  }
}

static const void *kernel_ptr(int mode, int r) {
  switch (r) {
    case 1: return kernel_for<1>(mode);
    case 2: return kernel_for<2>(mode);
    case 4: return kernel_for<4>(mode);
    default: return kernel_for<8>(mode);
  }
}

int force_max_blocks_per_sm(int mode, const Shape &sh) {
  int nb = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel_ptr(mode, sh.r), sh.bt, 0) !=
      cudaSuccess)
    return 0;
  return nb;
}

// One system's launches are links of a chain; those over a table of units (a
// pool's, or each pair once) follow copies and larger kernels and are plain.
template <class... P, class... A>
static cudaError_t launch_k(const DenseWork &, void (*k)(P...), dim3 grid, int bt, cudaStream_t st,
                            A... args) {
  return launch_chained(k, grid, bt, st, args...);
}
template <class... P, class... A>
static cudaError_t launch_k(const TableWork &, void (*k)(P...), dim3 grid, int bt, cudaStream_t st,
                            A... args) {
  k<<<grid, bt, 0, st>>>(args...);
  return cudaGetLastError();
}

template <int R, bool SPLIT, class W>
static cudaError_t launch_rw(int mode, const void *posm, const float4 *fpos, const float4 *anchor,
                             const W &w, dim3 grid, void *part, cudaStream_t st) {
  if (mode == NBODY_FP64)
    return launch_k(w, k_force_f64<BT_F64, R, T_F64, SPLIT ? IW_F64 : 1, W>, grid, BT_F64, st,
                    (const d4 *)posm, w, (d4 *)part);
  if (mode == NBODY_MIXED)
    return launch_k(w, k_force_mixed<BT_F32, R, T_F32, W>, grid, BT_F32, st, (const d4 *)posm, fpos,
                    anchor, w, (d4 *)part);
  if (mode == NBODY_F64E)
    return launch_k(w, k_force_f64e<BT_FF, (R < 4 ? R : 4), T_FF, SPLIT ? IW_FF : 1, W>, grid,
                    BT_FF, st, (const d4 *)posm, fpos, anchor, w, (d4 *)part);
  return launch_k(w, k_force_f32<BT_F32, R, T_F32, W>, grid, BT_F32, st,
                  (const float4 *)posm, w, (float4 *)part);
}

template <class W>
static cudaError_t launch_w(int mode, int r, const void *posm, const float4 *fpos,
                            const float4 *anchor, const W &w, dim3 grid, void *part,
                            cudaStream_t st) {
  switch (r) {
    case 1: return launch_rw<1, false>(mode, posm, fpos, anchor, w, grid, part, st);
    case 2: return launch_rw<2, false>(mode, posm, fpos, anchor, w, grid, part, st);
    case 4: return launch_rw<4, false>(mode, posm, fpos, anchor, w, grid, part, st);
    case 8: return launch_rw<8, false>(mode, posm, fpos, anchor, w, grid, part, st);
    default: return cudaErrorInvalidValue;
  }
}

// ---------------------------------------------------------------- binary64, each pair once: launches
// R = 3 (blocks of 384): 114 registers, 4 blocks of 4 warps per SM.  Measured on
// GB300 at N = 2^18 (this kernel alone, Gint/s): both potential sums in binary64
// R = 4 (148 registers, 3 blocks) 78.9, R = 3 81.6, R = 2 78.8; the row sum on the
// integer pipes R = 4 73.3, R = 3 85.6, R = 2 83.4; both sums on the integer
// pipes, k-loop not unrolled: R = 3 96.1, R = 2 96.3, R = 1 95.3 (unrolled twice:
// R = 2 92.2).
constexpr int SYM_BT = 128, SYM_R = 3, SYM_T = 128;
// softened systems: fixed point
constexpr int FXS_R = 2;

static bool fx_sym(double eps2) { return eps2 > 0.0; }
int sym_block_particles(double eps2) { return SYM_BT * (fx_sym(eps2) ? FXS_R : SYM_R); }
// the one-sided kernel's R for the pairs inside the diagonal blocks: the
// smallest supported R whose BT*R covers a block
int sym_units_r(double eps2) {
  const int r = fx_sym(eps2) ? FXS_R : SYM_R;
  return r <= 1 ? 1 : r <= 2 ? 2 : r <= 4 ? 4 : 8;
}

int sym_blocks_per_sm(double eps2) {
  int nb = 0;
  const void *k = fx_sym(eps2) ? (const void *)k_force_fx_sym<SYM_BT, FXS_R, SYM_T>
                               : (const void *)k_force_f64_sym<SYM_BT, SYM_R, SYM_T>;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, SYM_BT, 0) != cudaSuccess) return 0;
  return nb;
}

cudaError_t launch_force_f64_sym(const d4 *posm, int64_t n, double eps2, int M, int d0, int D,
                                 d4 *rows, d4 *cols, cudaStream_t st) {
  if (fx_sym(eps2))
    k_force_fx_sym<SYM_BT, FXS_R, SYM_T><<<D * M, SYM_BT, 0, st>>>(posm, n, eps2, M, d0, rows,
                                                                   cols);
  else
    k_force_f64_sym<SYM_BT, SYM_R, SYM_T><<<D * M, SYM_BT, 0, st>>>(posm, n, eps2, M, d0, rows,
                                                                    cols);
  return cudaGetLastError();
}

constexpr int SYMFF_BT = 128, SYMFF_R = 2, SYMFF_T = 256;

int sym_block_particles_ff() { return SYMFF_BT * SYMFF_R; }
int sym_r_ff() { return SYMFF_R; }

int sym_blocks_per_sm_ff() {
  int nb = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(
          &nb, k_force_f64e_sym<SYMFF_BT, SYMFF_R, SYMFF_T>, SYMFF_BT, 0) != cudaSuccess)
    return 0;
  return nb;
}

cudaError_t launch_force_f64e_sym(const d4 *posm, const float4 *jff, const float4 *anchor,
                                  int64_t n, double eps2, int M, int d0, int D, d4 *rows,
                                  d4 *cols, cudaStream_t st) {
  k_force_f64e_sym<SYMFF_BT, SYMFF_R, SYMFF_T><<<D * M, SYMFF_BT, 0, st>>>(
      posm, jff, anchor, n, eps2, M, d0, rows, cols);
  return cudaGetLastError();
}

cudaError_t launch_sym_combine(const d4 *rows, const d4 *cols, int D, int64_t n, d4 *acc_rows,
                               d4 *acc_cols, bool first, cudaStream_t st) {
  const int64_t blocks = std::min<int64_t>((n + 255) / 256, 4096);
  k_sym_combine<<<(unsigned)blocks, 256, 0, st>>>(rows, cols, D, n, acc_rows, acc_cols,
                                                  first ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t launch_force(int mode, const ForceIn &in, const Shape &sh, cudaStream_t st) {
  const int64_t rows = in.rows < 0 ? in.n : in.rows;
  if (!shape_supported(mode, sh) || in.n < 1 || rows < 1 || in.i0 < 0 || in.i0 + rows > in.n)
    return cudaErrorInvalidValue;
  const int64_t per_block = sh.per_block();
  const int64_t gx = (in.i0 % per_block + rows + per_block - 1) / per_block;
  if (gx > 0x7fffffff) return cudaErrorInvalidValue;
  DenseWork w;
  w.n = in.n;
  w.seg = in.seg;
  w.i_base = in.i0;
  w.rows = rows;
  w.eps2 = in.eps2;
  w.per_block = (int)per_block;
  w.tile = sh.t;
  const dim3 grid((unsigned)gx, (unsigned)sh.s);
  if (sh.iw > 1)
    return launch_rw<1, true>(mode, in.posm, in.fpos, in.anchor, w, grid, in.part, st);
  return launch_w(mode, sh.r, in.posm, in.fpos, in.anchor, w, grid, in.part, st);
}

cudaError_t launch_force_units(int mode, const void *posm, const float4 *fpos,
                               const float4 *anchor, const Unit *units, int64_t nunits, int r,
                               void *part, int64_t max_blocks, cudaStream_t st) {
  if (nunits < 1) return cudaErrorInvalidValue;
  TableWork w;
  w.units = units;
  w.n = nunits;
  int64_t g = nunits;
  if (max_blocks > 0 && g > max_blocks) g = max_blocks;
  if (g > 0x7fffffff) g = 0x7fffffff;
  return launch_w(mode, r, posm, fpos, anchor, w, dim3((unsigned)g), part, st);
}

cudaError_t launch_mixed_prep(const d4 *posm, int64_t n, int tile, float4 *fpos, float4 *anchor,
                              cudaStream_t st, bool ff) {
  if (tile != 256) return cudaErrorInvalidValue;  // one thread per tile member
  const int64_t nt = (n + tile - 1) / tile;
  DensePrep w;
  w.n = n;
  w.tile = tile;
  return launch_chained(ff ? k_mixed_prep<256, DensePrep, true> : k_mixed_prep<256, DensePrep, false>,
                        dim3((unsigned)nt), 256, st, posm, w, fpos, anchor);
}

cudaError_t launch_mixed_prep_units(const d4 *posm, const PrepUnit *units, int64_t nunits,
                                    float4 *fpos, float4 *anchor, cudaStream_t st, bool ff) {
  if (nunits < 1 || nunits > 0x7fffffff) return cudaErrorInvalidValue;
  TablePrep w;
  w.units = units;
  if (ff)
    k_mixed_prep<256, TablePrep, true><<<(unsigned)nunits, 256, 0, st>>>(posm, w, fpos, anchor);
  else
    k_mixed_prep<256, TablePrep, false><<<(unsigned)nunits, 256, 0, st>>>(posm, w, fpos, anchor);
  return cudaGetLastError();
}

}  // namespace nb
