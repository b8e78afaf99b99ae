// fx.cuh -- two-limb fixed-point complex arithmetic on the integer pipe.
//
// GB300 issues 2 DFMA per clock per SM but 32 IMAD.WIDE (32 x 32 + 64 bits; measured at 2070 MHz
// with operands from shared memory), so a product of two fixed-point numbers of two 27-bit limbs,
// three IMAD.WIDE, runs five times faster than one DFMA.  The member dots det = g . y
// and the triangular solves behind y are exactly the shape for it: sums of at most 36 products
// against one vector, whose accuracy is judged at the scale of the vectors' largest entries
// (the lemma guard; a solve's error bound), not entry by entry.
//
// A vector is stored with one binary exponent e above all its entries: entry x becomes the
// integer round(x 2^(b - e)), |.| <= 2^b (b = 54 .. 57, below), split as hi 2^27 + lo with lo in
// [-2^26, 2^26).  A sum accumulates hi hi and hi lo + lo hi in 64 bits and drops lo lo, at most
// 2^52 per product against 2^111 for the vectors' scale in a dot.  A dot is off by less than
// (2 n) 2^-56 |g|max |y|max then.  That is a quarter of what an FP64 chain may be off by when its
// largest product has that size, and more than FP64's error when all products are far smaller.  So a
// dot below a floor (accepted, below), below 2^-kc of the scale (kc: the lemma guard's exponent) or above
// eight times it is not used: the FP64 path forms that determinant again and applies its own guard, so
// which pairs the guard has refactored does not depend on this arithmetic.  (Random blocks of n = 6 to 18: the median dot is 2^-1.7 of the scale, one in a thousand
// lies above 2^0.6 to 2^1.)
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/mhc.h"
#include "device.cuh"

namespace mhc {
namespace fx {

constexpr int kBase = 27;               // bits of the low limb
constexpr int kFracBits = 56;           // a cached solve: |entry| <= 2^56
constexpr int kRowBits = 55;            // a propagator row: |entry| <= 2^55
constexpr int kDotBits = 57;            // a dot: 2^57 stands for the product of the scales
constexpr int kMaxHi = 1 << 28;         // high word of 2^60: a larger dot is not used
constexpr int kMulHi = 1 << 27;         // high word of 2^59: the largest factor of mul
constexpr int kNever = 0x7fffffff;      // a threshold that no value reaches
// Tables::align, other than the binades up to kMaxAlign: the member lies further below, adds nothing
// (its weight is zero, or there is no such member), or is evaluated by the FP64 path
enum : unsigned { kFar = 128, kMute = 129, kOnlyFp64 = 130 };
constexpr int kMaxAlign = 8;            // most bits of a dot that its family's common exponent may cost
constexpr int kFlush = 8;               // members per 64-bit sum of products (Acc2)
constexpr int kMaxMembers = 64;

// round(x 2^(b - e)) for |x| < 2^e, b <= 56
__device__ __forceinline__ long long quant(double x, int e, int b) {
  const long long w = __double_as_longlong(x);
  const int ex = (int)((w >> 52) & 0x7ff);
  long long m = (w & 0xfffffffffffffll) | (ex ? 0x10000000000000ll : 0ll);
  const int s = (ex ? ex : 1) - 1075 + b - e;  // <= 3 when |x| < 2^e
  m = s >= 0 ? m << min(s, 3) : (s < -54 ? 0ll : (m + (1ll << (-s - 1))) >> -s);
  return w < 0 ? -m : m;
}

// limbs of a complex entry: (re hi, re lo, im hi, im lo)
__device__ __forceinline__ int4 limbs(long long re, long long im) {
  constexpr long long half = 1ll << (kBase - 1);
  const int rh = (int)((re + half) >> kBase), ih = (int)((im + half) >> kBase);
  return make_int4(rh, (int)re - (rh << kBase), ih, (int)im - (ih << kBase));
}
__device__ __forceinline__ int4 quant(dev::cd z, int e, int b) { return limbs(quant(z.x, e, b), quant(z.y, e, b)); }

// back to FP64 (entries made from FP64 values hold at most 53 significant bits: exact)
__device__ __forceinline__ double pow2(int e) {  // 2^e for normal e, else saturated to 0 / inf
  return e < -1022 ? 0.0 : __longlong_as_double((long long)min(e + 1023, 2047) << 52);
}
__device__ __forceinline__ double scale2(double x, int e) {  // x 2^e without intermediate overflow
  e = min(e, 2046);  // more is infinite as well, and 0 stays 0
  const int h = e >> 1;
  return x * pow2(h) * pow2(e - h);
}
__device__ __forceinline__ dev::cd value(int4 v, int e) {
  const long long re = ((long long)v.x << kBase) + v.y, im = ((long long)v.z << kBase) + v.w;
  return make_double2(scale2((double)re, e - kFracBits), scale2((double)im, e - kFracBits));
}

// Sums of complex products.  The real part's positive and negative products have sums of
// their own: IMAD.WIDE adds its product, and a negated operand would cost an instruction each.
struct Acc {
  long long rp = 0, rn = 0, lp = 0, ln = 0, ih = 0, il = 0;
};
// a b + c.  As inline PTX it comes out as a multiplication and an addition on two pipes; the one
// instruction that the compiler makes of the C expression has half the rate and a longer latency
// (forward of 512 x 512 terms of n = 3 with these dots: 58 us with this, 64 us with that).
__device__ __forceinline__ long long madw(int a, int b, long long c) {
#ifdef __CUDA_ARCH__
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(c) : "r"(a), "r"(b));
  return c;
#else
  return (long long)a * b + c;
#endif
}
__device__ __forceinline__ void mac(Acc& s, int4 a, int4 b) {
  s.rp = madw(a.x, b.x, s.rp);
  s.rn = madw(a.z, b.z, s.rn);
  s.lp = madw(a.x, b.y, s.lp);
  s.ln = madw(a.z, b.w, s.ln);
  s.ih = madw(a.x, b.z, s.ih);
  s.il = madw(a.x, b.w, s.il);
  s.lp = madw(a.y, b.x, s.lp);
  s.ln = madw(a.w, b.z, s.ln);
  s.ih = madw(a.z, b.x, s.ih);
  s.il = madw(a.y, b.z, s.il);
  s.il = madw(a.z, b.y, s.il);
  s.il = madw(a.w, b.x, s.il);
}

// a value: a dot of a row (2^55) and a solve (2^56) in units of 2^54
struct Val {
  long long re, im;
};
__device__ __forceinline__ Val finish(const Acc& s) {
  constexpr long long half = 1ll << (kBase - 1);
  return Val{(s.rp - s.rn) + ((s.lp - s.ln + half) >> kBase), s.ih + ((s.il + half) >> kBase)};
}
// max(|re|, |im|) / 2^32 by the high words (a negative value's complement is its magnitude less
// one unit), and whether that lies in [thr, top)
__device__ __forceinline__ int magnitude(Val v) {
  const int a = (int)(v.re >> 32), b = (int)(v.im >> 32);
  return max(a ^ (a >> 31), b ^ (b >> 31));
}
__device__ __forceinline__ bool usable(int mag, int thr, int top = kMaxHi) { return mag >= thr && mag < top; }
// High word of the smallest usable |value|, at or above the point where the FP64 lemma guard
// can fire: |det| < 2^(e(row) + e(y) - kc) with floor exponents, here against exponents above the
// entries.  Rank 1: e(row) + e(y) <= r + e_y - 2, and a complex factor det B taken out of y moves
// either side by up to sqrt 2: 2^(57 - 1 - kc) covers both, and one binade more is kept.  Rank 2:
// two rows and two null vectors, e <= r_1 + r_2 + 2 e_z - 4, with 2^56 for the scales: 2^(53 - kc).
// At least 1: below 2^32 the FP64 path decides.
__device__ __forceinline__ int threshold(int kc, int rank) {
  const int t = (rank == 1 ? kDotBits : 53) - 32 - kc;
  return t >= 28 ? kNever : t <= 0 ? 1 : 1 << t;
}

// High word of the smallest |value| that is used: the guard's threshold, and a floor that no guard lowers.  A
// dot is off by a few units of 2^57 2^-56 times the square root of n, so a value of 2^(57 - kFloorBits)
// by some 2^-46 of itself (2^-45 for n > 8); a two-row determinant's two dots are each off by as little.  A
// smaller one may be a sum of large products that cancel, where FP64 is off as much, or all its products may
// be far below the scale: the FP64 path tells (fx_member64).  Of the dots of random blocks one in 20 000 lies
// below 2^-9 of the scale, one in 80 000 below 2^-10, where the default lemma guard sends it there anyway; an
// evaluation takes its warp as long as 10 to 20 members in fixed point, and more for n > 8.  (4096 x 4096
// terms of n = 6: floors of 2^-10, 2^-9, 2^-8 1095, 1112, 1150 us; small pairs queued for refactors, of which an
// item has one at a time, 1360 to 1520 us.)
constexpr int kFloorBits = 9, kFloorBitsLarge = 10;  // n <= 8; above
constexpr int kFloorBits2 = 12;  // of a two-row determinant, 2^56 for the scales
constexpr int kCarryBits = 4;    // a product this many binades below the scale still carries a small value
__device__ __forceinline__ int accepted(int n, int kc, int rank) {
  const int bits = rank == 2 ? 1 + kFloorBits2 : n <= 8 ? kFloorBits : kFloorBitsLarge;
  return max(threshold(kc, rank), 1 << (kDotBits - 32 - bits));
}

// Products of two dots.  A dot's scale is an upper bound that it stays a few binades below: the product
// keeps 57 bits of the scale of each factor, and its lo lo terms.  (With 54 bits and without them the
// correlator of 1291 x 977 terms of n = 5, 4 was off by 8e-14, against 1.8e-15 in FP64.)
// Limbs in base 2^30 of value / 2, |value| < 2^60: |hi| <= 2^29, lo in [-2^29, 2^29); kFlush products
// of four cross terms each stay below 2^63.
constexpr int kSplitBits = kDotBits - 1;  // 2^56 stands for the scale then
__device__ __forceinline__ int4 split(Val v) {
  const int rh = (int)((v.re + (1ll << 30)) >> 31), ih = (int)((v.im + (1ll << 30)) >> 31);
  return make_int4(rh, (int)(v.re >> 1) - (rh << 30), ih, (int)(v.im >> 1) - (ih << 30));
}
// A member whose product lies d binades below its family's exponent: its first dot in that exponent's units.
// Beside the larger members' own errors the bits it loses are nothing; where those members vanish, kMaxAlign
// leaves it 2^-49 of its scale.  A member further down (one in 100 with normal weights) is summed in
// FP64 by itself.  The shift rounds down: its mean of half a unit is multiplied by the second dot, whose
// phase it does not know; a single dot is rounded to the nearest instead.
__device__ __forceinline__ Val aligned(Val v, int d) { return Val{v.re >> d, v.im >> d}; }
__device__ __forceinline__ Val rounded(Val v, int d) {
  const unsigned half = (1u << d) >> 1;
  return aligned(Val{v.re + half, v.im + half}, d);
}
struct Acc2 : Acc {
  long long qp = 0, qn = 0, qi = 0;  // lo lo
  // the sums in units of 2^60 and 2^30
  __device__ __forceinline__ long long hi_re() const { return rp - rn; }
  __device__ __forceinline__ long long lo_re() const { return lp - ln + ((qp - qn) >> 30); }
  __device__ __forceinline__ long long hi_im() const { return ih; }
  __device__ __forceinline__ long long lo_im() const { return il + (qi >> 30); }
};
__device__ __forceinline__ void mac(Acc2& s, int4 a, int4 b) {
  mac(static_cast<Acc&>(s), a, b);
  s.qp = madw(a.y, b.y, s.qp);
  s.qn = madw(a.w, b.w, s.qn);
  s.qi = madw(a.y, b.w, s.qi);
  s.qi = madw(a.w, b.y, s.qi);
}
// a b / 2 with 2^56 for the product of the scales (a, b: limbs of values below 2^59)
__device__ __forceinline__ Val mul(int4 a, int4 b) {
  Acc2 s;
  mac(s, a, b);
  constexpr long long half = 1ll << 25;
  return Val{(s.hi_re() << 4) + ((s.lo_re() + half) >> 26), (s.hi_im() << 4) + ((s.lo_im() + half) >> 26)};
}

// ---- triangular solves ------------------------------------------------------------------
// The solve of one sink against a two-sided block's factors P B = L U (device.cuh, kapply):
// z = -B^{-1} a by L w = P a and U z = -w, with w and z as fixed-point vectors in the sink's
// shared-memory column.  The factors are stored as 54-bit limbs: L with exponent 1 (partial
// pivoting: |l| <= sqrt 2), row i of U with its own exponent eU_i, the pivot's reciprocal r_i
// with er_i.  w keeps the unit of a, 2^(ea - 55).  z's unit is chosen per sink so that the largest
// |r_i w_i| is at 2^54; entries may grow to 2^58 (on random blocks of n = 3 to 18 w grew by at most
// 2^2 and z by 2^3.5).  Every sum is exact but for the dropped lo lo products, below one unit.
// What one unit for all of a vector costs is bounded by checks; a sink or block that fails one is
// reported and takes the one-sided FP64 factorisation, ten times the work, so the limits lie where
// random blocks hardly ever come:
//   - the rows of a block have exponents within kBlockSpread, and its columns too (block_fits, by the
//     kfac routines): a row far below the others has its part of a, w and L in that many bits less, and
//     a column its part of U, against larger entries of z;
//   - w keeps kMinBits bits (a column far below its exponent), one less where it is a single entry;
//   - the largest r_i w_i is at least 2^kLeadBits units of w times the largest r_i: one unit of any w_i
//     moves z by at most 2^-kLeadBits of its largest entry.  product_exponent reads high limbs only;
//     with this a w_i without one is below 2^-20 of the largest product, and no T overflows;
//   - nothing grows above its limit.
// The error against the exact solve is the FP64 one's (both are the factors': mean 1.8e-15 at n = 18,
// 1.0e-15 at n = 12, of the largest entry).
//   layout: LU[M][M] limbs (diagonal: r_i) | (S row offset of the row's label, eU_i, er_i, e of
//           -U1^{-1} u) [M] | ... | -det B | det B (FP64)
constexpr int kFactBits = 54;
constexpr int kABits = 55;   // |a| <= 2^55
constexpr int kZBits = 54;   // the largest |r_i w_i|, within a factor of two
constexpr int kTopBits = 58;
constexpr int kMinBits = 52;
constexpr int kLeadBits = 47;
constexpr int kBlockSpread = 3;

__device__ __forceinline__ int4 factor_limbs(dev::cd z, int e) { return quant(z, e, kFactBits); }
// row i's exponents: normal, and |U_i| / |pivot| within the shifts of sum_shifted
__device__ __forceinline__ bool exponents_ok(int eu, int er) {
  return eu > -900 && eu < 900 && er > -900 && er < 900 && eu + er <= 20;
}

// lowest and highest exponent of a block's rows, or columns (each its largest entry's)
__device__ __forceinline__ bool block_fits(int lo, int hi) { return hi - lo <= kBlockSpread; }

__device__ __forceinline__ int bits(long long x) { return 64 - __clzll(x ^ (x >> 63)); }
__device__ __forceinline__ Val joined(int4 l) {
  return Val{((long long)l.x << kBase) + l.y, ((long long)l.z << kBase) + l.w};
}
__device__ __forceinline__ int4 limbs(Val v) { return limbs(v.re, v.im); }
// (sum of factor x vector products) 2^-(54 - k), 0 <= k <= 20
__device__ __forceinline__ Val sum_shifted(const Acc& s, int k) {
  const int r = kBase - k;
  const long long half = 1ll << (r - 1);
  return Val{((s.rp - s.rn) << k) + ((s.lp - s.ln + half) >> r), (s.ih << k) + ((s.il + half) >> r)};
}
// |v| < 7/8 2^58: 34 products with 2^27 sum to less than 2^63, and the high limb fits 32 bits
constexpr int kFits = 7 << (kTopBits - 35);
// exponent above max(|re|, |im|) of w times that of r (limbs, exponent er), within a factor of two
__device__ __forceinline__ int product_exponent(int4 w, int4 r, int er) {
  const float a = (float)max(abs(w.x), abs(w.z)), b = (float)max(abs(r.x), abs(r.z));
  return (__float_as_int(a * b) >> 23) - 126 + 2 * kBase - kFactBits + er;
}
__device__ __forceinline__ long long shift(long long x, int right) {  // x 2^-right, |right| <= 63
  return right >= 0 ? x >> min(right, 63) : x << -right;
}

// Solves one sink; Y: its column (stride ys), entries 0 .. M - 1 become z.  K: the block's factors,
// in shared memory (SM) or global; a: the sink's changed column of the propagator at its own
// exponent ea (Tables::sc).  zlo: the unit's exponent is at least zlo - 55 (so that the caller's
// other entries of z, below 2^zlo, fit).  Two rows share each load of the vector.  *unit: z's
// unit exponent, *mag: the magnitude of its largest entry.  Returns false when the sink has to
// take the FP64 path.
template <bool SM>
__device__ __forceinline__ bool solve(int M, const int4* __restrict__ a, int ea, int zlo, const int4* __restrict__ K,
                                      int4* Y, int ys, int* unit, int* mag) {
  auto ld = [](const int4* q) { return SM ? *q : __ldg(q); };
  int mx = -100000, top = 0, lead = -100000;
  for (int i = 0; i < M; i += 2) {
    const bool two = i + 1 < M;
    const int i1 = two ? i + 1 : i;
    const int4 t0 = ld(K + M * M + i), t1 = ld(K + M * M + i1);
    const Val a0 = joined(__ldg(a + t0.x)), a1 = joined(__ldg(a + t1.x));
    const int4 *k0 = K + i * M, *k1 = K + i1 * M;
    Acc s0, s1;
#pragma unroll 1
    for (int t = 0; t < i; t++) {
      const int4 w = Y[t * ys];
      mac(s0, ld(k0 + t), w);
      mac(s1, ld(k1 + t), w);
    }
    const Val q0 = sum_shifted(s0, 1), w0{a0.re - q0.re, a0.im - q0.im};
    const int4 l0 = limbs(w0);
    Y[i * ys] = l0;
    top = max(top, magnitude(w0));
    mx = max(mx, product_exponent(l0, ld(k0 + i), t0.z));
    lead = max(lead, max(t0.z, t1.z));
    if (two) {
      mac(s1, ld(k1 + i), l0);
      const Val q1 = sum_shifted(s1, 1), w1{a1.re - q1.re, a1.im - q1.im};
      const int4 l1 = limbs(w1);
      Y[i1 * ys] = l1;
      top = max(top, magnitude(w1));
      mx = max(mx, product_exponent(l1, ld(k1 + i1), t1.z));
    }
  }
  bool ok = top < kFits && top >= 1 << (kMinBits - (M > 1 ? 33 : 34)) && mx >= lead + kLeadBits;
  // unit exponent u of z: largest r_i w_i (2^(mx + ea - 55)) at 2^54
  const int u = max(mx + ea - kABits - kZBits, zlo - 55);
  *unit = u;
  mx = u + kABits - ea;
  int over = 0;  // largest magnitude of T and z
  top = 0;
  for (int i = M - 1; i >= 0; i -= 2) {
    const bool two = i >= 1;
    const int i1 = two ? i - 1 : i;
    const int4 t0 = ld(K + M * M + i), t1 = ld(K + M * M + i1);
    const int4 *k0 = K + i * M, *k1 = K + i1 * M;
    Acc s0, s1;
#pragma unroll 1
    for (int t = i + 1; t < M; t++) {
      const int4 z = Y[t * ys];
      mac(s0, ld(k0 + t), z);
      mac(s1, ld(k1 + t), z);
    }
    // row i: T = w + U z in units of 2^(u + eU_i), z_i = -r_i T
    auto row = [&](const Acc& s, int4 t, int at, const int4* k) {
      const Val w = joined(Y[at * ys]), q = sum_shifted(s, 0);
      const int sh = mx + t.y;
      const Val T{shift(w.re, sh) + q.re, shift(w.im, sh) + q.im};
      over = max(over, magnitude(T));
      Acc p;
      mac(p, ld(k + at), limbs(T));
      const int kk = t.y + t.z;  // |U_i| / |pivot| in binades, 0 .. 20
      ok = ok && bits(p.rp - p.rn) <= kTopBits - kk && bits(p.ih) <= kTopBits - kk;
      const Val z = sum_shifted(p, kk);
      const Val n{-z.re, -z.im};
      top = max(top, magnitude(n));
      const int4 l = limbs(n);
      Y[at * ys] = l;
      return l;
    };
    const int4 l = row(s0, t0, i, k0);
    if (two) {
      mac(s1, ld(k1 + i), l);
      row(s1, t1, i1, k1);
    }
  }
  *mag = top;
  return ok && max(over, top) < kFits;
}

// One sink's solve from its block's factors: z in Y (rank 1: n entries, the last 1; rank 2: z1 and z2),
// scaled so that the largest entry just fills 2^56.  F: the block's limbs (staged when SM), K: the same
// block in global memory, for its FP64 entries.  *e2: 2 e_y + 1 (an entry of 2^56 stands for 2^e_y; det
// B is a factor); *sd: rank 2, the FP64 factor.
template <bool SM>
__device__ __forceinline__ bool solve_sink(int n, int rho, const int4* __restrict__ a, int ea, const int4* __restrict__ F,
                                           const dev::cd* __restrict__ K, int4* Y, int ys, int* e2, dev::cd* sd) {
  const int M = n - rho;
  if (ea > 900 || ea < -900) return false;
  int4* z = Y + (rho == 2 ? n * ys : 0);
  const int zlo = rho == 2 ? max(0, __ldg(reinterpret_cast<const int4*>(K) + M * M).w) : 0;
  int u = zlo - 55, mag = 0;
  if (M > 0 && !solve<SM>(M, a, ea, zlo, F, z, ys, &u, &mag)) return false;
  // the unit entries; u >= -55, and an entry 1 below the unit is lost against the others
  const Val unit{u <= 0 ? 1ll << -u : 0ll, 0ll};
  const int4 one = limbs(unit), zero = make_int4(0, 0, 0, 0);
  mag = max(mag, magnitude(unit));
  if (rho == 2) {
    z[M * ys] = zero;
    z[(M + 1) * ys] = one;
    for (int q = 0; q < M; q++) {
      const int4 v = quant(__ldg(K + M * M + M + q), u + kFracBits, kFracBits);
      Y[q * ys] = v;
      mag = max(mag, magnitude(joined(v)));
    }
    Y[M * ys] = one;
    Y[(M + 1) * ys] = zero;
    *sd = __ldg(K + M * M + 2 * M);
  } else {
    z[M * ys] = one;
  }
  // the largest entry just below 2^56 (its bits by the high word: 32 when below 2^32)
  const int sh = 64 - __clz(mag) - kFracBits;
  for (int q = 0; q < rho * n; q++) {
    const Val x = joined(Y[q * ys]);
    Y[q * ys] = limbs(shift(x.re, sh), shift(x.im, sh));
  }
  *e2 = 2 * (u + sh + kFracBits) + 1;
  return true;
}

// ---- propagators for this arithmetic -----------------------------------------------------
// A row or column has one exponent, so entries far below its largest keep fewer bits than FP64 gives
// them.  Single dots, solves and blocks where that matters are found above; where it is the rule -- rows
// or columns of very different sizes, entries that decay with distance -- the whole call takes the FP64
// kernels' path: fxprep decides it for every call, over the labels that the plan's terms use.  Random
// rows with a diagonal (L = 24 to 96) have exponents within two binades and 1 to 2 % of small entries.  The
// accepted determinants' median error by FP64's: 0.95 to 1 on those, up to 1.08 with rows and columns
// scaled over 2^1, 1.35 over 2^2, 20 over 2^10.
constexpr int kFlatSpread = 2;  // binades between the rows' exponents, and between the columns'
constexpr int kSmallBits = 6;   // an entry is small below 2^-kSmallBits of its row's exponent
constexpr int kSmallShare = 8;  // at most one in kSmallShare is
__device__ __forceinline__ bool small_entry(dev::cd z, int e) { return dev::expo(z) < e - kSmallBits; }
struct Scan {
  int rlo = 4096, rhi = -4096, clo = 4096, chi = -4096;  // exponents of the rows and columns
  int small = 0, total = 0;                              // entries
  __device__ __forceinline__ void row(int e, int n_small, int n) {
    if (e <= -1022) return;  // all zero, or as good as that
    rlo = min(rlo, e);
    rhi = max(rhi, e);
    small += n_small;
    total += n;
  }
  __device__ __forceinline__ void column(int e) {
    if (e <= -1022) return;
    clo = min(clo, e);
    chi = max(chi, e);
  }
  __device__ __forceinline__ bool flat() const {  // (an exponent above 1023: not finite)
    return max(rhi, chi) <= 1023 && rhi - rlo <= kFlatSpread && chi - clo <= kFlatSpread && small <= total / kSmallShare;
  }
};

// Tables of one plan for one set of propagators and weights, rebuilt by every call.
struct Tables {
  const int* used[MHC_FMAX];    // [L_f] bit 0: a source term has the label (its row is used), bit 1: a
                                // sink term (its column); rows and columns below are the used entries
  const int4* s[MHC_FMAX];      // [L_f][L_f] propagator rows, each with its own exponent
  const int4* sc[MHC_FMAX];     // [L_f][L_f] the same entries with one exponent per column
  const int* cexp[MHC_FMAX];    // [L_f] that exponent (above every entry of the column)
  const int4* scan[MHC_FMAX];   // [L_f] exponent of the row, of the column, small entries and entries of
                                // the row
  int* state;                   // [0] 1: the propagators are flat (Scan), [1] rows scanned, 0 between calls
  const int4* ws;               // [members][L_f0] first flavour's first member row times the weight (as
                                // it is where that is zero), with an exponent of its own
  const unsigned* align;        // [members] at a family's member 0, 4, 8 ...: a byte for it and the next
                                // three, binades by which the member's product scale lies below its
                                // family's, or kFar, kMute, kOnlyFp64
  const int* below;             // [members] those binades of a kFar member
  const int* fexp;              // [W] exponent of the family's products: its largest member's
  int f0, nf;                   // first flavour with n_f > 0; flavours with n_f > 0 (0: no tables)
};

}  // namespace fx
}  // namespace mhc
