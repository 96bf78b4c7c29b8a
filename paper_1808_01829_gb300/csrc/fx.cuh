// FP64-accurate sums of products on the integer units.  This GPU issues two
// FP64 operations per clock and SM (a warp's DFMA takes 64 clocks); a 32 x 32 ->
// 64 bit integer multiply-add of a warp takes four (measured), so a dot product whose
// operands are first brought to a common exponent runs several times faster as
// integers than as FP64 FMAs.
//
// A block of reals x with |x| < 2^E is held as q = x 2^(55 - E), truncated, in
// two signed words q = hi 2^27 + lo with |hi| <= 2^28 and -2^26 <= lo < 2^26.
// Values within a factor of 4 of the block's largest are exact; smaller ones lose
// what lies below 2^-55 of 2^E (an FP64 sum rounds every step at 2^-53 of the
// running sum).  A product of two such numbers is
//   2^(E1 + E2 - 56) [h1 h2 + (h1 l2 + l1 h2) 2^-27 + l1 l2 2^-54],
// whose last term is below 2^-58 of 2^(E1 + E2) and dropped.  The sums A = sum h h
// and B = sum (h l + l h) are exact.
//
// A complex product (a + i b)(c + i d) takes three real ones, a c, b d and
// (a + b)(c + d); as integers nothing is lost in their differences.  Over up to
// 24 complex products |A| <= 24 2^58 < 2^63 and, with the second factor's words
// aligned (|lo| < 1.25 2^27), |B| <= 24 (2^29 1.25 2^28 + 2^27 2^29) < 2^63.
//
// A field in this form has one int4 (re hi, re lo, im hi, im lo) per complex, as
// large as its FP64 form, and one word per (site, column) with the exponent E of the three
// colours and how far the smallest colour lies below it (code, exponent, least).  Blocks with
// infinities, NaN or subnormals keep their FP64 values in the int4 under the exponent
// kSpecial; kZero marks a block of zeros.
//
// The error of a sum is absolute, 2^-55 of the largest operands, that of FP64 FMAs relative to
// sum |U_cb| |v_b| of each output c.  The two agree unless that sum is small for some c, as where
// unit-like links keep colours of very different size apart.  A hop therefore takes the integer
// form only where one of the eight neighbours has all three colours within 2^kApart of
// the largest (a row c of unitary links has an entry of order one there, which stage_links_fx
// checks), or else where for every output that sum, formed from the leading words, is
// at least half of largest link times largest value.  Measured against
// extended precision, largest error over sum |U_cb| |v_b| (integers; FP64 FMAs): Gaussian fields
// 7.6e-17; 4.1e-16, unit links and colours 1, 1/8, 1/8 4.1e-16; 2.6e-16, 1, 1/16, 1/16 5.0e-16; 2.6e-16.
#pragma once

namespace rhmc {
namespace fx {

constexpr int kLow = 27;              // bits of the low word
constexpr int kBits = 55;             // magnitude bits
constexpr int kSpecial = 1 << 20;     // exponent code: the block holds FP64 values
constexpr int kZero = -(1 << 20);     // exponent code: all zeros
constexpr int kApart = 3;             // see above; Gaussian colours: all but one (site, column) in a million

// A block's word: its exponent and, in the low five bits, the distance to that of its smallest colour
__device__ __forceinline__ int code(int e, int apart) { return e * 32 + min(apart, 31); }
__device__ __forceinline__ int exponent(int c) { return c >> 5; }
__device__ __forceinline__ int least(int c) { return (c >> 5) - (c & 31); }

// biased exponent field (0: zero or subnormal, 0x7ff: infinity or NaN)
__device__ __forceinline__ int expo(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }
__device__ __forceinline__ bool nonzero(double x) {
  return (((unsigned)__double2hiint(x) << 1) | (unsigned)__double2loint(x)) != 0u;
}

// the two words of q
__device__ __forceinline__ int2 words(long long q) {
  const int lo = (int)((unsigned)q << 5) >> 5;  // the low 27 bits, signed
  return make_int2((int)((q - (long long)lo) >> kLow), lo);
}
// x 2^(55 - E) for the block's largest exponent field ef (E = ef - 1022)
__device__ __forceinline__ int2 split(double x, int ef) {
  const unsigned hw = (unsigned)__double2hiint(x), lw = (unsigned)__double2loint(x);
  const int e = (int)(hw >> 20) & 0x7ff;
  const unsigned mh = (hw & 0xfffffu) | (e ? 0x100000u : 0u);
  // mantissa left-justified below bit 63, subnormals shifted out
  const unsigned long long m = ((unsigned long long)((mh << 10) | (lw >> 22)) << 32) | (lw << 10);
  const unsigned long long mag = m >> (e ? min(63, ef - e + 8) : 63);
  const long long sg = (long long)((int)hw >> 31);
  return words((long long)(mag ^ (unsigned long long)sg) - sg);
}

// x 2^55 rounded, for |x| < 2
__device__ __forceinline__ long long fixed55(double x) {
  const unsigned hw = (unsigned)__double2hiint(x), lw = (unsigned)__double2loint(x);
  const int e = (int)(hw >> 20) & 0x7ff;
  const unsigned long long m = ((unsigned long long)((hw & 0xfffffu) | (e ? 0x100000u : 0u)) << 32) | lw;
  const int s = 1023 + 52 - 55 - e;  // x = m 2^(e - 1075), 2^55 x = m 2^(e - 1020)
  const unsigned long long mag = s <= 0 ? m << -s : ((m >> min(63, s - 1)) + 1) >> 1;
  const long long sg = (long long)((int)hw >> 31);
  return (long long)(mag ^ (unsigned long long)sg) - sg;
}

// Three complex numbers (a site's column) as they are; returns the block's word.
__device__ __forceinline__ int keep3(const double2 *v, int4 *o) {
  bool any = false;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    any = any || nonzero(v[c].x) || nonzero(v[c].y);
    o[c] = *reinterpret_cast<const int4 *>(&v[c]);
  }
  return code(any ? kSpecial : kZero, 0);
}
// Three complex numbers as one block; returns its word.
__device__ __forceinline__ int pack3(const double2 *v, int4 *o) {
  int ef = 0, em = 0x7ff;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int e = max(expo(v[c].x), expo(v[c].y));
    ef = max(ef, e);
    em = min(em, e);
  }
  if (ef == 0x7ff || ef == 0) return keep3(v, o);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int2 re = split(v[c].x, ef), im = split(v[c].y, ef);
    o[c] = make_int4(re.x, re.y, im.x, im.y);
  }
  return code(ef - 1022, em ? ef - em : 31);
}
// The FP64 value of one complex of a block with exponent e.
__device__ __forceinline__ double2 unpack(int4 q, int e) {
  if (e == kSpecial) return *reinterpret_cast<const double2 *>(&q);
  if (e == kZero) return make_double2(0.0, 0.0);
  const long long re = ((long long)q.x << kLow) + q.y, im = ((long long)q.z << kLow) + q.w;
  return make_double2(ldexp((double)re, e - kBits), ldexp((double)im, e - kBits));
}

// The words of q 2^-sh, 0 <= sh <= kAlign: the bits that leave the high word enter the low
// one (lo then lies in [-2^26, 2^27 + 2^25)).
constexpr int kAlign = 26;
__device__ __forceinline__ void align(int &hi, int &lo, int sh) {
  // the low sh bits of hi at the top of a word (nothing for sh = 0), then down to bits 26 ..
  const unsigned out = __funnelshift_r(0u, (unsigned)hi, sh);
  lo = (lo >> sh) + (int)(out >> 5);
  hi >>= sh;
}

// A += h h, B += h l + l h
__device__ __forceinline__ void mac2(long long &A, long long &B, int ah, int al, int bh, int bl) {
  A += (long long)ah * bh;
  B += (long long)ah * bl;
  B += (long long)al * bh;
}
// (A + B 2^-27) for the sums of a product
__device__ __forceinline__ long long join(long long A, long long B) { return A + (B >> kLow); }

// |re| or |im| is 2^bits or more
__device__ __forceinline__ bool reaches(long long re, long long im, int bits) {
  return ((re ^ (re >> 63)) | (im ^ (im >> 63))) >> bits != 0;
}

// r 2^k rounded to FP64
__device__ __forceinline__ double value(long long r, int k) {
  if (r == 0) return 0.0;
  const double d = __ll2double_rn(r);
  const int hw = __double2hiint(d);
  const int e = ((hw >> 20) & 0x7ff) + k;
  if ((unsigned)(e - 1) < 2045u) return __hiloint2double(hw + (k << 20), __double2loint(d));
  return ldexp(d, max(-4000, min(4000, k)));
}

// r 2^-right, rounded
__device__ __forceinline__ long long shift(long long r, int right) {
  return right > 0 ? (r + (1ll << (right - 1))) >> right : (long long)((unsigned long long)r << -right);
}
// Six reals r 2^k (three complex) as a block: brought to 55 bits by the leading bit of the
// largest.
__device__ __forceinline__ int renorm3(const long long *r, int k, int4 *o) {
  int len = 0, least = 64;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    // |r| <= m + 1 <= 2^l
    const unsigned long long m = (unsigned long long)((r[2 * c] ^ (r[2 * c] >> 63)) | (r[2 * c + 1] ^ (r[2 * c + 1] >> 63)));
    const int l = 64 - __clzll((long long)m);
    len = max(len, l);
    least = min(least, l);
  }
  const int sh = len - kBits;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int2 re = words(shift(r[2 * c], sh));
    const int2 im = words(shift(r[2 * c + 1], sh));
    o[c] = make_int4(re.x, re.y, im.x, im.y);
  }
  bool any = len != 0;
#pragma unroll
  for (int c = 0; c < 6; ++c) any = any || r[c] != 0;  // (all -1 has m = 0)
  return code(any ? k + len : kZero, any ? len - least : 0);
}

}  // namespace fx
}  // namespace rhmc
