// modarith.cuh -- exact modular arithmetic on u64 residues (q < 2^58).
//
// Two published methods, both exact (the result is the canonical residue):
//  * Shoup's precomputed-quotient product for multiplication by a known
//    constant w:  w' = floor(w 2^64 / q);  a w - floor(a w' / 2^64) q lies in
//    [0, 2q) for every a < 2^64 (V. Shoup, NTL; D. Harvey, "Faster arithmetic
//    for number-theoretic transforms", J. Symb. Comp. 2014, which also gives
//    the lazy butterflies used by the NTT);
//  * Barrett reduction (P. Barrett 1986) of a 128-bit value x < 2^(2b+3),
//    b = bitlength(q): t = floor(x / 2^(b-2)), mu = floor(2^(2b+4) / q),
//    qhat = floor(t mu / 2^(b+6)) satisfies x/q - 2 < qhat <= x/q, so
//    x - qhat q lies in [0, 3q).  That bound admits sums of up to eight
//    products of canonical residues before one reduction.
// Every function is __host__ __device__ so the library's CPU self-test checks
// the very code the kernels run.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define FHE_HD __host__ __device__ __forceinline__
#else
#define FHE_HD inline
#endif

typedef uint64_t u64;
typedef unsigned __int128 u128;

FHE_HD u64 fhe_mulhi(u64 a, u64 b)
{
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (u64)(((u128)a * b) >> 64);
#endif
}

// 32 x 32 -> 64 products as single wide multiplications.  Sums of them are
// written with two products a statement, which become three-input additions
// on the addition pipe; a C product added to one accumulator at a time puts
// half of its 64-bit addition on the multiplier pipe (register-resident
// probes: conversions 531 -> 814 G residues/s, half-word products 6.3 -> 8.5
// T/s).
FHE_HD u64 wide_mul(uint32_t a, uint32_t b)
{
#ifdef __CUDA_ARCH__
    u64 p;
    asm("mul.wide.u32 %0, %1, %2;" : "=l"(p) : "r"(a), "r"(b));
    return p;
#else
    return (u64)a * b;
#endif
}
FHE_HD int64_t wide_mul_s(int32_t a, int32_t b)
{
#ifdef __CUDA_ARCH__
    int64_t p;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(p) : "r"(a), "r"(b));
    return p;
#else
    return (int64_t)a * b;
#endif
}

// Per-prime constants used by the kernels.
struct ModQ {
    u64 q;       // the prime
    u64 q2;      // 2q
    u64 mu;      // floor(2^(2b+4) / q) * 2^(58-b): Barrett constant, pre-shifted
    int bshift;  // b - 2, the shift that forms t
    int half;    // ceil(b / 2): the width of a half word (see HalfAcc)
    u64 mu64;    // floor(2^64 / q)
    uint32_t hlo, hhi;  // q = hhi 2^half + hlo
    uint32_t hninv;     // -q^-1 mod 2^half
    uint32_t qmu;       // floor(2^(32 + qsh) / q): quotients below 2^11 (see reduce_few)
    int qsh;            // b - 20 (0 for b <= 20)
    int32_t qinv;       // q^-1 mod 2^32
    int32_t nql, nqh;   // -q = nqh 2^32 + nql, nql signed
};

// a * w mod q in [0, 2q), w < q, ws = floor(w 2^64 / q), any a < 2^64.
FHE_HD u64 shoup_lazy(u64 a, u64 w, u64 ws, u64 q) { return a * w - fhe_mulhi(a, ws) * q; }

// Shoup's product with a cheaper quotient (the NTT butterflies' form): with
// a = ah 2^32 + al and ws = wh 2^32 + wl, floor(a ws / 2^64) = ah wh +
// floor((ah wl + al wh) / 2^32 + al wl / 2^64), and the estimate
// ah wh + floor(ah wl / 2^32) + floor(al wh / 2^32) drops three fractions
// below 1 each, so it is 0, 1 or 2 below the exact quotient.  Shoup's bound
// a w - floor(a ws / 2^64) q in [0, 2q) then gives a w - qhat q in [0, 4q),
// for any a < 2^64; the difference fits in 64 bits, so the arithmetic mod
// 2^64 is exact.  One 32x32->64 and two 32x32->hi products instead of the
// four 32x32->64 products (and their carries) of the exact high half.
//
// On the device the product is one multiply-add chain: with nq = 2^64 - q,
// a w - qhat q = a w + qhat nq (mod 2^64), so the low words of a w and of
// qhat nq are summed by a wide multiply-add and the high word by four 32-bit
// multiply-adds, with no separate 64-bit subtraction; the two high partial
// products of the quotient are summed by a wide multiply-add too (t1 * 1 +
// t2), so the whole product runs on the multiply-add pipe.
FHE_HD u64 shoup_lazy4_chain(u64 a, u64 w, u64 ws, u64 nq)
{
#ifdef __CUDA_ARCH__
    u64 r;
    asm("{\n\t"
        ".reg .u32 al, ah, wl, wh, sl, sh, ql, qh, t1, t2, hl, hh, rl, rh;\n\t"
        ".reg .u64 qhat, t12, lo, t2w;\n\t"
        "mov.b64 {al, ah}, %1;\n\t"
        "mov.b64 {wl, wh}, %2;\n\t"
        "mov.b64 {sl, sh}, %3;\n\t"
        "mov.b64 {ql, qh}, %4;\n\t"
        "mul.hi.u32 t1, ah, sl;\n\t"
        "mul.hi.u32 t2, al, sh;\n\t"
        "cvt.u64.u32 t2w, t2;\n\t"
        "mad.wide.u32 t12, t1, 1, t2w;\n\t"
        "mad.wide.u32 qhat, ah, sh, t12;\n\t"
        "mov.b64 {hl, hh}, qhat;\n\t"
        "mul.wide.u32 lo, al, wl;\n\t"
        "mad.wide.u32 lo, hl, ql, lo;\n\t"
        "mov.b64 {rl, rh}, lo;\n\t"
        "mad.lo.u32 rh, ah, wl, rh;\n\t"
        "mad.lo.u32 rh, al, wh, rh;\n\t"
        "mad.lo.u32 rh, hh, ql, rh;\n\t"
        "mad.lo.u32 rh, hl, qh, rh;\n\t"
        "mov.b64 %0, {rl, rh};\n\t"
        "}"
        : "=l"(r)
        : "l"(a), "l"(w), "l"(ws), "l"(nq));
    return r;
#else
    const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32), wl = (uint32_t)ws, wh = (uint32_t)(ws >> 32);
    const u64 qhat = (u64)ah * wh + ((((u64)ah * wl) >> 32) + (((u64)al * wh) >> 32));
    return a * w + qhat * nq;
#endif
}

FHE_HD u64 shoup(u64 a, u64 w, u64 ws, u64 q)
{
    u64 r = shoup_lazy(a, w, ws, q);
    return r >= q ? r - q : r;
}

// Canonical residue of x < 2^(2b+3).
FHE_HD u64 barrett128(u128 x, const ModQ &m)
{
    u64 lo = (u64)x, hi = (u64)(x >> 64);
    int s = m.bshift;                                   // 1 <= s <= 56
    u64 t = (hi << (64 - s)) | (lo >> s);               // floor(x / 2^(b-2)) < 2^(b+5)
    u64 qhat = fhe_mulhi(t, m.mu);                      // floor(t mu / 2^(b+6))
    u64 r = lo - qhat * m.q;                            // in [0, 3q)
    if (r >= m.q2) r -= m.q2;
    if (r >= m.q) r -= m.q;
    return r;
}

FHE_HD u64 mulmod(u64 a, u64 b, const ModQ &m) { return barrett128((u128)a * b, m); }

FHE_HD u64 addmod(u64 a, u64 b, u64 q)
{
    u64 r = a + b;
    return r >= q ? r - q : r;
}

FHE_HD u64 submod(u64 a, u64 b, u64 q) { return a >= b ? a - b : a + q - b; }

FHE_HD u64 negmod(u64 a, u64 q) { return a ? q - a : 0; }

// Any v < 2^64 -> [0, q): v - floor(v mu64 / 2^64) q lies in [0, 2q).
FHE_HD u64 reduce64(u64 v, const ModQ &m)
{
    const u64 r = v - fhe_mulhi(v, m.mu64) * m.q;
    return r >= m.q ? r - m.q : r;
}

// ---- sums with small centred scalars, in 64 bits -----------------------------
// sum_j k_j a_j mod q for canonical a_j without 128-bit arithmetic, where
// q sum |k_j| < 2^64 (small_fits); reduce64 then gives [0, q).  Term by term:
// a k = (q - a) |k| (mod q) for k < 0, and every term (q - a or a) |k| is at
// most q |k|.  Or all products mod 2^64 on top of q times the negative
// scalars' sum of |k|: the total is the same non-negative number.
FHE_HD bool small_fits(u64 qmax, u128 ksum) { return ksum * qmax < ((u128)1 << 64); }
FHE_HD u64 small_scaled(u64 a, int64_t k, u64 q) { return (k < 0 ? q - a : a) * (u64)(k < 0 ? -k : k); }
FHE_HD u64 small_start(u64 q, uint32_t neg) { return q * neg; }
FHE_HD u64 small_add(u64 acc, u64 a, int32_t k) { return acc + a * (u64)(int64_t)k; }

// x < 2^11 q -> [0, (1 + 2^-12 x/q) q + 1], below 2q: the quotient estimate
// qhat = floor(floor(x / 2^qsh) qmu / 2^32) never exceeds floor(x / q), and
// qmu >= 2^12 keeps it above x/q (1 - 2^-12) - 2^-19 - 1.  One 32-bit high
// product in place of reduce64's 64-bit one.
FHE_HD u64 reduce_few(u64 x, const ModQ &m)
{
    const uint32_t xs = (uint32_t)(x >> m.qsh);
#ifdef __CUDA_ARCH__
    const uint32_t qhat = __umulhi(xs, m.qmu);
#else
    const uint32_t qhat = (uint32_t)(((u64)xs * m.qmu) >> 32);
#endif
    return x - (u64)qhat * m.q;
}

// ---- half words -----------------------------------------------------------
// Residues of b bits as two halves of h = ceil(b/2) <= 29 bits.  A product's
// low, high and cross terms are summed over up to eight products in three
// 64-bit words, with no carry between them; the cross terms come from one
// product of the halves' sums (A. Karatsuba 1962: (xl + xh)(yl + yh) - xl yl
// - xh yh, the two subtractions once per sum; eight products of h + 1 bits
// stay below 2^63), so a product is three wide multiplications.  The
// multiplier pipe is what bounds these kernels: a 32 x 32 -> 64 product
// takes two of its slots, a 128-bit multiply-add four such products.
// One factor is kept as a constant times 2^(2h) mod q (half_const), and
// half_mont divides the sum by 2^(2h) again (P. Montgomery, Math. Comp. 1985,
// with two digits of h bits): it adds the multiples of q that clear the low
// and then the middle word.
struct HalfAcc {
    u64 lo, mid, hi;  // mid: the products of the halves' sums
};

// the two halves of x in the two 32-bit words of the result
FHE_HD u64 half_pack(u64 x, int h) { return ((x >> h) << 32) | (x & (((u64)1 << h) - 1)); }

// one factor's halves and their sum
struct Halves {
    uint32_t l, h, s;
};
FHE_HD Halves halves(uint32_t l, uint32_t h) { return Halves{l, h, l + h}; }
FHE_HD Halves halves_of(u64 packed) { return halves((uint32_t)packed, (uint32_t)(packed >> 32)); }

// acc += x y
FHE_HD void half_mac(HalfAcc &a, const Halves &x, const Halves &y)
{
    a.lo += wide_mul(x.l, y.l);
    a.hi += wide_mul(x.h, y.h);
    a.mid += wide_mul(x.s, y.s);
}

// acc += x y + u v
FHE_HD void half_mac2(HalfAcc &a, const Halves &x, const Halves &y, const Halves &u, const Halves &v)
{
    a.lo = a.lo + wide_mul(x.l, y.l) + wide_mul(u.l, v.l);
    a.hi = a.hi + wide_mul(x.h, y.h) + wide_mul(u.h, v.h);
    a.mid = a.mid + wide_mul(x.s, y.s) + wide_mul(u.s, v.s);
}

// The sum S of n <= 8 products of canonical residues, divided by 2^(2h):
// a residue below S / 2^(2h) + q <= (n + 1) q.
FHE_HD u64 half_mont(HalfAcc a, const ModQ &m)
{
    const uint32_t mask = ((uint32_t)1 << m.half) - 1;
    a.mid -= a.lo + a.hi;
    const uint32_t t0 = ((uint32_t)a.lo * m.hninv) & mask;
    a.lo += (u64)t0 * m.hlo;
    a.mid += (u64)t0 * m.hhi;
    a.mid += a.lo >> m.half;
    const uint32_t t1 = ((uint32_t)a.mid * m.hninv) & mask;
    a.mid += (u64)t1 * m.hlo;
    a.hi += (u64)t1 * m.hhi;
    return a.hi + (a.mid >> m.half);
}

// ---- sums of constant products ----------------------------------------------
// sum_i x_i c_i mod q for constants c_i: x = xh 2^h + xl (half words), so
// x c = xl c + xh (c 2^h mod q), and with both factors kept as the centred
// residues w of c 2^32 and v of c 2^(32 + h) the sum S = sum xl w + xh v is
// below n 2^h q in size -- 32 bits above q, which one 32-bit Montgomery step
// (P. Montgomery 1985, signed) removes: t = S q^-1 mod 2^32 in [-2^31, 2^31),
// (S - t q) / 2^32 = sum x_i c_i (mod q).  w and v are split into a signed low
// and a high word, so each x_i takes four wide multiply-adds into two 64-bit
// sums, without carries.
//
// Ranges: |low sum| <= 2^31 (sum xl + xh), plus 2^62 for t q's low word, stays
// below 2^63 while sum (xl + xh) <= 2^31: eight canonical residues up to 54
// bits, four at 56, two at 57 (dot_fold may be applied in between: its result
// is the next sum's high word).  The result lies within
// q/2 + 2^-33 q sum (xl + xh) of 0.
struct DotC {
    int32_t wl, wh, vl, vh;
};

struct DotAcc {
    int64_t l, h;
};

// x in half words: xl = x mod 2^h, xh = x >> h, below 2^31 each
FHE_HD void dot_mac(DotAcc &a, uint32_t xl, uint32_t xh, const DotC &c)
{
    a.l = a.l + wide_mul_s((int32_t)xl, c.wl) + wide_mul_s((int32_t)xh, c.vl);
    a.h = a.h + wide_mul_s((int32_t)xl, c.wh) + wide_mul_s((int32_t)xh, c.vh);
}

FHE_HD void dot_mac(DotAcc &a, u64 x, const DotC &c, int h)
{
    dot_mac(a, (uint32_t)x & (((uint32_t)1 << h) - 1), (uint32_t)(x >> h), c);
}

FHE_HD int64_t dot_fold(const DotAcc &a, const ModQ &m)
{
    const int32_t t = (int32_t)((uint32_t)a.l * (uint32_t)m.qinv);
    const int64_t c = a.l + (int64_t)t * m.nql;  // a multiple of 2^32
    return a.h + (int64_t)t * m.nqh + (c >> 32);
}

// (-q, q) -> [0, q)
FHE_HD u64 centred_mod(int64_t v, u64 q) { return (u64)(v + (int64_t)((u64)(v >> 63) & q)); }

// [0, 2q) -> [0, q)
FHE_HD u64 reduce2q(u64 a, u64 q) { return a >= q ? a - q : a; }

// [0, 4q) -> [0, q)
FHE_HD u64 reduce4q(u64 a, u64 q2, u64 q)
{
    if (a >= q2) a -= q2;
    return a >= q ? a - q : a;
}

// Host-side constructors.
inline ModQ make_modq(u64 q)
{
    ModQ m;
    int b = 0;
    while (b < 64 && (q >> b)) b++;
    m.q = q;
    m.q2 = 2 * q;
    u128 mu = ((u128)1 << (2 * b + 4)) / q;             // < 2^(b+5)
    m.mu = (u64)(mu << (58 - b));
    m.bshift = b - 2;
    m.mu64 = (u64)((((u128)1) << 64) / q);
    m.half = (b + 1) / 2;
    const uint32_t mask = ((uint32_t)1 << m.half) - 1;
    m.hlo = (uint32_t)q & mask;
    m.hhi = (uint32_t)(q >> m.half);
    uint32_t inv = 1;                                   // q^-1 mod 2^32 by Newton's iteration
    for (int i = 0; i < 5; i++) inv *= 2 - (uint32_t)q * inv;
    m.hninv = (0 - inv) & mask;
    m.qsh = b > 20 ? b - 20 : 0;
    m.qmu = (uint32_t)((((u128)1) << (32 + m.qsh)) / q);
    m.qinv = (int32_t)inv;
    m.nql = (int32_t)(0 - (uint32_t)q);
    m.nqh = (int32_t)((-(int64_t)q - m.nql) >> 32);
    return m;
}

// c 2^(2h) mod q, packed: the constant factor of half_mac
inline u64 half_const(u64 c, const ModQ &m)
{
    return half_pack((u64)((((u128)c << (2 * m.half)) % m.q)), m.half);
}

inline DotC dot_const(u64 c, const ModQ &m)
{
    auto centred = [&m](u64 x) { return x > m.q / 2 ? (int64_t)x - (int64_t)m.q : (int64_t)x; };
    const int64_t w = centred((u64)((((u128)c) << 32) % m.q));
    const int64_t v = centred((u64)((((u128)c % m.q) << (32 + m.half)) % m.q));
    DotC d;
    d.wl = (int32_t)(uint32_t)w;
    d.wh = (int32_t)((w - d.wl) >> 32);
    d.vl = (int32_t)(uint32_t)v;
    d.vh = (int32_t)((v - d.vl) >> 32);
    return d;
}

inline u64 shoup_const(u64 w, u64 q) { return (u64)(((u128)w << 64) / q); }
