// hc_arith.cuh -- uint64 modular arithmetic on the integer pipes, built from
// 32-bit partial products.
//
// Residues live in 64-bit words with q < 2^50, leaving 14 bits of head room:
// butterflies run lazily and reductions happen once, at the end.
//
// Cost model (measured on GB300): a 32x32->64 multiply-add (mad.wide.u32)
// issues at the same rate as a 32-bit multiply-add, while the high half
// alone (mad.hi.u32) costs twice as much, and the compiler's 64-bit mul.lo /
// mul.hi cost about 4 and 8 multiply-adds.  So every product below is formed
// from wide 32-bit multiply-adds, and high halves are taken from the wide
// results instead of being computed separately.
//
// Shoup multiplication (V. Shoup; D. Harvey, "Faster arithmetic for
// number-theoretic transforms", JSC 2014): for a constant w < q with
// companion w' = floor(w * 2^64 / q) and any y < 2^64,
//     y*w - floor(y*w' / 2^64) * q   lies in [0, 2q).
// shoup_lazy drops the lowest partial product y_lo*w'_lo and the carry of
// the two middle ones from the quotient, which makes the quotient at most 2
// too small: the result is congruent to y*w and lies in [0, 4q).
#pragma once

#include <cstdint>

namespace hc {

// y*w mod q, lazily: result in [0, 4q) for any y < 2^64, w < q < 2^62,
// wp = floor(w*2^64/q), nq = 2^64 - q.
__device__ __forceinline__ uint64_t shoup_lazy(uint64_t y, uint64_t w, uint64_t wp, uint64_t nq)
{
    uint64_t r;
    asm("{\n\t"
        ".reg .u32 yl, yh, wl, wh, pl, ph, nl, nh, al, ah, bl, bh, ql, qh, rl, rh, h, c;\n\t"
        ".reg .u64 a, b, t;\n\t"
        "mov.b64 {yl, yh}, %1;\n\t"
        "mov.b64 {wl, wh}, %2;\n\t"
        "mov.b64 {pl, ph}, %3;\n\t"
        "mov.b64 {nl, nh}, %4;\n\t"
        "mul.wide.u32 a, yh, pl;\n\t"
        "mul.wide.u32 b, yl, ph;\n\t"
        "mov.b64 {al, ah}, a;\n\t"
        "mov.b64 {bl, bh}, b;\n\t"
        "add.cc.u32 al, ah, bh;\n\t"       // hi(a) + hi(b): 33 bits
        "addc.u32 c, 0, 0;\n\t"
        "mov.b64 t, {al, c};\n\t"
        "mad.wide.u32 t, yh, ph, t;\n\t"   // quotient estimate Q
        "mov.b64 {ql, qh}, t;\n\t"
        "mul.wide.u32 a, yl, wl;\n\t"      // low 64 bits of y*w + Q*nq
        "mad.wide.u32 a, ql, nl, a;\n\t"
        "mul.lo.u32 h, yl, wh;\n\t"
        "mad.lo.u32 h, yh, wl, h;\n\t"
        "mad.lo.u32 h, ql, nh, h;\n\t"
        "mad.lo.u32 h, qh, nl, h;\n\t"
        "mov.b64 {rl, rh}, a;\n\t"
        "add.u32 rh, rh, h;\n\t"
        "mov.b64 %0, {rl, rh};\n\t"
        "}"
        : "=l"(r)
        : "l"(y), "l"(w), "l"(wp), "l"(nq));
    return r;
}

// y mod q, lazily: result in [0, 3q) for any y < 2^64.  ones = floor(2^64/q)
// (< 2^32 since q > 2^32); the quotient floor(y_hi * ones / 2^32) is at most
// one below floor(y * ones / 2^64).
__device__ __forceinline__ uint64_t reduce_lazy(uint64_t y, uint32_t ones, uint64_t nq)
{
    uint64_t r;
    asm("{\n\t"
        ".reg .u32 yl, yh, nl, nh, ql, qh, rl, rh, h;\n\t"
        ".reg .u64 a;\n\t"
        "mov.b64 {yl, yh}, %1;\n\t"
        "mov.b64 {nl, nh}, %3;\n\t"
        "mul.wide.u32 a, yh, %2;\n\t"
        "mov.b64 {ql, qh}, a;\n\t"          // Q = qh
        "mad.wide.u32 a, qh, nl, %1;\n\t"   // y + Q*nq (low 64 bits)
        "mul.lo.u32 h, qh, nh;\n\t"
        "mov.b64 {rl, rh}, a;\n\t"
        "add.u32 rh, rh, h;\n\t"
        "mov.b64 %0, {rl, rh};\n\t"
        "}"
        : "=l"(r)
        : "l"(y), "r"(ones), "l"(nq));
    return r;
}

__device__ __forceinline__ uint64_t csub(uint64_t x, uint64_t m)
{
    return x >= m ? x - m : x;
}

// canonical residue of x < 3q
__device__ __forceinline__ uint64_t canon3(uint64_t x, uint64_t q)
{
    return csub(csub(x, 2 * q), q);
}

// canonical residue of x < 4q
__device__ __forceinline__ uint64_t canon4(uint64_t x, uint64_t q)
{
    return csub(csub(x, 2 * q), q);
}

// ---- twiddle products ---------------------------------------------------------------
// TwArith<false>: any q, unsigned lazy values, Shoup products (twiddle = {w, w'}).
//
// TwArith<true>: q = 2^50 - c with 0 < c < 2^22 (LimbConst::special_c), signed lazy
// values, folded products.  The constant w < q is kept as two residues, w and
// v = w * 2^32 mod q, each cut at 2^20 (fold_twiddle).  With y = yl + 2^32 yh (yl
// unsigned, yh signed),
//     y*w = yl*w + yh*v = lo + 2^20 mid    (mod q),
//     lo = yl*wl + yh*vl,  mid = yl*wh + yh*vh,
// and, because 2^52 = 4c (mod q), mid's high word folds down as it stands:
//     t = lo + 2^20 lo32(mid) + 4c hi32(mid).
// For every signed 64-bit y: -2^51 <= lo < 2^52 + 2^51 and -2^61 <= mid < 2^62 + 2^61,
// so -10 * 2^50 <= t < 34 * 2^50, i.e. |t| <= kFoldMax q.  Six wide multiply-adds and
// no other instruction: the cut at 2^20 puts the fold at 2^52 on a word boundary of
// mid, so nothing is shifted, masked or carried, and signed values need no multiple of
// q added to a difference (two more instructions on the same pipes per butterfly).
// Bound by the multiply pipe (24 of its cycles per warp).  Measured on GB300, a
// radix-32 round in registers at 16 warps per SM: 28.6 cycles per warp butterfly and SM
// sub-partition, 33.5 with unsigned values, 41.6 with Shoup products (5 wide and 4
// narrow multiply-adds, 5 additions and moves).
constexpr uint64_t kFoldMax = 35;
// The most, in multiples of q, that a folded inverse stage's inputs may reach: their sums and
// differences are below 8190 q < 2^63 - 2^50, which leaves div_canon's k c < 2^36 room.
constexpr uint64_t kFoldStage = 4095;

template <bool SP>
struct TwArith;

template <>
struct TwArith<false> {
    uint64_t q, nq;
    uint32_t ones;  // floor(2^64 / q)
    __device__ __forceinline__ TwArith(uint64_t q_, uint64_t, uint64_t one_s)
        : q(q_), nq(0ull - q_), ones((uint32_t)one_s)
    {
    }
    // y*w mod q, < 4q
    __device__ __forceinline__ uint64_t mul(uint64_t y, ulonglong2 w) const { return shoup_lazy(y, w.x, w.y, nq); }
    __device__ __forceinline__ uint64_t mul_canon(uint64_t y, ulonglong2 w) const { return canon4(mul(y, w), q); }
    // canonical y / 2^LOGN, wn = 2^-LOGN
    template <int LOGN>
    __device__ __forceinline__ uint64_t div_canon(uint64_t y, ulonglong2 wn) const { return mul_canon(y, wn); }
    // x - y for a product y, and for y <= b
    __device__ __forceinline__ uint64_t sub(uint64_t x, uint64_t y) const { return x - y + 4 * q; }
    __device__ __forceinline__ uint64_t sub(uint64_t x, uint64_t y, uint64_t b) const { return x - y + b; }
    // canonical residue of any x < 2^64
    __device__ __forceinline__ uint64_t canon(uint64_t x) const { return canon3(reduce_lazy(x, ones, nq), q); }
};

template <>
struct TwArith<true> {
    uint64_t q;
    uint32_t c, c4, p20;
    __device__ __forceinline__ TwArith(uint64_t q_, uint64_t c_, uint64_t)
        : q(q_), c((uint32_t)c_), c4(4 * (uint32_t)c_)
    {
        // 2^20 as a register the compiler does not see through: a visible power of two
        // becomes shifts and carries, five instructions for one
        asm("mov.u32 %0, 0x100000;" : "=r"(p20));
    }
    // y*w + add mod q for any signed y, |result - add| <= kFoldMax q.  Each lo / hi pair
    // is one wide multiply-add, written by halves because the compiler gives
    // mad.wide.u32's result a fresh register pair and moves it back (2 moves a product).
    __device__ __forceinline__ uint64_t mul(uint64_t y, ulonglong2 w, uint64_t add = 0) const
    {
        uint64_t t;
        asm("{\n\t"
            ".reg .u32 yl, yh, wl, wh, vl, vh, ml, mh, ll, lh;\n\t"
            "mov.b64 {yl, yh}, %1;\n\t"
            "mov.b64 {wl, wh}, %2;\n\t"
            "mov.b64 {vl, vh}, %3;\n\t"
            "mov.b64 {ll, lh}, %6;\n\t"
            "mul.lo.u32 ml, yl, wh;\n\t"        // mid
            "mul.hi.u32 mh, yl, wh;\n\t"
            "mad.lo.cc.s32 ml, yh, vh, ml;\n\t"
            "madc.hi.s32 mh, yh, vh, mh;\n\t"
            "mad.lo.cc.u32 ll, yl, wl, ll;\n\t" // lo
            "madc.hi.u32 lh, yl, wl, lh;\n\t"
            "mad.lo.cc.s32 ll, yh, vl, ll;\n\t"
            "madc.hi.s32 lh, yh, vl, lh;\n\t"
            "mad.lo.cc.u32 ll, ml, %5, ll;\n\t"
            "madc.hi.u32 lh, ml, %5, lh;\n\t"
            "mad.lo.cc.s32 ll, mh, %4, ll;\n\t"
            "madc.hi.s32 lh, mh, %4, lh;\n\t"
            "mov.b64 %0, {ll, lh};\n\t"
            "}"
            : "=l"(t)
            : "l"(y), "l"(w.x), "l"(w.y), "r"(c4), "r"(p20), "l"(add));
        return t;
    }
    __device__ __forceinline__ uint64_t mul_canon(uint64_t y, ulonglong2 w) const
    {
        return canon_pos(mul(y, w, 16 * q));  // -10 * 2^50 + 16 q > 0
    }
    // canonical y / 2^LOGN for 2^LOGN | q - 1 and |y| <= 2 kFoldStage q.  Then c = -1 mod 2^LOGN, so
    // with k = -y mod 2^LOGN the sum y + k q = (y - k c) + 2^50 k is a multiple of 2^LOGN
    // in both terms: one wide product in place of the six of a product with N^-1.
    // |(y - k c) / 2^LOGN| <= 2^51 + 2^23 for LOGN >= 12, hence 4 q to make it positive.
    // Inverse transforms on GB300: 2048 limbs at N = 16384 275 -> 268 us, 4096 limbs at
    // N = 4096 98.6 -> 97.4; at N = 8192, in 128 registers with 32 residues, 1536 limbs
    // 93.3 -> 96.1, so there the product with N^-1 stays.
    template <int LOGN>
    __device__ __forceinline__ uint64_t div_canon(uint64_t y, ulonglong2 wn) const
    {
        static_assert(LOGN >= 12 && LOGN <= 15, "ring degrees");
        if constexpr (LOGN == 13) return mul_canon(y, wn);
        const uint32_t k = (0u - (uint32_t)y) & ((1u << LOGN) - 1);
        uint64_t t;
        asm("{\n\t"
            ".reg .u32 l, h;\n\t"
            "mov.b64 {l, h}, %1;\n\t"
            "mad.lo.cc.s32 l, %2, %3, l;\n\t"
            "madc.hi.s32 h, %2, %3, h;\n\t"
            "mov.b64 %0, {l, h};\n\t"
            "}"
            : "=l"(t)
            : "l"(y), "r"(k), "r"(0u - c));
        return canon_pos((uint64_t)((int64_t)t >> LOGN) + ((uint64_t)k << (50 - LOGN)) + 4 * q);
    }
    __device__ __forceinline__ uint64_t sub(uint64_t x, uint64_t y, uint64_t = 0) const { return x - y; }
    // a value congruent to x, > -2^36 and < 2^52 + 2^36 (< 5 q), for any signed x
    __device__ __forceinline__ uint64_t fold(uint64_t x) const
    {
        const int64_t h = (int32_t)(x >> 32) >> 20;  // x >> 52
        return (x & ((1ull << 52) - 1)) + (uint64_t)(h * (int64_t)c4);
    }
    // canonical residue of x >= 0: the fold at 2^50 leaves less than 2^50 + 2^36 < 2 q
    __device__ __forceinline__ uint64_t canon_pos(uint64_t x) const
    {
        return csub((x & ((1ull << 50) - 1)) + (uint64_t)(uint32_t)(x >> 50) * c, q);
    }
    // canonical residue of any x, |x| <= 2047 q
    __device__ __forceinline__ uint64_t canon(uint64_t x) const { return canon_pos(x + 2048 * q); }
};

// Multiply-accumulate of products x*w with x < 2^56, w < 2^50, as three
// partial sums of 32x32 products:
//   V = s0 + 2^64 c0 + 2^32 s1 + 2^64 s2,
//   s0 = sum xl*wl (carries counted in c0), s1 = sum xl*wh + xh*wl, s2 = sum xh*wh.
// s1, s2 cannot overflow for fewer than 2^7 terms with x < 2^56 (2^13 with x < 2^50).
struct MacAcc {
    uint64_t s0, s1, s2;
    uint32_t c0;
};

__device__ __forceinline__ void mac_zero(MacAcc &a)
{
    a.s0 = a.s1 = a.s2 = 0;
    a.c0 = 0;
}

__device__ __forceinline__ void mac_add(MacAcc &a, uint64_t x, uint64_t w)
{
    asm("{\n\t"
        ".reg .u32 xl, xh, wl, wh;\n\t"
        ".reg .u64 p;\n\t"
        "mov.b64 {xl, xh}, %4;\n\t"
        "mov.b64 {wl, wh}, %5;\n\t"
        "mul.wide.u32 p, xl, wl;\n\t"
        "add.cc.u64 %0, %0, p;\n\t"
        "addc.u32 %3, %3, 0;\n\t"
        "mad.wide.u32 %1, xl, wh, %1;\n\t"
        "mad.wide.u32 %1, xh, wl, %1;\n\t"
        "mad.wide.u32 %2, xh, wh, %2;\n\t"
        "}"
        : "+l"(a.s0), "+l"(a.s1), "+l"(a.s2), "+r"(a.c0)
        : "l"(x), "l"(w));
}

// V = lo + 2^64 hi of an accumulator: lo = s0 + 2^32 lo32(s1), hi = c0 + s2 + hi32(s1) + carry
__device__ __forceinline__ void mac_value(const MacAcc &a, uint64_t &lo, uint64_t &hi)
{
    asm("{\n\t"
        ".reg .u32 sl, sh, l0, l1, h0;\n\t"
        ".reg .u64 t;\n\t"
        "mov.b64 {sl, sh}, %3;\n\t"
        "mov.b64 {l0, l1}, %2;\n\t"
        "add.cc.u32 l1, l1, sl;\n\t"
        "addc.u32 h0, %5, sh;\n\t"          // c0 + hi32(s1) + carry (< 2^32)
        "mov.b64 %0, {l0, l1};\n\t"
        "cvt.u64.u32 t, h0;\n\t"
        "add.u64 %1, %4, t;\n\t"
        "}"
        : "=l"(lo), "=l"(hi)
        : "l"(a.s0), "l"(a.s1), "l"(a.s2), "r"(a.c0));
}

// canonical (lo + 2^64 hi) mod q for any hi < 2^64.  r64 = 2^64 mod q with companion r64_s.
__device__ __forceinline__ uint64_t reduce128(uint64_t lo, uint64_t hi, uint64_t q, uint64_t nq, uint64_t r64,
                                              uint64_t r64_s, uint32_t ones)
{
    const uint64_t x = shoup_lazy(hi, r64, r64_s, nq);  // < 4q
    const uint64_t y = reduce_lazy(lo, ones, nq);        // < 3q
    uint64_t s = x + y;                                  // < 7q
    s = csub(s, 4 * q);
    return canon4(s, q);
}

// canonical V mod q
__device__ __forceinline__ uint64_t mac_reduce(const MacAcc &a, uint64_t q, uint64_t nq, uint64_t r64,
                                               uint64_t r64_s, uint32_t ones)
{
    uint64_t lo, hi;
    mac_value(a, lo, hi);
    return reduce128(lo, hi, q, nq, r64, r64_s, ones);
}

// canonical V = lo + 2^64 hi mod q for q = 2^50 - c with 0 < c < 2^22, V < 2^104 (at most 16
// terms of products of residues below 2^50): with A = V >> 50 and
// B = V mod 2^50, V = A*2^50 + B = A*c + B (mod q); folding A*c (< 2^76) once
// more the same way leaves B + B2 + A2*c < 2.25 * 2^50 < 3q.  Three wide
// 32-bit products instead of the generic reduction's Shoup step.
__device__ __forceinline__ uint64_t reduce128_special(uint64_t lo, uint64_t hi, uint64_t q, uint32_t c)
{
    constexpr uint64_t M50 = (1ull << 50) - 1;
    const uint64_t A = (hi << 14) | (lo >> 50);  // < 2^54
    const uint64_t B = lo & M50;
    const uint64_t p0 = (uint64_t)(uint32_t)A * c;          // < 2^54
    const uint64_t p1 = (uint64_t)(uint32_t)(A >> 32) * c;  // < 2^44
    const uint64_t plo = p0 + (p1 << 32);
    const uint64_t phi = (p1 >> 32) + (plo < p0 ? 1 : 0);
    const uint64_t A2 = (phi << 14) | (plo >> 50);          // < 2^26
    const uint64_t r = B + (plo & M50) + (uint64_t)(uint32_t)A2 * c;
    return canon3(r, q);
}

__device__ __forceinline__ uint64_t mac_reduce_special(const MacAcc &a, uint64_t q, uint32_t c)
{
    uint64_t lo, hi;
    mac_value(a, lo, hi);
    return reduce128_special(lo, hi, q, c);
}

// ---- sums of products of canonical residues --------------------------------------------
// Residues below 2^50 cut at 2^25, x = x0 + 2^25 x1: a sum of products is
//   V = s0 + 2^25 (sm - s0 - s2) + 2^50 s2,
//   s0 = sum x0 w0,  s2 = sum x1 w1,  sm = sum (x0 + x1)(w0 + w1)      (Karatsuba 1962),
// three wide multiply-adds a product and, because the halves leave room, no carries:
// s0, s2 < G 2^50 and sm < G 2^52 fit 64 bits for G < 4096 terms.  MacAcc's cut at 2^32
// takes four and a carry chain.
struct MacAcc25 {
    uint64_t s0, s2, sm;
};
constexpr uint32_t kCut25 = (1u << 25) - 1;
constexpr uint32_t kMacSpecialTerms = 256;  // most terms mac25_reduce_special takes

__device__ __forceinline__ void mac25_zero(MacAcc25 &a) { a.s0 = a.s2 = a.sm = 0; }

// x = {x0, x1} in the low and high 32 bits
__device__ __forceinline__ uint64_t split25(uint64_t x)
{
    const uint32_t lo = (uint32_t)x, hi = (uint32_t)(x >> 32);
    return (uint64_t)(__funnelshift_r(lo, hi, 25)) << 32 | (lo & kCut25);
}

// a += b * c, in place: by halves, because the compiler gives mad.wide.u32's result a
// fresh register pair and moves it back
__device__ __forceinline__ void mad_wide(uint64_t &a, uint32_t b, uint32_t c)
{
    asm("{\n\t"
        ".reg .u32 l, h;\n\t"
        "mov.b64 {l, h}, %0;\n\t"
        "mad.lo.cc.u32 l, %1, %2, l;\n\t"
        "madc.hi.u32 h, %1, %2, h;\n\t"
        "mov.b64 %0, {l, h};\n\t"
        "}"
        : "+l"(a)
        : "r"(b), "r"(c));
}

// both operands split
__device__ __forceinline__ void mac25_add(MacAcc25 &a, uint64_t x, uint32_t xs, uint64_t w, uint32_t ws)
{
    mad_wide(a.s0, (uint32_t)x, (uint32_t)w);
    mad_wide(a.s2, (uint32_t)(x >> 32), (uint32_t)(w >> 32));
    mad_wide(a.sm, xs, ws);
}

// canonical V mod q, any q < 2^50
__device__ __forceinline__ uint64_t mac25_reduce(const MacAcc25 &a, uint64_t q, uint64_t nq, uint64_t r64,
                                                 uint64_t r64_s, uint32_t ones)
{
    const uint64_t s1 = a.sm - a.s0 - a.s2;
    const uint64_t t = a.s0 + (s1 << 25), lo = t + (a.s2 << 50);
    const uint64_t hi = (s1 >> 39) + (a.s2 >> 14) + (t < a.s0) + (lo < t);
    return reduce128(lo, hi, q, nq, r64, r64_s, ones);
}

// canonical V mod q for q = 2^50 - c, 0 < c < 2^22, at most 256 terms.  s0 < 2^58 and
// s1 < 2^59; with s1 = l + 2^25 h, V = s0 + 2^25 l + c (s2 + h) (mod q), and with
// s2 + h = tl + 2^28 th, th < 2^31, and u = c th = ul + 2^22 uh, 2^28 u = 2^28 ul + c uh:
//   V = s0 + 2^25 l + c tl + 2^28 ul + c uh < 2^58 + 2^54,
// whose fold at 2^50 leaves less than 2^50 + 2^31 < 2 q.  p25, p28: powers of two the
// compiler does not see through, for the shifted sums on the multiply pipe.
__device__ __forceinline__ uint64_t mac25_reduce_special(const MacAcc25 &a, uint64_t q, uint32_t c, uint32_t p25,
                                                         uint32_t p28)
{
    const uint64_t s1 = a.sm - a.s0 - a.s2;
    const uint64_t t = a.s2 + (s1 >> 25);
    const uint64_t u = (uint64_t)(uint32_t)(t >> 28) * c;
    uint64_t r = a.s0;
    mad_wide(r, (uint32_t)s1 & kCut25, p25);
    mad_wide(r, (uint32_t)t & ((1u << 28) - 1), c);
    mad_wide(r, (uint32_t)u & ((1u << 22) - 1), p28);
    mad_wide(r, (uint32_t)(u >> 22), c);
    uint64_t v = r & ((1ull << 50) - 1);
    mad_wide(v, (uint32_t)(r >> 50), c);
    return csub(v, q);
}

// canonical x*w mod q of a lazy forward-transform value x and a residue w < q.  The
// folded form's x (|x| < 2^60) is first brought into [0, 2^53), so that x*w < 2^104.
__device__ __forceinline__ uint64_t mul_slot(const TwArith<false> &ar, uint64_t x, uint64_t w, uint64_t r64,
                                             uint64_t r64_s)
{
    MacAcc a;
    mac_zero(a);
    mac_add(a, x, w);
    return mac_reduce(a, ar.q, ar.nq, r64, r64_s, ar.ones);
}
__device__ __forceinline__ uint64_t mul_slot(const TwArith<true> &ar, uint64_t x, uint64_t w, uint64_t, uint64_t)
{
    MacAcc a;
    mac_zero(a);
    mac_add(a, ar.fold(x + 2048 * ar.q), w);
    return mac_reduce_special(a, ar.q, ar.c);
}

}  // namespace hc
