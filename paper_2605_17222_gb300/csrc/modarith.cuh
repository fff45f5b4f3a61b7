// Modular arithmetic on uint64 RNS residues for sm_103a.
//
// The paper's PE modes (Sec. V: CM, CWPM, CM-ACC, CWPM-ACC, CWPA-CM) all reduce
// to three device primitives here:
//   * Shoup multiplication by a constant w with precomputed w' = floor(w 2^64 / q)
//     (twiddles, per-limb constants);
//   * a lazy 128-bit multiply-accumulate (mad.lo.cc / madc.hi), reduced once
//     at the end of an inner product;
//   * Barrett reduction of a 128-bit value with mu = floor(2^128 / q).
// Every modulus is below 2^60, so a product is below 2^120 and up to 256
// products fit one 128-bit accumulator.  Outputs are canonical in [0, q).
#pragma once
#include <cstdint>

typedef uint64_t u64;
typedef uint32_t u32;

struct ModC {
    u64 q;
    u64 mu_hi;  // floor(2^128 / q) >> 64
    u64 mu_lo;  // floor(2^128 / q) mod 2^64
    u64 mu_s;   // floor(2^(64 + bits - 1) / q), below 2^64
    // byte offset of the modulus's limb in a key, and in a diagonal among the Q
    // limbs (for a P limb: among the P limbs, which follow the Q limbs of the
    // diagonals' level)
    u64 koff, doff;
    u32 bits;  // bit length of q
    u32 pad;
};

struct U128 {
    u64 lo, hi;
};

__device__ __forceinline__ u64 add_mod(u64 a, u64 b, u64 q) {
    u64 s = a + b;
    return s >= q ? s - q : s;
}

__device__ __forceinline__ u64 sub_mod(u64 a, u64 b, u64 q) {
    return a >= b ? a - b : a + q - b;
}

// a * w mod q for w < q, wp = floor(w * 2^64 / q); valid for any a < 2^64 and q < 2^63.
__device__ __forceinline__ u64 mul_shoup(u64 a, u64 w, u64 wp, u64 q) {
    u64 t = __umul64hi(a, wp);
    u64 r = a * w - t * q;
    return r >= q ? r - q : r;
}

// acc += a * b.  The four 32x32 partial products are added into the four
// 32-bit words of the accumulator along explicit carry chains: ten 32-bit
// multiply-add instructions, cheaper than the 64-bit mad.lo/madc.hi forms.
// The caller keeps the 128-bit sum from overflowing.
__device__ __forceinline__ void mac128(U128& acc, u64 a, u64 b) {
    asm("{\n\t.reg .u32 a0, a1, a2, a3, x0, x1, y0, y1;\n\t"
        "mov.b64 {a0, a1}, %0;\n\t"
        "mov.b64 {a2, a3}, %1;\n\t"
        "mov.b64 {x0, x1}, %2;\n\t"
        "mov.b64 {y0, y1}, %3;\n\t"
        "mad.lo.cc.u32 a0, x0, y0, a0;\n\t"
        "madc.hi.cc.u32 a1, x0, y0, a1;\n\t"
        "madc.lo.cc.u32 a2, x1, y1, a2;\n\t"
        "madc.hi.u32 a3, x1, y1, a3;\n\t"
        "mad.lo.cc.u32 a1, x0, y1, a1;\n\t"
        "madc.hi.cc.u32 a2, x0, y1, a2;\n\t"
        "addc.u32 a3, a3, 0;\n\t"
        "mad.lo.cc.u32 a1, x1, y0, a1;\n\t"
        "madc.hi.cc.u32 a2, x1, y0, a2;\n\t"
        "addc.u32 a3, a3, 0;\n\t"
        "mov.b64 %0, {a0, a1};\n\t"
        "mov.b64 %1, {a2, a3};\n\t}"
        : "+l"(acc.lo), "+l"(acc.hi)
        : "l"(a), "l"(b));
}

// A 96-bit accumulator (low 64 bits, high 32 bits) for products of operands
// below 2^41.
struct U96 {
    u64 lo;
    u32 hi;
};

// acc += a * b for a, b < 2^41; the caller keeps the sum below 2^96.  With
// a = a1 2^32 + a0 and b = b1 2^32 + b0 (a1, b1 < 2^9), a1 b1 is below 2^18
// and the high halves of a0 b1 and a1 b0 below 2^9, so the top word takes
// them with no carry out of it: seven 32-bit multiply-adds along three short
// carry chains instead of mac128's ten.
__device__ __forceinline__ void mac96(U96& acc, u64 a, u64 b) {
    asm("{\n\t.reg .u32 w0, w1, x0, x1, y0, y1;\n\t"
        "mov.b64 {w0, w1}, %0;\n\t"
        "mov.b64 {x0, x1}, %2;\n\t"
        "mov.b64 {y0, y1}, %3;\n\t"
        "mad.lo.cc.u32 w0, x0, y0, w0;\n\t"
        "madc.hi.cc.u32 w1, x0, y0, w1;\n\t"
        "madc.lo.u32 %1, x1, y1, %1;\n\t"
        "mad.lo.cc.u32 w1, x0, y1, w1;\n\t"
        "madc.hi.u32 %1, x0, y1, %1;\n\t"
        "mad.lo.cc.u32 w1, x1, y0, w1;\n\t"
        "madc.hi.u32 %1, x1, y0, %1;\n\t"
        "mov.b64 %0, {w0, w1};\n\t}"
        : "+l"(acc.lo), "+r"(acc.hi)
        : "l"(a), "l"(b));
}

__device__ __forceinline__ void add128(U128& acc, u64 v) {
    asm("add.cc.u64 %0, %0, %2;\n\t"
        "addc.u64 %1, %1, 0;"
        : "+l"(acc.lo), "+l"(acc.hi)
        : "l"(v));
}

// x mod q for any 128-bit x (q < 2^62).  The quotient estimate
//   qe = x1*m1 + hi(x1*m0) + hi(x0*m1)            (mod 2^64)
// drops the low partial products, so it is below floor(x/q) by at most 3 and
// x - qe*q < 4q fits 64 bits.
__device__ __forceinline__ u64 reduce128_lazy(U128 x, const ModC& m) {  // x mod q up to 3q, in [0, 4q)
    const u64 qe = x.hi * m.mu_hi + __umul64hi(x.hi, m.mu_lo) + __umul64hi(x.lo, m.mu_hi);
    return x.lo - qe * m.q;
}
__device__ __forceinline__ u64 reduce128(U128 x, const ModC& m) {
    u64 r = reduce128_lazy(x, m);
    r = r >= 2 * m.q ? r - 2 * m.q : r;
    r = r >= m.q ? r - m.q : r;
    return r;
}

// x mod q up to 4q, in [0, 5q), for x = w3 w2 w1 w0 (32-bit words) below
// 2^(63 + bits): the quotient is estimated from x1 = floor(x / 2^(bits - 1)),
// which fits 64 bits, and mu_s.  Dropping the bits below x1 costs less than
// 1, mu_s's truncation less than 1, the low partial products at most 2 and the
// floor less than 1, so the estimate is at most 4 short.  Three 32-bit
// products for the estimate and three for the remainder, where
// reduce128_lazy's 128-bit product takes thirteen.
__device__ __forceinline__ u64 reduce_top(u32 w0, u32 w1, u32 w2, u32 w3, const ModC& m) {
    const u32 sh = m.bits - 1;
    const bool up = sh >= 32;
    const u32 a0 = up ? w1 : w0, a1 = up ? w2 : w1, a2 = up ? w3 : w2;
    const u32 x0 = __funnelshift_r(a0, a1, sh), x1 = __funnelshift_r(a1, a2, sh);  // shift modulo 32
    const u32 s0 = (u32)m.mu_s, s1 = (u32)(m.mu_s >> 32);
    u64 r;
    asm("{\n\t.reg .u32 n0, n1, e0, e1, t0, t1;\n\t.reg .u64 e, t;\n\t"
        "mov.b64 {n0, n1}, %7;\n\t"
        "mul.wide.u32 e, %2, %4;\n\tmov.b64 {e0, e1}, e;\n\t"
        "mad.hi.cc.u32 e0, %1, %4, e0;\n\taddc.u32 e1, e1, 0;\n\t"
        "mad.hi.cc.u32 e0, %2, %3, e0;\n\taddc.u32 e1, e1, 0;\n\t"
        "mov.b64 t, {%5, %6};\n\tmad.wide.u32 t, e0, n0, t;\n\tmov.b64 {t0, t1}, t;\n\t"
        "mad.lo.u32 t1, e0, n1, t1;\n\tmad.lo.u32 t1, e1, n0, t1;\n\t"
        "mov.b64 %0, {t0, t1};\n\t}" : "=l"(r) : "r"(x0), "r"(x1), "r"(s0), "r"(s1), "r"(w0), "r"(w1), "l"(0 - m.q));
    return r;
}

// x mod q up to 2q, in [0, 3q), for any 64-bit x and 2^32 < q < 2^40
// (mu32 = floor(2^64 / q) below 2^32): dropping x's low word costs less than
// 1, mu32's truncation less than 1, the floor less than 1.
// x + qe (2^64 - q) in three multiplies, spelled out (like Sum40's fold) because
// the 64-bit expressions leave moves on the multiplier pipe: the diagonal kernel
// at (1,64,4) takes 1.87 ms with them and 1.78 without.
__device__ __forceinline__ u64 reduce64_40(u64 x, u64 q, u32 mu32) {
    u64 r;
    asm("{\n\t.reg .u32 x0, x1, n0, n1, e, t0, t1;\n\t.reg .u64 t;\n\t"
        "mov.b64 {x0, x1}, %1;\n\tmov.b64 {n0, n1}, %2;\n\t"
        "mul.hi.u32 e, x1, %3;\n\tmad.wide.u32 t, e, n0, %1;\n\tmov.b64 {t0, t1}, t;\n\t"
        "mad.lo.u32 t1, e, n1, t1;\n\tmov.b64 %0, {t0, t1};\n\t}" : "=l"(r) : "l"(x), "l"(0 - q), "r"(mu32));
    return r;
}

// Sums of products without carries.  A carry chain costs an instruction per
// carry and serialises its multiplies; 64-bit accumulators of split operands
// need neither (register-only loops on GB300: 3.7e12 products/s in the 40-bit
// form and 3.2e12 in the three-product form, against 2.45e12 for mac96 and
// 2.0e12 for mac128).
//
// Sum40: products of a word d < 2^40 split at bit 20 by a word k < 2^40 split
// at bit 32 (the packed layout's own split).  At most 8 products: L and M stay
// below 2^55, P and Q (28-bit products) below 2^31.
struct Sum40 {
    u64 L = 0, M = 0;
    u32 P = 0, Q = 0;
    __device__ __forceinline__ void mac(u32 d0, u32 d1, u32 k0, u32 k1) {
        L += (u64)d0 * k0;
        M += (u64)d1 * k0;
        P += d0 * k1;
        Q += d1 * k1;
    }
    // L + 2^20 M + 2^32 P + 2^52 Q + add (add < 2^43) mod q, in [0, 3q).
    // M + 2^12 P + 2^32 Q is below 2^64; its residue m < 3q < 2^42 leaves
    // L + add + 2^20 m below 2^63.
    __device__ __forceinline__ u64 value(u64 add, u64 q, u32 mu32) const {
        u64 t;  // M + 2^12 P + 2^32 Q in 32-bit adds
        asm("{\n\t.reg .u32 t0, t1, p0, p1;\n\tmov.b64 {t0, t1}, %2;\n\tshl.b32 p0, %1, 12;\n\tshr.u32 p1, %1, 20;\n\tadd.u32 p1, p1, %3;\n\t"
            "add.cc.u32 t0, t0, p0;\n\taddc.u32 t1, t1, p1;\n\tmov.b64 %0, {t0, t1};\n\t}" : "=l"(t) : "r"(P), "l"(M), "r"(Q));
        const u64 m = reduce64_40(t, q, mu32);
        return reduce64_40(L + add + (m << 20), q, mu32);
    }
};
__device__ __forceinline__ void split20(u64 x, u32& l, u32& h) {  // x < 2^52
    l = (u32)x & 0xFFFFFu;
    h = __funnelshift_r((u32)x, (u32)(x >> 32), 20);
}

// Sum60: products of words below 2^60, both split at bit 30; at most 8.  L and
// H stay below 2^63, M (two products each) below 2^64.
struct Sum60 {
    u64 L = 0, M = 0, H = 0;
    __device__ __forceinline__ void mac(u32 d0, u32 d1, u32 k0, u32 k1) {
        asm("mad.wide.u32 %0, %3, %5, %0;\n\tmad.wide.u32 %1, %3, %6, %1;\n\t"
            "mad.wide.u32 %2, %4, %6, %2;\n\tmad.wide.u32 %1, %4, %5, %1;"
            : "+l"(L), "+l"(M), "+l"(H) : "r"(d0), "r"(d1), "r"(k0), "r"(k1));
    }
    // L + 2^30 M + 2^60 H + add (add < 2^63) mod q, in [0, 5q)
    __device__ __forceinline__ u64 value(u64 add, const ModC& m) const {
        const u64 l = L + add;
        u64 lo = l + (M << 30);
        u64 hi = (M >> 34) + (H >> 4) + (lo < l ? 1u : 0u);
        const u64 t = lo + (H << 60);
        hi += t < lo ? 1u : 0u;
        return reduce_top((u32)t, (u32)(t >> 32), (u32)hi, (u32)(hi >> 32), m);
    }
};
__device__ __forceinline__ void split30(u64 x, u32& l, u32& h) {  // x < 2^62
    l = (u32)x & 0x3FFFFFFFu;
    h = __funnelshift_r((u32)x, (u32)(x >> 32), 30);
}

// Products of a word below 5q by a word below q < 2^60 between two reductions of a 128-bit sum.
constexpr u32 FLUSH = 32;

// [0, 8q) -> [0, q), q < 2^60
__device__ __forceinline__ u64 canon8(u64 x, u64 q) {
    x = x >= 4 * q ? x - 4 * q : x;
    x = x >= 2 * q ? x - 2 * q : x;
    return x >= q ? x - q : x;
}

// Source index of the NTT-domain automorphism x -> x^g in bit-reversed
// storage (Eq. 7): output word s reads word brv(((g (2 brv(s) + 1)) mod 2N - 1) / 2).
// 2N divides 2^32, so the product may wrap.
__device__ __forceinline__ u32 auto_src(u32 s, u32 g, u32 log_n) {
    const u32 sh = 32u - log_n;
    u32 l = __brev(s) >> sh;
    u32 e = (g * (2u * l + 1u)) & ((2u << log_n) - 1u);
    return __brev((e - 1u) >> 1) >> sh;
}
