// Per-thread accumulation of the dot products of a sweep.
//
// A sweep forms a fixed set of dot products over the values of each row; a
// "pairs" type lists them (value a(k) times value b(k), k < np, of nv values),
// and an accumulator takes the values of one row at a time.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#include "portable.cuh"

namespace pbcg {

// Algorithm 9, first reduction: values q y r0 s z; (q,y) (y,y) (q,q) (r0,s) (r0,z)
struct PairsPipeA {
    static constexpr int nv = 5, np = 5;
    PBCG_HD static constexpr int a(int k) { return k == 0 || k == 2 ? 0 : k == 1 ? 1 : 2; }
    PBCG_HD static constexpr int b(int k) { return k == 0 || k == 1 ? 1 : k == 2 ? 0 : k; }
};
// Algorithm 9, second reduction: values r0 r w; (r0,r) (r0,w) (r,r)
struct PairsPipeB {
    static constexpr int nv = 3, np = 3;
    PBCG_HD static constexpr int a(int k) { return k == 2 ? 1 : 0; }
    PBCG_HD static constexpr int b(int k) { return k == 1 ? 2 : 1; }
};
// Algorithm 7: values r0 s; (r0,s)
struct PairsOne {
    static constexpr int nv = 2, np = 1;
    PBCG_HD static constexpr int a(int) { return 0; }
    PBCG_HD static constexpr int b(int) { return 1; }
};
// Algorithm 7: values q y; (q,y) (y,y) (q,q)
struct PairsOmega {
    static constexpr int nv = 2, np = 3;
    PBCG_HD static constexpr int a(int k) { return k == 1 ? 1 : 0; }
    PBCG_HD static constexpr int b(int k) { return k == 2 ? 0 : 1; }
};
// Algorithm 7: values r0 r; (r0,r) (r,r)
struct PairsRho {
    static constexpr int nv = 2, np = 2;
    PBCG_HD static constexpr int a(int k) { return k; }
    PBCG_HD static constexpr int b(int) { return 1; }
};

PBCG_HD uint32_t wide_mulhi(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
    return __umulhi(a, b);
#else
    return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}
// v >> s, 0 for s < 0 and from 64 on (the instruction takes s as unsigned and clamps it)
PBCG_HD uint64_t wide_shr(uint64_t v, int s) {
#ifdef __CUDA_ARCH__
    uint64_t r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
    return r;
#else
    return s < 0 || s > 63 ? 0 : v >> s;
#endif
}
// v << s, 0 for s < 0 and from 32 on
PBCG_HD uint32_t wide_shl(uint32_t v, int s) {
#ifdef __CUDA_ARCH__
    uint32_t r;
    asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(s));
    return r;
#else
    return s < 0 || s > 31 ? 0 : v << s;
#endif
}
PBCG_HD double wide_from_bits(uint64_t u) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)u);
#else
    double v;
    memcpy(&v, &u, 8);
    return v;
#endif
}
PBCG_HD int wide_clz(uint32_t v) {   // 32 for 0
#ifdef __CUDA_ARCH__
    return __clz((int)v);
#else
    return v ? __builtin_clz(v) : 32;
#endif
}

// A dot product of doubles summed in a 96-bit fixed-point number on the
// integer pipes, which the FP64 sweeps leave nearly idle: on this GPU a
// warp-wide FP64 instruction occupies its sub-partition's FP64 pipe for 64
// cycles, and 8 of the 37 FP64 operations of an Algorithm 9 row (7-point
// stencil) are these sums. Measured alone, the five dot products of a row take
// 195 cycles per warp here and 321 as FP64 FMAs, on other pipes: FP64 and
// integer instructions of different warps overlap fully.
//
// A product of two 53-bit significands (each shifted to the top of 63 bits) is
// formed to 62 bits by three 32-bit multiplies, 3 units too small at most,
// shifted right by the distance of its exponent to a reference exponent, and
// added with its sign; kWideRoom bits above it leave room for kWideThreadRows
// products. The reference is kWideMargin binades above the largest product of
// the WARP's first rows; a product above it moves it to kWideMargin binades
// above itself and shifts the sum. (A reference from each thread's own first
// row moved in some lane of the warp at every other row, and the sweep was
// slower than with FP64 sums.) A term keeps all bits down to the unit of the
// sum, which is at most 2^-73 of the largest product that the warp has met:
// all units that the 32 x kWideThreadRows terms of a warp can lose (one at the
// addition, one at a move) add up to less than 2^-53 of that product, so the
// warp's common reference costs no accuracy next to the rounding of one
// thread's sum to a double, whatever the ratio between its lanes. An FP64 FMA
// chain rounds the running sum at every step. Largest error of a warp's sum,
// relative to the sum of its absolute products, over 107, 1000 and 13000 rows a
// thread of normal values with one of 1, 1e2, 1e4 or 1e6 times that among the
// first: 1.1e-16, against 1.3e-14 with FP64 chains. (With the product aligned
// to the upper two words, a unit of 2^-54 of the warp's largest product, the
// outlier cost the other lanes their low bits: 4e-12 at 13000 rows and 1e4.)
// A product with an infinite or NaN factor is noted and decides the result as
// in an FP64 sum.
constexpr int kWideMargin = 6;
constexpr int kWideRoom = 13;               // products below 2^(95 - 14): 2^14 of them and a sign
constexpr int kWideThreadRows = 1 << 14;    // most rows of a thread
constexpr int kWideBias = 2106 + 32 - kWideRoom;
constexpr int kWideAbsent = -8192;   // exponent of a value whose products vanish

// A fixed-point number (w2 w1 w0) 2^(ref - kWideBias), two's complement: the sum of
// one dot product over the rows of a thread.
struct alignas(16) WideSlot {
    uint32_t w0, w1, w2;
    int ref;
};

// Move the reference up to `ref`: floor(sum / 2^shift).
PBCG_HD void wide_move(WideSlot &c, int ref) {
    const int d = ref - c.ref;
    c.ref = ref;
    const uint32_t sign = (uint32_t)((int)c.w2 >> 31);
    if (d >= 96) {
        c.w0 = c.w1 = c.w2 = sign;
        return;
    }
    if (d >= 64) {
        c.w0 = c.w2;
        c.w1 = c.w2 = sign;
    } else if (d >= 32) {
        c.w0 = c.w1;
        c.w1 = c.w2;
        c.w2 = sign;
    }
    const int r = d & 31;
    const uint64_t lo = (uint64_t)c.w1 << 32 | c.w0, hi = (uint64_t)c.w2 << 32 | c.w1;
    c.w0 = (uint32_t)(lo >> r);
    c.w1 = (uint32_t)(hi >> r);
    c.w2 = (uint32_t)((int)c.w2 >> r);
}

// The number as a double, rounded to nearest; f: flags of the terms it met (1 NaN, 2 +inf, 4 -inf).
PBCG_HD double wide_value(const WideSlot &c, unsigned f) {
    const uint32_t sign = (uint32_t)((int)c.w2 >> 31);
    uint64_t t = (uint64_t)(c.w0 ^ sign) + (sign & 1u);
    uint32_t a0 = (uint32_t)t;
    t = (uint64_t)(c.w1 ^ sign) + (t >> 32);
    uint32_t a1 = (uint32_t)t;
    uint32_t a2 = (c.w2 ^ sign) + (uint32_t)(t >> 32);
    int ex = c.ref - kWideBias + 64;   // |sum| = (a2 a1 a0) 2^(ex - 64); move its leading word to a2
    if (a2 == 0) {
        a2 = a1;
        a1 = a0;
        a0 = 0;
        ex -= 32;
    }
    if (a2 == 0) {
        a2 = a1;
        a1 = 0;
        ex -= 32;
    }
    if (f) {
        return wide_from_bits((f & 1) || f == 6 ? 0x7ff8000000000000ull
                                                : f == 2 ? 0x7ff0000000000000ull : 0xfff0000000000000ull);
    }
    if (a2 == 0) return 0.0;
    const int z = wide_clz(a2);
    uint64_t m = ((uint64_t)a2 << 32 | a1) << z;
    m |= (uint64_t)a0 << z >> 32;
    ex -= z;             // |sum| = m 2^(ex - 32), m in [2^63, 2^64)
    m += 1ull << 10;     // round to 53 bits
    if (m < (1ull << 63)) {   // carried out of the top
        m = 1ull << 63;
        ex += 1;
    }
    const int be = ex + 1054;   // biased exponent of the result
    const uint64_t s64 = (uint64_t)(sign & 1u) << 63, frac = (m >> 11) & 0xfffffffffffffull;
    if (be >= 1 && be <= 2046) return wide_from_bits(s64 | (uint64_t)be << 52 | frac);
    if (be > 2046) return wide_from_bits(s64 | 0x7ff0000000000000ull);
    if (be < -60) return wide_from_bits(s64);
    return wide_from_bits(s64 | (uint64_t)(be + 120) << 52 | frac) * wide_from_bits((1023ull - 120) << 52);
}

// A value taken apart: sign in bit 31 of hi, exponent, significand in the top of 63 bits.
struct WideParts {
    uint32_t hi, mh, ml;
    int e;
};
PBCG_HD WideParts wide_parts(double v) {
    WideParts p;
    const uint64_t u = bits_of(v);
    p.hi = (uint32_t)(u >> 32);
    p.e = (int)((p.hi >> 20) & 0x7ffu);
    const uint64_t m = ((uint64_t)((p.hi & 0xfffffu) | 0x100000u) << 32 | (uint32_t)u) << 10;
    p.mh = (uint32_t)(m >> 32);
    p.ml = (uint32_t)m;
    return p;
}

// The parts of a zero (exponent kWideAbsent) or subnormal value.
PBCG_HD void wide_subnormal(double v, WideParts &p) {
    const uint64_t f = bits_of(v) & 0xfffffffffffffull;
    if (f == 0) {
        p.e = kWideAbsent;
        return;
    }
    const uint32_t hi = (uint32_t)(f >> 32);
    const int z = hi ? wide_clz(hi) : 32 + wide_clz((uint32_t)f);
    const uint64_t m = f << (z - 1);   // the leading bit to bit 62; that of a normal number of exponent e is 2^(e - 1023)
    p.e = 12 - z;
    p.mh = (uint32_t)(m >> 32);
    p.ml = (uint32_t)m;
}

// Add the product of a and b (square: a times itself) to c; its exponent is `distance` below the reference.
PBCG_HD void wide_add(WideSlot &c, const WideParts &a, const WideParts &b, bool square, int distance) {
    const uint32_t mid = square ? 2u * wide_mulhi(a.mh, a.ml) : wide_mulhi(a.mh, b.ml) + wide_mulhi(a.ml, b.mh);
    const uint64_t q = (uint64_t)a.mh * b.mh + mid;
    const uint32_t sg = square ? 0u : (uint32_t)((int)(a.hi ^ b.hi) >> 31);
    // the words of q 2^32 >> shift; the lowest from the left shift below 32 and from the right one above
    const int shift = distance + kWideRoom;
    const uint64_t top = wide_shr(q, shift);
    const uint32_t q0 = (wide_shl((uint32_t)q, 32 - shift) | (uint32_t)wide_shr(q, shift - 32)) ^ sg;
    const uint32_t q1 = (uint32_t)top ^ sg, q2 = (uint32_t)(top >> 32) ^ sg;   // ~q for a negative product
#ifdef __CUDA_ARCH__
    if (square)
        asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
            : "+r"(c.w0), "+r"(c.w1), "+r"(c.w2)
            : "r"(q0), "r"(q1), "r"(q2));
    else   // the first addition only makes the carry, 1 for a negative product: -q = ~q + 1
        asm("{\n\t.reg .u32 t;\n\tadd.cc.u32 t, %6, %6;\n\taddc.cc.u32 %0, %0, %3;\n\t"
            "addc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;\n\t}"
            : "+r"(c.w0), "+r"(c.w1), "+r"(c.w2)
            : "r"(q0), "r"(q1), "r"(q2), "r"(sg));
#else
    const uint64_t t0 = (uint64_t)c.w0 + q0 + (sg & 1u), t1 = (uint64_t)c.w1 + q1 + (t0 >> 32);
    c.w0 = (uint32_t)t0;
    c.w1 = (uint32_t)t1;
    c.w2 += q2 + (uint32_t)(t1 >> 32);
#endif
}

// The dot products P of a thread's rows. Slots live in memory (shared memory
// in a kernel, `stride` slots apart), so that they hold no registers while a
// row's vectors are loaded and its product with A is formed.
template <class P>
struct WideDots {
    WideSlot *slot;
    int stride;
    unsigned special;   // 3 bits a dot product: NaN, +inf, -inf met
    unsigned lanes;     // lanes of the warp that have a first row, 0 once it is done

    PBCG_HD WideDots(WideSlot *s, int st, unsigned with_rows) : slot(s), stride(st), special(0u), lanes(with_rows) {}

    PBCG_HD void add(const double (&v)[P::nv]) {
        WideParts p[P::nv];
        int emin = 2047, emax = 0;
#pragma unroll
        for (int j = 0; j < P::nv; ++j) {
            p[j] = wide_parts(v[j]);
            emin = p[j].e < emin ? p[j].e : emin;
            emax = p[j].e > emax ? p[j].e : emax;
        }
        if (emin == 0 || emax == 2047) unusual(v, p, emax);
        if (lanes) first(p);
#pragma unroll
        for (int k = 0; k < P::np; ++k) {
            const WideParts &a = p[P::a(k)], &b = p[P::b(k)];
            WideSlot c = slot[k * stride];
            int s = c.ref - a.e - b.e;
            if (s < 0) {
                wide_move(c, a.e + b.e + kWideMargin);
                s = kWideMargin;
            }
            wide_add(c, a, b, P::a(k) == P::b(k), s);
            slot[k * stride] = c;
        }
    }

    // Zeros vanish; infinite and NaN values are noted and vanish; subnormal ones get their
    // leading bit in place and the exponent that goes with it.
    PBCG_HD void unusual(const double (&v)[P::nv], WideParts (&p)[P::nv], int emax) {
        if (emax == 2047) {
#pragma unroll
            for (int k = 0; k < P::np; ++k)
                if (p[P::a(k)].e == 2047 || p[P::b(k)].e == 2047) {
                    const double t = v[P::a(k)] * v[P::b(k)];
                    special |= (t != t ? 1u : t > 0.0 ? 2u : 4u) << (3 * k);
                }
        }
#pragma unroll
        for (int j = 0; j < P::nv; ++j) {
            if (p[j].e == 0) wide_subnormal(v[j], p[j]);
            else if (p[j].e == 2047) p[j].e = kWideAbsent;
        }
    }

    // Exponent of product k of a row.
    PBCG_HD static int product_exponent(const WideParts (&p)[P::nv], int k) {
        const int e = p[P::a(k)].e + p[P::b(k)].e;
        return e < 0 ? 0 : e;
    }
    // Empty sums with their references above the largest product of the warp's first rows.
    PBCG_HD void first(const WideParts (&p)[P::nv]) {
#pragma unroll
        for (int k = 0; k < P::np; ++k) {
            int top = product_exponent(p, k);
#ifdef __CUDA_ARCH__
            top = __reduce_max_sync(lanes, top);
#endif
            begin(k, top);
        }
        lanes = 0u;
    }
    PBCG_HD void begin(int k, int top) { slot[k * stride] = WideSlot{0u, 0u, 0u, top + kWideMargin}; }

    // The sums (a thread without a row has none to read).
    PBCG_HD void values(bool any, double (&d)[P::np]) const {
#pragma unroll
        for (int k = 0; k < P::np; ++k) d[k] = any ? wide_value(slot[k * stride], (special >> (3 * k)) & 7u) : 0.0;
    }
};

}  // namespace pbcg
