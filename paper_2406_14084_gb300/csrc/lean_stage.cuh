// lean_stage.cuh -- the in-place register-stage engine.
//
// Runs the records that lower.cpp writes: shear pairs (real 2x2 matrices without their diagonal
// factor), diagonal tables, phases and X.  Each record is one straight run of updates that
// overwrite their inputs, so a thread needs its 2^RB amplitudes (64 registers) and little else,
// two 256-thread CTAs fit one SM, and one dispatch covers a shear pair on every register bit.
// (The general engine of slab_common.cuh dispatches per 2x2 matrix and copies results through
// temporaries; it needs about 250 registers and stays for 4x4 and controlled matrices.)
//
// What bounds a record (ns per slab and SM with two CTAs on it, 2^13 complex64 / 2^12 complex128
// amplitudes; the same slab through the general engine takes about 500 ns per complex64 gate):
//   complex64    stage without records 570 (shared memory: 1024 of 1100 cycles), shears on all five
//                bits 413 (FMA pipe, about 80 % busy), on one bit 114, table 292-400 (L1 to
//                registers: 256 B per thread), X 190
//   complex128   2x2 matrix 1980, table 4330, half table 2170: the FP64 pipe, 2.0 FMA per SM and clock
//   double-float table 1030-1130 (FMA pipe)
#pragma once

#include "slab_common.cuh"

namespace qs {
namespace {

__device__ __forceinline__ unsigned long long pack2(float x, float y)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
// two FP32 operations per instruction
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c)
{
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint32_t xor_bits(float a, uint32_t s) { return __float_as_uint(a) ^ s; }

// Exchange a and b where m is all ones, in place.  Written as asm so that the compiler cannot turn
// the 25 target / control variants into register renamings that meet in one set of moves (spills).
__device__ __forceinline__ void cswap(uint32_t &a, uint32_t &b, uint32_t m)
{
    asm("{\n\t.reg .b32 t;\n\t"
        "lop3.b32 t, %0, %1, %2, 0x28;\n\t"  // (a ^ b) & m
        "xor.b32 %0, %0, t;\n\t"
        "xor.b32 %1, %1, t;\n\t}"
        : "+r"(a), "+r"(b)
        : "r"(m));
}
__device__ __forceinline__ void cswap(float &a, float &b, uint32_t m)
{
    uint32_t x = __float_as_uint(a), y = __float_as_uint(b);
    cswap(x, y, m);
    a = __uint_as_float(x);
    b = __uint_as_float(y);
}
__device__ __forceinline__ void cswap(unsigned long long &a, unsigned long long &b, uint32_t m)
{
    float2 x = unpack2(a), y = unpack2(b);
    cswap(x.x, y.x, m);
    cswap(x.y, y.y, m);
    a = pack2(x.x, x.y);
    b = pack2(y.x, y.y);
}
__device__ __forceinline__ void cswap(double &a, double &b, uint32_t m)
{
    unsigned long long x = __double_as_longlong(a), y = __double_as_longlong(b);
    cswap(x, y, m);
    a = __longlong_as_double(x);
    b = __longlong_as_double(y);
}

// Calls f(e) for the register elements of a pattern: 0 = all, 1 + 2 j + v = those whose bit j is v.
// Written out per pattern: a test per element is turned into predicated arithmetic, which takes the
// FP64 pipe as long as if it were done (a half table cost 4334 ns per slab and SM, as a full one).
template <int RB, int J, int V, typename F>
__device__ __forceinline__ void for_half(F &&f)
{
#pragma unroll
    for (int e = 0; e < (1 << RB); ++e)
        if ((e >> J & 1) == V) f(e);
}
template <int RB, bool HALVES, typename F>
__device__ __forceinline__ void for_pattern(uint32_t pat, F &&f)
{
    switch (HALVES ? pat : 0u) {
    case 1: for_half<RB, 0, 0>(f); break;
    case 2: for_half<RB, 0, 1>(f); break;
    case 3: for_half<RB, 1, 0>(f); break;
    case 4: for_half<RB, 1, 1>(f); break;
    case 5: for_half<RB, 2, 0>(f); break;
    case 6: for_half<RB, 2, 1>(f); break;
    case 7: if constexpr (RB > 3) for_half<RB, 3, 0>(f); break;
    case 8: if constexpr (RB > 3) for_half<RB, 3, 1>(f); break;
    default:
#pragma unroll
        for (int e = 0; e < (1 << RB); ++e) f(e);
        break;
    }
}

// The 2^RB amplitudes of one group in registers, with the engine's operations.
template <typename C, int RB> struct LeanRegs;

// complex64: real and imaginary parts apart, two elements (register bit 0 clear and set) per 64-bit
// pair, so that fma.rn.f32x2 serves the shears on every other bit and the complex multiplies of a
// table alike (a table word holds the two real parts, then the two imaginary parts).  With (re, im)
// pairs instead, a complex multiply needs its operands exchanged or four scalar FMAs per element:
// a table then took 361 ns per 2^13-amplitude slab and SM instead of 292.
template <int RB> struct LeanRegs<float2, RB> {
    static constexpr int E = 1 << RB, P = E / 2;
    static constexpr int kConstWords = P, kScaleWords = E / 4;  // words of the records
    unsigned long long X[P], Y[P];

    __device__ __forceinline__ void load(const float2 *sm, const uint32_t (&a)[E])
    {
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const float2 u = sm[a[2 * p]], v = sm[a[2 * p + 1]];
            X[p] = pack2(u.x, v.x);
            Y[p] = pack2(u.y, v.y);
        }
    }
    __device__ __forceinline__ void store(float2 *sm, const uint32_t (&a)[E]) const
    {
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const float2 x = unpack2(X[p]), y = unpack2(Y[p]);
            sm[a[2 * p]] = make_float2(x.x, y.x);
            sm[a[2 * p + 1]] = make_float2(x.y, y.y);
        }
    }
    // w: (y, x)
    template <int J> __device__ __forceinline__ void shear(unsigned long long w)
    {
        const float2 f = unpack2(w);
        if constexpr (J == 0) {
            const float cy = f.x, cx = f.y;
#pragma unroll
            for (int p = 0; p < P; ++p) {
                float2 x = unpack2(X[p]), y = unpack2(Y[p]);
                x.y = fmaf(cy, x.x, x.y);
                y.y = fmaf(cy, y.x, y.y);
                x.x = fmaf(cx, x.y, x.x);
                y.x = fmaf(cx, y.y, y.x);
                X[p] = pack2(x.x, x.y);
                Y[p] = pack2(y.x, y.y);
            }
        } else {
            constexpr int B = 1 << (J - 1);
            const unsigned long long yy = pack2(f.x, f.x), xx = pack2(f.y, f.y);
#pragma unroll
            for (int p = 0; p < P; ++p) {
                if (p & B) continue;
                X[p | B] = fma2(yy, X[p], X[p | B]);
                Y[p | B] = fma2(yy, Y[p], Y[p | B]);
                X[p] = fma2(xx, X[p | B], X[p]);
                Y[p] = fma2(xx, Y[p | B], Y[p]);
            }
        }
    }
    static constexpr int kRotWords = 1;
    template <int J, bool NEG, typename W> __device__ __forceinline__ void rot(const W &words, uint32_t at)
    {
        shear<J>(words(at).y);
    }
    template <typename W> __device__ __forceinline__ void rot_all(const W &words, uint32_t at)
    {
        const ulonglong2 w1 = words(at + 1);
        shear<0>(words(at).y);
        shear<1>(w1.x);
        shear<2>(w1.y);
        if constexpr (RB > 3) {
            const ulonglong2 w2 = words(at + 2);
            shear<3>(w2.x);
            if constexpr (RB > 4) shear<4>(w2.y);
        }
    }
    // word p: both real parts, both imaginary parts of the factors of pair p
    template <bool HALVES, typename W> __device__ __forceinline__ void table(const W &words, uint32_t at, uint32_t nl, uint32_t pat)
    {
        // (patterns of register bit 0, inside the pairs, are not used here)
        for_pattern<RB - 1, HALVES>(pat > 2 ? pat - 2 : 0, [&](int p) {
            const ulonglong2 q = words.bulk(at + (uint32_t(p) << nl));
            times(p, q.x, q.y);
        });
    }
    // pair p times (re, im), each for both elements
    __device__ __forceinline__ void times(int p, unsigned long long re, unsigned long long im)
    {
        const unsigned long long m = mul2(im ^ 0x8000000080000000ull, Y[p]), w = mul2(im, X[p]);
        X[p] = fma2(re, X[p], m);
        Y[p] = fma2(re, Y[p], w);
    }
    // separable table: f[0] = s, f[1 + j] = phi_j
    struct Sep {
        float2 f[RB + 1];
        template <typename W> __device__ __forceinline__ void group(const W &words, uint32_t at, uint32_t nl, bool first)
        {
#pragma unroll
            for (int k = 0; k <= RB; k += 2) {
                const ulonglong2 q = words.bulk(at + (uint32_t(k >> 1) << nl));
                const float2 a = unpack2(q.x), b = unpack2(q.y);
                f[k] = first ? a : cmul(a, f[k]);
                if (k + 1 <= RB) f[k + 1] = first ? b : cmul(b, f[k + 1]);
            }
        }
    };
    static constexpr int kSepWords = (RB + 2) / 2;
    // the factors of the pairs come from a walk over the register bits, one multiply per step down
    template <int BIT> __device__ __forceinline__ void sep_walk(const Sep &t, int p, unsigned long long re, unsigned long long im)
    {
        if constexpr (BIT == RB - 1) {
            times(p, re, im);
        } else {
            sep_walk<BIT + 1>(t, p, re, im);
            const float2 g = t.f[BIT + 2];
            const unsigned long long gx = pack2(g.x, g.x), gy = pack2(g.y, g.y), ny = pack2(-g.y, -g.y);
            sep_walk<BIT + 1>(t, p | (1 << BIT), fma2(gx, re, mul2(ny, im)), fma2(gx, im, mul2(gy, re)));
        }
    }
    template <bool ONE> __device__ __forceinline__ void sep(const Sep &t)
    {
        const float2 u = cmul(t.f[0], t.f[1]);
        sep_walk<0>(t, 0, pack2(t.f[0].x, u.x), pack2(t.f[0].y, u.y));
    }
    template <typename W> __device__ __forceinline__ void scale(const W &words, uint32_t at)
    {
#pragma unroll
        for (int p = 0; p < P; p += 2) {
            const ulonglong2 q = words(at + p / 2);
            X[p] = mul2(q.x, X[p]);
            Y[p] = mul2(q.x, Y[p]);
            X[p + 1] = mul2(q.y, X[p + 1]);
            Y[p + 1] = mul2(q.y, Y[p + 1]);
        }
    }
    // m: elements whose sign changes
    __device__ __forceinline__ void sign(uint32_t m)
    {
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const uint32_t s0 = (m << (31 - 2 * p)) & 0x80000000u, s1 = (m << (30 - 2 * p)) & 0x80000000u;
            const float2 x = unpack2(X[p]), y = unpack2(Y[p]);
            X[p] = pack2(__uint_as_float(xor_bits(x.x, s0)), __uint_as_float(xor_bits(x.y, s1)));
            Y[p] = pack2(__uint_as_float(xor_bits(y.x, s0)), __uint_as_float(xor_bits(y.y, s1)));
        }
    }
    __device__ __forceinline__ void phase(uint32_t elems, uint32_t /*pat*/, ulonglong2 w, bool on)
    {
        if (!on) return;
        const float2 t = unpack2(w.x);
#pragma unroll
        for (int p = 0; p < P; ++p) {
            if (!(elems >> (2 * p) & 3u)) continue;
            const float c0 = elems >> (2 * p) & 1u ? t.x : 1.f, c1 = elems >> (2 * p) & 2u ? t.x : 1.f;
            const float s0 = elems >> (2 * p) & 1u ? t.y : 0.f, s1 = elems >> (2 * p) & 2u ? t.y : 0.f;
            const unsigned long long m = mul2(pack2(-s0, -s1), Y[p]), w = mul2(pack2(s0, s1), X[p]);
            X[p] = fma2(pack2(c0, c1), X[p], m);
            Y[p] = fma2(pack2(c0, c1), Y[p], w);
        }
    }
    template <int J, int CT> __device__ __forceinline__ void x_bit(uint32_t m)
    {
        if constexpr (J == 0) {
#pragma unroll
            for (int p = 0; p < P; ++p) {
                if (CT > 0 && !(p >> (CT > 0 ? CT - 1 : 0) & 1)) continue;
                float2 x = unpack2(X[p]), y = unpack2(Y[p]);
                cswap(x.x, x.y, m);
                cswap(y.x, y.y, m);
                X[p] = pack2(x.x, x.y);
                Y[p] = pack2(y.x, y.y);
            }
        } else {
            constexpr int B = 1 << (J - 1);
#pragma unroll
            for (int p = 0; p < P; ++p) {
                if (p & B) continue;
                if (CT > 0 && !(p >> (CT > 0 ? CT - 1 : 0) & 1)) continue;
                if (CT == 0) {  // only the elements with register bit 0 set: the pairs' upper halves
                    float2 a = unpack2(X[p]), b = unpack2(X[p | B]);
                    cswap(a.y, b.y, m);
                    X[p] = pack2(a.x, a.y);
                    X[p | B] = pack2(b.x, b.y);
                    a = unpack2(Y[p]), b = unpack2(Y[p | B]);
                    cswap(a.y, b.y, m);
                    Y[p] = pack2(a.x, a.y);
                    Y[p | B] = pack2(b.x, b.y);
                } else {
                    cswap(X[p], X[p | B], m);
                    cswap(Y[p], Y[p | B], m);
                }
            }
        }
    }
};

// complex128: one element per entry.
__device__ __forceinline__ void sign_of(double &v, uint32_t s)
{
    v = __longlong_as_double(__double_as_longlong(v) ^ (long long)((unsigned long long)s << 32));
}
template <int RB> struct LeanRegs<double2, RB> {
    using C = double2;
    static constexpr int E = 1 << RB;
    static constexpr int kConstWords = E, kScaleWords = E;
    C v[E];

    __device__ __forceinline__ void load(const C *sm, const uint32_t (&a)[E])
    {
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = sm[a[e]];
    }
    __device__ __forceinline__ void store(C *sm, const uint32_t (&a)[E]) const
    {
#pragma unroll
        for (int e = 0; e < E; ++e) sm[a[e]] = v[e];
    }
    static constexpr int kRotWords = 2;
    template <int J, bool NEG, typename W> __device__ __forceinline__ void rot(const W &words, uint32_t at)
    {
        const C c = factor(words(at + 1));
#pragma unroll
        for (int e = 0; e < E; ++e) {
            if (e & (1 << J)) continue;
            const C a = v[e], b = v[e | (1 << J)];
            v[e] = rfma(c.y, b, a);
            v[e | (1 << J)] = NEG ? rfms(c.x, a, b) : rfma(c.x, a, b);
        }
    }
    static __device__ __forceinline__ C factor(ulonglong2 w)
    {
        return make_double2(__longlong_as_double((long long)w.x), __longlong_as_double((long long)w.y));
    }
    // elements outside the pattern have the factor 1
    template <bool HALVES, typename W> __device__ __forceinline__ void table(const W &words, uint32_t at, uint32_t nl, uint32_t pat)
    {
        for_pattern<RB, HALVES>(pat, [&](int e) { v[e] = cmul(factor(words(at + (uint32_t(e) << nl))), v[e]); });
    }
    struct Sep {
        C f[RB + 1];
        template <typename W> __device__ __forceinline__ void group(const W &words, uint32_t at, uint32_t nl, bool first)
        {
#pragma unroll
            for (int k = 0; k <= RB; ++k) {
                const C a = factor(words(at + (uint32_t(k) << nl)));
                f[k] = first ? a : cmul(a, f[k]);
            }
        }
    };
    static constexpr int kSepWords = RB + 1;
    // ONE: the factor so far is 1
    template <int BIT, bool ONE> __device__ __forceinline__ void sep_walk(const Sep &t, int e, C f)
    {
        if constexpr (BIT == RB) {
            if (!ONE) v[e] = cmul(f, v[e]);
        } else {
            sep_walk<BIT + 1, ONE>(t, e, f);
            sep_walk<BIT + 1, false>(t, e | (1 << BIT), ONE ? t.f[BIT + 1] : cmul(t.f[BIT + 1], f));
        }
    }
    template <bool ONE> __device__ __forceinline__ void sep(const Sep &t) { sep_walk<0, ONE>(t, 0, t.f[0]); }
    template <typename W> __device__ __forceinline__ void scale(const W &words, uint32_t at)
    {
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = rmul(factor(words(at + e)).x, v[e]);
    }
    __device__ __forceinline__ void sign(uint32_t m)
    {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const uint32_t s = (m << (31 - e)) & 0x80000000u;
            sign_of(v[e].x, s);
            sign_of(v[e].y, s);
        }
    }
    // elems within the pattern: the others of the pattern are multiplied by 1
    __device__ __forceinline__ void phase(uint32_t elems, uint32_t pat, ulonglong2 w, bool on)
    {
        if (!on) return;
        const C t = factor(w);
        for_pattern<RB, true>(pat, [&](int e) {
            const bool in = elems >> e & 1u;
            v[e] = cmul(make_double2(in ? t.x : 1.0, in ? t.y : 0.0), v[e]);
        });
    }
    template <int J, int CT> __device__ __forceinline__ void x_bit(uint32_t m)
    {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            if (e & (1 << J)) continue;
            if (CT >= 0 && !(e >> (CT < 0 ? 0 : CT) & 1)) continue;
            cswap(v[e].x, v[e | (1 << J)].x, m);
            cswap(v[e].y, v[e | (1 << J)].y, m);
        }
    }
};

// complex128 in double-float form (df_arith.cuh) with both parts of an amplitude packed: h holds the
// leading FP32 numbers of the real and the imaginary part, l the trailing ones, so that each step of
// the double-float operations is one f32x2 instruction for both.  The steps and their roundings are
// those of df_arith.cuh (negated products stand for subtractions).
struct __align__(16) dfp {
    unsigned long long h, l;
};

__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long sub2(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long neg2(unsigned long long a)
{
    const float2 f = unpack2(a);
    return pack2(-f.x, -f.y);
}
// a double-float factor for each part, with its negative
struct df_factor {
    unsigned long long h, nh, nl;
    __device__ __forceinline__ df_factor(unsigned long long ph, unsigned long long pl) : h(ph), nh(neg2(ph)), nl(neg2(pl)) {}
    __device__ __forceinline__ df_factor(float ch, float cl) : df_factor(pack2(ch, ch), pack2(cl, cl)) {}
};
// a b: p + e with e = -g
__device__ __forceinline__ void df_prod(const df_factor &a, const dfp &b, unsigned long long &p, unsigned long long &g)
{
    p = mul2(a.h, b.h);
    g = fma2(a.nh, b.h, p);
    g = fma2(a.nh, b.l, g);
    g = fma2(a.nl, b.h, g);
}
// p - g + c, or p - g - c
template <bool SUB> __device__ __forceinline__ dfp df_sum(unsigned long long p, unsigned long long g, const dfp &c)
{
    const unsigned long long s = SUB ? sub2(p, c.h) : add2(p, c.h), bb = sub2(s, p);
    const unsigned long long e = sub2(p, sub2(s, bb));
    const unsigned long long t = SUB ? sub2(sub2(e, add2(c.h, bb)), add2(c.l, g)) : add2(add2(e, sub2(c.h, bb)), sub2(c.l, g));
    dfp r;
    r.h = add2(s, t);
    r.l = sub2(t, sub2(r.h, s));
    return r;
}
__device__ __forceinline__ dfp df_fma(const df_factor &a, const dfp &b, const dfp &c)
{
    unsigned long long p, g;
    df_prod(a, b, p, g);
    return df_sum<false>(p, g, c);
}
__device__ __forceinline__ dfp df_mul(const df_factor &a, const dfp &b)
{
    unsigned long long p, g;
    df_prod(a, b, p, g);
    dfp r;
    r.h = sub2(p, g);
    r.l = sub2(sub2(p, r.h), g);
    return r;
}

template <int RB> struct LeanRegs<dfp, RB> {
    static constexpr int E = 1 << RB;
    static constexpr int kConstWords = E, kScaleWords = E;
    dfp v[E];

    __device__ __forceinline__ void load(const dfp *sm, const uint32_t (&a)[E])
    {
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = sm[a[e]];
    }
    __device__ __forceinline__ void store(dfp *sm, const uint32_t (&a)[E]) const
    {
#pragma unroll
        for (int e = 0; e < E; ++e) sm[a[e]] = v[e];
    }
    static constexpr int kRotWords = 2;
    template <int J, bool NEG, typename W> __device__ __forceinline__ void rot(const W &words, uint32_t at)
    {
        const float4 c = factor(words(at + 1));
        const df_factor y(c.x, c.y), x(c.z, c.w);
#pragma unroll
        for (int e = 0; e < E; ++e) {
            if (e & (1 << J)) continue;
            // both products before either sum: they hold what the sums need of the old values (26 qubits, 12
            // layers: 37.7 ms, 38.1 with one result after the other)
            dfp &a = v[e], &b = v[e | (1 << J)];
            unsigned long long p, g, q, f;
            df_prod(x, b, p, g);
            df_prod(y, a, q, f);
            a = df_sum<false>(p, g, a);
            b = df_sum<NEG>(q, f, b);
        }
    }
    static __device__ __forceinline__ float4 factor(ulonglong2 w)
    {
        const float2 a = unpack2(w.x), b = unpack2(w.y);
        return make_float4(a.x, a.y, b.x, b.y);
    }
    // (re, im) <- t (re, im): t.re (re, im) + (-t.im, t.im) (im, re)
    static __device__ __forceinline__ void times(dfp &v, float4 t)
    {
        const float2 h = unpack2(v.h), l = unpack2(v.l);
        dfp w;
        w.h = pack2(h.y, h.x);
        w.l = pack2(l.y, l.x);
        v = df_fma(df_factor(t.x, t.y), v, df_mul(df_factor(pack2(-t.z, t.z), pack2(-t.w, t.w)), w));
    }
    template <bool HALVES, typename W> __device__ __forceinline__ void table(const W &words, uint32_t at, uint32_t nl, uint32_t pat)
    {
        for_pattern<RB, HALVES>(pat, [&](int e) { times(v[e], factor(words(at + (uint32_t(e) << nl)))); });
    }
    static __device__ __forceinline__ dfp as_dfp(float4 t) { return dfp{pack2(t.x, t.z), pack2(t.y, t.w)}; }
    static __device__ __forceinline__ float4 as_factor(const dfp &a)
    {
        const float2 h = unpack2(a.h), l = unpack2(a.l);
        return make_float4(h.x, l.x, h.y, l.y);
    }
    struct Sep {
        dfp f[RB + 1];
        template <typename W> __device__ __forceinline__ void group(const W &words, uint32_t at, uint32_t nl, bool first)
        {
#pragma unroll
            for (int k = 0; k <= RB; ++k) {
                const float4 a = factor(words(at + (uint32_t(k) << nl)));
                if (first) f[k] = as_dfp(a);
                else times(f[k], a);
            }
        }
    };
    static constexpr int kSepWords = RB + 1;
    template <int BIT, bool ONE> __device__ __forceinline__ void sep_walk(const Sep &t, int e, dfp f)
    {
        if constexpr (BIT == RB) {
            if (!ONE) times(v[e], as_factor(f));
        } else {
            sep_walk<BIT + 1, ONE>(t, e, f);
            dfp g = t.f[BIT + 1];
            if (!ONE) times(g, as_factor(f));
            sep_walk<BIT + 1, false>(t, e | (1 << BIT), g);
        }
    }
    template <bool ONE> __device__ __forceinline__ void sep(const Sep &t) { sep_walk<0, ONE>(t, 0, t.f[0]); }
    template <typename W> __device__ __forceinline__ void scale(const W &words, uint32_t at)
    {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const float4 t = factor(words(at + e));
            v[e] = df_mul(df_factor(t.x, t.y), v[e]);
        }
    }
    __device__ __forceinline__ void sign(uint32_t m)
    {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const uint32_t s = (m << (31 - e)) & 0x80000000u;
            const unsigned long long ss = (unsigned long long)s << 32 | s;
            v[e].h ^= ss;
            v[e].l ^= ss;
        }
    }
    __device__ __forceinline__ void phase(uint32_t elems, uint32_t pat, ulonglong2 w, bool on)
    {
        if (!on) return;
        const float4 t = factor(w);
        for_pattern<RB, true>(pat, [&](int e) {
            const bool in = elems >> e & 1u;
            times(v[e], make_float4(in ? t.x : 1.f, in ? t.y : 0.f, in ? t.z : 0.f, in ? t.w : 0.f));
        });
    }
    template <int J, int CT> __device__ __forceinline__ void x_bit(uint32_t m)
    {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            if (e & (1 << J)) continue;
            if (CT >= 0 && !(e >> (CT < 0 ? 0 : CT) & 1)) continue;
            cswap(v[e].h, v[e | (1 << J)].h, m);
            cswap(v[e].l, v[e | (1 << J)].l, m);
        }
    }
};

template <typename V, int RB, int J>
__device__ __forceinline__ void x_target(V &v, uint32_t ctrl, uint32_t m)
{
    switch (ctrl) {
    case 0: if (J != 0) v.template x_bit<J, (J != 0 ? 0 : 1)>(m); break;
    case 1: if (J != 1) v.template x_bit<J, (J != 1 ? 1 : 0)>(m); break;
    case 2: if (J != 2) v.template x_bit<J, (J != 2 ? 2 : 0)>(m); break;
    case 3: if (J != 3 && RB > 3) v.template x_bit<J, (J != 3 && RB > 3 ? 3 : (J != 0 ? 0 : 1))>(m); break;
    case 4: if (J != 4 && RB > 4) v.template x_bit<J, (J != 4 && RB > 4 ? 4 : (J != 0 ? 0 : 1))>(m); break;
    default: v.template x_bit<J, -1>(m); break;
    }
}

// Element addresses: the address of e is that of e without its lowest set bit, XORed with that
// bit's offset (the swizzle is linear over GF(2)).
template <int RB>
__device__ __forceinline__ void group_addresses(uint32_t (&a)[1 << RB], uint32_t a0, const uint32_t (&bo)[RB])
{
    a[0] = a0;
#pragma unroll
    for (int e = 1; e < (1 << RB); ++e) a[e] = a[e & (e - 1)] ^ bo[lowest_bit(e)];
}

// A lowered stage is a stream of 16-byte words (format: qs_internal.h).  GlobalWords reads it from
// device memory; the pass kernel also has a form that carries it in its parameters (k_lean.cuh), where
// bulk(), used for the factors of tables, still reads device memory.
//
// load_word: written as asm so that the two 64-bit halves land in the register pairs that f32x2
// instructions take; through __ldg of a vector type the compiler copies them (117 instead of 87
// instructions on the FMA pipe per table of 2^5 elements, 345 instead of 292 ns per slab and SM).
__device__ __forceinline__ ulonglong2 load_word(const ulonglong2 *p)
{
    ulonglong2 w;
    asm volatile("ld.global.nc.v2.b64 {%0, %1}, [%2];" : "=l"(w.x), "=l"(w.y) : "l"(p));
    return w;
}
struct GlobalWords {
    const ulonglong2 *p;
    __device__ __forceinline__ ulonglong2 operator()(uint32_t i) const { return __ldg(p + i); }
    __device__ __forceinline__ ulonglong2 bulk(uint32_t i) const { return load_word(p + i); }
};
__device__ __forceinline__ uint4 as_u4(ulonglong2 w)
{
    return make_uint4(uint32_t(w.x), uint32_t(w.x >> 32), uint32_t(w.y), uint32_t(w.y >> 32));
}

// Values of a record's condition bits: x = those inside the slab (nl of them), y = those outside it,
// which are the same for the whole slab.
__device__ __forceinline__ uint2 condition_index(ulonglong2 cw, uint32_t nl, uint32_t ndl, uint32_t base, uint64_t cta_base)
{
    unsigned long long codes = cw.x;
    uint32_t hl = 0, ho = 0, k = 0;
    for (; k < nl; ++k, codes = k == 8 ? cw.y : codes >> 8) hl |= ((base >> (codes & 0x7fu)) & 1u) << k;
    for (; k < ndl; ++k, codes = k == 8 ? cw.y : codes >> 8) ho |= uint32_t((cta_base >> (codes & 0x7fu)) & 1u) << (k - nl);
    return make_uint2(hl, ho);
}

// Whether some thread of this one's warp has a group of a stage over 2^nrest of them.
__device__ __forceinline__ bool with_groups(uint32_t tid, int nrest) { return ((tid & ~31u) >> nrest) == 0; }

// Runs the stage whose words start at `at` on the slab in shared memory (addressing: run_stage) and
// returns the index after its last word.  One group per thread, the caller has at least 2^nrest threads.
// (With a loop over groups the compiler keeps the 31 address offsets live across it, which costs
// spills at 128 registers.)  Threads without a group work on a copy of one and store nothing, so that
// control flow stays the same for the whole warp; what they load may be stored by its owner at the same time, and is
// never used.  In complex128 warps without any group should not come here (with_groups): their copies would
// take the FP64 pipe as long as real work (10 qubits, 4 layers: 188 us, 125 without; slabs of 8 bits 3.2 times).
// FULL = false: stages without separable tables, X and half tables, in complex64 without phases too.  The larger set
// costs the common records registers and moves (layered-28 complex64: 41.2 ms with one set, 37.8 with two).
template <typename C, int RB, bool FULL = true, typename Words>
__device__ __forceinline__ uint32_t run_lean_stage(C *sm, const Words &words, uint32_t at, const C *__restrict__ pool,
                                                   uint64_t cta_base, uint32_t tid)
{
    using V = LeanRegs<C, RB>;
    constexpr int E = 1 << RB;
    constexpr int SW = sizeof(C) == 8 ? 1 : 2;
    constexpr int PL = sizeof(C) == 8 ? 1 : 0;  // table entries per 16-byte word, log2
    const uint4 hd = as_u4(words(at++));
    const uint32_t nrest = hd.z & 0xffu, flip = hd.z >> 8, end = hd.w + at;
    const bool mine = !(tid >> nrest);
    uint32_t bo[RB], fl = 0, base = tid & ((1u << nrest) - 1u);
#pragma unroll
    for (int j = 0; j < RB; ++j) {
        const uint32_t sb = j < 4 ? (hd.x >> (8 * j)) & 0xff : (hd.y >> (8 * (j - 4))) & 0xff;
        bo[j] = swz<SW>(1u << sb);
        if (flip >> j & 1) fl ^= bo[j];
        const uint32_t low = base & ((1u << sb) - 1u);
        base = ((base ^ low) << 1) | low;
    }
    const uint32_t pb = swz<SW>(base);
    V v;
    {
        uint32_t a[E];
        group_addresses<RB>(a, pb, bo);
        v.load(sm, a);
    }
#pragma unroll 1
    while (at != end) {
        const ulonglong2 hw = words(at);
        const uint4 h = as_u4(hw);
        switch (h.x & 0xffu) {
        case L_ROTA:  // every register bit (complex64)
            if constexpr (PL == 1) v.rot_all(words, at);
            at += 1 + RB / 2;
            break;
        case L_ROT0: v.template rot<0, false>(words, at); at += V::kRotWords; break;
        case L_ROT1: v.template rot<1, false>(words, at); at += V::kRotWords; break;
        case L_ROT2: v.template rot<2, false>(words, at); at += V::kRotWords; break;
        case L_ROT3: if constexpr (RB > 3) v.template rot<3, false>(words, at); at += V::kRotWords; break;
        case L_ROT4: if constexpr (RB > 4) v.template rot<4, false>(words, at); at += V::kRotWords; break;
        case L_ROTM0: if constexpr (PL == 0) v.template rot<0, true>(words, at); at += V::kRotWords; break;
        case L_ROTM1: if constexpr (PL == 0) v.template rot<1, true>(words, at); at += V::kRotWords; break;
        case L_ROTM2: if constexpr (PL == 0) v.template rot<2, true>(words, at); at += V::kRotWords; break;
        case L_ROTM3: if constexpr (PL == 0 && RB > 3) v.template rot<3, true>(words, at); at += V::kRotWords; break;
        case L_CONST:  // a table without conditions: its factors follow
            v.template table<FULL>(words, at + 1, 0, h.z);
            at += 1 + V::kConstWords;
            break;
        case L_TABLE: {
            const uint32_t nl = (h.x >> 16) & 0xffu;
            const uint2 i = condition_index(words(at + 1), nl, h.x >> 24, base, cta_base);
            v.template table<FULL>(GlobalWords{reinterpret_cast<const ulonglong2 *>(pool) + (h.y + (i.y << (RB - PL + nl)) + i.x)}, 0, nl, h.z);
            at += 2;
            break;
        }
        case L_SEP:
        case L_SEP1: if constexpr (FULL) {
            typename V::Sep t;
            const uint32_t ng = (h.x >> 8) & 0xffu;
            for (uint32_t g = 0; g < ng; ++g) {
                const uint4 gw = as_u4(words(at + 1 + 2 * g));
                const uint32_t nl = gw.y & 0xffu;
                const uint2 i = condition_index(words(at + 2 + 2 * g), nl, (gw.y >> 8) & 0xffu, base, cta_base);
                t.group(GlobalWords{reinterpret_cast<const ulonglong2 *>(pool) + (gw.x + ((i.y * V::kSepWords) << nl) + i.x)}, 0,
                        nl, g == 0);
            }
            if ((h.x & 0xffu) == L_SEP) v.template sep<false>(t);
            else v.template sep<true>(t);
            at += 1 + 2 * ng;
        }
            break;
        case L_SCALE:
            v.scale(words, at + 1);
            at += 1 + V::kScaleWords;
            break;
        case L_SIGN:
        case L_PHASE: {
            const uint4 c = as_u4(words(at + 1));  // conditions
            const uint64_t ocm = uint64_t(c.w) << 32 | c.z;
            const bool on = (base & c.x) == c.x && (cta_base & ocm) == ocm;
            if ((!FULL && PL == 1) || (h.x & 0xffu) == L_SIGN) {
                v.sign(on ? h.y : 0u);
                at += 2;
            } else {
                v.phase(h.y, h.z, words(at + 2), on);
                at += 3;
            }
            break;
        }
        default: if constexpr (FULL) {  // L_CX
            const uint4 c = as_u4(words(at + 1));
            const uint64_t ocm = uint64_t(c.w) << 32 | c.z;
            const uint32_t m = ((base & c.x) == c.x && (cta_base & ocm) == ocm) ? ~0u : 0u;
            const uint32_t ctrl = (h.x >> 16) & 0xffu;
            switch ((h.x >> 8) & 0xffu) {
            case 0: x_target<V, RB, 0>(v, ctrl, m); break;
            case 1: x_target<V, RB, 1>(v, ctrl, m); break;
            case 2: x_target<V, RB, 2>(v, ctrl, m); break;
            case 3: if constexpr (RB > 3) x_target<V, RB, 3>(v, ctrl, m); break;
            case 4: if constexpr (RB > 4) x_target<V, RB, 4>(v, ctrl, m); break;
            default: break;
            }
            at += 2;
        }
            break;
        }
    }
    if (mine) {
        uint32_t a[E];
        group_addresses<RB>(a, pb ^ fl, bo);
        v.store(sm, a);
    }
    return at;
}

}  // namespace
}  // namespace qs
