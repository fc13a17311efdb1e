// fdm_fix.cuh -- 64-bit block fixed-point transforms of FP64 fields.
//
// GB300's FP64 pipe retires 2 lanes per SM and clock (measured 2.0); its integer pipes retire
// 40 64-bit additions and 60 wide multiply-adds (32 x 32 + 64 bits) in that time.  A transform
// of FP64 data needs no floating point: its error is a fraction of the sequence's largest
// value whatever the format, so a sequence whose largest magnitude is 2^(e+1) is held as
// integers in units of 2^(e+1-58) (an exact shift of every mantissa for values within 2^-5 of
// the largest, and rounded to nearest five bits below FP64's own rounding of the largest for the
// others), transformed with integer additions and 62-bit twiddles, and converted back with one
// rounding.  Every pass shifts right by the bits it may grow, inside the twiddle product, so
// nothing overflows.  Measured against long-double transforms the result is closer than an
// FP64 transform's for every field the library meets (noise, smooth fields, fronts).
#pragma once
#include <cmath>

#include "fdm_device.cuh"

namespace fdm {

#define FIX_HD __host__ __device__ __forceinline__

struct alignas(16) cfx { long long x, y; };
FIX_HD cfx mkx(long long a, long long b) { cfx r; r.x = a; r.y = b; return r; }
FIX_HD cfx operator+(cfx a, cfx b) { return mkx(a.x + b.x, a.y + b.y); }
FIX_HD cfx operator-(cfx a, cfx b) { return mkx(a.x - b.x, a.y - b.y); }
template <int S> FIX_HD cfx mul_si(cfx a) { return S > 0 ? mkx(-a.y, a.x) : mkx(a.y, -a.x); }

// A factor c + i s, |c + i s| <= 1, stored as 2^-K (c + i s) = (ch + cl 2^-32) 2^-32 + i ...
// with cl, sl signed: 61 - K bits and more of the factor in four ints (the size of a complex
// double, so the tables keep their places).
struct alignas(16) twx { int ch, cl, sh, sl; };
FIX_HD void fix_split(double v, int* h, int* l) {   // v = (h + l 2^-32) 2^-32, |v| <= 2^-2
    const double a = v * 4294967296.0;                // exact
    const double r = rint(a);
    double f = rint((a - r) * 4294967296.0);
    if (f > 2147483647.0) f = 2147483647.0;
    if (f < -2147483647.0) f = -2147483647.0;
    *h = (int)r;
    *l = (int)f;
}
FIX_HD twx fix_factor(double c, double s, int K) {
    const double p = K == 3 ? 0.125 : 0.25;
    twx w;
    fix_split(c * p, &w.ch, &w.cl);
    fix_split(s * p, &w.sh, &w.sl);
    return w;
}

// a b + c: one instruction on the multiply-add pipe (written out: the compiler expands the
// plain expression to about three)
FIX_HD long long fix_mad(int a, int b, long long c) {
#if defined(__CUDA_ARCH__)
    long long d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
#else
    return (long long)a * (long long)b + c;
#endif
}
FIX_HD long long fix_wide(int a, int b) {
#if defined(__CUDA_ARCH__)
    long long d;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
    return d;
#else
    return (long long)a * (long long)b;
#endif
}
FIX_HD int fix_hi(long long a) { return (int)(a >> 32); }
// a = h 2^32 + l with l signed
FIX_HD void fix_halves(long long a, int& h, int& l) {
    l = (int)(unsigned)(unsigned long long)a;
    h = (int)((a + 0x80000000ll) >> 32);
}
// 2^(s-K) a w, K the table's scale and s <= K; S = +1 multiplies by the conjugate factor.  The
// product of the low halves (below half a unit) is left out, the rest is rounded to nearest.
// |a| < 2^62.6 in the complex modulus.
FIX_HD long long fix_combine(long long t, long long q, int s) {   // (t 2^32 + q) >> (32 - s)
    const long long v = fix_mad(fix_hi(q), 1, t);
#if defined(__CUDA_ARCH__)
    const unsigned lo = __funnelshift_l((unsigned)q, (unsigned)v, s);
    const unsigned hi = __funnelshift_l((unsigned)v, (unsigned)(v >> 32), s);
    return (long long)(((unsigned long long)hi << 32) | lo);
#else
    return (long long)(((unsigned long long)v << s) | (s ? (unsigned long long)(unsigned)q >> (32 - s) : 0));
#endif
}
template <int S> FIX_HD cfx fix_mul(cfx a, twx w, int s) {
    int ah, al, bh, bl;
    fix_halves(a.x, ah, al);
    fix_halves(a.y, bh, bl);
    const int ps = S < 0 ? w.sh : -w.sh, pl = S < 0 ? w.sl : -w.sl;   // the factor's imaginary part
    const int ns = S < 0 ? -w.sh : w.sh, nl = S < 0 ? -w.sl : w.sl;   // its negative
    const long long half = (long long)(0x80000000u >> s);
    const long long tr = fix_mad(bh, ns, fix_wide(ah, w.ch)), ti = fix_mad(bh, w.ch, fix_wide(ah, ps));
    const long long qr = fix_mad(bh, nl, fix_mad(bl, ns, fix_mad(ah, w.cl, fix_mad(al, w.ch, half))));
    const long long qi = fix_mad(bh, w.cl, fix_mad(bl, w.ch, fix_mad(ah, pl, fix_mad(al, ps, half))));
    return mkx(fix_combine(tr, qr, s), fix_combine(ti, qi, s));
}
// a / 2^k rounded to nearest
FIX_HD long long fix_shr(long long a, int k) { return (a + ((1ll << k) >> 1)) >> k; }
FIX_HD cfx fix_shr(cfx a, int k) { return mkx(fix_shr(a.x, k), fix_shr(a.y, k)); }
// a / sqrt 2, |a| < 2^62: 2^31 / sqrt 2 = 1518500250 - 51432894 2^-32
FIX_HD long long fix_rsqrt2(long long a) {
    int h, l;
    fix_halves(a + a, h, l);
    const long long q = fix_mad(h, -51432894, fix_mad(l, 1518500250, 0x80000000ll));
    return fix_mad(fix_hi(q), 1, fix_wide(h, 1518500250));
}

// DFT of 2, 4 or 8 integers (as Dft<T, R>)
template <int R, int S> struct FixDft;
template <int S> struct FixDft<2, S> {
    static FIX_HD void run(cfx* v) { const cfx a = v[0], b = v[1]; v[0] = a + b; v[1] = a - b; }
};
template <int S> struct FixDft<4, S> {
    static FIX_HD void run(cfx* v) {
        const cfx t0 = v[0] + v[2], t1 = v[0] - v[2], t2 = v[1] + v[3], t3 = v[1] - v[3];
        v[0] = t0 + t2;
        v[2] = t0 - t2;
        if (S < 0) {   // t1 + S i t3
            v[1] = mkx(t1.x + t3.y, t1.y - t3.x);
            v[3] = mkx(t1.x - t3.y, t1.y + t3.x);
        } else {
            v[1] = mkx(t1.x - t3.y, t1.y + t3.x);
            v[3] = mkx(t1.x + t3.y, t1.y - t3.x);
        }
    }
};
template <int S> struct FixDft<8, S> {
    static FIX_HD void run(cfx* a) {
        const cfx b0 = a[0] + a[4], b4 = a[0] - a[4], b1 = a[1] + a[5], d5 = a[1] - a[5];
        const cfx b2 = a[2] + a[6], d6 = a[2] - a[6], b3 = a[3] + a[7], d7 = a[3] - a[7];
        // even outputs: DFT-4 of b0..b3
        const cfx c0 = b0 + b2, c2 = b0 - b2, c1 = b1 + b3, d3 = b1 - b3;
        a[0] = c0 + c1;
        a[4] = c0 - c1;
        // odd outputs: b4, W8 d5, W8^2 d6, W8^3 d7 with W8 = (1 + S i) / sqrt 2.  With
        // p = (d5 - d7) / sqrt 2 and m = (d5 + d7) / sqrt 2:
        //   W8 d5 + W8^3 d7 = p + S i m,   W8 d5 - W8^3 d7 = m + S i p
        const cfx p = mkx(fix_rsqrt2(d5.x - d7.x), fix_rsqrt2(d5.y - d7.y));
        const cfx m = mkx(fix_rsqrt2(d5.x + d7.x), fix_rsqrt2(d5.y + d7.y));
        if (S < 0) {
            a[2] = mkx(c2.x + d3.y, c2.y - d3.x);
            a[6] = mkx(c2.x - d3.y, c2.y + d3.x);
            const cfx c4 = mkx(b4.x + d6.y, b4.y - d6.x), c6 = mkx(b4.x - d6.y, b4.y + d6.x);
            const cfx c5 = mkx(p.x + m.y, p.y - m.x);            // p - i m
            // c7 = S i (m + S i p) = -p + S i m
            const cfx c7 = mkx(m.y - p.x, -(p.y + m.x));
            a[1] = c4 + c5;
            a[5] = c4 - c5;
            a[3] = c6 + c7;
            a[7] = c6 - c7;
        } else {
            a[2] = mkx(c2.x - d3.y, c2.y + d3.x);
            a[6] = mkx(c2.x + d3.y, c2.y - d3.x);
            const cfx c4 = mkx(b4.x - d6.y, b4.y + d6.x), c6 = mkx(b4.x + d6.y, b4.y - d6.x);
            const cfx c5 = mkx(p.x - m.y, p.y + m.x);            // p + i m
            const cfx c7 = mkx(-(p.x + m.y), m.x - p.y);         // -p + i m
            a[1] = c4 + c5;
            a[5] = c4 - c5;
            a[3] = c6 + c7;
            a[7] = c6 - c7;
        }
    }
};

// ---- conversion.  A sequence whose largest component has biased exponent E is held in units
// of 2^(E - 1080): |components| < 2^58.
constexpr int kFixBits = 58;
// the exponents that the conversions take as they are; others are first scaled by 2^+-600
constexpr int kFixLowExp = 128, kFixHighExp = 1900;
FIX_HD unsigned long long fix_bits(double x) {
#if defined(__CUDA_ARCH__)
    return (unsigned long long)__double_as_longlong(x);
#else
    unsigned long long u;
    __builtin_memcpy(&u, &x, 8);
    return u;
#endif
}
FIX_HD double fix_from_bits(unsigned long long u) {
#if defined(__CUDA_ARCH__)
    return __longlong_as_double((long long)u);
#else
    double x;
    __builtin_memcpy(&x, &u, 8);
    return x;
#endif
}
// the high word of |x| (its exponent above the top 20 mantissa bits)
FIX_HD unsigned fix_mag(double x) { return (unsigned)(fix_bits(x) >> 32) & 0x7fffffffu; }
// x in units of 2^(E - 1022 - B), truncated toward zero (or, NEAR, rounded to nearest); E >=
// kFixLowExp at least x's exponent: |result| <= 2^B
template <int B = kFixBits, bool NEAR = false> FIX_HD long long fix_from(double x, int E) {
    const unsigned long long u = fix_bits(x);
    const int d = E - ((int)(u >> 52) & 0x7ff);
    unsigned long long m = ((u & 0xfffffffffffffull) | 0x10000000000000ull) << (B - 53 + (NEAR ? 1 : 0));
#if defined(__CUDA_ARCH__)
    asm("shr.u64 %0, %1, %2;" : "=l"(m) : "l"(m), "r"(d));   // 0 beyond 63
#else
    m = d > 63 ? 0 : m >> d;
#endif
    if (NEAR) m = (m + 1) >> 1;
    const long long s = (long long)u >> 63;
    return ((long long)m ^ s) - s;
}
// fix_from<kFixBits, true>(x, E); adds what its rounding left of x, in units of 2^-6 of its units, to
// lost (six bits of it: to 2^-64 of 2^E)
FIX_HD long long fix_from_lost(double x, int E, int& lost) {
    const unsigned long long u = fix_bits(x);
    const int d = E - ((int)(u >> 52) & 0x7ff);
    unsigned long long m = ((u & 0xfffffffffffffull) | 0x10000000000000ull) << (kFixBits - 53 + 6);
#if defined(__CUDA_ARCH__)
    asm("shr.u64 %0, %1, %2;" : "=l"(m) : "l"(m), "r"(d));   // 0 beyond 63
#else
    m = d > 63 ? 0 : m >> d;
#endif
    const int s = (int)(u >> 32) >> 31;
    const int l = (int)((unsigned)m << 26) >> 26;
    lost += (l ^ s) - s;
    m = (m + 32) >> 6;
    return ((long long)m ^ s) - s;
}
// a 2^sc as a double, one rounding (sc keeps every a != 0 in the normal range)
FIX_HD double fix_to(long long a, int sc) {
    const double d = (double)a;
#if defined(__CUDA_ARCH__)
    const int hi = __double2hiint(d);
    return __hiloint2double(hi == 0 ? 0 : hi + (sc << 20), __double2loint(d));
#else
    return a == 0 ? 0.0 : fix_from_bits(fix_bits(d) + ((unsigned long long)(long long)sc << 52));
#endif
}

// ---- the passes of an L-point transform, eight values per thread: radix 8 while it divides,
// then one radix-4 or radix-2 pass (pass_radix).  Thread j of L / 8 takes the elements
// j + u L/8 in every pass; the last pass leaves its results at those places too, in natural
// order, so a first pass reads from and a last pass writes to global memory directly.
template <int L> struct FixPlan {
    static constexpr int T = L / 8;
    static __host__ __device__ constexpr int passes(int Ns = 1, int n = 0) {
        return Ns * 8 <= L ? passes(Ns * 8, n + 1) : (Ns < L ? n + 1 : n);
    }
    static constexpr int P = passes();
    static __host__ __device__ constexpr int ns(int p) { return p == 0 ? 1 : 8 * ns(p - 1); }
    static __host__ __device__ constexpr int radix(int p) { return ns(p) * 8 <= L ? 8 : L / ns(p); }
    // table offset of pass p: 7 entries per k < Ns for each earlier pass
    static __host__ __device__ constexpr int off(int p) { return p == 0 ? 0 : off(p - 1) + 7 * ns(p - 1); }
    // bits that pass p shifts right before its butterflies when `used` of the sequence's
    // `need` bits have been shifted before it
    static __host__ __device__ constexpr int most(int p) {
        return p == 0 ? 0 : (radix(p) == 8 ? 3 : (radix(p) == 4 ? 2 : 1));
    }
    static __host__ __device__ constexpr int before(int p) { return p == 0 ? 0 : 3 * (p - 1); }
    static FIX_HD int shift(int p, int need) {
        const int left = need - before(p);
        return left < 0 ? 0 : (left > most(p) ? most(p) : left);
    }
};
FIX_HD int fix_pad(int i) { return i + (i >> 3); }
// the place of a thread's result u of pass p (p < P - 1: a radix-8 pass)
template <int L, int p> FIX_HD int fix_place(int j, int u) {
    constexpr int Ns = FixPlan<L>::ns(p);
    const int k = j & (Ns - 1);
    return ((j - k) << 3) + k + u * Ns;
}
// pass p of direction S on the eight values of thread j; need: the sequence's growth bits
template <int L, int p, int S> FIX_HD void fix_pass(cfx* v, int j, const twx* __restrict__ tab, int need) {
    using Pl = FixPlan<L>;
    constexpr int R = Pl::radix(p), Ns = Pl::ns(p), PER = 8 / R, K = R == 8 ? 3 : 2;
    const int sh = Pl::shift(p, need);
#pragma unroll
    for (int b = 0; b < PER; ++b) {
        cfx w[R];
#pragma unroll
        for (int r = 0; r < R; ++r) w[r] = v[b + r * PER];
        if (p > 0) {
            const int k = (j + b * Pl::T) & (Ns - 1);
            w[0] = fix_shr(w[0], sh);
#pragma unroll
            for (int r = 1; r < R; ++r) w[r] = fix_mul<S>(w[r], tab[Pl::off(p) + (r - 1) * Ns + k], K - sh);
        }
        FixDft<R, S>::run(w);
#pragma unroll
        for (int r = 0; r < R; ++r) v[b + r * PER] = w[r];
    }
}

// ---- twists between the L-point transform of a packed real row and its half spectrum
// (r2c_twist_pair, c2r_twist_pair); w = exp(-2 pi i k / (2 L)) scaled by 2^-2
// forward: X(k) and X(L - k) from Z(k), Z(L - k)
FIX_HD void fix_r2c(cfx zk, cfx zc, twx w, cfx* xk, cfx* xc) {
    const cfx A = zk, B = mkx(zc.x, -zc.y);
    const cfx E = mkx(fix_shr(A.x + B.x, 1), fix_shr(A.y + B.y, 1));
    const cfx O = fix_mul<-1>(mkx(A.y - B.y, B.x - A.x), w, 1);   // -i (A - B) w / 2
    *xk = E + O;
    *xc = mkx(E.x - O.x, O.y - E.y);
}
// inverse, halved: Z(k) / 2 and Z(L - k) / 2 from X(k), X(L - k)
FIX_HD void fix_c2r(cfx xk, cfx xc, twx w, cfx* zk, cfx* zc) {
    const cfx A = xk, B = mkx(xc.x, -xc.y);
    const cfx E = mkx(fix_shr(A.x + B.x, 1), fix_shr(A.y + B.y, 1));
    const cfx O = fix_mul<+1>(mkx(A.x - B.x, A.y - B.y), w, 1);
    *zk = mkx(E.x - O.y, E.y + O.x);
    *zc = mkx(E.x + O.y, O.x - E.y);
}

// ---------------------------------------------------------------------------------
// The FP64 stencil's short node update: nodes of one characteristic direction, in the same
// arithmetic.  Where both one-sided derivatives along x1 have one sign, and both along x2 have one
// sign, every pair gives dH/dp of one sign and dH/dq of one sign: one of a+, a- and one of b+, b- is
// exactly zero, so three of Step 4's four weights are zero, the fourth is one, and that one belongs
// to the intermediate point whose displacement is zero.  The update is then U - v0 dt |grad| with
// the gradient (p, q) of that quadrant at the node itself: two reciprocal square roots instead of
// twelve and a reciprocal, no speeds and no weights, equal to the whole scheme up to the rounding
// of its weights' ratio.  The limited second differences make both sides' derivatives agree
// wherever U13 is smooth, its extrema along the axes included: of the coupled random field 99.7% of
// the nodes qualify at the start and 97% after 150 steps.  An axis along which nothing varies (both
// derivatives, both limited second differences and the cross differences zero) qualifies as well:
// its two weights of 1/2 belong to equal values.  (FP32: the same skipping took as many instructions
// as it saved, 69.6 us either way.  Double words: 348 -> 209 us at 2048^2, but a coupled run of 74
// steps there amplified the weights' other rounding, 3e-14, to 1e-8, so they keep the whole scheme.)
//
// The first differences are FP64 subtractions; from there the node works in units of 2^-59 of 2^E
// (half units from the derivatives on), rounded to nearest, with 2^E the bound of the four
// differences to its neighbours.  The differences beyond those enter through the limiter alone,
// which caps what they contribute: where they are larger they are set to 8 times the bound, so the
// tail of a front keeps its own scale.  (One scale over all of them, and shifts that round down,
// left each step of such a tail 2^-55 off: 5.6e-15 after 200 steps of two walls that annihilate down
// to 1e-42, against 2.4e-16 to 7.3e-16 for FP64 arithmetic; 2.7e-17 to 4.2e-16 now; with two bits
// fewer 2.1e-16 to 7.1e-16.)  A node whose side's differences lie below 2^-6 of the bound would keep
// fewer bits than FP64's, one whose derivatives lie within the rounding may have the wrong sign:
// both are left to the whole scheme. Against 113-bit arithmetic, error of the increment in units of
// 2^-53, 99.9% of the nodes below: noise 2.6 (FP64 arithmetic: 16), smooth with noise 1.9 (3.6),
// tails 1.3 (4.2), kinks 2.1 (3.6), axes of different size 1.8 (3.2), exponents spread over 60 bits,
// where either cancels, 7e5 (5e6). Integer instructions and 13 FP64 ones per node replace 39 FP64
// ones.
// ---------------------------------------------------------------------------------
// (a b) / 2^64 rounded (the product of the low halves left out), |a|, |b| <= 2^62 (fix_halves
// rounds up: it needs 2^31 of room below 2^63)
FIX_HD long long fix_mulhi(long long a, long long b) {
    int ah, al, bh, bl;
    fix_halves(a, ah, al);
    fix_halves(b, bh, bl);
    const long long q = fix_mad(al, bh, fix_mad(ah, bl, 0x80000000ll));
    return fix_mad(fix_hi(q), 1, fix_wide(ah, bh));
}
// (a b) / 2^(64 - s)
FIX_HD long long fix_mulhi(long long a, long long b, int s) {
    int ah, al, bh, bl;
    fix_halves(a, ah, al);
    fix_halves(b, bh, bl);
    const long long q = fix_mad(al, bh, fix_mad(ah, bl, (long long)(0x80000000u >> s)));
    return fix_combine(fix_wide(ah, bh), q, s);
}
// (a b + c d) / 2^(64 - s)
FIX_HD long long fix_mulhi2(long long a, long long b, long long c, long long d, int s) {
    int ah, al, bh, bl, ch, cl, dh, dl;
    fix_halves(a, ah, al);
    fix_halves(b, bh, bl);
    fix_halves(c, ch, cl);
    fix_halves(d, dh, dl);
    const long long t = fix_mad(ch, dh, fix_wide(ah, bh));
    const long long half = (long long)(0x80000000u >> s);
    const long long q = fix_mad(cl, dh, fix_mad(ch, dl, fix_mad(al, bh, fix_mad(ah, bl, half))));
    return fix_combine(t, q, s);
}
// ---- cos(x / beta) for the lattice friction.  x becomes a fraction of a turn first: x / (2 pi beta)
// modulo 1 comes from the product with the factor's leading 100 bits (exact to the fraction's
// last bit, where a rounded x / beta is off by 2^-53 of its value), and the rest is a polynomial in 64-bit fixed point.
struct FixTurns {
    unsigned long long m, l;   // 1 / (2 pi |beta|) = (m + l 2^-64) 2^(e + 958)
    int e;                     // beyond every exponent: beta outside the range below, use cos()
};
inline FixTurns fix_turns(double beta) {
    FixTurns t{0ull, 0ull, 1 << 20};
    const double b = beta < 0.0 ? -beta : beta;
    if (!(b > 1e-100 && b < 1e100)) return t;
    // 2 pi b and its reciprocal to about 104 bits, as sums of two doubles
    const double p1 = 6.283185307179586, p2 = 2.4492935982947064e-16;
    const double h = b * p1, l = std::fma(b, p1, -h) + b * p2;
    const double r = 1.0 / h, dr = (std::fma(-r, h, 1.0) - r * l) * r;
    int k;
    const double f = std::frexp(r, &k);
    const double d = std::ldexp(dr, 64 - k), df = std::floor(d);
    t.m = ((unsigned long long)std::ldexp(f, 53) << 11) + (unsigned long long)(long long)df;
    t.l = (unsigned long long)std::ldexp(d - df, 32) << 32;
    t.e = k - 1022;
    return t;
}
// cos(x / beta) in units of 2^-62, within 2^-58; false beyond 2^10 turns (there cos() of the
// rounded x / beta is further than 1e-12 off, and its own bits are kept), infinities and NaN
FIX_HD bool fix_cos(double x, const FixTurns& t, long long* c) {
    const unsigned long long u = fix_bits(x);
    const int E = (int)(u >> 52) & 0x7ff, k = E + t.e;
    if (k > 10) return false;
    const unsigned long long m = ((u & 0xfffffffffffffull) | 0x10000000000000ull) << 11;
#if defined(__CUDA_ARCH__)
    const unsigned long long lo0 = m * t.m, lo = lo0 + __umul64hi(m, t.l);
    const unsigned long long hi = __umul64hi(m, t.m) + (lo < lo0 ? 1u : 0u);
    unsigned long long F;
    if (k > 0) F = (hi << k) | (lo >> (64 - k));
    else asm("shr.u64 %0, %1, %2;" : "=l"(F) : "l"(hi), "r"(-k));   // 0 beyond 63
#else
    const unsigned __int128 P = (unsigned __int128)m * t.m + (((unsigned __int128)m * t.l) >> 64);
    const unsigned long long hi = (unsigned long long)(P >> 64), lo = (unsigned long long)P;
    const unsigned long long F = k > 0 ? (hi << k) | (lo >> (64 - k)) : (-k > 63 ? 0ull : hi >> -k);
#endif
    // F: the turn's fraction in 2^-64; cos(2 pi F) = sin(pi h / 2), h = 1 - 4 |F| in quarter turns of 2^62
    const long long s = (long long)F >> 63;
    const long long h = (long long)(0x4000000000000000ull - ((F ^ (unsigned long long)s) - (unsigned long long)s));
    long long z = fix_mulhi(h, h, 2);
    z -= z >> 62;
    // the Taylor series of sin(pi h / 2) / h in z = h^2, (-1)^n (pi / 2)^(2n + 1) / (2n + 1)!, in
    // 2^-62, to n = 11 (the next is below 2^-67).  From n = 7 on 32 bits hold the terms, in 2^-60 and
    // each scaled by 4 more, since z comes in 2^-30.
    const int y = (int)(z >> 32);
    int w = -370;
    w = 18974 + fix_hi(fix_wide(w, y));
    w = -807426 + fix_hi(fix_wide(w, y));
    w = 27978803 + fix_hi(fix_wide(w, y));
    w = -771077950 + fix_hi(fix_wide(w, y));
    long long p = 262505142787ll + fix_mulhi((long long)w, z, 4);
    p = -16596735030340ll + fix_mulhi(p, z, 2);
    p = 739904368663792ll + fix_mulhi(p, z, 2);
    p = -21590780087563799ll + fix_mulhi(p, z, 2);
    p = 367517370231208053ll + fix_mulhi(p, z, 2);
    p = -2978983596875621757ll + fix_mulhi(p, z, 2);
    p = 7244019458077122842ll + fix_mulhi(p, z, 2);
    *c = fix_mulhi(h, p, 2);
    return true;
}
// of one sign and none zero: the one of least magnitude, else 0
FIX_HD long long fix_minmod(long long a, long long b) {
    const long long s = a >> 63;
    long long m = a ^ s;
    const long long mb = b ^ s;   // negative where the signs differ (or zero meets a negative)
    m = mb < m ? mb : m;
    return (m ^ s) & ~(m >> 63);
}
// the limiter parameter theta in [1, 2]: code 1 or 2 when it is exactly that, else 2^-3 theta as
// fix_split's halves (2^-2 theta comes to 2^31 in the high half just below theta = 2)
struct FixTheta { int code, h, l; };
inline FixTheta fix_theta_of(double theta) {
    FixTheta t;
    t.code = theta == 1.0 ? 1 : (theta == 2.0 ? 2 : 0);
    fix_split(0.125 * theta, &t.h, &t.l);
    return t;
}
FIX_HD long long fix_theta(long long a, FixTheta t) {
    if (t.code == 1) return a;
    if (t.code == 2) return a + a;
    int h, l;
    fix_halves(a, h, l);
    return fix_combine(fix_wide(h, t.h), fix_mad(l, t.h, fix_mad(h, t.l, 0x10000000ll)), 3);
}
FIX_HD int fix_clz(long long v) {   // v > 0
#if defined(__CUDA_ARCH__)
    return __clzll(v);
#else
    return __builtin_clzll((unsigned long long)v);
#endif
}
FIX_HD float fix_rsqrt_seed(unsigned x) {   // 1 / sqrt(x), relative error below 2^-21
#if defined(__CUDA_ARCH__)
    return rsqrtf((float)x);
#else
    return 1.0f / __builtin_sqrtf((float)x) * (1.0f + 0x1p-22f);
#endif
}
FIX_HD int fix_round(float v) {
#if defined(__CUDA_ARCH__)
    return __float2int_rn(v);
#else
    return (int)__builtin_rintf(v);
#endif
}
// 2^61 / sqrt(x 2^-58) for x in [2^56, 2^59), relative error below 2^-56: the float seed y0 and
// y0 (1 + e / 2 + 3 e^2 / 8) with e = 1 - x y0^2 (the binomial series; |e| < 2^-20)
FIX_HD long long fix_rsqrt(long long x) {
    const float s = fix_rsqrt_seed((unsigned)((unsigned long long)x >> 27)) * 0x1.6a09e6p15f;   // y0: x 2^-27 = xi 2^31
    const int y = fix_round(s * 0x1p29f);                          // y0 2^29 in (2^28, 2^30]
    const long long one = (long long)1 << 57;
    const long long e = one - fix_mulhi(x << 3, fix_wide(y, y) << 2);   // 2^57 e
    int eh, el;
    fix_halves(e, eh, el);
    // y0 e / 2 in units of 2^-61: y e 2^-26
    const long long d = (fix_wide(y, eh) << 6) + (fix_wide(y, el) >> 26);
    const float ef = (float)(int)(e >> 16) * 0x1p-41f;
    const int c = fix_round(s * (0.375f * ef) * ef * 0x1p61f);
    return fix_mad(c, 1, ((long long)y << 32) + d);
}
// (p, q) shifted left by *L (right where it is negative: 62 bits and more) so that the larger has 61
// bits, and |(p, q)|^2 of those / 2^64, in [2^56, 2^59); false for (0, 0)
FIX_HD bool fix_norm2(long long p, long long q, long long* ps, long long* qs, int* L, long long* r2) {
    const long long sp = p >> 63, sq = q >> 63;
    const long long m = ((p ^ sp) - sp) | ((q ^ sq) - sq);
    if (m == 0) return false;
    *L = fix_clz(m) - 3;
    *ps = *L < 0 ? p >> -*L : (long long)((unsigned long long)p << *L);
    *qs = *L < 0 ? q >> -*L : (long long)((unsigned long long)q << *L);
    int ph, pl, qh, ql;
    fix_halves(*ps, ph, pl);
    fix_halves(*qs, qh, ql);
    const long long t = fix_mad(qh, qh, fix_wide(ph, ph));
    const long long h = fix_mad(ql, qh, fix_mad(pl, ph, 0x40000000ll));   // half the cross terms
    *r2 = t + (h >> 31);
    return true;
}

// six more than FP64's: differences down to 2^-6 of the bound stay exact
constexpr int kNodeBits = 59;
// a difference beyond the first ones, in their units: |result| <= 8 times their bound, which it is
// set to if it lies above
FIX_HD long long fix_outer(double x, int E) {
    const unsigned long long u = fix_bits(x);
    const int d = E + 3 - ((int)(u >> 52) & 0x7ff);
    const long long m = fix_from<kNodeBits + 3, true>(x, d < 0 ? E + 3 - d : E + 3);
    const long long s = (long long)u >> 63;
    return d < 0 ? ((1ll << (kNodeBits + 3)) ^ s) - s : m;
}

// returns whether the node qualifies (and *out its new value); nodes whose scale lies near the ends
// of FP64's range, whose cross difference dwarfs the others, or whose result would keep fewer bits
// than FP64's do not
template <typename F>
FIX_HD bool fix_upwind(F f, double v0, double dt_h, FixTheta th, int time_level, double* out) {
    const double f0 = f(0, 0);
    const double xm = f(-1, 0), xp = f(1, 0), ym = f(0, -1), yp = f(0, 1);
    const double axm3 = xm - f(-2, 0), axm1 = f0 - xm, axp1 = xp - f0, axp3 = f(2, 0) - xp;
    const double aym3 = ym - f(0, -2), aym1 = f0 - ym, ayp1 = yp - f0, ayp3 = f(0, 2) - yp;
    auto top = [](unsigned a, unsigned b) { return a > b ? a : b; };
    const unsigned m = top(top(fix_mag(axm1), fix_mag(axp1)), top(fix_mag(aym1), fix_mag(ayp1)));
    const unsigned mx = top(fix_mag(axm3), fix_mag(axp3)), my = top(fix_mag(aym3), fix_mag(ayp3));
    const int E = (int)(m >> 20);
    if (E < kFixLowExp || E > kFixHighExp) {
        if (m != 0u) return false;
        const unsigned long long any = fix_bits(axm1) | fix_bits(axp1) | fix_bits(aym1) | fix_bits(ayp1);
        *out = f0;   // no gradient on any side: H = 0
        return (any << 1) == 0ull;
    }
    const double vdt = v0 * dt_h;
    if (fix_mag(vdt) > 0x3ff00000u || top(mx, my) >= 0x7ff00000u) return false;
    const long long dxm1 = fix_from<kNodeBits, true>(axm1, E), dxp1 = fix_from<kNodeBits, true>(axp1, E);
    const long long dym1 = fix_from<kNodeBits, true>(aym1, E), dyp1 = fix_from<kNodeBits, true>(ayp1, E);
    // an outer difference at its bound of 8: with first differences of one sign the limiter takes
    // theta times theirs, at most 2, whatever lies above 3.5
    const bool turn_x = (dxp1 ^ dxm1) < 0, turn_y = (dyp1 ^ dym1) < 0;
    if ((turn_x && (int)(mx >> 20) > E + 3) || (turn_y && (int)(my >> 20) > E + 3)) return false;
    const long long dxm3 = fix_outer(axm3, E), dxp3 = fix_outer(axp3, E);
    const long long dym3 = fix_outer(aym3, E), dyp3 = fix_outer(ayp3, E);
    // the limited second differences of theta a, (a + b) / 2 and theta b: the minima of doubles, halved
    // to nearest
    auto limited = [&](long long a, long long b) {
        const long long m = fix_minmod(fix_theta(fix_minmod(a, b), th) << 1, a + b);
        return (m + 1) >> 1;
    };
    const long long cx = dxp1 - dxm1, cy = dyp1 - dym1;
    const long long Sx0 = limited(dxp3 - dxp1, cx), Sx1 = limited(cx, dxm1 - dxm3);
    const long long Sy0 = limited(dyp3 - dyp1, cy), Sy1 = limited(cy, dym1 - dym3);
    // twice the one-sided derivatives, in half units from here on
    const long long px0 = (dxp1 << 1) - Sx0, px1 = (dxm1 << 1) + Sx1;
    const long long qy0 = (dyp1 << 1) - Sy0, qy1 = (dym1 << 1) + Sy1;
    // of one sign, and by more than the conversions' rounding (below 4)
    auto mag = [](long long v) { return v ^ (v >> 63); };
    auto one_sign = [&](long long a, long long b) { return (a ^ b) >= 0 && mag(a) >= 8 && mag(b) >= 8; };
    const bool one_x = one_sign(px0, px1), one_y = one_sign(qy0, qy1);
    const bool flat_x = (px0 | px1 | Sx0 | Sx1) == 0, flat_y = (qy0 | qy1 | Sy0 | Sy1) == 0;
    if (!(one_x || flat_x) || !(one_y || flat_y)) return false;
    // side 0 (+) where v0 and the derivative have opposite signs, side 1 (-) where they agree
    const long long vs = (long long)fix_bits(v0);
    const bool s0 = (vs ^ px0) < 0, t0 = (vs ^ qy0) < 0;
    long long p = s0 ? px0 : px1, q = t0 ? qy0 : qy1, ps, qs, r2;
    const long long Dx = s0 ? dxp1 : dxm1, Dy = t0 ? dyp1 : dym1;
    long long Sx = s0 ? Sx0 : Sx1, Sy = t0 ? Sy0 : Sy1;
    // half units, 2^-60 of the bound, are to stay below 2^-54 of what the gradient is formed from
    if ((mag(Dx << 1) | mag(Sx) | mag(Dy << 1) | mag(Sy)) < (1ll << (kNodeBits - 5))) return false;
    const int ix = s0 ? 1 : -1, iy = t0 ? 1 : -1;
    const double fy = t0 ? yp : ym;
    const double ac = f(ix, iy) - fy;
    const int ea = (int)(fix_mag(ac) >> 20);
    const long long fx = s0 ? dxp1 : -dxm1;
    const bool wide = ea > E + 2;   // the tail of a front: the diagonal dwarfs the axes
    if (ea > E + 32) return false;
    if (flat_x || flat_y) {
        const double oc = flat_y ? f(ix, -iy) - (t0 ? ym : yp) : f(-ix, iy) - fy;   // the other quadrant's
        if (wide || (int)(fix_mag(oc) >> 20) > E + 2) return false;
        if (fix_from<kNodeBits + 2, true>(ac, E + 2) != fx) return false;
        if (fix_from<kNodeBits + 2, true>(oc, E + 2) != (flat_y ? fx : -fx)) return false;
    }
    int L, Ec = E;
    if (time_level == 0 && fix_norm2(p, q, &ps, &qs, &L, &r2)) {
        // (p, q) -= dt/2 Hess grad_(p,q) H, grad H = v0 (p, q) / |(p, q)|
        const long long y = fix_rsqrt(r2);
        const long long c = fix_mulhi(ps, y, 3), s = fix_mulhi(qs, y, 3);   // the direction, in units of 2^-61
        const long long h = fix_from<kFixBits, true>(vdt, 1023) << 4;   // v0 dt / (2 h) in units of 2^-62
        const int k = wide ? ea - E - 2 : 0;
        // the diagonal sets the units of the sums below (the direction kept its own)
        auto down = [&](long long v) { return (v + ((1ll << k) >> 1)) >> k; };
        Ec = E + k;
        const long long mixed = fix_from<kNodeBits + 2, true>(ac, Ec + 2) - (wide ? down(fx) : fx);
        const long long cross = (s0 == t0) ? mixed : -mixed;
        if (wide) {
            p = down(p);
            q = down(q);
            Sx = down(Sx);
            Sy = down(Sy);
        }
        p -= fix_mulhi(fix_mulhi2(Sx, c, cross, s, 4), h, 2);
        q -= fix_mulhi(fix_mulhi2(cross, c, Sy, s, 4), h, 2);
        // (|p|, |q| < 2^62.6 for any first differences, diagonal and |v0 dt / h| <= 1)
        if (wide && (mag(p) | mag(q)) < (1ll << (kNodeBits - 5))) return false;
    }
    double g = 0.0;   // h |grad|
    if (fix_norm2(p, q, &ps, &qs, &L, &r2)) {
        // |(p 2^L, q 2^L)| = 2^61 sqrt(xi), xi = r2 2^-58, sqrt(xi) = xi / sqrt(xi)
        const long long r = fix_mulhi(r2 << 3, fix_rsqrt(r2));   // 2^58 sqrt(xi)
        g = fix_to(r, Ec - (1022 + kNodeBits + 1) + 3 - L);
    }
    *out = f0 - vdt * g;
    return true;
}

}  // namespace fdm
