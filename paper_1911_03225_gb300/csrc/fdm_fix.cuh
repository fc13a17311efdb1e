// fdm_fix.cuh -- 64-bit block fixed-point transforms of FP64 fields.
//
// GB300's FP64 pipe retires 2 lanes per SM and clock (measured 2.0); its integer pipes retire
// 40 64-bit additions and 60 wide multiply-adds (32 x 32 + 64 bits) in that time.  A transform
// of FP64 data needs no floating point: its error is a fraction of the sequence's largest
// value whatever the format, so a sequence whose largest magnitude is 2^(e+1) is held as
// integers in units of 2^(e+1-58) (an exact shift of every mantissa for values within 2^-5 of
// the largest, and a truncation five bits below FP64's own rounding of the largest for the
// others), transformed with integer additions and 62-bit twiddles, and converted back with one
// rounding.  Every pass shifts right by the bits it may grow, inside the twiddle product, so
// nothing overflows.  Measured against long-double transforms the result is closer than an
// FP64 transform's for every field the library meets (noise, smooth fields, fronts).
#pragma once
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
// x in units of 2^(E - 1080), truncated toward zero; E >= kFixLowExp at least x's exponent
FIX_HD long long fix_from(double x, int E) {
    const unsigned long long u = fix_bits(x);
    const int d = E - ((int)(u >> 52) & 0x7ff);
    unsigned long long m = ((u & 0xfffffffffffffull) | 0x10000000000000ull) << 5;
#if defined(__CUDA_ARCH__)
    asm("shr.u64 %0, %1, %2;" : "=l"(m) : "l"(m), "r"(d));   // 0 beyond 63
#else
    m = d > 63 ? 0 : m >> d;
#endif
    const long long s = (long long)u >> 63;
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
    static __host__ __device__ constexpr int most(int p) { return p == 0 ? 0 : (radix(p) == 8 ? 3 : (radix(p) == 4 ? 2 : 1)); }
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

}  // namespace fdm
