// FP64 transforms of one axis in fixed point: the values of a line (a row or a
// column) are aligned to the line's largest exponent as 64-bit integers, run
// through all radix stages with integer additions and 64 x 64 -> 64-bit
// products, and are rounded back to FP64 once, after the last stage.
//
// Why: an SM executes 2 FP64 operations per clock but 64 integer ones (and 13
// 32 x 32 + 64-bit multiply-adds), and a transform is mostly additions.  Per SM
// a radix-16 butterfly with its 15 twiddles takes 127 clocks in FP64 and 48
// clocks here with both conversions; conversions are half of that, hence one
// each way per line and not per stage.
// Precision: the aligned values carry 57 (first radix 16) to 60 bits below the
// line's largest; a later stage shifts its inputs down by what its growth needs
// (stage_shift), while sums grow; shifts and products round to the nearest.  One
// rounding to 53 bits at the end replaces one per addition.  Relative L2 error
// against an extended-precision reference (one tensor row, mean stress twice the
// fluctuation), FP64 butterflies -> integers: projections 16^3 2.4e-16 -> 1.3e-16,
// 64^3 3.7e-16 -> 1.8e-16, 54 x 90 x 100 4.3e-16 -> 2.7e-16, 128 x 64 x 80 2.8e-16 ->
// 2.8e-16; operators with their contraction 64^3 5.1e-16 -> 2.6e-16, 54 x 90 x 100
// 6.4e-16 -> 3.7e-16, 108 x 96 x 50 6.0e-16 -> 3.1e-16.
// Range: a line whose largest exponent is near overflow or the subnormals, or
// which holds an infinity or a NaN, runs its stages in FP64 instead (fp64_bfly),
// so those propagate as they always did.
//
// Headroom: a stage's inputs have moduli of at most 2^62.5 / R, so every partial
// sum of R of them (times unit-modulus factors) stays below 2^62.5.
#pragma once

#include <cuda_runtime.h>

namespace gff {
namespace fx {

struct Cq {
    long long x, y;
};

// Fixed-point constant c (|c| <= 1, 62 fractional bits) as c = h 2^32 + l with l a signed 32-bit number.
struct Limbs {
    int h, l;
};
__host__ __device__ constexpr Limbs limbs_of(long long c) {
    const long long l = c - (((c + 0x80000000LL) >> 32) << 32);
    return Limbs{(int)((c - l) >> 32), (int)l};
}
__device__ __forceinline__ void split(long long a, int& h, int& l) {
    l = (int)a;
    h = (int)((unsigned)(a >> 32) + ((unsigned)l >> 31));
}
// The product (r 2^32 + p) / 2^62 from its partial sums r (high by high) and p (the cross terms, in units 2^32 lower),
// to the nearest integer: p starts at HALF, and the two low bits come from p.  (Left at zero, as the high word of the
// product shifted up by two has them, every product is a multiple of four units and about two too small, a bias that
// adds up over the stages of a plan.)
constexpr long long HALF = 1LL << 29;
__device__ __forceinline__ long long join(long long r, long long p) {
    r += (int)(p >> 32);
    const unsigned lo = __funnelshift_l((unsigned)p, (unsigned)r, 2);
    const unsigned hi = __funnelshift_l((unsigned)r, (unsigned)((unsigned long long)r >> 32), 2);
    return (long long)((unsigned long long)hi << 32 | lo);
}
// a c / 2^62 for |a| < 2^62.5: the low-by-low partial product (below a quarter unit) is dropped
__device__ __forceinline__ long long mul1(long long a, Limbs c) {
    int ah, al;
    split(a, ah, al);
    const long long p = HALF + (long long)ah * c.l + (long long)al * c.h;
    return join((long long)ah * c.h, p);
}
// (a ca + b cb) / 2^62 for |a|, |b| < 2^61.2 (two inputs of radix 5) and |ca| + |cb| <= 1.54 (its sines): the high
// halves are below 2^29.2 and the low ones at most 2^31, so |p| < 2 2^60.2 + 1.54 2^61 < 2^62.5 and |r| < 1.54 2^59.2
__device__ __forceinline__ long long mul2(long long a, Limbs ca, long long b, Limbs cb) {
    int ah, al, bh, bl;
    split(a, ah, al);
    split(b, bh, bl);
    const long long p = HALF + (long long)ah * ca.l + (long long)al * ca.h + (long long)bh * cb.l + (long long)bl * cb.h;
    return join((long long)ah * ca.h + (long long)bh * cb.h, p);
}

// Twiddle w = (x + i y), 62 fractional bits, as limbs (xh, xl, yh, yl); a w, or a conj(w) when CONJ, for |a| < 2^62.5
template <bool CONJ> __device__ __forceinline__ Cq twmul(Cq a, int4 w) {
    int xh, xl, yh, yl;
    split(a.x, xh, xl);
    split(a.y, yh, yl);
    const int nh = -w.z, nl = -w.w;  // (l > -2^31: limbs_of)
    const int rh = CONJ ? w.z : nh, rl = CONJ ? w.w : nl;  // re = ax wx + ay r
    const int ih = CONJ ? nh : w.z, il = CONJ ? nl : w.w;  // im = ay wx + ax i
    const long long p = HALF + (long long)xh * w.y + (long long)xl * w.x + (long long)yh * rl + (long long)yl * rh;
    const long long q = HALF + (long long)yh * w.y + (long long)yl * w.x + (long long)xh * il + (long long)xl * ih;
    return Cq{join((long long)xh * w.x + (long long)yh * rh, p), join((long long)yh * w.x + (long long)xh * ih, q)};
}
// the twiddle as FP64 (for the butterflies that stay in FP64)
__device__ __forceinline__ double2 tw_fp64(int4 w) {
    constexpr double s32 = 4294967296.0, s62 = 1.0 / 4611686018427387904.0;
    return make_double2(fma((double)w.x, s32, (double)w.y) * s62, fma((double)w.z, s32, (double)w.w) * s62);
}

__device__ __forceinline__ Cq add(Cq a, Cq b) { return Cq{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ Cq sub(Cq a, Cq b) { return Cq{a.x - b.x, a.y - b.y}; }
template <bool INV> __device__ __forceinline__ Cq rot90(Cq a) { return INV ? Cq{-a.y, a.x} : Cq{a.y, -a.x}; }
// a exp(-+ i theta), c = cos theta, s = sin theta
template <bool INV> __device__ __forceinline__ Cq turn(Cq a, long long c, long long s) {
    const Limbs lc = limbs_of(c), ls = limbs_of(s), ln = limbs_of(-s);
    return INV ? Cq{mul2(a.x, lc, a.y, ln), mul2(a.y, lc, a.x, ls)} : Cq{mul2(a.x, lc, a.y, ls), mul2(a.y, lc, a.x, ln)};
}
constexpr long long COS_PI8 = 4260642322793532497LL;  // round(2^62 cos(pi / 8)), sin(pi / 8), cos(pi / 4)
constexpr long long SIN_PI8 = 1764815834521887442LL;
constexpr long long COS_PI4 = 3260954456333195553LL;
template <bool INV> __device__ __forceinline__ Cq turn45(Cq a) {
    const Limbs h = limbs_of(COS_PI4);
    return INV ? Cq{mul1(a.x - a.y, h), mul1(a.x + a.y, h)} : Cq{mul1(a.x + a.y, h), mul1(a.y - a.x, h)};
}

template <int R> struct Top;  // a line entering radix R: bit of the leading one of its largest value
template <> struct Top<2> { static constexpr int v = 60; };
template <> struct Top<16> { static constexpr int v = 57; };
template <> struct Top<8> { static constexpr int v = 58; };
template <> struct Top<5> { static constexpr int v = 58; };
template <> struct Top<4> { static constexpr int v = 59; };
template <> struct Top<3> { static constexpr int v = 59; };

// Bits by which the stage after others shifts its inputs down: what takes their moduli from 2^bound to 2^62.5 / R; bound
// (log2, after the first stage Top + 1.5 + log2 R) becomes the stage's own.  The fractions count: a plan 4, 5, 5 gives up
// 3 + 2 bits, not twice the 3 that a radix 5 may grow by, which halves the rounding of its last stage.
inline double log2_radix(int R) {
    return R == 16 ? 4.0 : R == 8 ? 3.0 : R == 5 ? 2.321928094887362 : R == 4 ? 2.0 : R == 3 ? 1.584962500721156 : 1.0;
}
inline int stage_shift(int R, double& bound) {
    int k = 0;
    while (bound - k > 62.5 - log2_radix(R) + 1e-9) ++k;
    bound += log2_radix(R) - k;
    return k;
}
// stage_shift of the second stage of a plan of two powers of two or one and a 3 or 5, either way round
__host__ __device__ constexpr int headroom(int R) { return R == 16 ? 4 : R == 8 || R == 5 ? 3 : R == 4 || R == 3 ? 2 : 1; }

// The butterflies of the FP64 code (fft_proj.cu), on integers.
template <int R, bool INV> struct Bq;
template <bool INV> struct Bq<2, INV> {
    static __device__ __forceinline__ void run(Cq* v) {
        const Cq a = v[0], b = v[1];
        v[0] = add(a, b);
        v[1] = sub(a, b);
    }
};
template <bool INV> struct Bq<4, INV> {
    static __device__ __forceinline__ void run(Cq* v) {
        const Cq a0 = add(v[0], v[2]), a1 = sub(v[0], v[2]);
        const Cq a2 = add(v[1], v[3]), a3 = rot90<INV>(sub(v[1], v[3]));
        v[0] = add(a0, a2);
        v[2] = sub(a0, a2);
        v[1] = add(a1, a3);
        v[3] = sub(a1, a3);
    }
};
template <bool INV> struct Bq<8, INV> {
    static __device__ __forceinline__ void run(Cq* v) {
        Cq e[4] = {v[0], v[2], v[4], v[6]};
        Cq o[4] = {v[1], v[3], v[5], v[7]};
        Bq<4, INV>::run(e);
        Bq<4, INV>::run(o);
        const Cq o1 = turn45<INV>(o[1]), o2 = rot90<INV>(o[2]), o3 = rot90<INV>(turn45<INV>(o[3]));
        v[0] = add(e[0], o[0]);
        v[4] = sub(e[0], o[0]);
        v[1] = add(e[1], o1);
        v[5] = sub(e[1], o1);
        v[2] = add(e[2], o2);
        v[6] = sub(e[2], o2);
        v[3] = add(e[3], o3);
        v[7] = sub(e[3], o3);
    }
};
template <bool INV> struct Bq<16, INV> {
    static __device__ __forceinline__ void run(Cq* v) {
        Cq y[4][4];
#pragma unroll
        for (int n2 = 0; n2 < 4; ++n2) {
            Cq a[4] = {v[n2], v[4 + n2], v[8 + n2], v[12 + n2]};
            Bq<4, INV>::run(a);
#pragma unroll
            for (int k1 = 0; k1 < 4; ++k1) y[n2][k1] = a[k1];
        }
        y[1][1] = turn<INV>(y[1][1], COS_PI8, SIN_PI8);
        y[1][2] = turn45<INV>(y[1][2]);
        y[1][3] = turn<INV>(y[1][3], SIN_PI8, COS_PI8);
        y[2][1] = turn45<INV>(y[2][1]);
        y[2][2] = rot90<INV>(y[2][2]);
        y[2][3] = rot90<INV>(turn45<INV>(y[2][3]));
        y[3][1] = turn<INV>(y[3][1], SIN_PI8, COS_PI8);
        y[3][2] = rot90<INV>(turn45<INV>(y[3][2]));
        y[3][3] = turn<INV>(y[3][3], -COS_PI8, -SIN_PI8);
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) {
            Cq b[4] = {y[0][k1], y[1][k1], y[2][k1], y[3][k1]};
            Bq<4, INV>::run(b);
#pragma unroll
            for (int k2 = 0; k2 < 4; ++k2) v[k1 + 4 * k2] = b[k2];
        }
    }
};
template <bool INV> struct Bq<3, INV> {
    static __device__ __forceinline__ void run(Cq* v) {
        const Limbs s3 = limbs_of(3993837246235628775LL);  // round(2^62 sin(2 pi / 3))
        const Cq t1 = add(v[1], v[2]), d = sub(v[1], v[2]);
        const Cq t2 = Cq{v[0].x - (t1.x >> 1), v[0].y - (t1.y >> 1)};
        const Cq t3 = rot90<INV>(Cq{mul1(d.x, s3), mul1(d.y, s3)});
        v[0] = add(v[0], t1);
        v[1] = add(t2, t3);
        v[2] = sub(t2, t3);
    }
};
template <bool INV> struct Bq<5, INV> {
    static __device__ __forceinline__ void run(Cq* v) {
        // cos(2 pi / 5) = -1/4 + sqrt(5)/4, cos(4 pi / 5) = -1/4 - sqrt(5)/4
        const Limbs q = limbs_of(2578010857022246787LL);   // round(2^62 sqrt(5) / 4)
        const Limbs s1 = limbs_of(4385974038932618941LL), n1 = limbs_of(-4385974038932618941LL);  // sin(2 pi / 5)
        const Limbs s2 = limbs_of(2710681029835013083LL);  // sin(4 pi / 5)
        const Cq t1 = add(v[1], v[4]), t2 = add(v[2], v[3]);
        const Cq t3 = sub(v[1], v[4]), t4 = sub(v[2], v[3]);
        const Cq t = add(t1, t2), u = sub(t1, t2);
        const Cq d = Cq{mul1(u.x, q), mul1(u.y, q)};
        const Cq m = Cq{v[0].x - (t.x >> 2), v[0].y - (t.y >> 2)};
        const Cq a1 = add(m, d), a2 = sub(m, d);
        const Cq b1 = rot90<INV>(Cq{mul2(t3.x, s1, t4.x, s2), mul2(t3.y, s1, t4.y, s2)});
        const Cq b2 = rot90<INV>(Cq{mul2(t3.x, s2, t4.x, n1), mul2(t3.y, s2, t4.y, n1)});
        v[0] = add(v[0], t);
        v[1] = add(a1, b1);
        v[4] = sub(a1, b1);
        v[2] = add(a2, b2);
        v[3] = sub(a2, b2);
    }
};

// ---- conversions.  me: the largest biased exponent of the line; values of that exponent get their leading
// one at bit TOP.
__device__ __forceinline__ long long to_fixed(double d, int key) {
    // key = ((me + 63 - TOP) << 20) | 0xfffff, so (key - |hi|) >> 20 is the distance of d's leading
    // one from bit 63; zeros and subnormals are shifted out
    const int hi = __double2hiint(d), lo = __double2loint(d);
    const unsigned th = __funnelshift_l((unsigned)lo, (unsigned)hi, 11) | 0x80000000u;
    const unsigned long long t = ((unsigned long long)th << 32) | ((unsigned)lo << 11);
    const unsigned s = (unsigned)(key - (hi & 0x7fffffff)) >> 20;
    unsigned long long m;
    asm("shr.u64 %0, %1, %2;" : "=l"(m) : "l"(t), "r"(s));  // PTX: 0 for s > 63
    const long long sg = (long long)(hi >> 31);
    return ((long long)m ^ sg) - sg;
}
// FP64 nearest to v 2^(e62 - 1023 - 62), |v| < 2^63 (e62: the biased exponent of bit 62), halves rounded away
// from zero.  By integer operations: the conversion instructions run at the FP64 pipe's rate.
__device__ __forceinline__ double from_fixed(long long v, int e62) {
    const int sg = (int)(v >> 32) >> 31;
    const unsigned long long a = (unsigned long long)((v ^ (long long)sg) - (long long)sg);
    unsigned ah = (unsigned)(a >> 32), al = (unsigned)a;
    int e = e62;
    if (ah == 0) {          // (heavy cancellation) 31 bits up, so that ah < 2^31
        ah = al >> 1;
        al <<= 31;
        e -= 31;
    }
    const int z = __clz((int)ah) - 1;  // puts the leading one at bit 62
    const unsigned long long n = (((unsigned long long)ah << 32 | al) << z) + 0x200ull;
    const unsigned long long r = n >> 10;  // 53 bits, the leading one at bit 52 (53 after a carry)
    const unsigned hi = (unsigned)(r >> 32) + ((unsigned)(e - z - 1) << 20);
    const unsigned h = v == 0 ? 0u : hi | ((unsigned)sg & 0x80000000u);
    return __hiloint2double((int)h, (int)(unsigned)r);
}

// Largest exponent key of a line's values: their high words without the sign, and bit 0 where a low word is not zero
// (below 2^-1042 the high word is zero), so that only a line of zeros has key 0.
struct Key {
    int m = 0, low = 0;
    __device__ __forceinline__ void add(const double2& v) {
        m = max(max(m, __double2hiint(v.x) & 0x7fffffff), __double2hiint(v.y) & 0x7fffffff);
        low |= __double2loint(v.x) | __double2loint(v.y);
    }
    __device__ __forceinline__ int get() const { return m | (low != 0 ? 1 : 0); }
};

// v / 2^k to the nearest integer
__device__ __forceinline__ long long shift_down(long long v, int k) { return (v + ((1LL << k) >> 1)) >> k; }

// exponents this far from both ends of the range leave room for the growth of a line and for its last bit
constexpr int ME_MIN = 80, ME_MAX = 0x7f0;

}  // namespace fx
}  // namespace gff
