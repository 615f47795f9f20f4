// sg_fx.cuh -- 64-bit block fixed-point complex arithmetic and FFT for the
// FP64 and compensated plans' passes.
//
// Why.  GB300 has two FP64 lanes per SM (1.7 operations per clock and SM
// measured, 0.6 TFLOP/s of adds), against 118 lanes of 32-bit integer
// addition and 24-31 of 32 x 32 + 64-bit multiply-adds.  An FFT is additions
// (two instructions per 64-bit integer sum) and products by factors of
// modulus 1, so in fixed point a butterfly with its twiddles takes about a
// tenth of the FP64 pipe's time, at better accuracy: 59 bits below the largest
// element, where FP64 sums round at 53 below their own size.
//
// Numbers.  A transform's elements share one exponent: value = (x + i y)
// 2^E with 64-bit integers x, y.  Before a pass (radix 8 at most) every
// component is at most 2^59, so |z| <= 2^59.5 and no sum of the pass exceeds
// 2^62.5; after it the block's largest component is found (an OR over the
// sign-folded high words, one shared-memory word per pass) and the next pass's
// twiddle products shift by what it grew (s <= 4).  The largest modulus never
// shrinks through an orthogonal pass, so no shift to the left is needed.
//
// Products.  Both operands are split in signed 32-bit digits a = ah 2^32 + al,
// and with the factor w held as W = 2^(64 - s) w
//   a w 2^-s = a W 2^-64 = ah Wh + (ah Wl + al Wh) 2^-32
// without al Wl (a quarter of a unit at most).  The digit products accumulate
// in 64 bits over a complex product's two terms, so that its parts take six
// multiply-adds and one addition of a high word each, no shifts: the twiddles
// are tabled for s = 2, 3, 4, and a block that grew by less is moved up first
// (s = 2).  Karatsuba's three real products would save three of the twelve
// multiply-adds for seven more additions, digits and one bit of headroom.
#pragma once
#include <math.h>
#include <stdint.h>

#include <vector>

#define FXHD __host__ __device__ __forceinline__

struct __align__(16) fx2 {
    long long x, y;
};

namespace sg {

constexpr int FX_T = 59;      // bits of the largest component before a pass
constexpr int FX_PROD = 64;              // a product's scale below its factors'
constexpr int FX_SMIN = 2, FX_SMAX = 4;  // a product's shifts s

FXHD int fx_h(long long a) { return (int)(a >> 32) + (int)((unsigned)a >> 31); }
FXHD int fx_l(long long a) { return (int)(unsigned)a; }
// a b + c, as one instruction: left to the compiler, a negated digit is
// widened before its sign is changed, and its product becomes one of 64 x 64 bits
FXHD long long fx_wide(int a, int b, long long c)
{
#ifdef __CUDA_ARCH__
    long long r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
#else
    return (long long)((unsigned long long)((long long)a * b) + (unsigned long long)c);
#endif
}

// hi + mid 2^-32, rounded: the sums start at FX_HI and FX_MID, which hold the
// rounding and 2^63 more in mid, so that its high word is added unsigned
constexpr long long FX_MID = (long long)(0x8000000080000000ull), FX_HI = -(1ll << 31);
FXHD long long fx_join(long long hi, long long mid) { return hi + (long long)((unsigned long long)mid >> 32); }

// a factor's digits: W = (rh + i ih) 2^32 + (rl + i il), no digit -2^31
struct __align__(16) fxw {
    int rh, rl, ih, il;
};
FXHD fxw fx_digits(long long wr, long long wi) { return fxw{fx_h(wr), fx_l(wr), fx_h(wi), fx_l(wi)}; }
// a W 2^-64 (DIR < 0) or a conj(W) 2^-64 (DIR > 0).  The middle sums stay
// below 2^63: |ah| sqrt 2 2^31 + sqrt 2 2^31 |Wh| with |a| <= 2^(59.5 + s),
// |W| <= 2^(64 - s) for a twiddle, |a| <= 2^62.5, |W| <= 2^61.5 for a spectrum
template <int DIR>
FXHD fx2 fx_cmul(fx2 a, fxw w)
{
    const int xh = fx_h(a.x), xl = fx_l(a.x), yh = fx_h(a.y), yl = fx_l(a.y);
    const int uh = DIR < 0 ? -w.ih : w.ih, ul = DIR < 0 ? -w.il : w.il;  // times y, into the real part
    const int vh = DIR < 0 ? w.ih : -w.ih, vl = DIR < 0 ? w.il : -w.il;  // times x, into the imaginary part
    const long long rm = fx_wide(xl, w.rh, fx_wide(xh, w.rl, fx_wide(yl, uh, fx_wide(yh, ul, FX_MID))));
    const long long im = fx_wide(yl, w.rh, fx_wide(yh, w.rl, fx_wide(xl, vh, fx_wide(xh, vl, FX_MID))));
    return fx2{fx_join(fx_wide(xh, w.rh, fx_wide(yh, uh, FX_HI)), rm),
               fx_join(fx_wide(yh, w.rh, fx_wide(xh, vh, FX_HI)), im)};
}
// a / sqrt 2, as a - a (1 - 1 / sqrt 2): that factor fits 2^64 times itself
FXHD long long fx_rmul(long long a)
{
    constexpr long long r = 0x4AFB0CCC06219B7Cll;  // round(2^64 (1 - 1 / sqrt 2))
    const int ah = fx_h(a), al = fx_l(a), rh = fx_h(r), rl = fx_l(r);
    return a - fx_join(fx_wide(ah, rh, FX_HI), fx_wide(al, rh, fx_wide(ah, rl, FX_MID)));
}

// (a + b) / 2 and (a - b) / 2 without the sum's extra bit, off by half a unit at
// most and by nothing on average: the sum's halves are rounded one down, one
// up, the difference's both down
FXHD long long fx_half_sum(long long a, long long b) { return (a >> 1) + (b >> 1) + (b & 1); }
FXHD long long fx_half_diff(long long a, long long b) { return (a >> 1) - (b >> 1); }

FXHD fx2 fx_add(fx2 a, fx2 b) { return fx2{a.x + b.x, a.y + b.y}; }
FXHD fx2 fx_sub(fx2 a, fx2 b) { return fx2{a.x - b.x, a.y - b.y}; }
// x + DIR i d
template <int DIR>
FXHD fx2 fx_addi(fx2 x, fx2 d) { return DIR > 0 ? fx2{x.x - d.y, x.y + d.x} : fx2{x.x + d.y, x.y - d.x}; }

template <int DIR>
FXHD void fx_dft4(fx2& a0, fx2& a1, fx2& a2, fx2& a3)
{
    const fx2 t0 = fx_add(a0, a2), t1 = fx_sub(a0, a2), t2 = fx_add(a1, a3), d = fx_sub(a1, a3);
    a0 = fx_add(t0, t2);
    a2 = fx_sub(t0, t2);
    a1 = fx_addi<DIR>(t1, d);
    a3 = fx_addi<-DIR>(t1, d);
}
// a e^{DIR i pi k / 4}, k = 1, 3
template <int DIR, int K>
FXHD fx2 fx_w8(fx2 a)
{
    if (K == 1) return fx2{fx_rmul(a.x - DIR * a.y), fx_rmul(a.y + DIR * a.x)};
    return fx2{fx_rmul(-a.x - DIR * a.y), fx_rmul(-a.y + DIR * a.x)};
}
template <int R, int DIR>
FXHD void fx_dft(fx2* a)
{
    if (R == 2) {
        const fx2 t = a[0];
        a[0] = fx_add(t, a[1]);
        a[1] = fx_sub(t, a[1]);
    }
    if (R == 4) fx_dft4<DIR>(a[0], a[1], a[2], a[3]);
    if (R == 8) {
        fx_dft4<DIR>(a[0], a[2], a[4], a[6]);
        fx_dft4<DIR>(a[1], a[3], a[5], a[7]);
        const fx2 o1 = fx_w8<DIR, 1>(a[3]), o3 = fx_w8<DIR, 3>(a[7]);
        const fx2 e0 = a[0], e1 = a[2], e2 = a[4], e3 = a[6], o0 = a[1], d = a[5];
        a[0] = fx_add(e0, o0);
        a[4] = fx_sub(e0, o0);
        a[1] = fx_add(e1, o1);
        a[5] = fx_sub(e1, o1);
        a[2] = fx_addi<DIR>(e2, d);
        a[6] = fx_addi<-DIR>(e2, d);
        a[3] = fx_add(e3, o3);
        a[7] = fx_sub(e3, o3);
    }
}

// sign-folded high word: its OR over a block bounds every |component| < 2^(64 - clz)
FXHD unsigned fx_fold(long long a) { return (unsigned)((int)(a >> 32) ^ (int)(a >> 63)); }
FXHD unsigned fx_fold(fx2 a) { return fx_fold(a.x) | fx_fold(a.y); }
FXHD int fx_clz32(unsigned v)
{
#ifdef __CUDA_ARCH__
    return __clz((int)v);
#else
    return v ? __builtin_clz(v) : 32;
#endif
}
FXHD int fx_clz64(unsigned long long v)
{
#ifdef __CUDA_ARCH__
    return __clzll((long long)v);
#else
    return v ? __builtin_clzll(v) : 64;
#endif
}
// the same bound for eight values, from the extremes of their high words
FXHD unsigned fx_fold(const fx2 (&v)[8])
{
    int hi = (int)(v[0].x >> 32), lo = hi;
#pragma unroll
    for (int e = 0; e < 8; e++) {
        const int a = (int)(v[e].x >> 32), b = (int)(v[e].y >> 32);
#ifdef __CUDA_ARCH__
        hi = __vimax3_s32(hi, a, b);
        lo = __vimin3_s32(lo, a, b);
#else
        hi = hi > a ? hi : a;
        hi = hi > b ? hi : b;
        lo = lo < a ? lo : a;
        lo = lo < b ? lo : b;
#endif
    }
    return (unsigned)(hi > ~lo ? hi : ~lo);
}
// bits of the block's largest component from the OR of fx_fold
FXHD int fx_bits(unsigned folded) { return 64 - fx_clz32(folded); }

// x 2^-d, rounded, or x 2^-d for d < 0; |x| <= 2^62, so that d >= 63 gives 0;
// a tie goes up, or down for odd = 1
FXHD long long fx_shift(long long x, int d, int odd = 0)
{
    const int l = d > 0 ? 0 : d > -63 ? -d : 63, r = d < 0 ? 0 : d < 63 ? d : 63;
    return ((x << l) + (long long)(((1ull << r) - (unsigned)odd) >> 1)) >> r;
}

FXHD unsigned long long fx_dbits(double d)
{
#ifdef __CUDA_ARCH__
    return (unsigned long long)__double_as_longlong(d);
#else
    unsigned long long u;
    __builtin_memcpy(&u, &d, 8);
    return u;
#endif
}
FXHD double fx_dmake(unsigned long long u)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)u);
#else
    double d;
    __builtin_memcpy(&d, &u, 8);
    return d;
#endif
}
// |high word| of a double: its maximum over a block gives the block's exponent
FXHD unsigned fx_abshi(double d) { return (unsigned)(fx_dbits(d) >> 32) & 0x7fffffffu; }
// the exponent field of a block from the largest fx_abshi (subnormals count as 1)
FXHD int fx_field(unsigned abshi)
{
    const int f = (int)(abshi >> 20);
    return f > 0 ? f : 1;
}
// the double as a component of a block whose largest exponent field is F:
// value = result 2^(F - 1081), rounded, |result| <= 2^59
FXHD long long fx_from_double(double d, int F)
{
    const unsigned long long u = fx_dbits(d);
    const int f = (int)(u >> 52) & 0x7ff;
    unsigned long long m = u & 0xfffffffffffffull;
    if (f) m |= 0x10000000000000ull;
    const int sh = F - (f ? f : 1);
    m = sh < 63 ? (((m << 7) >> sh) + 1) >> 1 : 0;
    const long long sg = (long long)u >> 63;
    return ((long long)m ^ sg) - sg;
}
FXHD int fx_exp_of_field(int F) { return F - 1081; }
constexpr int FX_BAD = 1 << 20;  // the exponent of a block with an infinity or NaN

// x 2^E as a double (round to nearest); E in [-1022, 960] (fx_exp_safe)
FXHD bool fx_exp_safe(int E) { return E >= -1022 && E <= 960; }
FXHD double fx_to_double(long long x, int E)
{
    const unsigned long long sg = (unsigned long long)(x >> 63);
    unsigned long long m = ((unsigned long long)x ^ sg) - sg;
    const int lz = fx_clz64(m);
    m = (m << (lz - 1)) + 512;
    const unsigned long long bits = ((unsigned long long)(unsigned)(E - lz + 1085) << 52) + (m >> 10);
    return fx_dmake(x == 0 ? 0ull : bits | (sg << 63));
}
// any exponent: overflow to infinity, gradual underflow, NaN for a bad block
FXHD double fx_to_double_any(long long x, int E)
{
    if (E >= FX_BAD / 2) return fx_dmake(0x7ff8000000000000ull);
    if (fx_exp_safe(E)) return fx_to_double(x, E);
    return scalbn(fx_to_double(x, 0), E);
}

// ---------------------------------------------------------------------------
// Kernel spectra in fixed point: per mode m a row of N_u + 2 entries, kappa =
// 0 .. N_u and the row's exponent.  Entry kappa holds (x, y) with K = (x + i
// y) 2^(e_row - dE): |x|, |y| <= 2^61, dE in 0..63 in the low three bits of x
// and y (59 bits below the entry's own modulus are left, rounded).
// ---------------------------------------------------------------------------
FXHD long long fx_spec_round(long long x)
{
    x = (x + 4) & ~7ll;
    return fx_l(x) == INT32_MIN ? x + 8 : x;  // no low digit of -2^31
}
FXHD fx2 fx_spec_entry(double kx, double ky, int Frow)
{
    const unsigned hx = fx_abshi(kx), hy = fx_abshi(ky);
    const int f = fx_field(hx > hy ? hx : hy);
    int dE = Frow - f;
    dE = dE > 63 ? 63 : dE;
    const int F = Frow - dE;  // >= f
    const long long x = fx_from_double(kx, F) * 4, y = fx_from_double(ky, F) * 4;
    return fx2{fx_spec_round(x) | (dE & 7), fx_spec_round(y) | (dE >> 3)};
}
FXHD int fx_spec_drop(fx2 w) { return ((int)w.x & 7) | ((int)w.y & 7) << 3; }  // dE
FXHD fx2 fx_spec_mant(fx2 w) { return fx2{w.x & ~7ll, w.y & ~7ll}; }
FXHD int fx_spec_exp(int Frow) { return fx_exp_of_field(Frow) - 2; }  // e_row: K = x 2^(e_row - dE)

// twiddle tables: for a transform of 2^LG points the radix-8 passes after the
// first (radix 2, 4 or 8) take w^r, w = e^{-2 pi i k / (8 Ns)}, k < Ns the
// place in the Ns points done before, at fx_tw_base(LG, pass) + (r - 1) Ns +
// k, so that a warp's loads of one power are contiguous; one such table for
// each shift s, fx_tw_entries() apart
// (64 points: eight threads, below which the exchanges hold what FP64 passes
// cost; 64 x 128 forward call 95.6 -> 29.9 us against FP64 rows and columns)
constexpr int FX_MIN_LG = 6, FX_MAX_LG = 12;
FXHD constexpr int fx_first_lg(int LG) { return LG % 3 ? LG % 3 : 3; }
FXHD constexpr int fx_passes(int LG) { return (LG - 1) / 3; }  // radix-8 passes after the first
FXHD constexpr int fx_tw_base(int LG, int pass)
{
    int at = 0;
    for (int lg = FX_MIN_LG; lg <= LG; lg++)
        for (int p = 0; p < fx_passes(lg); p++) {
            if (lg == LG && p == pass) return at;
            at += 7 << (fx_first_lg(lg) + 3 * p);
        }
    return at;
}
FXHD constexpr int fx_tw_entries() { return fx_tw_base(FX_MAX_LG, 99); }

// 2^62 (cos, sin) of 2 pi j / 4096, j = 0 .. 512, rounded: Taylor series in
// double-double (two-term sums and FMA products), good to about 2^-100.
// Twiddles rounded at 53 bits would leak 2^-54 of a strong mode into all
// others, several times what the transforms' own rounding leaves.
inline std::vector<long long> fx_octant()
{
    struct dd {
        double h, l;
        static dd norm(double a, double b)
        {
            const double s = a + b;
            return dd{s, b - (s - a)};
        }
        dd mul(dd o) const
        {
            const double p = h * o.h;
            return norm(p, fma(h, o.h, -p) + (h * o.l + l * o.h));
        }
        dd add(dd o) const
        {
            const double s = h + o.h, t = s - h;
            return norm(s, ((h - (s - t)) + (o.h - t)) + (l + o.l));
        }
        dd div(double n) const
        {
            const double q = h / n;
            return norm(q, (fma(-q, n, h) + l) / n);
        }
        long long fixed() const
        {
            const double a = h * 0x1p62, whole = floor(a);
            return (long long)whole + llrint((a - whole) + l * 0x1p62);
        }
    };
    std::vector<long long> t(2 * 513);
    const dd step = dd{0x1.921fb54442d18p-10, 0x1.1a62633145c07p-64};  // pi / 2048
    for (int j = 0; j <= 512; j++) {
        const dd a = step.mul(dd{(double)j, 0.0}), m = a.mul(dd{-a.h, -a.l});
        dd c{1.0, 0.0}, s{1.0, 0.0}, tc{1.0, 0.0}, ts{1.0, 0.0};
        for (int n = 1; n <= 11; n++) {
            tc = tc.mul(m).div((2.0 * n - 1.0) * (2.0 * n));
            ts = ts.mul(m).div((2.0 * n) * (2.0 * n + 1.0));
            c = c.add(tc);
            s = s.add(ts);
        }
        t[2 * j] = c.fixed();
        t[2 * j + 1] = s.mul(a).fixed();
    }
    return t;
}
// the twiddle tables ((FX_SMAX - FX_SMIN + 1) fx_tw_entries() factors)
inline std::vector<fxw> fx_twiddle_table()
{
    const std::vector<long long> q = fx_octant();
    std::vector<fxw> out((FX_SMAX - FX_SMIN + 1) * fx_tw_entries());
    for (int lg = FX_MIN_LG; lg <= FX_MAX_LG; lg++)
        for (int p = 0; p < fx_passes(lg); p++) {
            const int ns = 1 << (fx_first_lg(lg) + 3 * p);
            for (int r = 1; r < 8; r++)
                for (int k = 0; k < ns; k++) {
                    const int j = r * k * (4096 / (8 * ns)) & 4095, o = j >> 9, i = j & 511;  // octant, place in it
                    const long long *e = &q[2 * ((o & 1) ? 512 - i : i)], c = (o + 1) & 2 ? e[1] : e[0],
                                    s = (o + 1) & 2 ? e[0] : e[1];
                    const long long wr = o >= 2 && o <= 5 ? -c : c, wi = o >= 4 ? s : -s;  // cos, -sin of 2 pi j / 4096
                    for (int t = FX_SMIN; t <= FX_SMAX; t++) {
                        long long x = fx_shift(wr, t - 2), y = fx_shift(wi, t - 2);
                        x += fx_l(x) == INT32_MIN;  // no low digit of -2^31
                        y += fx_l(y) == INT32_MIN;
                        out[(t - FX_SMIN) * fx_tw_entries() + fx_tw_base(lg, p) + (r - 1) * ns + k] = fx_digits(x, y);
                    }
                }
        }
    return out;
}

}  // namespace sg
