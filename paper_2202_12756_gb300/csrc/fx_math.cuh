// 64-bit block fixed-point arithmetic for the double-precision transforms.
//
// GB300 issues two FP64 instructions per SM and clock, but 64 integer ones
// on each of two pipes, and about 28 multiplications 32 x 32 -> 64 bit.  The
// FP64 passes were bound by FP64 issue (30 instructions per element, 15
// clocks, against 1.5 clocks for the element's HBM traffic), so double lines
// are transformed as integers instead: a line (or column) is scaled by one
// power of two, its FFT runs on 64-bit integers, and the result is rounded to
// double once.
//
// Accuracy.  Let g be such that the L1 norm of the elements of any one thread
// is below 2^g; the scale makes that 2^61.  Every first-stage butterfly lies
// within a thread, and the stage-s butterfly (radix R_s) adds R_s of its
// inputs, so multiplying by 2^-D_s <= 1 / R_s with the stage's twiddles (the
// table entries are scaled) keeps every value below 2^61, whatever the data.
// The rounding steps are then 2^-55 to 2^-57 of the rms of what they are added
// to for noise-like lines, and finer for lines with a few large entries,
// against 2^-53 of the value for each operation of an FP64 transform.  As
// there, an error is small against the line, not against each entry of it.
//
// Lines with non-finite values, or whose scale leaves the exponent range in
// which the conversions below work, take the FP64 path (the kernels' slow
// path), which keeps the behaviour of double arithmetic for them.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

namespace fft3d {

#define FX_HD __host__ __device__ __forceinline__

struct fx64 {  // tag of the fixed-point number type, as float and double are of theirs
    int64_t v;
};
struct fxc {  // complex value
    int64_t x, y;
};
// Twiddle factor w 2^(64 - d) (d: the table's scale), |components| <= 2^62, in
// balanced 32-bit limbs: component = h 2^32 + l, l in (-2^31, 2^31).
struct __align__(16) fxtw {
    int32_t xh, xl, yh, yl;
};

// values stay below 2^kFxBits in magnitude
constexpr int kFxBits = 61;

// table scale of the R2C rotation factors
constexpr int kFxRotShift = 2;
// scale 2^-D of the twiddles that go with a radix-r butterfly (r > 1)
__host__ __device__ constexpr int fx_stage_shift(int r) { return r <= 4 ? 2 : 1 + fx_stage_shift((r + 1) / 2); }

FX_HD int32_t fx_lo(int64_t a) { return (int32_t)(uint32_t)a; }
// high limb that goes with the low limb read as a signed number
FX_HD int32_t fx_hi(int64_t a) { return (int32_t)((uint64_t)a >> 32) + (int32_t)((uint32_t)a >> 31); }
// a b as one mul.wide, whose sums with other products are 64-bit additions.
// Measured on GB300 in registers, a complex product by a table twiddle takes 57
// issue cycles of an SM quarter (21 instructions) this way, against 67 (31) as
// mad.wide chains, which the compiler splits, and 54 instructions in plain C++,
// which it turns into 64 x 64-bit products where it sees the sign extensions
// apart from the multiplication.
FX_HD int64_t fx_mul(int32_t a, int32_t b)
{
#ifdef __CUDA_ARCH__
    int64_t r;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
    return r;
#else
    return (int64_t)a * b;
#endif
}

FX_HD fxc fx_make(int64_t x, int64_t y)
{
    fxc r;
    r.x = x;
    r.y = y;
    return r;
}

// z w 2^-d.  Products of limbs of weight 2^64 (hi) and 2^32 (mid, rounded
// into the result); low x low, below 1/4 unit, is left out.  Four mid terms
// stay below 2^63 for |z| < 2^62 and d >= 2.
FX_HD fxc cmul(fxc z, fxtw w)
{
    const int32_t xl = fx_lo(z.x), xh = fx_hi(z.x), yl = fx_lo(z.y), yh = fx_hi(z.y);
    const int32_t nh = -w.yh, nl = -w.yl;
    const int64_t half = 0x80000000LL;
    const int64_t mr = fx_mul(yl, nh) + fx_mul(yh, nl) + fx_mul(xl, w.xh) + fx_mul(xh, w.xl) + half;
    const int64_t mi = fx_mul(yl, w.xh) + fx_mul(yh, w.xl) + fx_mul(xl, w.yh) + fx_mul(xh, w.yl) + half;
    return fx_make(fx_mul(yh, nh) + fx_mul(xh, w.xh) + (mr >> 32), fx_mul(yh, w.xh) + fx_mul(xh, w.yh) + (mi >> 32));
}
// z conj(w) 2^-d
FX_HD fxc cmulc(fxc z, fxtw w)
{
    w.yh = -w.yh;
    w.yl = -w.yl;
    return cmul(z, w);
}
// z 2^-D, rounded
template <int D> FX_HD fxc fx_shr(fxc z)
{
    return fx_make((z.x + (1LL << (D - 1))) >> D, (z.y + (1LL << (D - 1))) >> D);
}

// cos(2 pi p / 96), p = 0..24, as (unit + k / 2^64) with |k| <= 2^63: 64-bit
// roundings of the mathematical values.
struct FxConst {
    int unit;
    int64_t k;
};
__host__ __device__ constexpr FxConst fx_cos96_q1(int p)
{
    constexpr int64_t k[25] = {0LL,
                               -39495895059648002LL,
                               -157814452752426473LL,
                               -354449014849699498LL,
                               -628557561968679382LL,
                               -978966319228692918LL,
                               -1404174782535421627LL,
                               -1902362143969795207LL,
                               -2471395088767036514LL,
                               -3108836930497996774LL,
                               -3811958045334532105LL,
                               -4577747560717795106LL,
                               -5402926248376769404LL,
                               -6283960566487162427LL,
                               -7217077790839976240LL,
                               -8198282170225769627LL,
                               -9223372036854775807LL - 1,
                               8158786275166121626LL,
                               7059263338087549767LL,
                               5929511551637462929LL,
                               4774368686408090022LL,
                               3598781241489102189LL,
                               2407783262799110479LL,
                               1206474786528201567LL,
                               0LL};
    return FxConst{p <= 16 ? 1 : 0, k[p]};
}
__host__ __device__ constexpr FxConst fx_neg(FxConst c)
{
    // -1/2 and 1/2 both carry k = -2^63
    return c.k == (-9223372036854775807LL - 1) ? FxConst{1 - c.unit, c.k} : FxConst{-c.unit, -c.k};
}
// cos(2 pi p / 96) for any p
__host__ __device__ constexpr FxConst fx_cos96(int p)
{
    const int q = ((p % 96) + 96) % 96;
    if (q <= 24) return fx_cos96_q1(q);
    if (q <= 48) return fx_neg(fx_cos96_q1(48 - q));
    if (q <= 72) return fx_neg(fx_cos96_q1(q - 48));
    return fx_cos96_q1(96 - q);
}
__host__ __device__ constexpr int32_t fx_limb_l(int64_t k) { return (int32_t)(uint32_t)(uint64_t)k; }
__host__ __device__ constexpr int32_t fx_limb_h(int64_t k)
{
    return (int32_t)((k >> 32) + (int64_t)((uint64_t)k >> 31 & 1));
}

// a cos(2 pi P / 96) for a real a, |a| < 2^62 (0 < P <= 16)
template <int P> FX_HD int64_t fx_scale96(int64_t a)
{
    constexpr FxConst C = fx_cos96(P);
    static_assert(C.unit == 1, "first eighth");
    constexpr int32_t cl = fx_limb_l(C.k), ch = fx_limb_h(C.k);
    const int32_t l = fx_lo(a), h = fx_hi(a);
    return a + fx_mul(h, ch) + ((fx_mul(l, ch) + fx_mul(h, cl) + 0x80000000LL) >> 32);
}
// z exp(-2 pi i / 8), z exp(-2 pi i 3 / 8)
FX_HD fxc w8_1(fxc z) { return fx_make(fx_scale96<12>(z.x + z.y), fx_scale96<12>(z.y - z.x)); }
FX_HD fxc w8_3(fxc z) { return fx_make(fx_scale96<12>(z.y - z.x), -fx_scale96<12>(z.x + z.y)); }

// z exp(-2 pi i P / 96) at full scale, for |z| < 2^61
template <int P> FX_HD fxc fx_rot96(fxc z)
{
    constexpr int p = ((P % 96) + 96) % 96;
    if constexpr (p == 0) {
        return z;
    } else if constexpr (p == 24) {
        return fx_make(z.y, -z.x);
    } else if constexpr (p == 48) {
        return fx_make(-z.x, -z.y);
    } else if constexpr (p == 72) {
        return fx_make(-z.y, z.x);
    } else if constexpr (p == 12) {
        return w8_1(z);
    } else if constexpr (p == 36) {
        return w8_3(z);
    } else if constexpr (p % 8 == 0 && p < 48) {
        // 30, 60, 120, 150 degrees: a half, and one product by sin 60 per component
        // (6 mul.wide instead of 12; with the 45 degrees above, 768^3 pair 15.4 -> 15.1 ms)
        const int64_t hx = (z.x + 1) >> 1, hy = (z.y + 1) >> 1, sx = fx_scale96<8>(z.x), sy = fx_scale96<8>(z.y);
        if constexpr (p == 8) return fx_make(sx + hy, sy - hx);
        else if constexpr (p == 16) return fx_make(hx + sy, hy - sx);
        else if constexpr (p == 32) return fx_make(sy - hx, -sx - hy);
        else return fx_make(hy - sx, -sy - hx);
    } else if constexpr (p > 48 && p % 4 == 0) {
        const fxc r = fx_rot96<p - 48>(z);
        return fx_make(-r.x, -r.y);
    } else {
        constexpr FxConst C = fx_cos96(p), S = fx_cos96(p - 24), M = fx_neg(fx_cos96(p - 24));
        // re = C x + S y, im = C y - S x
        constexpr int32_t cl = fx_limb_l(C.k), ch = fx_limb_h(C.k), sl = fx_limb_l(S.k), sh = fx_limb_h(S.k),
                          nl = fx_limb_l(M.k), nh = fx_limb_h(M.k);
        const int32_t xl = fx_lo(z.x), xh = fx_hi(z.x), yl = fx_lo(z.y), yh = fx_hi(z.y);
        const int64_t half = 0x80000000LL;
        const int64_t mr = fx_mul(yl, sh) + fx_mul(yh, sl) + fx_mul(xl, ch) + fx_mul(xh, cl) + half;
        const int64_t mi = fx_mul(xl, nh) + fx_mul(xh, nl) + fx_mul(yl, ch) + fx_mul(yh, cl) + half;
        int64_t re = mr >> 32, im = mi >> 32;
        if constexpr (C.unit == 1) re += z.x, im += z.y;
        if constexpr (C.unit == -1) re -= z.x, im -= z.y;
        if constexpr (S.unit == 1) re += z.y;
        if constexpr (S.unit == -1) re -= z.y;
        if constexpr (M.unit == 1) im += z.x;
        if constexpr (M.unit == -1) im -= z.x;
        return fx_make(fx_mul(yh, sh) + fx_mul(xh, ch) + re, fx_mul(xh, nh) + fx_mul(yh, ch) + im);
    }
}
// ------------------------------------------------------------ double <-> fixed point
FX_HD uint64_t fx_bits(double v)
{
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(v);
#else
    uint64_t u;
    memcpy(&u, &v, 8);
    return u;
#endif
}
FX_HD double fx_double(uint64_t u)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)u);
#else
    double v;
    memcpy(&v, &u, 8);
    return v;
#endif
}
FX_HD float fx_float(uint32_t u)
{
#ifdef __CUDA_ARCH__
    return __uint_as_float(u);
#else
    float v;
    memcpy(&v, &u, 4);
    return v;
#endif
}
FX_HD uint32_t fx_float_bits(float v)
{
#ifdef __CUDA_ARCH__
    return __float_as_uint(v);
#else
    uint32_t u;
    memcpy(&u, &v, 4);
    return u;
#endif
}
FX_HD int fx_clz(uint64_t a)
{
#ifdef __CUDA_ARCH__
    return __clzll((long long)a);
#else
    return a ? __builtin_clzll(a) : 64;
#endif
}

// |v| without its low word: sign cleared, exponent and 20 mantissa bits
FX_HD int32_t fx_top(double v) { return (int32_t)((uint32_t)(fx_bits(v) >> 32) & 0x7fffffffu); }

// Scale of a line.  A thread gathers the largest `top` of its values, then
// their sum as floats relative to that one's exponent; the scale code g (the
// biased exponent of a power of two above the L1 norm; 0 where all tops are zeros,
// kFxBad with a non-finite value) is combined by max over the line.
constexpr int kFxBad = 1 << 20;
// codes outside [kFxMinCode, kFxMaxCode] leave the exponent range of the conversions
constexpr int kFxMinCode = 128, kFxMaxCode = 1900, kFxZeroCode = 1023;

FX_HD float fx_mag(int32_t top, int32_t expo)  // |v| / 2^(expo's exponent), at least 2^-100
{
    const int32_t fl = expo - (100 << 20);
    const uint32_t t = (uint32_t)(top > fl ? top : fl), off = ((127u << 20) - (uint32_t)expo) * 8u;
#ifdef __CUDA_ARCH__
    uint32_t b;
    asm("mad.lo.u32 %0, %1, 8, %2;" : "=r"(b) : "r"(t), "r"(off));  // not on the pipe of the maxima
    return fx_float(b);
#else
    return fx_float(t * 8u + off);
#endif
}
FX_HD int fx_code(int32_t top_max, float sum)
{
    if (top_max >= 0x7ff00000) return kFxBad;
    // (1 + 2^-12): mantissas were cut to 20 bits, the sum rounded
    const uint32_t s = fx_float_bits(sum * 1.000244140625f);
    return top_max == 0 ? 0 : (top_max >> 20) + (int)(s >> 23) - 126;
}

// Scale code of a thread's n complex values.  (Bounding the L1 norm by twice the
// larger component of each takes 17 issue cycles of an SM quarter per value
// instead of 21, but a line with one large entry loses up to a bit: relative L2
// error 2.4e-16 at 2048 points, above the FP64 transform's 2.1e-16.)
template <int N> FX_HD int fx_thread_code(const double2 *v)
{
    int32_t tm = 0;
#pragma unroll
    for (int i = 0; i < N; ++i) tm = max(tm, max(fx_top(v[i].x), fx_top(v[i].y)));
    const int32_t ex = tm & 0x7ff00000;
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < N; ++i) s += fx_mag(fx_top(v[i].x), ex) + fx_mag(fx_top(v[i].y), ex);
    return fx_code(tm, s);
}

// A line is transformed in fixed point if its code is in range or it is one of zeros.
FX_HD bool fx_in_range(int g) { return (uint32_t)(g - kFxMinCode) <= (uint32_t)(kFxMaxCode - kFxMinCode); }
// Whether a thread of a line out of range speaks against it: code 0 also goes with
// values below 2^-1042, whose low words alone are set.  Left to this rare case
// because a look at the low words in every line, never taken, costs the column
// passes 2% (1024 x 1024 x 512 pair 15.97 -> 16.16 ms).
template <int N> FX_HD bool fx_unfit(int g, const double2 *v)
{
    uint32_t low = 0;
#pragma unroll
    for (int i = 0; i < N; ++i) low |= (uint32_t)fx_bits(v[i].x) | (uint32_t)fx_bits(v[i].y);
    return g != 0 || low != 0;
}

// v scaled so that 2^(g - 1023) becomes 2^bits, cut towards zero (|v| < 2^(g - 1023))
FX_HD int64_t fx_from(double v, int g, int bits)
{
    const uint64_t u = fx_bits(v);
    const uint32_t hi = (uint32_t)(u >> 32);
    const uint64_t m = (u << 11) | 0x8000000000000000ULL;
    const uint32_t sh = (uint32_t)(g + (63 - bits)) - ((hi & 0x7fffffffu) >> 20);
#ifdef __CUDA_ARCH__
    int64_t a;
    asm("{\n .reg .pred p;\n shr.u64 %0, %1, %2;\n"  // 0 from 64 on
        " setp.lt.s32 p, %3, 0;\n @p neg.s64 %0, %0;\n}\n"
        : "=&l"(a)
        : "l"(m), "r"(sh), "r"((int32_t)hi));
    return a;
#else
    const uint64_t a = sh > 63 ? 0 : m >> sh;
    return (int32_t)hi < 0 ? -(int64_t)a : (int64_t)a;
#endif
}

// Left shift that brings the leading bit of h that differs from its sign to bit
// 31, -1 without one.
FX_HD int32_t fx_lead_shift(int32_t h)
{
#ifdef __CUDA_ARCH__
    int32_t n;
    asm("bfind.shiftamt.s32 %0, %1;" : "=r"(n) : "r"(h));
    return n;
#else
    const uint32_t a = (uint32_t)(h ^ (h >> 31));
    return a ? __builtin_clz(a) : -1;
#endif
}
FX_HD uint32_t fx_shl_hi(uint32_t lo, uint32_t hi, uint32_t n)  // high word of hi:lo << n, n < 32
{
#ifdef __CUDA_ARCH__
    return __funnelshift_l(lo, hi, n);
#else
    return n ? hi << n | lo >> (32 - n) : hi;
#endif
}

// X 2^e, rounded to nearest (ties towards +infinity, so that they leave no
// bias), for |X| < 2^62 and e in [-1000, 900], on the integer pipes.  Serves
// |X| >= 2^32, else clears the sign bit of `big` and returns anything.  The
// exponent is a product by 2^20, which the multiply pipe takes off the adders
// (42 issue cycles of an SM quarter per complex value, 49 with shifts).
FX_HD double fx_to_big(int64_t X, int e, int32_t &big)
{
    const uint32_t hi = (uint32_t)((uint64_t)X >> 32), lo = (uint32_t)(uint64_t)X;
    const uint32_t s = (uint32_t)((int32_t)hi >> 31);
    const int32_t n1 = fx_lead_shift((int32_t)hi);
    big &= ~n1;
    const uint32_t n = (uint32_t)n1 - 1;
    // |X| 2^n with its leading bit at 62 (one less in the last place if X < 0)
    const uint64_t v = ((uint64_t)(fx_shl_hi(lo, hi, n & 31) ^ s) << 32 | ((lo << (n & 31)) ^ s)) + 512;
    const uint32_t r = (uint32_t)(v >> 42) + (((uint32_t)(e + 1084) << 20) - n * 1048576u);
    return fx_double((uint64_t)(r | (s & 0x80000000u)) << 32 | (uint32_t)(v >> 10));
}
// The same for any |X| < 2^62, with two FP64 additions (ties to even).
FX_HD double fx_to(int64_t X, int e)
{
    const uint32_t s = (uint32_t)e << 20;
    const double dh = fx_double((uint64_t)(0x45300000u + s) << 32 | ((uint32_t)((uint64_t)X >> 32) ^ 0x80000000u));
    const double dl = fx_double((uint64_t)(0x43300000u + s) << 32 | (uint32_t)X);
    const double d0 = fx_double((uint64_t)(0x45300000u + s) << 32 | 0x80100000u);
    return (dh - d0) + dl;
}

// ------------------------------------------------------------ twiddle tables
// cos and sin of 2 pi p / d (0 <= p < d <= 2^13) as integers of scale 2^62:
// exact octant reduction, then both Maclaurin series in 64-bit fixed point
// (errors of a few units of 2^-62).
FX_HD uint64_t fx_umulhi(uint64_t a, uint64_t b)
{
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (uint64_t)((unsigned __int128)a * b >> 64);
#endif
}
FX_HD void fx_cossin(uint32_t p, uint32_t d, int64_t *c_out, int64_t *s_out)
{
    uint32_t n = 2 * p, q = d;  // angle pi n / q
    bool neg_c = false, neg_s = false, swap = false;
    if (n >= q) {
        n -= q;
        neg_c = true;
        neg_s = true;
    }
    if (2 * n > q) {
        n = q - n;
        neg_c = !neg_c;
    }
    if (4 * n > q) {
        n = q - 2 * n;
        q = 2 * q;
        swap = true;
    }
    // x = pi n / q in units of 2^-62 (n / q <= 1/4 as a 64-bit fraction)
    const uint64_t q1 = ((uint64_t)n << 32) / q, r1 = ((uint64_t)n << 32) % q;
    const uint64_t frac = (q1 << 32) | ((r1 << 32) / q);
    const uint64_t x = fx_umulhi(frac, 0xC90FDAA22168C235ULL);  // pi 2^62
    const uint64_t x2 = fx_umulhi(x << 1, x << 1);
    uint64_t tc = 1ULL << 62, ts = x;
    int64_t c = (int64_t)tc, s = (int64_t)ts;
    for (uint32_t k = 1; k <= 12; ++k) {
        tc = (fx_umulhi(tc << 1, x2 << 1)) / ((2 * k - 1) * (2 * k));
        ts = fx_umulhi(ts << 1, x2 << 1) / ((2 * k) * (2 * k + 1));
        c += (k & 1) ? -(int64_t)tc : (int64_t)tc;
        s += (k & 1) ? -(int64_t)ts : (int64_t)ts;
    }
    int64_t cc = swap ? s : c, ss = swap ? c : s;
    *c_out = neg_c ? -cc : cc;
    *s_out = neg_s ? -ss : ss;
}
FX_HD void fx_limbs(int64_t v, int32_t *h, int32_t *l)
{
    if ((uint32_t)v == 0x80000000u) ++v;  // keep -l representable
    *l = fx_lo(v);
    *h = fx_hi(v);
}
// exp(-2 pi i p / d) 2^(64 - shift), shift >= 2
FX_HD fxtw fx_twiddle(uint32_t p, uint32_t d, int shift)
{
    int64_t c, s;
    fx_cossin(p, d, &c, &s);
    const int64_t half = shift > 2 ? 1LL << (shift - 3) : 0;
    fxtw w;
    fx_limbs((c + half) >> (shift - 2), &w.xh, &w.xl);
    fx_limbs((-s + half) >> (shift - 2), &w.yh, &w.yl);
    return w;
}
// component value h 2^32 + l of a table of scale `shift` (1 to 5), as a double.
// The FP64 path is bound by FP64 issue, so this is integer work: a component is
// 0 or, as sin(2 pi / 2^13) > 2^-11, at least 2^48.
FX_HD double fx_twiddle_value(int32_t h, int32_t l, int shift)
{
    const int64_t X = (int64_t)h * 4294967296LL + l;
    int32_t big = -1;
    const double v = fx_to_big(X, shift - 64, big);
    return X == 0 ? 0.0 : v;
}

}  // namespace fft3d
