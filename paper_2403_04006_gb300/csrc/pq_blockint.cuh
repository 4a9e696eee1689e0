// pq_blockint.cuh -- complex products in 64-bit block integers, the arithmetic
// of the walks' products.
//
// GB300 issues 2 FP64 lane operations per clock and SM, and the integer pipes
// 64 to 128; a 32 x 32 + 64 bit multiply-add (IMAD.WIDE) runs at 32 lanes per
// clock and SM.  A complex product in FP64 takes 4 FP64 instructions and the
// column update of a Gray step 2, 3.3 clocks per lane, column and term at the
// pipe's measured 1.8; the same work in the integers below takes 0.57.  So a
// lane's column sums and running products are integers, and FP64 is left
// with one conversion and one fused add per term and component.
//
// Column sums.  Column j of a permanent is scaled by 2^e_j, chosen so that
// every |Re S_j|, |Im S_j| the code can reach stays below 2^62 (the bound is
// sum_i r_i max(|Re b_ij|, |Im b_ij|), added up in integers of 21 bits: FP64
// would take the 16 warps of an SM longer than the rest of the staging), and its entries are rounded to
// integers once, when the base matrix is staged.  Every update of a column sum
// is then exact; in FP64 each of them rounded, at 2^-53 of the largest sum on
// the way against the single rounding at 2^-62 of the bound here.
//
// The real and imaginary parts of a column share its unit, and a product its
// error, so a part that is small beside the other keeps fewer bits than in FP64,
// where it has its own exponent.  That shows in a result only where all factors
// lie near an axis (one part below 2^-kAxisBits of the other in every entry, and
// not zero): one factor with two parts of like size gives the product two parts
// of like size.  Error of the small part, mean over random matrices of 4 to 12
// columns, against FP64: ratio 0.4 to 0.6 at parts of 2^-4, 1 to 2 at 2^-5, 10 to
// 14 at 2^-8, 240 at 2^-12.  Those matrices (complex steps, small phases on a real
// matrix, a real matrix with the rounding of its imaginary parts) are staged with
// a unit for each part (bmul_parts, SInt).  Telling them apart costs a task a
// comparison and two votes: 42504 permanents of 5 photons 161.5 -> 163.9 us.
//
// Products.  A complex number is two signed 64-bit integers with one binary
// exponent.  p s is formed from 32-bit limbs (high signed, low signed after
// moving its carry up): the four high products in 64 bits and the high words
// of the eight cross products, low times low left out: (p s) >> 64 with an
// absolute error of about one unit.  Every second product is normalised
// (shifted left until the larger component has its top bit at 61, the shift
// added to the exponent).  A product of two typical column sums has about 2^56,
// so two products cost an error of about 2^-55 of the product's magnitude, a
// third of what two FP64 complex products round.
//
// The multiply-adds are written as mul.wide plus a 64-bit add: ptxas fuses
// these, while mad.wide was split into more instructions (0.57 against 0.70
// clocks per lane, column and term in an isolated loop).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace pqi {

constexpr int kSumBits = 62;  // column sums stay below 2^kSumBits in magnitude
constexpr int kAxisBits = 4;  // parts this many binades apart: near an axis

// Complex number of two 64-bit integers in 32-bit words.
struct BInt {
    int rh, ih;
    uint32_t rl, il;
};

// re = a 2^32 + b, im = c 2^32 + d with signed low words.
struct BLimbs {
    int a, b, c, d;
};

__host__ __device__ __forceinline__ uint64_t bint_bits(double x)
{
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t u;
    __builtin_memcpy(&u, &x, sizeof(u));
    return u;
#endif
}

// The bound of a column's sums, in integers.  An entry counts with the high
// word of the larger of |Re|, |Im| (bint_mag).  With hmax the column's largest
// it is below bint_units(h, hmax) 2^(hmax's exponent field - 1043), and a
// column whose units (times multiplicity) add up to u is scaled by
// 2^bint_scale(hmax, u), which keeps its sums below 2^kSumBits (1 - 2^-21).
// A column of subnormal entries (hmax < 2^20) is added up exactly, in units of
// 2^-1074, so that it loses no bits (bint_scale_subnormal: at most 58 bits, and
// one to spare, since a sum that is exactly the bound would reach 2^kSumBits
// less a few units, where the high word of a negative number is -2^30 already
// and bnorm's shift would be negative).
__host__ __device__ __forceinline__ uint32_t bint_mag(double re, double im)
{
    const uint32_t x = (uint32_t)(bint_bits(re) >> 32) & 0x7fffffffu;
    const uint32_t y = (uint32_t)(bint_bits(im) >> 32) & 0x7fffffffu;
    return x > y ? x : y;
}

// The largest real and imaginary parts of a set of numbers: high words without
// sign, and whether any low word is set (a high word of zero is not a zero).
struct BParts {
    uint32_t re = 0, im = 0, re_low = 0, im_low = 0;
    __host__ __device__ __forceinline__ void add(double x, double y)
    {
        const uint64_t u = bint_bits(x), v = bint_bits(y);
        const uint32_t p = (uint32_t)(u >> 32) & 0x7fffffffu, q = (uint32_t)(v >> 32) & 0x7fffffffu;
        re = p > re ? p : re;
        im = q > im ? q : im;
        re_low |= (uint32_t)u;
        im_low |= (uint32_t)v;
    }
    __host__ __device__ __forceinline__ bool no_re() const { return (re | re_low) == 0; }
    __host__ __device__ __forceinline__ bool no_im() const { return (im | im_low) == 0; }
};

__host__ __device__ __forceinline__ int bint_width(uint64_t u)  // u < 2^width
{
#ifdef __CUDA_ARCH__
    return 64 - __clzll((long long)u);
#else
    int bits = 0;
    while (bits < 64 && (u >> bits) != 0)
        ++bits;
    return bits;
#endif
}

// Biased exponent of a high word, below 1 for subnormals.
__host__ __device__ __forceinline__ int bint_exponent(uint32_t h)
{
    return h >= 0x100000u ? (int)(h >> 20) : bint_width(h) - 20;
}

// Whether the larger parts re and im (high words) are kAxisBits binades apart.
__host__ __device__ __forceinline__ bool bint_apart(uint32_t re, uint32_t im)
{
    const int d = bint_exponent(re) - bint_exponent(im);
    return d >= kAxisBits || d <= -kAxisBits;
}

// Numbers near an axis: a part is small throughout, and not zero.
__host__ __device__ __forceinline__ bool bint_near_axis(const BParts& m)
{
    return bint_apart(m.re, m.im) && !m.no_re() && !m.no_im();
}

__host__ __device__ __forceinline__ uint32_t bint_units(uint32_t h, uint32_t hmax)
{
    const int f = (int)(h >> 20), d = (int)(hmax >> 20) - (f == 0 ? 1 : f);
    const uint32_t m = (h & 0xfffffu) + (f == 0 ? 1u : 0x100001u);  // rounded up
    return d <= 0 ? m : (d > 31 ? 1u : (m >> d) + 1u);
}

__host__ __device__ __forceinline__ int bint_scale(uint32_t hmax, uint32_t units)
{
    return kSumBits + 1043 - (int)(hmax >> 20) - bint_width(units);
}

__host__ __device__ __forceinline__ uint64_t bint_mag_subnormal(double re, double im)
{
    const uint64_t x = bint_bits(re) & 0xfffffffffffffull, y = bint_bits(im) & 0xfffffffffffffull;
    return x > y ? x : y;
}

__host__ __device__ __forceinline__ int bint_scale_subnormal(uint64_t sum)
{
    return kSumBits + 1073 - bint_width(sum);
}

// round(x 2^e) as an integer, ties away from zero; |x| 2^e < 2^63.
__host__ __device__ __forceinline__ int64_t bint_of(double x, int e)
{
    const uint64_t u = bint_bits(x);
    const int f = (int)((u >> 52) & 0x7ff);
    uint64_t m = u & 0xfffffffffffffull;
    if (f != 0)
        m |= 0x10000000000000ull;
    const int s = (f == 0 ? 1 : f) - 1075 + e;
    if (s >= 0)
        m <<= s;
    else if (s > -55)
        m = (m + (1ull << (-s - 1))) >> (-s);
    else
        m = 0;
    return (u >> 63) ? -(int64_t)m : (int64_t)m;
}

#ifdef __CUDACC__
// Column sums are kept with 2^31 added to each component, so that the high
// word already holds the carry of the signed low word.
constexpr int64_t kSumBias = int64_t(1) << 31;

__device__ __forceinline__ BLimbs sum_limbs(longlong2 s)
{
    BLimbs v;
    v.a = (int)(s.x >> 32);
    v.b = (int)((uint32_t)s.x ^ 0x80000000u);
    v.c = (int)(s.y >> 32);
    v.d = (int)((uint32_t)s.y ^ 0x80000000u);
    return v;
}

__device__ __forceinline__ BLimbs limbs(const BInt& p)
{
    BLimbs v;
    v.a = p.rh + (int)(p.rl >> 31);
    v.b = (int)p.rl;
    v.c = p.ih + (int)(p.il >> 31);
    v.d = (int)p.il;
    return v;
}

__device__ __forceinline__ int64_t mulw(int a, int b)
{
    int64_t r;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
    return r;
}

// (p s) >> 64.  High words within 2^30 in magnitude, low words within 2^31:
// the cross sums stay within [-2^63, 2^63).  (The differences are taken of
// the products: negating a low word would overflow at -2^31.)
__device__ __forceinline__ BInt bmul(const BLimbs& p, const BLimbs& s)
{
    const int64_t mr = (mulw(p.a, s.b) + mulw(p.b, s.a)) - (mulw(p.c, s.d) + mulw(p.d, s.c));
    const int64_t mi = (mulw(p.a, s.d) + mulw(p.b, s.c)) + (mulw(p.c, s.b) + mulw(p.d, s.a));
    const int64_t hr = mulw(p.a, s.a) - mulw(p.c, s.c) + (int64_t)(int)(mr >> 32);
    const int64_t hi = mulw(p.a, s.c) + mulw(p.c, s.a) + (int64_t)(int)(mi >> 32);
    BInt r;
    r.rh = (int)(hr >> 32);
    r.rl = (uint32_t)hr;
    r.ih = (int)(hi >> 32);
    r.il = (uint32_t)hi;
    return r;
}

// (p p) >> 64: the bits of bmul(p, p), from 7 wide multiplies instead of 12.
__device__ __forceinline__ BInt bsqr(const BLimbs& p)
{
    const int64_t mr = mulw(p.a, p.b) - mulw(p.c, p.d);
    const int64_t mi = mulw(p.a, p.d) + mulw(p.b, p.c);
    const int64_t m = mulw(p.a, p.c);
    const int64_t hr = mulw(p.a, p.a) - mulw(p.c, p.c) + (int64_t)(int)(mr >> 31);
    const int64_t hi = m + m + (int64_t)(int)(mi >> 31);
    BInt r;
    r.rh = (int)(hr >> 32);
    r.rl = (uint32_t)hr;
    r.ih = (int)(hi >> 32);
    r.il = (uint32_t)hi;
    return r;
}

// Shift left until the larger high word has its top bit at position 29; the
// shift (at most 30) is added to E.
__device__ __forceinline__ void bnorm(BInt& p, int& E)
{
    const uint32_t t = (uint32_t)abs(p.rh) | (uint32_t)abs(p.ih);
    int top;
    asm("bfind.u32 %0, %1;" : "=r"(top) : "r"(t));  // -1 for zero
    const int s = 29 - top;
    E += s;
    p.rh = (int)__funnelshift_l(p.rl, (uint32_t)p.rh, s);
    p.rl <<= s;
    p.ih = (int)__funnelshift_l(p.il, (uint32_t)p.ih, s);
    p.il <<= s;
}

__device__ __forceinline__ BInt bint_words(longlong2 s)
{
    BInt p;
    p.rh = (int)(s.x >> 32);
    p.rl = (uint32_t)s.x;
    p.ih = (int)(s.y >> 32);
    p.il = (uint32_t)s.y;
    return p;
}

__device__ __forceinline__ BInt bint_plain(longlong2 s)
{
    BInt p;
    s.x -= kSumBias;
    s.y -= kSumBias;
    p.rh = (int)(s.x >> 32);
    p.rl = (uint32_t)s.x;
    p.ih = (int)(s.y >> 32);
    p.il = (uint32_t)s.y;
    return p;
}

// +-w 2^(-kSumBits - E), the factor that takes a product's integers to a term
// of weight w (a double >= 1) in the range of FP64: integer work on w's
// exponent (zero below the smallest normal number).
__device__ __forceinline__ double bint_factor(double w, int E, bool neg)
{
    const int h = __double2hiint(w) - ((kSumBits + min(E, 1900)) << 20);
    return h >= 0x100000 ? __hiloint2double(h | (neg ? (int)0x80000000 : 0), __double2loint(w))
                         : 0.0;
}

__device__ __forceinline__ bool not_finite(double x)
{
    return (__double2hiint(x) & 0x7ff00000) == 0x7ff00000;
}

// ---- a unit for each part
// The high 64 bits of a real product of limbs, low times low left out.
__device__ __forceinline__ int64_t mulhi(int ah, int al, int bh, int bl)
{
    const int64_t m = mulw(ah, bl) + mulw(al, bh);
    return mulw(ah, bh) + (int64_t)(int)(m >> 32);
}

// (p s) >> 64 where im is in units 2^-f of re's, shift = min(63, 2 f): im times im is
// that much finer than re.
__device__ __forceinline__ BInt bmul_parts(const BLimbs& p, const BLimbs& s, int shift)
{
    const int64_t hr = mulhi(p.a, p.b, s.a, s.b) - (mulhi(p.c, p.d, s.c, s.d) >> shift);
    const int64_t hi = mulhi(p.a, p.b, s.c, s.d) + mulhi(p.c, p.d, s.a, s.b);
    BInt r;
    r.rh = (int)(hr >> 32);
    r.rl = (uint32_t)hr;
    r.ih = (int)(hi >> 32);
    r.il = (uint32_t)hi;
    return r;
}

// The walks' products: both parts in one unit, or im in units 2^-f of re's.
struct OneUnit {
    __device__ __forceinline__ BInt operator()(const BLimbs& p, const BLimbs& s) const
    {
        return bmul(p, s);
    }
    __device__ __forceinline__ BInt sqr(const BLimbs& p) const { return bsqr(p); }
};

struct PartUnits {
    int shift;
    __device__ __forceinline__ BInt operator()(const BLimbs& p, const BLimbs& s) const
    {
        return bmul_parts(p, s, shift);
    }
    __device__ __forceinline__ BInt sqr(const BLimbs& p) const { return bmul_parts(p, p, shift); }
};

// A product whose factors have different f (a gradient's, whose products leave out a
// column): p 2^-E, im in units 2^-f of re's.  f does not depend on the lane.
struct SInt {
    BInt p;
    int E, f;
};

// p s, normalised: each part's finer product is shifted down to the other's unit.
__device__ __forceinline__ SInt smul(const SInt& p, const SInt& s)
{
    const BLimbs x = limbs(p.p), y = limbs(s.p);
    SInt r;
    r.f = min(p.f, s.f);
    r.E = p.E + s.E;
    const int64_t hr =
        mulhi(x.a, x.b, y.a, y.b) - (mulhi(x.c, x.d, y.c, y.d) >> min(63, p.f + s.f));
    const int64_t hi = (mulhi(x.a, x.b, y.c, y.d) >> min(63, s.f - r.f)) +
                       (mulhi(x.c, x.d, y.a, y.b) >> min(63, p.f - r.f));
    r.p.rh = (int)(hr >> 32);
    r.p.rl = (uint32_t)hr;
    r.p.ih = (int)(hi >> 32);
    r.p.il = (uint32_t)hi;
    bnorm(r.p, r.E);
    return r;
}

// A column's scale when its parts have units of their own: 2^e for the larger part,
// 2^(e + f) for the smaller; turned: the imaginary part is the larger, and the
// column is staged divided by i.  f = kOnAxisF where a part is zero throughout.
constexpr int kOnAxisF = 1 << 14;
struct SScale {
    int e, f;
    bool turned;
    __host__ __device__ int32_t pack() const { return (e & 0xffff) | (f << 16) | (turned ? 1 << 31 : 0); }
};
__host__ __device__ __forceinline__ SScale sscale_of(int32_t v)
{
    return SScale{(int)(int16_t)(v & 0xffff), (v >> 16) & 0x7fff, v < 0};
}

// The scale of the sums of one part (im or re) of a column, whose largest high
// word is hmax: as bint_scale.
__device__ __forceinline__ int part_scale(const double2* col, int ld, int k, const int32_t* rmul,
                                          bool im, uint32_t hmax)
{
    uint32_t units = 0;
    uint64_t sum = 0;
    for (int i = 0; i < k; ++i) {
        const double x = im ? col[i * ld].y : col[i * ld].x;
        units += (uint32_t)rmul[i] * bint_units(bint_mag(x, 0.0), hmax);
        sum += (uint64_t)rmul[i] * bint_mag_subnormal(x, 0.0);
    }
    return hmax < 0x100000u ? bint_scale_subnormal(sum) : bint_scale(hmax, units);
}

// Stage the base matrix with a unit for each part (2 b, as bint_stage): cexp[j]
// receives column j's SScale.  one: all columns take the least f, which is that of
// the product of them all.  Returns the sum of c_j e_j.
static __device__ __noinline__ int sint_stage(double2* Md, int ld, int k, int l, const int32_t* rmul,
                                              const int32_t* cmul, int32_t* cexp, int lane, bool one)
{
    longlong2* M = reinterpret_cast<longlong2*>(Md);
    int x = 0, least = kOnAxisF;
    for (int j = lane; j < l; j += 32) {
        BParts parts;
        for (int i = 0; i < k; ++i)
            parts.add(Md[i * ld + j].x, Md[i * ld + j].y);
        const bool axis = parts.no_re() || parts.no_im();
        SScale s;
        s.turned = bint_exponent(parts.im) > bint_exponent(parts.re) || (axis && parts.no_re());
        s.e = part_scale(Md + j, ld, k, rmul, s.turned, s.turned ? parts.im : parts.re);
        s.f = kOnAxisF;
        if (!axis) {
            const int small =
                part_scale(Md + j, ld, k, rmul, !s.turned, s.turned ? parts.re : parts.im);
            s.e = min(s.e, small);
            s.f = small - s.e;
        }
        cexp[j] = s.pack();
        least = min(least, s.f);
        x += cmul[j] * s.e;
    }
    least = (int)__reduce_min_sync(0xffffffffu, (unsigned)least);
    for (int j = lane; j < l; j += 32) {
        SScale s = sscale_of(cexp[j]);
        if (one)
            s.f = least;
        for (int i = 0; i < k; ++i) {
            const double2 b = Md[i * ld + j];
            const double low = s.turned ? -b.x : b.y;
            M[i * ld + j] = make_longlong2(2 * bint_of(s.turned ? b.y : b.x, s.e),
                                           low == 0.0 ? 0 : 2 * bint_of(low, s.e + s.f));
        }
        cexp[j] = s.pack();
    }
    __syncwarp();
    return __reduce_add_sync(0xffffffffu, x);
}

// Multiplied back by i^turns.
__device__ __forceinline__ double2 turn(double re, double im, int turns)
{
    switch (turns & 3) {
    case 0: return make_double2(re, im);
    case 1: return make_double2(-im, re);
    case 2: return make_double2(-re, -im);
    default: return make_double2(im, -re);
    }
}

// How bint_stage leaves the base matrix.
enum {
    kStagedInt,    // integers, one unit for a column
    kStagedParts,  // near an axis: a unit for each part
    kStagedFp64    // not finite, or beyond FP64: the doubles as they came
};

// Turn a staged base matrix (k x l doubles in shared memory, row stride ld,
// row multiplicities rmul, column multiplicities cmul; one warp) into scaled
// integers 2 b_ij in place: cexp[j] receives column j's exponent and esum the
// sum of c_j cexp[j].  The matrix stays in doubles if a lane passes bad (a
// non-finite entry) or a column's sums can overflow FP64.  It is staged by
// sint_stage if a product of the columns can lie near an axis: no column is off
// the axes and one is near one.  omit: the products that leave out one copy of a
// column, too (a gradient's: one column off the axes, not repeated, decides
// nothing).
__device__ __forceinline__ int bint_stage(double2* Md, int ld, int k, int l, const int32_t* rmul,
                                          const int32_t* cmul, int32_t* cexp, bool bad, int lane,
                                          int& esum, bool omit)
{
    int x = 0;
    int off = 0;  // copies of this lane's columns off the axes
    bool near = false;
    for (int j = lane; j < l; j += 32) {
        uint32_t re = 0, im = 0, units = 0;
        for (int i = 0; i < k; ++i) {
            const double2 b = Md[i * ld + j];
            re = max(re, bint_mag(b.x, 0.0));
            im = max(im, bint_mag(b.y, 0.0));
        }
        const uint32_t hmax = max(re, im);
        if (!bint_apart(re, im)) {
            off += cmul[j];
        } else {
            BParts parts;
            for (int i = 0; i < k; ++i)
                parts.add(Md[i * ld + j].x, Md[i * ld + j].y);
            near = near || bint_near_axis(parts);
        }
        for (int i = 0; i < k; ++i) {
            const double2 b = Md[i * ld + j];
            units += (uint32_t)rmul[i] * bint_units(bint_mag(b.x, b.y), hmax);
        }
        int e = bint_scale(hmax, units);
        if (hmax < 0x100000u) {
            uint64_t sum = 0;
            for (int i = 0; i < k; ++i) {
                const double2 b = Md[i * ld + j];
                sum += (uint64_t)rmul[i] * bint_mag_subnormal(b.x, b.y);
            }
            e = bint_scale_subnormal(sum);
        }
        bad = bad || e < kSumBits - 1024;  // the sums can overflow FP64
        cexp[j] = e;
        x += cmul[j] * e;
    }
    if (__any_sync(0xffffffffu, bad))
        return kStagedFp64;
    const bool axes = omit ? __reduce_add_sync(0xffffffffu, off) <= 1
                           : !__any_sync(0xffffffffu, off > 0);
    if (axes && __any_sync(0xffffffffu, near)) {
        esum = sint_stage(Md, ld, k, l, rmul, cmul, cexp, lane, !omit);
        return kStagedParts;
    }
    esum = __reduce_add_sync(0xffffffffu, x);
    __syncwarp();
    longlong2* M = reinterpret_cast<longlong2*>(Md);
    for (int e = lane; e < k * l; e += 32) {
        const int i = e / l, j = e - i * l;
        const double2 b = Md[i * ld + j];
        const int c = cexp[j];
        M[i * ld + j] = make_longlong2(2 * bint_of(b.x, c), 2 * bint_of(b.y, c));
    }
    __syncwarp();
    return kStagedInt;
}

// sum_i r_i b_ij of a staged column (all Gray digits at zero), biased.
__device__ __forceinline__ longlong2 bint_base(const longlong2* Mj, int ld, int k,
                                               const int32_t* rmul)
{
    longlong2 s = make_longlong2(kSumBias, kSumBias);
    for (int i = 0; i < k; ++i) {
        const longlong2 b = Mj[i * ld];
        s.x += rmul[i] * (b.x >> 1);
        s.y += rmul[i] * (b.y >> 1);
    }
    return s;
}
#endif

}  // namespace pqi
