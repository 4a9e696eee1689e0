// hafnian.cu -- hafnians and loop hafnians of symmetric matrices with
// repeated indices (Sec. 4.1, Eq. (haf_def), Eq. (loop_hafnian), Figs.
// hafnian and loop_hafnian with (2, ..., 2) repetitions), on the same
// warp-uniform mixed-radix Gray walk and double-double accumulation as the
// permanent.
//
// Glynn-type formulas (a reading: the paper names the Glynn-type strategy but
// prints no formula).  For a sign vector d of the N expanded indices, the
// coefficient of d_1 ... d_N in exp(Q(d) + Lin(d)), Q = sum_{p<q} A_pq d_p d_q,
// Lin = sum_p A_pp d_p, counts every matching with loops once, and the mean of
// (prod d) times a polynomial in d is exactly that coefficient.  Without loops
// only Q^n / n! (N = 2n) has degree N.  With base index i repeated r_i times
// and g_i of its copies negative, x_i = r_i - 2 g_i and, B the base matrix and
// gamma the loop weights,
//   q(g) = 1/2 (x^T B x - sum_i r_i B_ii),   l(g) = gamma^T x,
//   haf  = 1 / (n! 2^{N-1}) sum_g s(g) q^n,
//   lhaf = 1 / 2^{N-1} sum_g s(g) sum_{j <= N/2} q^j l^{N-2j} / (j! (N-2j)!),
//   s(g) = (-1)^{sum g} prod_i C(top_i, g_i),
// one copy of the least repeated index keeping a + sign (top = r - 1 there;
// the summand is even under flipping every sign).  A Gray step changes one
// x_r by D = -+2:  q += D y_r + 2 B_rr with y = B x, then y_j += D B_jr and
// l += D gamma_r.  Inside a chunk only the J low digits move, so the walk
// reads y at the J low rows alone and keeps only those (2J adds a step
// instead of 2k); y is formed in full once per chunk for the start value of
// q.  q^n is taken by repeated squaring.  The loop polynomial is homogeneous
// of degree N/2 in (q, l^2): sum_j q^j s^{J-j} / (j! (N-2j)!) with s = l^2,
// J = floor(N/2), equals c_J prod_m (q - z_m s) (times l for odd N), where
// z_m = -1 / (2 x_m^2) and x_m runs over the positive roots of the Hermite
// polynomial He_N (substituting z = -1/(2x^2) turns the sum into
// x^{-N} He_N(x) / N!).  The roots are real, found once per N on the host by
// Sturm-count bisection on the Jacobi matrix of He_N, and the kernel
// multiplies the factors in pairs.
//
// The walk runs in 64-bit block integers (pq_blockint.cuh) on the integer
// pipes, as the permanent's does: q, y and l are scaled integers (every update
// is exact), the powers and polynomial factors are products of limbs, and FP64
// takes one conversion and one fused add per term and component.  All sums are
// taken modulo 2^64: only q and l themselves have to stay in range.  In FP64
// the walk was bound by the FP64 pipe (85 to 90% active): (2, ..., 2) at
// N = 36 took 19.1 ms (hafnian), N = 28 with loops 1.68 ms; in integers, bound
// by the wide multiplies and their adds, 4.67 ms and 0.34 ms.  A matrix
// without a scale (non-finite or subnormal entries, a bound beyond FP64) is
// walked in FP64.  Where the terms lie near the real or imaginary axis, one unit
// for both parts would round the small one (pq_blockint.cuh): a hafnian then has a
// unit for each part, a loop hafnian, whose factors add two terms of any ratio,
// keeps the FP64 walk.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <numeric>
#include <vector>

#include "../../include/pq.h"
#include "pq_blockint.cuh"
#include "pq_device.cuh"
#include "pq_fixsum.cuh"
#include "pq_kernels.h"

namespace pqi {

constexpr int kHafMaxHalf = PQ_MAX_N / 2;  // loop-polynomial factors j = 1 .. N/2
// integers of a loop polynomial of J = N/2 roots: 4 a pair, 2 for an odd root
__host__ __device__ constexpr int haf_integers(int J) { return 4 * (J / 2) + 2 * (J % 2); }
constexpr int kHafMaxInts = 48;
static_assert(haf_integers(kHafMaxHalf) <= kHafMaxInts && haf_integers(kHafMaxHalf - 1) <= kHafMaxInts,
              "room for the integers of every loop polynomial");

// Per (loop) hafnian: k kept base indices, digits as for the permanent.
struct alignas(16) HafDesc {
    int64_t T, nchunks, L, src_off, gam_off;
    int32_t k, n, N, ld;   // kept indices, N/2, expanded size, source row stride
    int32_t meta;          // ridx[k], rmul[k], drow[nd], drad[nd], dtop[nd]
    int32_t ndig, J, ntasks, slot0;
    int32_t gslot0;        // first counter of its task groups (more than 32 tasks)
    int32_t weighted, trivial;  // trivial: result = value (0 for odd N, 1 for N = 0)
    int32_t coef_off;           // loop hafnian: factors of its loop polynomial in loopc
    double value;               // final multiplier (or the trivial result)
};

struct HafArgs {
    const HafDesc* desc;
    const int32_t* meta;
    const Task* tasks;
    int64_t ntasks;
    const double2* src;
    const double2* gamma;  // loop weights (loop hafnian only)
    const double* loopc;   // loop-polynomial factors per distinct N (loop hafnian only):
                           // J + 1 doubles, then the integers of loop_integers
    double2* out;
    double* partials;
    int32_t* counters;  // [0] task queue head, [1 + b] finished tasks (or groups) of item b
    int32_t* groups;    // finished tasks of each group of 32
};

// Shared memory of one warp: M (k x k), y0 = B r (k), gamma (k), y (k x 32,
// lane-major), loop-polynomial factors (doubles and integers).  The planner
// puts the rows of the low digits first, so the walk's y and B at the low rows
// are the first J rows of these.
__host__ __device__ inline int haf_warp_smem_bytes(int kmax)
{
    const int bytes = (kmax * kmax + 2 * kmax + 32 * kmax) * 16 +
                      (kHafMaxHalf + 1 + kHafMaxInts) * 8;
    return (bytes + 15) & ~15;
}

// q^E by the binary method, unrolled at compile time.
template <int E>
__device__ __forceinline__ double2 cpow_c(double2 q)
{
    if constexpr (E == 1) {
        return q;
    } else if constexpr ((E & 1) == 0) {
        const double2 h = cpow_c<E / 2>(q);
        return cmul(h, h);
    } else {
        return cmul(cpow_c<E - 1>(q), q);
    }
}

// q^n for a warp-uniform 1 <= n <= PQ_MAX_N / 2: one uniform branch to
// straight-line code (a runtime bit loop would issue its conditional
// multiplies under false predicates).
__device__ __forceinline__ double2 cpow_n(double2 q, int n)
{
    switch (n) {
#define PQ_POW_CASE(E) \
    case E: return cpow_c<E>(q);
        PQ_POW_CASE(1) PQ_POW_CASE(2) PQ_POW_CASE(3) PQ_POW_CASE(4) PQ_POW_CASE(5)
        PQ_POW_CASE(6) PQ_POW_CASE(7) PQ_POW_CASE(8) PQ_POW_CASE(9) PQ_POW_CASE(10)
        PQ_POW_CASE(11) PQ_POW_CASE(12) PQ_POW_CASE(13) PQ_POW_CASE(14) PQ_POW_CASE(15)
        PQ_POW_CASE(16) PQ_POW_CASE(17) PQ_POW_CASE(18) PQ_POW_CASE(19) PQ_POW_CASE(20)
        PQ_POW_CASE(21) PQ_POW_CASE(22) PQ_POW_CASE(23) PQ_POW_CASE(24)
#undef PQ_POW_CASE
    default: return q;  // not reached: the planner bounds n by PQ_MAX_N / 2
    }
}
static_assert(PQ_MAX_N / 2 == 24, "cpow_n covers exponents up to 24");

// sum_{j=0}^{N/2} q^j l^{N-2j} / (j! (N-2j)!) from the factors cf = [c_J,
// a_0, b_0, a_1, b_1, ..., (z_last)]: each of the P = floor(N/4) pairs of
// roots gives q^2 + a q s + b s^2 (a = -(z1 + z2), b = z1 z2); an odd root
// count J leaves one factor q - z s; odd N one factor l.  JODD and NODD are
// template flags so that no factor is issued under a false predicate.
template <bool JODD, bool NODD>
__device__ __forceinline__ double2 loop_poly(double2 q, double2 l, int P, const double* cf)
{
    const double2 s = cmul(l, l);
    double2 h = make_double2(cf[0], 0.0);
    if (P) {
        const double2 q2 = cmul(q, q), qs = cmul(q, s), s2 = cmul(s, s);
#pragma unroll 1
        for (int p = 0; p < P; ++p) {
            const double a = cf[1 + 2 * p], b = cf[2 + 2 * p];
            double2 t;
            t.x = __fma_rn(b, s2.x, __fma_rn(a, qs.x, q2.x));
            t.y = __fma_rn(b, s2.y, __fma_rn(a, qs.y, q2.y));
            h = cmul(h, t);
        }
    }
    if (JODD) {
        const double z = cf[1 + 2 * P];
        double2 t;
        t.x = __fma_rn(-z, s.x, q.x);
        t.y = __fma_rn(-z, s.y, q.y);
        h = cmul(h, t);
    }
    if (NODD)
        h = cmul(h, l);
    return h;
}

// The pieces of a warp's shared memory; doubles for the FP64 walk, scaled
// integers for the other.
struct HafSmem {
    double2* M;    // k x k: b (FP64), 2 b (integers)
    double2* y0;   // k: B r
    double2* gam;  // k
    double2* Y;    // k x 32, lane-major
    double* cj;    // loop-polynomial factors
    int64_t* ci;   // and their integers
    __device__ HafSmem(unsigned char* raw, int kmax)
    {
        M = reinterpret_cast<double2*>(raw);
        y0 = M + kmax * kmax;
        gam = y0 + kmax;
        Y = gam + kmax;
        cj = reinterpret_cast<double*>(Y + 32 * kmax);
        ci = reinterpret_cast<int64_t*>(cj + kHafMaxHalf + 1);
    }
};

// Integer metadata of one item.
struct HafMeta {
    const int32_t *ridx, *rmul, *drow, *drad, *dtop;
    __device__ HafMeta(const HafArgs& a, const HafDesc& D)
    {
        ridx = a.meta + D.meta;
        rmul = ridx + D.k;
        drow = rmul + D.k;
        drad = drow + D.ndig;
        dtop = drad + D.ndig;
    }
};

// What a warp keeps about the item it has staged.
struct HafStaged {
    int item = -1;
    int mode = kStagedInt;
    int exp2 = 0;       // the terms' sum times 2^exp2 is the sum of s(g) times the polynomial
                        // (in integers: without its leading factor)
    int eq = 0, el = 0; // q and l times 2^eq, 2^el are the integers
    int ref2 = 0, ref1 = 0;  // loop hafnian: upper bounds of a factor's exponent (pair, odd root)
};

// The walk of this lane's chunk in FP64; returns the task's sum.
template <bool LOOP>
__device__ __noinline__ dd2 haf_walk_fp64(const HafDesc& D, const HafMeta& mt, const HafSmem& sm,
                                  int64_t c, bool active, int lane)
{
    const int k = D.k, J = D.J, nd = D.ndig;
    const double2 *M = sm.M, *y0 = sm.y0, *gam = sm.gam;
    const double* cj = sm.cj;
    const int32_t *rmul = mt.rmul, *drow = mt.drow, *drad = mt.drad, *dtop = mt.dtop;
    dd2 res;
    const int64_t c_first = c;
    double2* y = sm.Y + lane;
#pragma unroll 1
    for (int j = 0; j < k; ++j)
        y[j * 32] = y0[j];
    // High digits of this lane's chunk: x_row = r_row - 2 g.  y = B x is
    // finished before x^T y is formed in a second pass over the digits.
    uint64_t whigh_u = 1;
    int gpar = 0;
#pragma unroll 1
    for (int d = J; d < nd; ++d) {
        const int rad = drad[d];
        const int g = (int)(c % rad);
        c /= rad;
        if (!g)
            continue;
        const int row = drow[d];
        const double coef = (double)(-2 * g);
#pragma unroll 1
        for (int j = 0; j < k; ++j) {
            const double2 b = M[j * k + row];
            double2 v = y[j * 32];
            v.x = __fma_rn(coef, b.x, v.x);
            v.y = __fma_rn(coef, b.y, v.y);
            y[j * 32] = v;
        }
        whigh_u *= binom_u64(dtop[d], g);
        gpar += g;
    }
    // q = 1/2 (x^T y - sum_i r_i B_ii) and l = gamma^T x, low digits at 0
    double2 q = make_double2(0.0, 0.0), l = make_double2(0.0, 0.0);
#pragma unroll 1
    for (int i = 0; i < k; ++i) {
        const double2 v = y[i * 32];
        const double2 bii = M[i * k + i];
        const double r = (double)rmul[i];
        q.x = __fma_rn(r, __dsub_rn(v.x, bii.x), q.x);
        q.y = __fma_rn(r, __dsub_rn(v.y, bii.y), q.y);
        if (LOOP) {
            l.x = __fma_rn(r, gam[i].x, l.x);
            l.y = __fma_rn(r, gam[i].y, l.y);
        }
    }
    c = c_first;
#pragma unroll 1
    for (int d = J; d < nd; ++d) {
        const int rad = drad[d];
        const int g = (int)(c % rad);
        c /= rad;
        if (!g)
            continue;
        const int row = drow[d];
        const double2 v = y[row * 32];
        const double coef = (double)(-2 * g);
        q.x = __fma_rn(coef, v.x, q.x);
        q.y = __fma_rn(coef, v.y, q.y);
        if (LOOP) {
            l.x = __fma_rn(coef, gam[row].x, l.x);
            l.y = __fma_rn(coef, gam[row].y, l.y);
        }
    }
    q.x *= 0.5;
    q.y *= 0.5;
    double2* yl = y;  // rows 0 .. J - 1
    double whigh = active ? (double)whigh_u : 0.0;
    if (gpar & 1)
        whigh = -whigh;

    LowWalk wk;
    wk.v = 0;
    wk.g = 0;
    wk.dir = 0;
    wk.radm1 = 0;
    wk.topp = 0;
    for (int d = 0; d < J; ++d) {
        wk.radm1 |= uint64_t(drad[d] - 1) << (4 * d);
        wk.topp |= uint64_t(dtop[d]) << (4 * d);
    }
    const bool weighted = D.weighted != 0;
    const int n = D.n, N = D.N;
    const int form = ((N >> 1) & 1) * 2 + (N & 1), P = N >> 2;
    double wlow = 1.0;
    double2 acc = make_double2(0.0, 0.0);
    double rh = 0.0, rl = 0.0, ih = 0.0, il = 0.0;
    const int64_t L = D.L;
    // The term's polynomial value; the uniform switches pick straight-line
    // code for the exponent or the loop-polynomial shape, so no FP64
    // instruction is issued under a false predicate.
    auto value = [&]() -> double2 {
        if (LOOP) {
            switch (form) {
            case 0: return loop_poly<false, false>(q, l, P, cj);
            case 1: return loop_poly<false, true>(q, l, P, cj);
            case 2: return loop_poly<true, false>(q, l, P, cj);
            default: return loop_poly<true, true>(q, l, P, cj);
            }
        }
        return cpow_n(q, n);
    };
    auto term_pos = [&]() {
        const double2 p = value();
        acc.x = __fma_rn(wlow, p.x, acc.x);
        acc.y = __fma_rn(wlow, p.y, acc.y);
    };
    auto term_neg = [&]() {
        const double2 p = value();
        acc.x = __fma_rn(-wlow, p.x, acc.x);
        acc.y = __fma_rn(-wlow, p.y, acc.y);
    };
    // One Gray step: x_row moves by -+2.
    auto step = [&]() {
        int up;
        const int d = low_step(wk, up);
        const double delta = up > 0 ? -2.0 : 2.0;
        const double2 yr = yl[d * 32];
        const double2* Bd = M + d * k;
        const double2 brr = Bd[d];
        q.x = __fma_rn(delta, yr.x, q.x);
        q.y = __fma_rn(delta, yr.y, q.y);
        q.x = __fma_rn(2.0, brr.x, q.x);
        q.y = __fma_rn(2.0, brr.y, q.y);
        if (LOOP) {
            const double2 gr = gam[d];
            l.x = __fma_rn(delta, gr.x, l.x);
            l.y = __fma_rn(delta, gr.y, l.y);
        }
#pragma unroll 1
        for (int e = 0; e < J; ++e) {
            const double2 b = Bd[e];
            double2 v = yl[e * 32];
            v.x = __fma_rn(delta, b.x, v.x);
            v.y = __fma_rn(delta, b.y, v.y);
            yl[e * 32] = v;
        }
        if (weighted && ((wk.radm1 >> (4 * d)) & 15u) > 1u)
            wlow = (double)low_weight(wk, J);
    };
    // Term 0 has sign +; then pairs (odd: -, even: +), folded into the
    // double-double sums every 16 terms by the outer loop.
    term_pos();
    int64_t s = 1;
#pragma unroll 1
    while (s < L) {
        const int npairs = (int)min((L - s) >> 1, (int64_t)8);
#pragma unroll 1
        for (int i = 0; i < npairs; ++i) {
            step();
            term_neg();
            step();
            term_pos();
        }
        s += 2 * npairs;
        if (npairs == 0) {  // one (odd) term left
            step();
            term_neg();
            s += 1;
        }
        dd_acc(rh, rl, acc.x);
        dd_acc(ih, il, acc.y);
        acc = make_double2(0.0, 0.0);
    }
    dd_acc(rh, rl, acc.x);
    dd_acc(ih, il, acc.y);
    fast_two_sum(rh, rl, rh, rl);
    fast_two_sum(ih, il, ih, il);
    dd_mul_d(rh, rl, whigh);
    dd_mul_d(ih, il, whigh);
    // the lanes' sums added exactly in integers (pq_fixsum.cuh)
    warp_fix_sum(rh, rl, res.rh, res.rl);
    warp_fix_sum(ih, il, res.ih, res.il);
    return res;
}

// Whether the terms of an item can lie near an axis (pq_blockint.cuh): b the parts
// of the entries, g those of the loop weights, root the exponent of
// the loop polynomial's largest root (its first factor is q + 2^root l^2 or so).
// q^n is near an axis where q is; a factor of the loop polynomial where the larger
// of its two terms' parts are far apart, and N = 1 leaves l alone.
template <bool LOOP>
__device__ __forceinline__ bool haf_near_axis(const BParts& b, const BParts& g, int N, int root)
{
    if (!LOOP)
        return bint_near_axis(b);
    if (N == 1)
        return bint_near_axis(g);
    constexpr int kNone = -(1 << 20);
    int re = b.no_re() ? kNone : bint_exponent(b.re) - 1023;
    int im = b.no_im() ? kNone : bint_exponent(b.im) - 1023;
    const int x = g.no_re() ? kNone : bint_exponent(g.re) - 1023;
    const int y = g.no_im() ? kNone : bint_exponent(g.im) - 1023;
    re = max(re, 2 * max(x, y) + root);
    im = max(im, x + y + 1 + root);
    return min(re, im) > kNone / 2 && abs(re - im) >= kAxisBits;
}

// The power of two that brings the largest part near 1, leaving at most 900
// binades below it to the smaller one.
__device__ __forceinline__ int unit_scale(const BParts& m)
{
    const int x = bint_exponent(m.re), y = bint_exponent(m.im);
    const int hi = max(x, y), lo = m.no_re() || m.no_im() ? hi : min(x, y);
    return 1023 - hi + max(0, hi - lo - 900);
}

// A loop hafnian near an axis, for the FP64 walk: entries times 2^(2 t) and loop
// weights times 2^t, which multiplies every term by 2^(t N) and keeps the powers in
// range.  Returns t.
__device__ __noinline__ int haf_scale(const HafSmem& sm, int k, const BParts& b, const BParts& g,
                                      int lane)
{
    int t = b.no_re() && b.no_im() ? 1 << 20 : unit_scale(b) >> 1;
    if (!g.no_re() || !g.no_im())
        t = min(t, unit_scale(g));
    for (int e = lane; e < k * k; e += kWarp)
        sm.M[e] = make_double2(scalbn(sm.M[e].x, 2 * t), scalbn(sm.M[e].y, 2 * t));
    for (int i = lane; i < k; i += kWarp)
        sm.gam[i] = make_double2(scalbn(sm.gam[i].x, t), scalbn(sm.gam[i].y, t));
    __syncwarp();
    return t;
}

// The scale of the sums of one part (im or re) of q, hmax its entries' largest
// high word.
__device__ __forceinline__ int haf_part_scale(const HafMeta& mt, const HafSmem& sm, int k, bool im,
                                              uint32_t hmax, int lane)
{
    uint64_t units = 0;
    for (int i = lane; i < k; i += kWarp) {
        uint32_t row = 0;
        for (int j = 0; j < k; ++j) {
            const double2 v = sm.M[i * k + j];
            row += (uint32_t)(mt.rmul[j] + (j == i ? 1 : 0)) *
                   bint_units(bint_mag(im ? v.y : v.x, 0.0), hmax);
        }
        units += (uint64_t)mt.rmul[i] * row;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
        units += __shfl_xor_sync(0xffffffffu, units, off);
    units += (units >> 20) + 1;  // the rounding of the entries stays inside the bound
    return kSumBits + 1044 - (int)(hmax >> 20) - bint_width(units);
}

// A hafnian near an axis: M = 2 b with a unit for each part, divided by i where the
// imaginary part is the larger.  False if a part has no scale (subnormal).
__device__ __noinline__ bool haf_stage_parts(const HafMeta& mt, const HafSmem& sm, int k,
                                             const BParts& b, SScale& s, int lane)
{
    if (min(b.re, b.im) < 0x100000u)
        return false;
    s.turned = bint_exponent(b.im) > bint_exponent(b.re);
    const int big = haf_part_scale(mt, sm, k, s.turned, max(b.re, b.im), lane);
    const int small = haf_part_scale(mt, sm, k, !s.turned, min(b.re, b.im), lane);
    s.e = min(big, small);
    s.f = small - s.e;
    longlong2* M = reinterpret_cast<longlong2*>(sm.M);
    for (int e = lane; e < k * k; e += kWarp) {
        const double2 v = sm.M[e];
        M[e] = make_longlong2(2 * bint_of(s.turned ? v.y : v.x, s.e),
                              2 * bint_of(s.turned ? -v.x : v.y, s.e + s.f));
    }
    __syncwarp();
    return true;
}

__device__ __forceinline__ void warp_parts(BParts& m)
{
    m.re = __reduce_max_sync(0xffffffffu, m.re);
    m.im = __reduce_max_sync(0xffffffffu, m.im);
    m.re_low = __reduce_or_sync(0xffffffffu, m.re_low);
    m.im_low = __reduce_or_sync(0xffffffffu, m.im_low);
}

// Stage item D as scaled integers: M = 2 b, y0 = B r, gam; a hafnian near an axis
// with a unit for each part (ci[0]: its SScale).  Returns false if it stays in
// doubles: an item without a scale as it came, a loop hafnian near an axis scaled.
template <bool LOOP>
__device__ bool haf_stage_int(const HafDesc& D, const HafMeta& mt, const HafSmem& sm, HafStaged& st,
                              int lane)
{
    const int k = D.k;
    st.mode = kStagedInt;
    st.exp2 = 0;
    bool bad = false;
    BParts b, g;
    for (int e = lane; e < k * k; e += kWarp)
        b.add(sm.M[e].x, sm.M[e].y);
    warp_parts(b);
    const uint32_t hmax = max(b.re, b.im);
    uint32_t gmax = 0;
    // |q| <= 1/2 (sum_ij r_i r_j |b_ij| + sum_i r_i |b_ii|)
    uint64_t units = 0;
    for (int i = lane; i < k; i += kWarp) {
        uint32_t row = 0;
        for (int j = 0; j < k; ++j)
            row += (uint32_t)(mt.rmul[j] + (j == i ? 1 : 0)) *
                   bint_units(bint_mag(sm.M[i * k + j].x, sm.M[i * k + j].y), hmax);
        units += (uint64_t)mt.rmul[i] * row;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
        units += __shfl_xor_sync(0xffffffffu, units, off);
    units += (units >> 20) + 1;  // the rounding of the entries stays inside the bound
    const int eq = kSumBits + 1044 - (int)(hmax >> 20) - bint_width(units);
    bad = hmax < 0x100000u || hmax >= 0x7ff00000u || eq < kSumBits - 1023;
    int el = 0;
    if (LOOP) {
        for (int i = lane; i < k; i += kWarp)
            g.add(sm.gam[i].x, sm.gam[i].y);
        warp_parts(g);
        gmax = max(g.re, g.im);
        uint32_t gu = 0;
        for (int i = lane; i < k; i += kWarp)
            gu += (uint32_t)mt.rmul[i] * bint_units(bint_mag(sm.gam[i].x, sm.gam[i].y), gmax);
        gu = __reduce_add_sync(0xffffffffu, gu);
        if (!g.no_re() || !g.no_im()) {
            el = bint_scale(gmax, gu);
            bad = bad || gmax < 0x100000u || gmax >= 0x7ff00000u || el < kSumBits - 1023;
        }
    }
    if (bad)
        return false;
    const int root = LOOP && D.N > 1 ? (int)sm.ci[0] : 0;
    SScale ps{eq, 0, false};
    if (haf_near_axis<LOOP>(b, g, D.N, root)) {
        if (LOOP) {
            st.exp2 = -haf_scale(sm, k, b, g, lane) * D.N;
            return false;
        }
        if (!haf_stage_parts(mt, sm, k, b, ps, lane))
            return false;
        st.mode = kStagedParts;
        if (lane == 0)
            sm.ci[0] = ps.pack();
    }
    longlong2* M = reinterpret_cast<longlong2*>(sm.M);
    longlong2* y0 = reinterpret_cast<longlong2*>(sm.y0);
    longlong2* gam = reinterpret_cast<longlong2*>(sm.gam);
    if (st.mode == kStagedInt) {
        for (int e = lane; e < k * k; e += kWarp) {
            const double2 v = sm.M[e];
            M[e] = make_longlong2(2 * bint_of(v.x, eq), 2 * bint_of(v.y, eq));
        }
    }
    if (LOOP) {
        for (int i = lane; i < k; i += kWarp) {
            const double2 b = sm.gam[i];
            gam[i] = make_longlong2(bint_of(b.x, el), bint_of(b.y, el));
        }
    }
    __syncwarp();
    for (int j = lane; j < k; j += kWarp) {
        uint64_t x = 0, y = 0;
        for (int i = 0; i < k; ++i) {
            const longlong2 b = M[j * k + i];
            x += (uint64_t)mt.rmul[i] * (uint64_t)(b.x >> 1);
            y += (uint64_t)mt.rmul[i] * (uint64_t)(b.y >> 1);
        }
        y0[j] = make_longlong2((long long)x, (long long)y);
    }
    __syncwarp();
    st.eq = eq;
    st.el = el;
    if (LOOP) {
        const int P = D.N >> 2, jo = (D.N >> 1) & 1, no = D.N & 1;
        const int xq = -eq, xs = 64 - 2 * el;  // upper bounds; the largest root comes first
        st.ref2 = P == 0 ? 0
                         : 2 + max(64 + 2 * xq, 66 + xs + max(xq + (int)sm.ci[0], xs + (int)sm.ci[2]));
        st.ref1 = jo == 0 ? 0 : 2 + max(xq, xs + (int)sm.ci[4 * P] + 2);
        st.exp2 = kSumBits + 64 * (P + jo + no - 1) + P * st.ref2 + jo * st.ref1 - no * el;
    } else {
        st.exp2 = kSumBits + 64 * (D.n - 1) - D.n * ps.e;
    }
    return true;
}

__device__ __forceinline__ longlong2 bint_pair(const BInt& p)
{
    return make_longlong2((long long)(((uint64_t)(uint32_t)p.rh << 32) | p.rl),
                          (long long)(((uint64_t)(uint32_t)p.ih << 32) | p.il));
}

// h[i] = q[i]^n, n >= 1 (binary method from the top bit; n is uniform): the
// integers, normalised, and their exponents E.  M = 2 interleaves two terms,
// whose dependent chains of products then hide each other (N = 36: 4.87 -> 4.67
// ms; 14 warps fit on an SM by shared memory, which leaves 128 registers).
template <int M, class Mul>
__device__ __forceinline__ void haf_power(const longlong2 (&q)[M], int n, BInt (&h)[M], int (&E)[M],
                                          const Mul& mul)
{
    BLimbs lx[M];
    int Ex[M];
#pragma unroll
    for (int i = 0; i < M; ++i) {
        h[i] = bint_words(q[i]);
        Ex[i] = 0;
        bnorm(h[i], Ex[i]);
        lx[i] = limbs(h[i]);
        E[i] = Ex[i];
    }
#pragma unroll 1
    for (int bit = 30 - __clz(n); bit >= 0; --bit) {
#pragma unroll
        for (int i = 0; i < M; ++i) {
            h[i] = mul.sqr(limbs(h[i]));
            E[i] *= 2;
            bnorm(h[i], E[i]);
        }
        if ((n >> bit) & 1) {
#pragma unroll
            for (int i = 0; i < M; ++i) {
                h[i] = mul(limbs(h[i]), lx[i]);
                E[i] += Ex[i];
                bnorm(h[i], E[i]);
            }
        }
    }
}

// c v >> 64 for a real 0 <= c < 2^62 (the limbs of a larger c overflow).
__device__ __forceinline__ longlong2 real_scale(int64_t c, const BLimbs& v)
{
    const int ch = (int)((c + kSumBias) >> 32), cl = (int)(uint32_t)c;
    const int64_t mr = mulw(v.a, cl) + mulw(v.b, ch), mi = mulw(v.c, cl) + mulw(v.d, ch);
    const int64_t hr = mulw(v.a, ch) + (int64_t)(int)(mr >> 32);
    const int64_t hi = mulw(v.c, ch) + (int64_t)(int)(mi >> 32);
    return make_longlong2(hr, hi);
}

__device__ __forceinline__ longlong2 shift_right(longlong2 v, int n)
{
    n = min(n, 63);
    return make_longlong2(v.x >> n, v.y >> n);
}

// The loop polynomial of q and l without its leading factor: P pairs of roots
// q^2 + a q s + b s^2 with s = l^2, an odd root q + c s, an odd N one factor l.
// q^2, q s and s^2 are normalised once, and the coefficients are integers of 62
// bits with an exponent each (ci: ea, a, eb, b of each pair, ec and c of an odd
// root), so every product has its full bits whatever the ratio of q and s; the
// three terms of a factor are brought to the largest of their exponents and one
// more, which keeps the factor below 2^62.  E counts the factors' exponents
// against their upper bounds ref2 and ref1.
__device__ __forceinline__ BInt haf_loop_poly(longlong2 q, longlong2 l, int P, bool jodd, bool nodd,
                                              const int64_t* ci, const HafStaged& st, int& E)
{
    BInt lw = bint_words(l), h;
    int El = 0;
    bnorm(lw, El);
    E = 0;
    bool first = true;
    if (P > 0 || jodd) {
        BInt qw = bint_words(q);
        int Eq = 0;
        bnorm(qw, Eq);
        const BLimbs ll = limbs(lw);
        BInt sw = bsqr(ll);
        int Es = 0;
        bnorm(sw, Es);
        constexpr int kNone = -(1 << 18), kLeast = -(1 << 17);  // exponent of an exact zero
        const int xq = (qw.rh | qw.ih | qw.rl | qw.il) == 0 ? kNone : -st.eq - Eq;
        const int xs = (sw.rh | sw.ih | sw.rl | sw.il) == 0 ? kNone : 64 - 2 * (st.el + El) - Es;
        const BLimbs lq = limbs(qw), ls = limbs(sw);
        if (P > 0) {
            int n0 = 0, n1 = 0, n2 = 0;
            BInt v0 = bsqr(lq), v1 = bmul(lq, ls), v2 = bsqr(ls);
            bnorm(v0, n0);
            bnorm(v1, n1);
            bnorm(v2, n2);
            const int x0 = 2 * xq + 64 - n0, x1 = xq + xs + 66 - n1, x2 = 2 * xs + 66 - n2;
            const longlong2 q2 = bint_pair(v0);
            const BLimbs qs = limbs(v1), s2 = limbs(v2);
#pragma unroll 1
            for (int p = 0; p < P; ++p) {
                const int64_t* c = ci + 4 * p;
                const int f1 = x1 + (int)c[0], f2 = x2 + (int)c[2];
                const int f = max(max(x0 + 1, max(f1, f2)) + 1, kLeast);
                const longlong2 t0 = shift_right(q2, f - x0);
                const longlong2 t1 = shift_right(real_scale(c[1], qs), f - f1);
                const longlong2 t2 = shift_right(real_scale(c[3], s2), f - f2);
                const BInt t = bint_words(make_longlong2(t0.x + t1.x + t2.x, t0.y + t1.y + t2.y));
                h = first ? t : bmul(limbs(h), limbs(t));
                first = false;
                E += st.ref2 - f;
                bnorm(h, E);
            }
        }
        if (jodd) {
            const int64_t* c = ci + 4 * P;
            const int f1 = xs + (int)c[0] + 2, f = max(max(xq + 1, f1) + 1, kLeast);
            const longlong2 t0 = shift_right(bint_pair(qw), f - xq);
            const longlong2 t1 = shift_right(real_scale(c[1], ls), f - f1);
            const BInt t = bint_words(make_longlong2(t0.x + t1.x, t0.y + t1.y));
            h = first ? t : bmul(limbs(h), limbs(t));
            first = false;
            E += st.ref1 - f;
            bnorm(h, E);
        }
    }
    if (nodd) {
        h = first ? lw : bmul(limbs(h), limbs(lw));
        E += El;
    }
    return h;
}

// The walk of this lane's chunk in block integers; returns the task's sum.
// All sums are taken modulo 2^64 (unsigned): y may leave the range of 64 bits,
// q and l do not.
template <bool LOOP, class Mul>
__device__ __forceinline__ dd2 haf_walk_int(const HafDesc& D, const HafMeta& mt, const HafSmem& sm,
                                            const HafStaged& st, int64_t c, bool active, int lane,
                                            const Mul& mul)
{
    const int k = D.k, J = D.J, nd = D.ndig;
    const ulonglong2* M = reinterpret_cast<const ulonglong2*>(sm.M);
    const ulonglong2* y0 = reinterpret_cast<const ulonglong2*>(sm.y0);
    const ulonglong2* gam = reinterpret_cast<const ulonglong2*>(sm.gam);
    ulonglong2* y = reinterpret_cast<ulonglong2*>(sm.Y) + lane;
    // High digits of this lane's chunk: x_row = r_row - 2 g.  y = B x is
    // finished before x^T y is formed in a second pass over the digits.
#pragma unroll 1
    for (int j = 0; j < k; ++j)
        y[j * 32] = y0[j];
    uint64_t whigh_u = 1;
    int gpar = 0;
    const bool narrow = D.nchunks <= 0x7fffffff;
    int64_t cc = c;
#pragma unroll 1
    for (int d = J; d < nd; ++d) {
        const int g = next_digit(cc, mt.drad[d], narrow);
        if (!g)
            continue;
        const ulonglong2* Mr = M + mt.drow[d];
#pragma unroll 1
        for (int j = 0; j < k; ++j) {
            const ulonglong2 b = Mr[j * k];
            ulonglong2 v = y[j * 32];
            v.x -= (uint64_t)g * b.x;
            v.y -= (uint64_t)g * b.y;
            y[j * 32] = v;
        }
        whigh_u *= high_binom(mt.dtop[d], g);
        gpar += g;
    }
    // 2 q = x^T y - sum_i r_i B_ii and l = gamma^T x, low digits at 0
    ulonglong2 q = make_ulonglong2(0, 0), l = make_ulonglong2(0, 0);
#pragma unroll 1
    for (int i = 0; i < k; ++i) {
        const ulonglong2 v = y[i * 32], bii = M[i * k + i];
        const uint64_t r = (uint64_t)mt.rmul[i];
        q.x += r * (v.x - (uint64_t)((int64_t)bii.x >> 1));
        q.y += r * (v.y - (uint64_t)((int64_t)bii.y >> 1));
        if (LOOP) {
            l.x += r * gam[i].x;
            l.y += r * gam[i].y;
        }
    }
    cc = c;
#pragma unroll 1
    for (int d = J; d < nd; ++d) {
        const int g = next_digit(cc, mt.drad[d], narrow);
        if (!g)
            continue;
        const int row = mt.drow[d];
        const ulonglong2 v = y[row * 32];
        q.x -= 2 * (uint64_t)g * v.x;
        q.y -= 2 * (uint64_t)g * v.y;
        if (LOOP) {
            l.x -= 2 * (uint64_t)g * gam[row].x;
            l.y -= 2 * (uint64_t)g * gam[row].y;
        }
    }
    q.x = (uint64_t)((int64_t)q.x >> 1);
    q.y = (uint64_t)((int64_t)q.y >> 1);

    LowDigits lo;
    lo.radm1 = lo.topp = 0;
    lo.J = J;
    for (int d = 0; d < J; ++d) {
        lo.radm1 |= uint64_t(mt.drad[d] - 1) << (4 * d);
        lo.topp |= uint64_t(mt.dtop[d]) << (4 * d);
    }
    const bool weighted = D.weighted != 0;
    const int n = D.n, P = D.N >> 2;
    const bool jodd = ((D.N >> 1) & 1) != 0, nodd = (D.N & 1) != 0;
    uint32_t steps = 0;
    double step_w = 1.0, w = 1.0;
    double2 acc = make_double2(0.0, 0.0);
    double rh = 0.0, rl = 0.0, ih = 0.0, il = 0.0;
    const uint32_t L = (uint32_t)D.L;
    uint32_t s = 0;
    // step s - 1 -> s of the Gray code
    auto advance = [&]() {
        // the Gray steps 32 at a time, one per lane, as in the permanent's walk
        const int sq = (int)((s - 1u) & 31u);
        if (sq == 0) {
            bool up;
            uint64_t wu;
            const int d = gray_step_at(lo, s + (uint32_t)lane, weighted, up, wu);
            steps = ((uint32_t)d << 1) | (up ? 0u : 1u);
            if (weighted)
                step_w = (double)wu;
        }
        const uint32_t step = __shfl_sync(0xffffffffu, steps, sq);
        if (weighted)
            w = __shfl_sync(0xffffffffu, step_w, sq);
        // x_d moves by -+2: q += -+2 y_d + 2 B_dd, then y moves by -+2 B
        const int d = (int)(step >> 1);
        const ulonglong2 yd = y[d * 32];
        const ulonglong2* Bd = M + d * k;
        const ulonglong2 bdd = Bd[d];
        if (step & 1u) {
            q.x += 2 * yd.x + bdd.x;
            q.y += 2 * yd.y + bdd.y;
#pragma unroll 1
            for (int e = 0; e < J; ++e) {
                const ulonglong2 b = Bd[e];
                ulonglong2 v = y[e * 32];
                v.x += b.x;
                v.y += b.y;
                y[e * 32] = v;
            }
            if (LOOP) {
                l.x += 2 * gam[d].x;
                l.y += 2 * gam[d].y;
            }
        } else {
            q.x += bdd.x - 2 * yd.x;
            q.y += bdd.y - 2 * yd.y;
#pragma unroll 1
            for (int e = 0; e < J; ++e) {
                const ulonglong2 b = Bd[e];
                ulonglong2 v = y[e * 32];
                v.x -= b.x;
                v.y -= b.y;
                y[e * 32] = v;
            }
            if (LOOP) {
                l.x -= 2 * gam[d].x;
                l.y -= 2 * gam[d].y;
            }
        }
    };
    auto add_term = [&](const BInt& p, int E, uint32_t at, double wt) {
        const longlong2 pv = bint_pair(p);
        const double f = bint_factor(wt, E, (at & 1u) != 0);
        acc.x = __fma_rn(__ll2double_rn(pv.x), f, acc.x);
        acc.y = __fma_rn(__ll2double_rn(pv.y), f, acc.y);
    };
#pragma unroll 1
    for (;;) {
        const longlong2 q0 = make_longlong2((long long)q.x, (long long)q.y);
        if (LOOP) {
            int E;
            const BInt p =
                haf_loop_poly(q0, make_longlong2((long long)l.x, (long long)l.y), P, jodd, nodd,
                              sm.ci, st, E);
            add_term(p, E, s, w);
        } else if (s + 1 < L) {
            const double w0 = w;
            ++s;
            advance();
            const longlong2 q2[2] = {q0, make_longlong2((long long)q.x, (long long)q.y)};
            BInt p[2];
            int E[2];
            haf_power(q2, n, p, E, mul);
            add_term(p[0], E[0], s - 1, w0);
            add_term(p[1], E[1], s, w);
        } else {
            const longlong2 q1[1] = {q0};
            BInt p[1];
            int E[1];
            haf_power(q1, n, p, E, mul);
            add_term(p[0], E[0], s, w);
        }
        ++s;
        if (s == L || (s & 15u) == 0) {
            if (L <= 16u) {  // the only fold of a short chunk
                rh = acc.x;
                ih = acc.y;
                break;
            }
            dd_acc(rh, rl, acc.x);
            dd_acc(ih, il, acc.y);
            acc = make_double2(0.0, 0.0);
            if (s == L)
                break;
        }
        advance();
    }
    double whigh = active ? (double)whigh_u : 0.0;
    if (gpar & 1)
        whigh = -whigh;
    fast_two_sum(rh, rl, rh, rl);
    fast_two_sum(ih, il, ih, il);
    dd_mul_d(rh, rl, whigh);
    dd_mul_d(ih, il, whigh);
    // the lanes' sums added exactly in integers (pq_fixsum.cuh)
    dd2 res;
    warp_fix_sum(rh, rl, res.rh, res.rl);
    warp_fix_sum(ih, il, res.ih, res.il);
    return res;
}

__device__ __noinline__ dd2 haf_walk_parts(const HafDesc& D, const HafMeta& mt, const HafSmem& sm,
                                           const HafStaged& st, int64_t c, bool active, int lane)
{
    const PartUnits mul{min(63, 2 * sscale_of((int32_t)sm.ci[0]).f)};
    return haf_walk_int<false>(D, mt, sm, st, c, active, lane, mul);
}

template <bool LOOP>
__device__ void haf_task(const HafArgs& a, const Task& t, const HafSmem& sm, HafStaged& st, int lane)
{
    const HafDesc D = a.desc[t.perm];
    const int k = D.k;
    dd2 res = {0.0, 0.0, 0.0, 0.0};

    if (!D.trivial) {
        const HafMeta mt(a, D);
        if (st.item != t.perm) {
            __syncwarp();
            for (int e = lane; e < k * k; e += kWarp) {
                const int i = e / k, j = e - i * k;
                double2 b = a.src[D.src_off + (int64_t)mt.ridx[i] * D.ld + mt.ridx[j]];
                // q cancels the diagonal entry of a single index (x_i^2 = r_i = 1): left
                // out, so that a large one takes no bits from the others
                if (i == j && mt.rmul[i] == 1 && !not_finite(b.x) && !not_finite(b.y))
                    b = make_double2(0.0, 0.0);
                sm.M[e] = b;
            }
            if (LOOP) {
                const int nf = D.N / 2 + 1;
                for (int i = lane; i < k; i += kWarp)
                    sm.gam[i] = a.gamma[D.gam_off + mt.ridx[i]];
                for (int j = lane; j < nf; j += kWarp)
                    sm.cj[j] = a.loopc[D.coef_off + j];
                for (int j = lane; j < haf_integers(D.N / 2); j += kWarp)
                    sm.ci[j] = __double_as_longlong(a.loopc[D.coef_off + nf + j]);
            }
            __syncwarp();
            if (!haf_stage_int<LOOP>(D, mt, sm, st, lane)) {
                st.mode = kStagedFp64;
                for (int j = lane; j < k; j += kWarp) {  // y0 = B r
                    double2 s = make_double2(0.0, 0.0);
                    for (int i = 0; i < k; ++i) {
                        const double r = (double)mt.rmul[i];
                        s.x = __fma_rn(r, sm.M[j * k + i].x, s.x);
                        s.y = __fma_rn(r, sm.M[j * k + i].y, s.y);
                    }
                    sm.y0[j] = s;
                }
                __syncwarp();
            }
            st.item = t.perm;
        }
        const int64_t chunk0 = (int64_t)t.part * kWarp;
        const bool active = chunk0 + lane < D.nchunks;
        const int64_t c = active ? (chunk0 + lane) : 0;
        if (st.mode == kStagedFp64)
            res = haf_walk_fp64<LOOP>(D, mt, sm, c, active, lane);
        else if (LOOP || st.mode == kStagedInt)
            res = haf_walk_int<LOOP>(D, mt, sm, st, c, active, lane, OneUnit());
        else
            res = haf_walk_parts(D, mt, sm, st, c, active, lane);
    }

    auto finish = [&](dd2 v) {
        double2 o;
        if (D.trivial) {
            o = make_double2(D.value, 0.0);
        } else {
            // the FP64 walk's terms hold the loop polynomial's leading factor
            const double f = LOOP && st.mode == kStagedInt ? D.value * sm.cj[0] : D.value;
            const int x = st.exp2 + 1 - D.N;
            double h, e;
            fast_two_sum(v.rh, v.rl, h, e);
            o.x = scalbn((h + e) * f, x);
            fast_two_sum(v.ih, v.il, h, e);
            if (!LOOP && st.mode == kStagedParts) {
                const SScale ps = sscale_of((int32_t)sm.ci[0]);
                o = turn(o.x, scalbn((h + e) * f, x - ps.f), ps.turned ? D.n : 0);
            } else {
                o.y = scalbn((h + e) * f, x);
            }
        }
        a.out[t.perm] = o;
    };
    if (gather_partials(a.partials + 4 * (int64_t)D.slot0, a.counters + 1 + t.perm,
                        a.groups + D.gslot0, t.part, D.ntasks, res.rh, res.rl, res.ih, res.il,
                        lane) &&
        lane == 0)
        finish(res);
}

// Persistent: every warp takes tasks from a global queue (counters[0]).
template <bool LOOP>
__global__ void __launch_bounds__(256, 2) hafnian_kernel(HafArgs a, int kmax)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const HafSmem sm(smem_raw + warp * haf_warp_smem_bytes(kmax), kmax);
    HafStaged st;
    for (;;) {
        int q = 0;
        if (lane == 0)
            q = atomicAdd(a.counters, 1);
        q = __shfl_sync(0xffffffffu, q, 0);
        if (q >= a.ntasks)
            break;
        haf_task<LOOP>(a, a.tasks[q], sm, st, lane);
    }
}

// Positive roots of the Hermite polynomial He_N (He_{k+1} = x He_k - k He_{k-1}),
// ascending: bisection on the number of eigenvalues of its Jacobi matrix
// (zero diagonal, off-diagonal sqrt(k)) below t, counted by the signs of the
// LDL^T pivots of J - t, then Newton steps on He_N.
static std::vector<double> hermite_positive_roots(int N)
{
    auto count_below = [N](double t) {
        int c = 0;
        double d = -t;
        c += d < 0.0;
        for (int k = 1; k < N; ++k) {
            if (d == 0.0)
                d = 1e-300;
            d = -t - (double)k / d;
            c += d < 0.0;
        }
        return c;
    };
    const int J = N / 2;
    const double top = 2.0 * std::sqrt((double)N) + 2.0;  // every root lies below
    std::vector<double> x;
    for (int i = N - J + 1; i <= N; ++i) {  // i-th smallest root
        double lo = 0.0, hi = top;
        for (int it = 0; it < 2000; ++it) {
            const double mid = 0.5 * (lo + hi);
            if (mid <= lo || mid >= hi)
                break;
            if (count_below(mid) >= i)
                hi = mid;
            else
                lo = mid;
        }
        double r = 0.5 * (lo + hi);
        for (int it = 0; it < 2; ++it) {
            double p0 = 1.0, p1 = r;  // He_{k-1}, He_k
            for (int k = 1; k < N; ++k) {
                const double p2 = r * p1 - (double)k * p0;
                p0 = p1;
                p1 = p2;
            }
            if (p0 != 0.0)
                r -= p1 / ((double)N * p0);
        }
        x.push_back(r);
    }
    return x;
}

// Factors of the loop polynomial of size N for loop_poly: [c_J, a_0, b_0,
// ..., (z_last)], J + 1 numbers.
static std::vector<double> loop_factors(int N)
{
    const int J = N / 2;
    std::vector<double> cf;
    double cJ = 1.0;
    for (int i = 2; i <= J; ++i)
        cJ /= (double)i;  // 1 / (J! (N - 2J)!), N - 2J <= 1
    cf.push_back(cJ);
    const std::vector<double> x = hermite_positive_roots(N);
    std::vector<double> z;
    for (double v : x)
        z.push_back(-1.0 / (2.0 * v * v));
    int m = 0;
    for (; m + 1 < J; m += 2) {
        cf.push_back(-(z[m] + z[m + 1]));
        cf.push_back(z[m] * z[m + 1]);
    }
    if (m < J)
        cf.push_back(z[m]);
    return cf;
}

// The factors after the first as integers for haf_loop_poly: the exponent e
// and v 2^(62 - e) in [2^61, 2^62) of a and b of each pair, and of -z of an odd
// root.  The roots' sizes descend, so the first pair's exponents are the
// largest.
static std::vector<int64_t> loop_integers(const std::vector<double>& cf)
{
    const int J = (int)cf.size() - 1, P = J / 2;
    std::vector<int64_t> ci;
    auto add = [&](double v) {
        int e = 0;
        const double m = std::frexp(v, &e);
        ci.push_back(e);
        ci.push_back((int64_t)std::ldexp(m, 62));  // m < 1 has 53 bits: exact
    };
    for (int j = 1; j <= 2 * P; ++j)
        add(cf[j]);
    if (J % 2)
        add(-cf[1 + 2 * P]);
    return ci;
}

static double factorial_h(int n)
{
    double r = 1.0;
    for (int i = 2; i <= n; ++i)
        r *= (double)i;
    return r;
}

}  // namespace pqi

// A planned batch of (loop) hafnians: host schedule uploaded once, device
// workspace owned by the plan.
struct pq_haf_plan {
    int loop = 0;
    int64_t batch = 0, ntasks = 0, ngroups = 0;
    int kmax = 1, wpb = 1, blocks = 1, per_warp = 0;
    unsigned char* arena = nullptr;  // one allocation: the arrays below
    std::vector<unsigned char> image;  // its host copy, until the upload has been waited for
    pqi::HafDesc* desc_d = nullptr;
    int32_t* meta_d = nullptr;
    pqi::Task* tasks_d = nullptr;
    double* part_d = nullptr;
    int32_t* cnt_d = nullptr;
    double* loopc_d = nullptr;
};

namespace pqi {

static void haf_plan_free(pq_haf_plan* P)
{
    if (!P)
        return;
    dev_free(P->arena);
    delete P;
    host_object_freed();
}

// Plan: digits, chunks, tasks (longest first), loop-polynomial factors; uploads
// them on the stream (the caller waits for it before it drops P->image) and
// raises the kernel's shared-memory limit.
static int haf_plan_build(const int64_t* mat_off, const int32_t* k, const int32_t* rep,
                          const int64_t* rep_off, int64_t batch, bool loop, cudaStream_t st,
                          pq_haf_plan** out)
{
    *out = nullptr;
    if (batch < 0 || (batch > 0 && (!mat_off || !k || !rep || !rep_off)))
        return report(PQ_ERR_ARG, "null argument or negative batch");
    if (batch > (int64_t(1) << 30))
        return report(PQ_ERR_UNSUPPORTED, "batch above 2^30");
    int dev = 0, sms = 1;
    if (batch > 0 && (cudaGetDevice(&dev) != cudaSuccess ||
                      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) !=
                          cudaSuccess))
        return report(PQ_ERR_CUDA, "no CUDA device");
    struct Dg {
        int rad, row, top;
    };
    struct Item {
        std::vector<int32_t> ridx, rm;
        std::vector<Dg> dg;
    };
    std::vector<HafDesc> desc(batch);
    std::vector<Item> items(batch);
    double t_total = 0.0;
    // Pass 1: kept indices, digits and term counts.
    for (int64_t b = 0; b < batch; ++b) {
        HafDesc& D = desc[b];
        Item& it = items[b];
        std::memset(&D, 0, sizeof(D));
        if (k[b] < 0 || k[b] > PQ_MAX_DIM || mat_off[b] < 0 || rep_off[b] < 0)
            return report(PQ_ERR_ARG, "bad size or offset");
        const int32_t* r = rep + rep_off[b];
        int N = 0;
        for (int i = 0; i < k[b]; ++i) {
            if (r[i] < 0)
                return report(PQ_ERR_ARG, "negative repetition");
            if (r[i] > PQ_MAX_N)
                return report(PQ_ERR_UNSUPPORTED, "expanded size above PQ_MAX_N");
            if (r[i] > 0) {
                it.ridx.push_back(i);
                it.rm.push_back(r[i]);
                N += r[i];
            }
        }
        if (N > PQ_MAX_N)
            return report(PQ_ERR_UNSUPPORTED, "expanded size above PQ_MAX_N");
        D.src_off = mat_off[b];
        D.gam_off = rep_off[b];
        D.ld = k[b];
        D.N = N;
        D.n = N / 2;
        if (N == 0 || (!loop && (N & 1))) {
            D.trivial = 1;
            D.value = (N == 0) ? 1.0 : 0.0;
            continue;
        }
        const int kk = (int)it.ridx.size();
        D.k = kk;
        D.value = loop ? 1.0 : 1.0 / factorial_h(N / 2);
        // Digits: one copy of the least repeated index fixed (radix r_f), the
        // others radix r_i + 1; ascending radix so that small ones walk inside
        // a chunk.
        const int f = (int)(std::min_element(it.rm.begin(), it.rm.end()) - it.rm.begin());
        int64_t T = 1;
        for (int i = 0; i < kk; ++i) {
            const int rad = (i == f) ? it.rm[i] : it.rm[i] + 1;
            if (rad < 2)
                continue;
            it.dg.push_back({rad, i, (i == f) ? it.rm[i] - 1 : it.rm[i]});
            if (T > (int64_t(1) << 62) / rad)
                return report(PQ_ERR_UNSUPPORTED, "term count above 2^62");
            T *= rad;
        }
        std::stable_sort(it.dg.begin(), it.dg.end(),
                         [](const Dg& x, const Dg& y) { return x.rad < y.rad; });
        D.T = T;
        D.ndig = (int)it.dg.size();
        t_total += (double)T;
    }
    // Pass 2: chunks and tasks.  Every item gets a share of about 64 warp
    // tasks per SM in proportion to its terms, so that one large hafnian still
    // fills the GPU.
    const double want_tasks = 64.0 * sms;
    std::vector<int32_t> meta;
    std::vector<Task> tasks;
    std::vector<double> cost;
    std::vector<double> loopc;
    std::vector<int32_t> coef_at(PQ_MAX_N + 1, -1);
    int kmax = 1;
    int32_t slot = 0;
    int64_t ngroups = 0;
    for (int64_t b = 0; b < batch; ++b) {
        HafDesc& D = desc[b];
        Item& it = items[b];
        D.slot0 = slot;
        D.gslot0 = (int32_t)ngroups;
        if (D.trivial) {
            D.ntasks = 1;
            tasks.push_back(Task{(int32_t)b, 0});
            cost.push_back(0.0);
            slot += 1;
            continue;
        }
        const int kk = D.k, N = D.N;
        const int64_t T = D.T;
        kmax = std::max(kmax, kk);
        if (loop) {
            if (coef_at[N] < 0) {
                coef_at[N] = (int32_t)loopc.size();
                const std::vector<double> cf = loop_factors(N);
                loopc.insert(loopc.end(), cf.begin(), cf.end());
                for (int64_t v : loop_integers(cf)) {
                    double bits;
                    std::memcpy(&bits, &v, sizeof(bits));
                    loopc.push_back(bits);
                }
            }
            D.coef_off = coef_at[N];
        }
        // Chunk length L = product of the J low radices, at most 4096 terms,
        // at most T / (32 x the item's task share), and J minimising the work per
        // term, 2J + 8 for the walk plus 2k(ndig - J) + 4k + 64 per chunk for the
        // start value: the FP64 walk's counts, which leave out a task's staging
        // and lane sums.  With J - 1, J and J + 1, in ms: hafnian (2, ..., 2), k =
        // 18, 4.76, 4.65, 4.97; k = 14 0.60, 0.25, 0.14; (3, ..., 3), k = 10 0.234,
        // 0.235, 0.101; loop hafnian (2, ..., 2), k = 14 0.71, 0.35, 0.23.  So the
        // share of 64 tasks per SM is the larger part of the smaller items' time.
        const double share = std::max(1.0, std::ceil(want_tasks * (double)T / t_total));
        const int64_t cap = std::max<int64_t>(
            1, std::min<int64_t>(4096, (int64_t)((double)T / (kWarp * share))));
        int J = 0;
        int64_t L = 1;
        {
            double best = 1e300;
            int64_t Lc = 1;
            for (int j = 0;; ++j) {
                const double c = 2.0 * j + 8.0 + (2.0 * kk * (D.ndig - j) + 4.0 * kk + 64.0) / Lc;
                if (c < best) {
                    best = c;
                    J = j;
                    L = Lc;
                }
                if (j >= D.ndig || j >= kMaxLowDigits || it.dg[j].rad > kMaxLowRadix ||
                    Lc * it.dg[j].rad > cap)
                    break;
                Lc *= it.dg[j].rad;
            }
        }
        D.J = J;
        D.L = L;
        D.nchunks = T / L;
        for (int d = 0; d < J; ++d)
            if (it.dg[d].rad > 2)
                D.weighted = 1;
        const int64_t nt = (D.nchunks + kWarp - 1) / kWarp;
        if (nt + slot > (int64_t(1) << 30))
            return report(PQ_ERR_UNSUPPORTED, "too many tasks");
        D.ntasks = (int32_t)nt;
        if (nt > 32)
            ngroups += (nt + 31) / 32;
        D.meta = (int32_t)meta.size();
        // rows of the low digits first, in digit order
        {
            std::vector<int32_t> at(kk, -1), idx(kk), rm(kk);
            int next = 0;
            for (int d = 0; d < J; ++d)
                at[it.dg[d].row] = next++;
            for (int i = 0; i < kk; ++i)
                if (at[i] < 0)
                    at[i] = next++;
            for (int i = 0; i < kk; ++i) {
                idx[at[i]] = it.ridx[i];
                rm[at[i]] = it.rm[i];
            }
            it.ridx = idx;
            it.rm = rm;
            for (Dg& d : it.dg)
                d.row = at[d.row];
        }
        meta.insert(meta.end(), it.ridx.begin(), it.ridx.end());
        meta.insert(meta.end(), it.rm.begin(), it.rm.end());
        for (const Dg& d : it.dg)
            meta.push_back(d.row);
        for (const Dg& d : it.dg)
            meta.push_back(d.rad);
        for (const Dg& d : it.dg)
            meta.push_back(d.top);
        // relative cost of a term, for the tasks' order
        const double per_term = loop ? (2.0 * J + 10.0 * (N / 2) + 12.0) : (2.0 * J + 24.0);
        for (int64_t q = 0; q < nt; ++q) {
            tasks.push_back(Task{(int32_t)b, (int32_t)q});
            cost.push_back((double)L * per_term);
        }
        slot += (int32_t)nt;
    }
    if (!host_object_alloc_ok())
        return report(PQ_ERR_NOMEM, "host allocation failed");
    pq_haf_plan* P = new (std::nothrow) pq_haf_plan();
    if (!P) {
        host_object_freed();
        return report(PQ_ERR_NOMEM, "host allocation failed");
    }
    P->loop = loop ? 1 : 0;
    P->batch = batch;
    if (batch == 0) {
        *out = P;
        return PQ_OK;
    }
    // longest task first
    std::vector<int64_t> order(tasks.size());
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(),
                     [&](int64_t x, int64_t y) { return cost[x] > cost[y]; });
    std::vector<Task> sorted(tasks.size());
    for (size_t q = 0; q < order.size(); ++q)
        sorted[q] = tasks[order[q]];
    P->ntasks = (int64_t)sorted.size();
    P->ngroups = ngroups;
    P->kmax = kmax;
    int rc = PQ_OK;
    // One allocation and one upload: six of the one and four of the other, with
    // the frees, were most of a one-shot call (300 small hafnians: 400 us, the
    // kernel 29 of them).  The counters come zeroed with the upload.  It is made
    // on the stream that the kernel runs on: a plain cudaMemcpy from pageable
    // memory may return before the data has arrived, and streams that do not wait
    // for the default one would read what the memory held before.
    std::vector<unsigned char>& image = P->image;
    auto place = [&](const void* src, size_t bytes) {
        const size_t at = (image.size() + 255) & ~size_t(255);
        image.resize(at + std::max<size_t>(bytes, 1));
        if (src && bytes)
            std::memcpy(image.data() + at, src, bytes);
        return at;
    };
    const size_t at_desc = place(desc.data(), sizeof(HafDesc) * batch);
    const size_t at_tasks = place(sorted.data(), sizeof(Task) * sorted.size());
    const size_t at_loopc = place(loopc.data(), sizeof(double) * loopc.size());
    const size_t at_meta = place(meta.data(), sizeof(int32_t) * meta.size());
    const size_t at_cnt = place(nullptr, sizeof(int32_t) * (size_t)(batch + 1 + ngroups));
    const size_t at_part = (image.size() + 255) & ~size_t(255);
    const size_t total = at_part + sizeof(double) * 4 * (size_t)std::max<int32_t>(slot, 1);
    if (dev_alloc((void**)&P->arena, total) != cudaSuccess)
        rc = report(PQ_ERR_NOMEM, "hafnian workspace allocation failed");
    if (rc == PQ_OK &&
        cudaMemcpyAsync(P->arena, image.data(), image.size(), cudaMemcpyHostToDevice, st) !=
            cudaSuccess)
        rc = report(PQ_ERR_CUDA, "hafnian upload failed");
    if (rc == PQ_OK) {
        P->desc_d = reinterpret_cast<HafDesc*>(P->arena + at_desc);
        P->tasks_d = reinterpret_cast<Task*>(P->arena + at_tasks);
        P->loopc_d = reinterpret_cast<double*>(P->arena + at_loopc);
        P->meta_d = reinterpret_cast<int32_t*>(P->arena + at_meta);
        P->cnt_d = reinterpret_cast<int32_t*>(P->arena + at_cnt);
        P->part_d = reinterpret_cast<double*>(P->arena + at_part);
    }
    if (rc == PQ_OK) {
        P->per_warp = haf_warp_smem_bytes(kmax);
        cudaFuncAttributes fa{};
        const cudaError_t ea = loop ? cudaFuncGetAttributes(&fa, hafnian_kernel<true>)
                                    : cudaFuncGetAttributes(&fa, hafnian_kernel<false>);
        // as many resident warps as fit: a product waits on its own chain
        int wpb = 1, bps = 1;
        launch_geometry_max(ea == cudaSuccess ? fa.numRegs : 128, P->per_warp, 8, wpb, bps);
        P->wpb = wpb;
        const int64_t want_blocks = (P->ntasks + wpb - 1) / wpb;
        P->blocks = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)sms * bps, want_blocks));
        // raise (never lower) the dynamic shared-memory limit of the kernel
        cudaFuncAttributes at{};
        cudaError_t e = loop ? cudaFuncGetAttributes(&at, hafnian_kernel<true>)
                             : cudaFuncGetAttributes(&at, hafnian_kernel<false>);
        const int need = wpb * P->per_warp;
        if (e == cudaSuccess && at.maxDynamicSharedSizeBytes < need)
            e = loop ? cudaFuncSetAttribute(hafnian_kernel<true>,
                                            cudaFuncAttributeMaxDynamicSharedMemorySize, need)
                     : cudaFuncSetAttribute(hafnian_kernel<false>,
                                            cudaFuncAttributeMaxDynamicSharedMemorySize, need);
        if (e != cudaSuccess)
            rc = report(PQ_ERR_CUDA, "hafnian kernel attribute setup failed");
    }
    if (rc != PQ_OK) {
        cudaStreamSynchronize(st);  // the upload may be in flight
        haf_plan_free(P);
        return rc;
    }
    *out = P;
    return PQ_OK;
}

// Execution: clear the counters (unless they are as uploaded) and launch;
// allocates nothing, no sync.
static int haf_plan_launch(pq_haf_plan* P, const pq_c128* mats, const pq_c128* gamma,
                           pq_c128* out, cudaStream_t st, bool reset)
{
    if (P->batch == 0)
        return PQ_OK;
    if (reset &&
        cudaMemsetAsync(P->cnt_d, 0, sizeof(int32_t) * (P->batch + 1 + P->ngroups), st) !=
            cudaSuccess)
        return report(PQ_ERR_CUDA, "hafnian counter reset failed");
    HafArgs a;
    a.desc = P->desc_d;
    a.meta = P->meta_d;
    a.tasks = P->tasks_d;
    a.ntasks = P->ntasks;
    a.src = reinterpret_cast<const double2*>(mats);
    a.gamma = reinterpret_cast<const double2*>(gamma);
    a.loopc = P->loopc_d;
    a.out = reinterpret_cast<double2*>(out);
    a.partials = P->part_d;
    a.counters = P->cnt_d;
    a.groups = P->cnt_d + P->batch + 1;
    const int smem = P->wpb * P->per_warp;
    if (P->loop)
        hafnian_kernel<true><<<P->blocks, 32 * P->wpb, smem, st>>>(a, P->kmax);
    else
        hafnian_kernel<false><<<P->blocks, 32 * P->wpb, smem, st>>>(a, P->kmax);
    if (cudaGetLastError() != cudaSuccess)
        return report(PQ_ERR_CUDA, "hafnian kernel launch failed");
    return PQ_OK;
}

// The one-shot calls: plan, run, synchronise, free.
static int run_hafnians(const pq_c128* mats, const int64_t* mat_off, const int32_t* k,
                        const int32_t* rep, const int64_t* rep_off, const pq_c128* gamma,
                        int64_t batch, pq_c128* out, void* stream)
{
    if (batch > 0 && (!mats || !out))
        return report(PQ_ERR_ARG, "null argument");
    cudaStream_t st = (cudaStream_t)stream;
    pq_haf_plan* P = nullptr;
    int rc = haf_plan_build(mat_off, k, rep, rep_off, batch, gamma != nullptr, st, &P);
    if (rc != PQ_OK)
        return rc;
    rc = haf_plan_launch(P, mats, gamma, out, st, false);
    if (cudaStreamSynchronize(st) != cudaSuccess && rc == PQ_OK)
        rc = report(PQ_ERR_CUDA, "hafnian kernel failed");
    haf_plan_free(P);
    return rc;
}

}  // namespace pqi

extern "C" int pq_hafnian_repeated(const pq_c128* mats, const int64_t* mat_off, const int32_t* k,
                                   const int32_t* rep, const int64_t* rep_off, int64_t batch,
                                   pq_c128* out, void* stream)
{
    return pqi::run_hafnians(mats, mat_off, k, rep, rep_off, nullptr, batch, out, stream);
}

extern "C" int pq_loop_hafnian_repeated(const pq_c128* mats, const pq_c128* gamma,
                                        const int64_t* mat_off, const int32_t* k,
                                        const int32_t* rep, const int64_t* rep_off, int64_t batch,
                                        pq_c128* out, void* stream)
{
    if (batch > 0 && !gamma)
        return pqi::report(PQ_ERR_ARG, "null gamma");
    return pqi::run_hafnians(mats, mat_off, k, rep, rep_off, gamma, batch, out, stream);
}

extern "C" int pq_loop_poly_factors(int32_t N, double* out)
{
    if (N < 0 || N > PQ_MAX_N || !out)
        return pqi::report(PQ_ERR_ARG, "N outside [0, PQ_MAX_N] or null output");
    const std::vector<double> cf = pqi::loop_factors(N);
    for (size_t i = 0; i < cf.size(); ++i)
        out[i] = cf[i];
    return PQ_OK;
}

extern "C" int pq_hafnian_plan_create(const int64_t* mat_off, const int32_t* k, const int32_t* rep,
                                      const int64_t* rep_off, int64_t batch, int32_t loop,
                                      pq_haf_plan** out)
{
    if (!out)
        return pqi::report(PQ_ERR_ARG, "null output");
    int rc = pqi::haf_plan_build(mat_off, k, rep, rep_off, batch, loop != 0, nullptr, out);
    // a run may come on any stream: the upload is complete when the plan exists
    if (rc == PQ_OK && (*out)->arena) {
        if (cudaStreamSynchronize(nullptr) != cudaSuccess) {
            pqi::haf_plan_free(*out);
            *out = nullptr;
            return pqi::report(PQ_ERR_CUDA, "hafnian upload failed");
        }
        std::vector<unsigned char>().swap((*out)->image);
    }
    return rc;
}

extern "C" int pq_hafnian_plan_run(pq_haf_plan* plan, const pq_c128* mats, const pq_c128* gamma,
                                   pq_c128* out, void* stream)
{
    if (!plan)
        return pqi::report(PQ_ERR_ARG, "null plan");
    if (plan->batch > 0 && (!mats || !out || (plan->loop && !gamma)))
        return pqi::report(PQ_ERR_ARG, "null argument");
    return pqi::haf_plan_launch(plan, mats, plan->loop ? gamma : nullptr, out,
                                (cudaStream_t)stream, true);
}

extern "C" int pq_hafnian_plan_destroy(pq_haf_plan* plan)
{
    if (plan) {
        cudaDeviceSynchronize();
        pqi::haf_plan_free(plan);
    }
    return PQ_OK;
}
