// glynn_fwd.cuh -- the forward walk: permanents with repeated rows and columns by
// the BB/FG formula over a mixed-radix Gray code (paper Sec. 4.2, "Boson
// Sampling"; Eq. (per_def) for the permanent, Eq. (BS_prob) for the
// probabilities written by the final reduction).
//
// One thread walks one chunk of the Gray code.  The FP64 pipe (2 lane
// operations per clock and SM) would bound the walk, so its column sums and
// products are 64-bit block integers (pq_blockint.cuh) on the integer pipes:
//   * a lane's column sums S_j = sum_i (r_i - 2 g_i) b_ij are scaled integers,
//     in shared memory, lane-major (one 16-byte pair per lane per column, so a
//     warp access is conflict-free), or in registers;
//   * a Gray step changes one row's sign count by +-1 for all lanes at once:
//     S_j += -+2 b_ij, one 64-bit add per component, 2 b read as a broadcast;
//     the shared-memory walk makes it in the loop that forms the next term;
//   * product columns are sorted by non-increasing multiplicity, so
//     prod_j S_j^{c_j} = prod_m P(n_m) with P(q) = S_0 ... S_{q-1}: l - 1
//     complex products for P(l) plus one per extra prefix, instead of n - 1;
//     without repeated columns they are taken in pairs, p (S_j S_{j+1}),
//     which halves the dependent chain;
//   * a term is converted to FP64 and added to a running FP64 sum with its
//     sign (-1)^step, the binomial weight of the low digits and its power of
//     two in one DFMA per component;
//   * every 32 terms the FP64 running sum is folded into a double-double
//     accumulator with TwoSum.
// A base matrix with a non-finite entry, or a column whose bound overflows, has
// no such scale: its tasks walk in FP64 (fp64_walk), so that infinities and
// NaNs propagate as FP64 arithmetic gives them.  Matrices whose columns all lie
// near the real or imaginary axis have a unit for each part (other_task), so that
// the small part keeps its bits: 16384 ragged permanents 2.03 ms (1.52 with parts
// of like size, 5.34 for the FP64 walk), one n = 24 permanent 0.91 (0.60, 2.64).
// A warp task is up to 32 chunks of one permanent (one per lane).  The lanes'
// sums are added exactly, in 128-bit integers (pq_fixsum.cuh), and the tasks
// of one permanent in task order by the warp that finishes last, so results
// do not depend on scheduling.
//
// Bound: the multiplier pipe (a wide multiply takes 4 cycles of a
// sub-partition, 12 to a complex product) and the adds and shifts beside it,
// 0.57 clocks per lane, column and term and SM, against 3.3 for the FP64 walk.
// Measured, FP64 walk -> now: 65536 ragged permanents (n = 4..20) 20.95 ->
// 5.78 ms, 4096 permanents of 12 columns 914 -> 194 us, one n = 30 permanent
// 165.7 -> 35.3 ms.
#pragma once
#include <cuda_runtime.h>

#include "../../include/pq.h"
#include "pq_blockint.cuh"
#include "pq_device.cuh"
#include "pq_fixsum.cuh"
#include "pq_kernels.h"

namespace pqi {

// Shared memory of one warp: base matrix (kmax x ld pairs), base column sums
// (ld pairs), the column sums of the 32 lanes (ld x 32 pairs; only the
// shared-memory walk), low-digit rows (16 ints), extra-factor counts and scale
// exponents (ld ints each).
__host__ __device__ inline int warp_smem_bytes(int kmax, int ld)
{
    int bytes = (kmax * ld + ld + 32 * ld) * 16 + (16 + 2 * ld) * 4;
    return (bytes + 15) & ~15;
}

__host__ __device__ inline int reg_warp_smem_bytes(int kmax, int ld)
{
    int bytes = (kmax * ld + ld) * 16 + (16 + 2 * ld) * 4;
    return (bytes + 15) & ~15;
}

struct WarpSmem {
    longlong2* M;     // kmax x ld: 2 b_ij scaled (b_ij itself, as doubles, for fp64_walk)
    longlong2* base;  // ld: column sums at all digits zero (biased; doubles for fp64_walk)
    longlong2* S;     // ld x 32, S[j * 32 + lane] (shared-memory walk)
    int32_t* lowrow;  // 16
    int32_t* ecnt;    // ld
    int32_t* cexp;    // ld: scale exponent of each column
    int ld;
    __device__ WarpSmem(unsigned char* raw, int kmax, int ld_, bool sums)
    {
        ld = ld_;
        M = reinterpret_cast<longlong2*>(raw);
        base = M + kmax * ld;
        S = base + ld;
        lowrow = reinterpret_cast<int32_t*>(S + (sums ? 32 * ld : 0));
        ecnt = lowrow + 16;
        cexp = ecnt + ld;
    }
    // of a walk with its column sums elsewhere
    __device__ WarpSmem(longlong2* M_, longlong2* base_, int32_t* lowrow_, int ld_)
        : M(M_), base(base_), S(nullptr), lowrow(lowrow_), ecnt(lowrow_ + 16),
          cexp(lowrow_ + 16 + ld_), ld(ld_)
    {
    }
};

// What a warp keeps about the permanent it has staged.
struct Staged {
    int perm = -1;
    int mode = kStagedInt;
    int exp2 = 0;       // the terms' sum times 2^exp2 is the sum of prod_j S_j^{c_j}
    uint32_t emask = 0; // bit j: column j < 32 has extra prefixes
};

// Copy the oriented base matrix of permanent D into shared memory as scaled
// integers and form base_j = sum_i r_i b_ij (all Gray digits at zero).
static __device__ void stage_perm(const ExecArgs& a, const PermDesc& D, const MetaView& mv, WarpSmem& sm,
                           Staged& st, int lane)
{
    const int k = D.k, l = D.l;
    double2* Md = reinterpret_cast<double2*>(sm.M);
    bool bad = false;
    for (int e = lane; e < k * l; e += kWarp) {
        const int i = e / l, j = e - i * l;
        const int64_t off = D.src_off + (int64_t)mv.ridx[i] * D.si + (int64_t)mv.cidx[j] * D.sj;
        const double2 b = a.src[off];
        bad = bad || not_finite(b.x) || not_finite(b.y);
        Md[i * sm.ld + j] = b;
    }
    for (int d = lane; d < D.J; d += kWarp)
        sm.lowrow[d] = mv.drow[d];
    for (int j = lane; j < l; j += kWarp)
        sm.ecnt[j] = mv.ecnt[j];
    __syncwarp();
    int esum = 0;
    st.perm = -1;
    st.mode = bint_stage(Md, sm.ld, k, l, mv.rmul, mv.cmul, sm.cexp, bad, lane, esum, false);
    if (st.mode == kStagedFp64) {
        double2* base = reinterpret_cast<double2*>(sm.base);
        for (int j = lane; j < l; j += kWarp) {
            double2 s = make_double2(0.0, 0.0);
            for (int i = 0; i < k; ++i) {
                const double r = (double)mv.rmul[i];
                const double2 b = Md[i * sm.ld + j];
                s.x = __fma_rn(r, b.x, s.x);
                s.y = __fma_rn(r, b.y, s.y);
            }
            base[j] = s;
        }
        st.exp2 = 0;
        __syncwarp();
        return;
    }
    uint32_t em = 0;
    for (int j = lane; j < l; j += kWarp) {
        sm.base[j] = bint_base(sm.M + j, sm.ld, k, mv.rmul);
        if (j < 32 && sm.ecnt[j] > 0)
            em |= 1u << j;
    }
    st.emask = __reduce_or_sync(0xffffffffu, em);
    // n - 1 products, each shifted down by 64; the terms carry 2^-kSumBits
    st.exp2 = kSumBits + 64 * (D.n - 1) - esum;
    __syncwarp();
}

// The column sums of one term, after its Gray step.  Shared memory: column j is
// read, moved by the changed row's 2 b_j (STEP 1: the digit went up, 2: down,
// 0: the chunk's first term) and written back as the term needs it.
template <int STEP, int STRIDE>
struct SharedCols {
    longlong2* S;        // this lane's
    const longlong2* b;  // the changed row
    __device__ __forceinline__ longlong2 operator()(int j) const
    {
        longlong2 s = S[j * STRIDE];
        if (STEP != 0) {
            const longlong2 d = b[j];
            s.x = STEP == 1 ? s.x - d.x : s.x + d.x;
            s.y = STEP == 1 ? s.y - d.y : s.y + d.y;
            S[j * STRIDE] = s;
        }
        return s;
    }
};

template <int NL>
struct RegCols {
    const longlong2 (&S)[NL];
    __device__ __forceinline__ longlong2 operator()(int j) const { return S[j]; }
};

// prod_j S_j without repeated columns, 2^E times the integers returned: S_0 S_1,
// then the columns in pairs, p (S_j S_{j+1}).  NL > 0: registers, unrolled,
// l <= NL; NL = 0: shared memory.
template <int NL, class Mul, class Cols>
__device__ __forceinline__ BInt unit_product(const Mul& mul, const Cols& col, int l, int& E)
{
    const longlong2 s0 = col(0);
    if (l == 1)
        return bint_plain(s0);
    BInt p = mul(sum_limbs(s0), sum_limbs(col(1)));
    if constexpr (NL == 0) {
        int j = 2;
#pragma unroll 1
        for (; j + 1 < l; j += 2) {
            const BLimbs x = sum_limbs(col(j)), y = sum_limbs(col(j + 1));
            const BInt q = mul(x, y);
            bnorm(p, E);
            p = mul(limbs(p), limbs(q));
        }
        if (j < l) {
            bnorm(p, E);
            p = mul(limbs(p), sum_limbs(col(j)));
        }
    } else {
#pragma unroll
        for (int j = 2; j < NL; j += 2) {  // NL is even
            if (j + 1 < l) {
                const BInt q = mul(sum_limbs(col(j)), sum_limbs(col(j + 1)));
                bnorm(p, E);
                p = mul(limbs(p), limbs(q));
            } else if (j < l) {
                bnorm(p, E);
                p = mul(limbs(p), sum_limbs(col(j)));
            }
        }
    }
    return p;
}

// The extra factors of a prefix (n_extra = ecnt[j] copies at column j, > 0): at
// the first column with extras (jf) ex starts as that prefix, and every further
// extra multiplies it in.
template <class Mul>
__device__ __forceinline__ void extra_factors(const Mul& mul, BInt& pre, int& E, BInt& ex, int& Ex,
                                              int j, int jf, int n_extra)
{
    bnorm(pre, E);
    const BLimbs lp = limbs(pre);
    int e = 0;
    if (j == jf) {
        ex = pre;
        Ex = E;
        e = 1;
    }
#pragma unroll 1
    for (; e < n_extra; ++e) {
        ex = mul(limbs(ex), lp);
        Ex += E;
        bnorm(ex, Ex);
    }
}

// Columns j and j + 1 (j + 1 < l, or j alone) of a term with repeated columns:
// as one pair, p (S_j S_{j+1}), where no extra factor falls between them.
// has(j): column j has extras.
template <class Mul, class Cols, class Has>
__device__ __forceinline__ void prefix_pair(const Mul& mul, const Cols& col, const Has& has,
                                            BInt& pre, int& E, BInt& ex, int& Ex, int j, int l,
                                            int jf, const int32_t* ecnt)
{
    bnorm(pre, E);
    if (j + 1 < l && !has(j)) {
        const BInt q = mul(sum_limbs(col(j)), sum_limbs(col(j + 1)));
        pre = mul(limbs(pre), limbs(q));
    } else {
        pre = mul(limbs(pre), sum_limbs(col(j)));
        if (has(j))
            extra_factors(mul, pre, E, ex, Ex, j, jf, ecnt[j]);
        if (j + 1 >= l)
            return;
        pre = mul(limbs(pre), sum_limbs(col(j + 1)));
    }
    if (has(j + 1))
        extra_factors(mul, pre, E, ex, Ex, j + 1, jf, ecnt[j + 1]);
}

// prod_j S_j^{c_j}; UNIT: no repeated column, else from the prefixes.
template <int NL, bool UNIT, class Mul, class Cols>
__device__ __forceinline__ BInt term_product(const Mul& mul, const Cols& col, int l, int jf,
                                             uint32_t emask, const int32_t* ecnt, int& E)
{
    E = 0;
    if constexpr (UNIT)
        return unit_product<NL>(mul, col, l, E);
    BInt pre = bint_plain(col(0)), ex = pre;
    int Ex = 0;
    if constexpr (NL == 0) {
        auto has = [&](int j) { return ecnt[j] > 0; };
        if (has(0))
            extra_factors(mul, pre, E, ex, Ex, 0, jf, ecnt[0]);
#pragma unroll 1
        for (int j = 1; j < l; j += 2)
            prefix_pair(mul, col, has, pre, E, ex, Ex, j, l, jf, ecnt);
    } else {
        auto has = [&](int j) { return ((emask >> j) & 1u) != 0; };
        if (has(0))
            extra_factors(mul, pre, E, ex, Ex, 0, jf, ecnt[0]);
#pragma unroll
        for (int j = 1; j < NL; j += 2)
            if (j < l)
                prefix_pair(mul, col, has, pre, E, ex, Ex, j, j + 1 < NL ? l : j + 1, jf, ecnt);
    }
    E += Ex;
    return mul(limbs(pre), limbs(ex));
}

// acc +-= w 2^(-kSumBits - E) p
__device__ __forceinline__ void add_term(const BInt& p, int E, double w, bool neg, double2& acc)
{
    const double f = bint_factor(w, E, neg);
    const long long re = (long long)(((uint64_t)(uint32_t)p.rh << 32) | p.rl);
    const long long im = (long long)(((uint64_t)(uint32_t)p.ih << 32) | p.il);
    acc.x = __fma_rn(__ll2double_rn(re), f, acc.x);
    acc.y = __fma_rn(__ll2double_rn(im), f, acc.y);
}

// A run of equally weighted terms ends: run += wlow * acc, and the walk's new
// weight becomes wlow.
__device__ __forceinline__ void reweight(const LowWalk& wk, int J, double& wlow, double2& acc,
                                         double2& run)
{
    run.x = __fma_rn(wlow, acc.x, run.x);
    run.y = __fma_rn(wlow, acc.y, run.y);
    acc = make_double2(0.0, 0.0);
    wlow = (double)low_weight(wk, J);
}

// Write per = 2^{-(n-1)} * sum, and |per|^2 * norm, the sum being v times 2^exp2, with
// PARTS its imaginary part times 2^-f more and the whole times i^turns; a sharded plan
// writes its unscaled double-double sum instead.
template <bool PARTS>
__device__ __forceinline__ void finalize(const ExecArgs& a, const PermDesc& D, dd2 v, int exp2,
                                         int f, int turns)
{
    const int exp2_im = PARTS ? exp2 - f : exp2;
    auto turned = [&](double re, double im) {
        return PARTS ? turn(re, im, turns) : make_double2(re, im);
    };
    if (a.out_partial) {
        double* o = a.out_partial + 4 * (int64_t)D.out;
        if (D.trivial) {
            o[0] = 1.0;
            o[1] = o[2] = o[3] = 0.0;
        } else {
            const double2 h = turned(scalbn(v.rh, exp2), scalbn(v.ih, exp2_im));
            const double2 e = turned(scalbn(v.rl, exp2), scalbn(v.il, exp2_im));
            o[0] = h.x;
            o[1] = e.x;
            o[2] = h.y;
            o[3] = e.y;
        }
        return;
    }
    double2 per = make_double2(1.0, 0.0);
    if (!D.trivial)
        per = turned(scale_exp2(__dadd_rn(v.rh, v.rl), exp2 + 1 - D.n),
                     scale_exp2(__dadd_rn(v.ih, v.il), exp2_im + 1 - D.n));
    if (a.out_amp)
        a.out_amp[D.out] = per;
    if (a.out_prob)
        a.out_prob[D.out] = (per.x * per.x + per.y * per.y) * D.norm;
}

// The task's sum: every lane's chunk sum (rh + rl, ih + il) times its
// high-digit weight (-1)^neg whigh_u (zero for a lane without a chunk), added
// over the warp exactly in integer arithmetic (pq_fixsum.cuh); every lane gets
// it.  When no lane's weight is above 1 the weight is a sign, applied to the
// bit patterns, and the double-double product (14 FP64 operations) is skipped.
__device__ __forceinline__ dd2 task_sum(double rh, double rl, double ih, double il,
                                        uint64_t whigh_u, bool neg, bool active)
{
    if (__any_sync(0xffffffffu, active && whigh_u != 1)) {
        double w = active ? (double)whigh_u : 0.0;
        if (neg)
            w = -w;
        fast_two_sum(rh, rl, rh, rl);
        fast_two_sum(ih, il, ih, il);
        dd_mul_d(rh, rl, w);
        dd_mul_d(ih, il, w);
    } else if (!active) {
        rh = rl = ih = il = 0.0;
    } else if (neg) {
        const uint64_t s = 1ull << 63;
        rh = fix_double(fix_bits(rh) ^ s);
        rl = fix_double(fix_bits(rl) ^ s);
        ih = fix_double(fix_bits(ih) ^ s);
        il = fix_double(fix_bits(il) ^ s);
    }
    dd2 res;
    warp_fix_sum(rh, rl, res.rh, res.rl);
    warp_fix_sum(ih, il, res.ih, res.il);
    return res;
}

// The task's sum res (the same on every lane) goes to the permanent's output
// if the permanent has one task; otherwise to its slot, and the warps that
// finish last add the slots (gather_partials).
template <bool PARTS>
static __device__ void combine_task(const ExecArgs& a, const Task& t, const PermDesc& D, dd2 res,
                                    int exp2, int f, int turns, int lane)
{
    if (gather_partials(a.partials + 4 * (int64_t)D.slot0, a.counters + 1 + t.perm,
                        a.groups + D.gslot0, t.part - D.part0, D.ntasks, res.rh, res.rl, res.ih,
                        res.il, lane) &&
        lane == 0)
        finalize<PARTS>(a, D, res, exp2, f, turns);
}

// ---------------------------------------------------------------- the walk
__device__ __forceinline__ void start_walk(LowWalk& wk, const MetaView& mv, int J)
{
    wk.v = 0;
    wk.g = 0;
    wk.dir = 0;
    wk.radm1 = 0;
    wk.topp = 0;
    for (int d = 0; d < J; ++d) {
        wk.radm1 |= uint64_t(mv.drad[d] - 1) << (4 * d);
        wk.topp |= uint64_t(mv.dtop[d]) << (4 * d);
    }
}

// The walk of this lane's chunk; returns the task's sum over the warp
// (task_sum).  NL = 0: column sums in shared memory; NL > 0: in registers.
// With and without repeated columns are walks of their own: one loop holding
// both bodies took half as many instructions again per column.
// S: this lane's column sums with the given stride (NL = 0).
template <int NL, bool UNIT, int STRIDE = 32, class Mul>
__device__ __forceinline__ dd2 int_walk(const Mul& mul, longlong2* S, const PermDesc& D,
                                        const MetaView& mv, const WarpSmem& sm, uint32_t emask,
                                        int64_t chunk, bool active, int lane)
{
    const int l = D.l, J = D.J, ndig = D.ndig, ld = NL > 0 ? NL : sm.ld;
    constexpr int kRegs = NL > 0 ? NL : 1;
    longlong2 R[kRegs];
    if constexpr (NL > 0) {
#pragma unroll
        for (int j = 0; j < NL; ++j)
            R[j] = j < l ? sm.base[j] : make_longlong2(0, 0);
    } else {
#pragma unroll 1
        for (int j = 0; j < l; ++j)
            S[j * STRIDE] = sm.base[j];
    }
    const bool narrow = D.nchunks <= 0x7fffffff;
    uint64_t whigh_u = 1;
    int gpar = 0;
#pragma unroll 1
    for (int d = J; d < ndig; ++d) {
        const int g = next_digit(chunk, mv.drad[d], narrow);
        if (g == 0)  // no sign flip in this row: nothing to do (for the whole warp, often)
            continue;
        const longlong2* Mr = sm.M + mv.drow[d] * ld;
        if constexpr (NL > 0) {
#pragma unroll
            for (int j = 0; j < NL; ++j) {
                if (j < l) {
                    const longlong2 b = Mr[j];
                    R[j].x -= g * b.x;
                    R[j].y -= g * b.y;
                }
            }
        } else {
#pragma unroll 1
            for (int j = 0; j < l; ++j) {
                const longlong2 b = Mr[j];
                longlong2 s = S[j * STRIDE];
                s.x -= g * b.x;
                s.y -= g * b.y;
                S[j * STRIDE] = s;
            }
        }
        whigh_u *= high_binom(mv.dtop[d], g);
        gpar += g;
    }

    const LowDigits lo = low_digits(mv, J);
    const bool weighted = D.weighted != 0;
    const int jf = D.jf;
    // The Gray steps are the same for all lanes.  Every 32 steps each lane
    // works out one of them (the changed row's offset in M, bit 0: down, and
    // the weight after it) and the walk takes them by shuffle: about a quarter
    // of the instructions that carrying the digits from step to step takes on
    // every lane.
    uint32_t steps = 0;
    double step_w = 1.0, w = 1.0;
    // every 32 terms acc is folded into the double-double rh/rl, ih/il
    double2 acc = make_double2(0.0, 0.0);
    double rh = 0.0, rl = 0.0, ih = 0.0, il = 0.0;
    const uint32_t L = (uint32_t)D.L;  // at most 2^30 (the planner's cap)
    int E;
    BInt p;
    if constexpr (NL > 0)
        p = term_product<NL, UNIT>(mul, RegCols<kRegs>{R}, l, jf, emask, sm.ecnt, E);
    else
        p = term_product<0, UNIT>(mul, SharedCols<0, STRIDE>{S, sm.M}, l, jf, emask, sm.ecnt, E);
    uint32_t s = 0;
#pragma unroll 1
    for (;;) {
        add_term(p, E, w, (s & 1u) != 0, acc);
        ++s;
        if (s == L || (s & 31u) == 0) {
            if (L <= 32u) {  // the only fold of a short chunk
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
        const int q = (int)((s - 1u) & 31u);
        if (q == 0) {
            bool up;
            uint64_t wu;
            const int d = gray_step_at(lo, s + (uint32_t)lane, weighted, up, wu);
            steps = ((uint32_t)(sm.lowrow[d] * ld) << 1) | (up ? 0u : 1u);
            if (weighted)
                step_w = (double)wu;
        }
        const uint32_t step = __shfl_sync(0xffffffffu, steps, q);
        if (weighted)
            w = __shfl_sync(0xffffffffu, step_w, q);
        const longlong2* Mr = sm.M + (step >> 1);
        if constexpr (NL > 0) {
            if (step & 1u) {
#pragma unroll
                for (int j = 0; j < NL; ++j) {
                    const longlong2 b = Mr[j];
                    R[j].x += b.x;
                    R[j].y += b.y;
                }
            } else {
#pragma unroll
                for (int j = 0; j < NL; ++j) {
                    const longlong2 b = Mr[j];
                    R[j].x -= b.x;
                    R[j].y -= b.y;
                }
            }
            p = term_product<NL, UNIT>(mul, RegCols<kRegs>{R}, l, jf, emask, sm.ecnt, E);
        } else if (step & 1u) {
            p = term_product<0, UNIT>(mul, SharedCols<2, STRIDE>{S, Mr}, l, jf, emask, sm.ecnt, E);
        } else {
            p = term_product<0, UNIT>(mul, SharedCols<1, STRIDE>{S, Mr}, l, jf, emask, sm.ecnt, E);
        }
    }
    return task_sum(rh, rl, ih, il, whigh_u, (gpar & 1) != 0, active);
}

// The same walk in FP64, for a base matrix without integer scales (non-finite
// entries, a column bound beyond FP64): column sums in local memory, products
// in the same order.  Speed is not the point here: infinities and NaNs are
// combined as FP64 arithmetic does.
static __device__ void fp64_term(const double2* S, int l, int jf, const int32_t* ecnt, bool neg,
                          double2& acc)
{
    double2 pre = S[0], ex = make_double2(neg ? -1.0 : 1.0, 0.0);
    if (jf < 0) {
        if (l == 1) {  // n = 1: the product is S_0 itself
            acc.x = neg ? __dsub_rn(acc.x, pre.x) : __dadd_rn(acc.x, pre.x);
            acc.y = neg ? __dsub_rn(acc.y, pre.y) : __dadd_rn(acc.y, pre.y);
            return;
        }
        for (int j = 1; j < l - 1; ++j)
            pre = cmul(pre, S[j]);
        ex = S[l - 1];
    } else {
        for (int j = 0; j < l; ++j) {
            if (j > 0)
                pre = cmul(pre, S[j]);
            if (j == jf)
                ex = pre;
            for (int e = j == jf ? 1 : 0; e < ecnt[j]; ++e)
                ex = cmul(ex, pre);
        }
    }
    if (neg)
        cfma_acc<true>(acc, pre, ex);
    else
        cfma_acc<false>(acc, pre, ex);
}

static __device__ dd2 fp64_walk(const PermDesc& D, const MetaView& mv, const WarpSmem& sm,
                                      int64_t chunk, bool active)
{
    const int l = D.l, J = D.J, ndig = D.ndig;
    const double2* M = reinterpret_cast<const double2*>(sm.M);
    const double2* base = reinterpret_cast<const double2*>(sm.base);
    double2 S[PQ_MAX_PRODUCT_COLS];
    for (int j = 0; j < l; ++j)
        S[j] = base[j];
    auto add_row = [&](int row, double coef) {
        for (int j = 0; j < l; ++j) {
            const double2 b = M[row * sm.ld + j];
            S[j].x = __fma_rn(coef, b.x, S[j].x);
            S[j].y = __fma_rn(coef, b.y, S[j].y);
        }
    };
    uint64_t whigh_u = 1;
    int gpar = 0;
    for (int d = J; d < ndig; ++d) {
        const int g = next_digit(chunk, mv.drad[d], false);
        if (g == 0)
            continue;
        add_row(mv.drow[d], (double)(-2 * g));
        whigh_u *= binom_u64(mv.dtop[d], g);
        gpar += g;
    }
    LowWalk wk;
    start_walk(wk, mv, J);
    double wlow = 1.0;
    double2 acc = make_double2(0.0, 0.0), run = make_double2(0.0, 0.0);
    double rh = 0.0, rl = 0.0, ih = 0.0, il = 0.0;
    for (int64_t s = 0;;) {
        fp64_term(S, l, D.jf, sm.ecnt, (s & 1) != 0, acc);
        ++s;
        if (s == D.L || (s & 31) == 0) {
            run.x = __fma_rn(wlow, acc.x, run.x);
            run.y = __fma_rn(wlow, acc.y, run.y);
            dd_acc(rh, rl, run.x);
            dd_acc(ih, il, run.y);
            acc = run = make_double2(0.0, 0.0);
            if (s == D.L)
                break;
        }
        int up;
        const int d = low_step(wk, up);
        if (((wk.radm1 >> (4 * d)) & 15u) > 1u)
            reweight(wk, J, wlow, acc, run);
        add_row(sm.lowrow[d], up > 0 ? -2.0 : 2.0);
    }
    return task_sum(rh, rl, ih, il, whigh_u, (gpar & 1) != 0, active);
}

// The tasks of a permanent that is not staged as integers of one unit: the whole
// rest of the task, so that the main path keeps nothing for it (with the walks
// alone called and their sum combined on the main path, a class at its register
// limit spilled more: one n = 26 permanent 1.98 -> 2.26 ms).
static __device__ __noinline__ void other_task(const ExecArgs& a, Task t, longlong2* M,
                                               longlong2* base, int32_t* lowrow, int ld, int mode,
                                               int exp2, uint32_t emask, int lane)
{
    const PermDesc D = a.desc[t.perm];
    const MetaView mv = meta_view(a.meta, D);
    const WarpSmem sm(M, base, lowrow, ld);
    const int64_t chunk0 = (int64_t)t.part * kWarp;
    const bool active = chunk0 + lane < D.nchunks;
    const int64_t chunk = active ? (chunk0 + lane) : 0;
    if (mode == kStagedFp64) {
        const dd2 res = fp64_walk(D, mv, sm, chunk, active);
        combine_task<false>(a, t, D, res, exp2, 0, 0, lane);
        return;
    }
    // a unit for each part; column sums in local memory
    longlong2 S[PQ_MAX_PRODUCT_COLS];
    const int f = sscale_of(sm.cexp[0]).f;
    int turns = 0;
    for (int j = 0; j < D.l; ++j)
        turns += sscale_of(sm.cexp[j]).turned ? mv.cmul[j] : 0;
    const PartUnits mul{min(63, 2 * f)};
    const dd2 res = D.jf < 0 ? int_walk<0, true, 1>(mul, S, D, mv, sm, emask, chunk, active, lane)
                             : int_walk<0, false, 1>(mul, S, D, mv, sm, emask, chunk, active, lane);
    combine_task<true>(a, t, D, res, exp2, f, turns, lane);
}

// Whether the end of a task reads the descriptor again, so that the walk does not
// hold it in registers: in the classes whose registers are short.  Held / read again:
// n = 26 permanent 2.20 / 1.94 ms, 28 8.78 / 8.58, 30 35.7 / 35.4, 4096 patterns of 12
// photons 195.5 / 193.7 us; but class 24 0.593 / 0.608 ms and, in shared memory, 65536
// ragged permanents 5.74 / 5.80.
constexpr bool fwd_reads_again(int nl) { return nl > 0 && nl != 24; }

template <int NL>
__device__ __forceinline__ void process_task(const ExecArgs& a, const Task& t, WarpSmem& sm,
                                             Staged& st, int lane)
{
    const PermDesc D = a.desc[t.perm];
    const MetaView mv = meta_view(a.meta, D);
    dd2 res = {0.0, 0.0, 0.0, 0.0};
    if (!D.trivial) {
        if (st.perm != t.perm) {
            __syncwarp();
            stage_perm(a, D, mv, sm, st, lane);
            st.perm = t.perm;
        }
        if (st.mode != kStagedInt) {
            other_task(a, t, sm.M, sm.base, sm.lowrow, sm.ld, st.mode, st.exp2, st.emask, lane);
            return;
        }
        const int64_t chunk0 = (int64_t)t.part * kWarp;
        const bool active = chunk0 + lane < D.nchunks;
        const int64_t chunk = active ? (chunk0 + lane) : 0;
        if (D.jf < 0)
            res = int_walk<NL, true>(OneUnit(), sm.S + lane, D, mv, sm, st.emask, chunk, active, lane);
        else
            res = int_walk<NL, false>(OneUnit(), sm.S + lane, D, mv, sm, st.emask, chunk, active, lane);
    }
    if (fwd_reads_again(NL)) {
        asm volatile("" ::: "memory");
        const PermDesc E = a.desc[t.perm];
        combine_task<false>(a, t, E, res, st.exp2, 0, 0, lane);
    } else {
        combine_task<false>(a, t, D, res, st.exp2, 0, 0, lane);
    }
}

// Task ti of the list, once its guards pass (a failing task is skipped and
// recorded in the error record).
template <int NL>
__device__ __forceinline__ void run_task(const ExecArgs& a, int64_t ti, WarpSmem& sm, int kmax,
                                         int ld, Staged& st, int lane)
{
    const Task t = a.tasks[ti];
    const int32_t bad = task_guard(t, a.desc, a.nperm, a.nmeta, a.nslots, kmax, ld, kMaxLowDigits,
                                   a.ngroups);
    if (bad) {
        if (lane == 0)
            record_error(a.err, bad, ti);
        return;
    }
    process_task<NL>(a, t, sm, st, lane);
}

// The register-resident kernel of column bound NL: tasks as in
// glynn_fwd_kernel, each of a permanent with at most NL product columns (a
// task beyond that is skipped and recorded as a layout error).  Batches of one
// column class run it, so that the warps of an
// SM run one instantiation of the walk: warps running different ones (a
// single kernel dispatching on l) ran 1.6 times slower.
// Resident warps per SM of a class, in blocks of 4 warps (the register file is
// split over 4 sub-partitions): 96, 128, 168 and 255 registers at 20, 16, 12 and
// 8 warps.  The column sums take 4 NL, the rest of the walk about 50.  (Blocks of
// 8 warps round the warps down to a multiple of 8: with 4-warp blocks and the
// walk of unit columns, 65536 ragged permanents 6.90 -> 5.98 ms, n = 30 49.1 ->
// 35.2 ms.)
constexpr int fwd_reg_blocks(int nl) { return nl <= 6 ? 5 : nl <= 14 ? 4 : nl <= 26 ? 3 : 2; }

template <int NL>
__global__ void __launch_bounds__(128, fwd_reg_blocks(NL)) glynn_fwd_reg_kernel(const __grid_constant__ ExecArgs a,
                                                             int64_t t_begin,
                                                             int64_t t_end, int kmax, int ld,
                                                             int queue)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (NL > ld) {  // the launch's shared-memory rows are narrower than this class's
        if (threadIdx.x == 0)
            record_error(a.err, kErrDescLayout, t_begin);
        return;
    }
    WarpSmem sm(smem_raw + warp * reg_warp_smem_bytes(kmax, ld), kmax, NL, false);
    Staged st;
    if (!queue) {
        const int64_t ti = t_begin + (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
        if (ti < t_end)
            run_task<NL>(a, ti, sm, kmax, NL, st, lane);
        return;
    }
    for (;;) {
        int q = 0;
        if (lane == 0)
            q = atomicAdd(a.counters, 1);
        q = __shfl_sync(0xffffffffu, q, 0);
        const int64_t ti = t_begin + q;
        if (ti >= t_end)
            break;
        run_task<NL>(a, ti, sm, kmax, NL, st, lane);
    }
}

}  // namespace pqi
