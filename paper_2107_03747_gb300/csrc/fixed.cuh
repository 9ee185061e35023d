// fixed.cuh -- products of unitary matrices in 58-bit fixed point on the integer pipe.
//
// Why.  GB300 issues a warp's FP64 FMA every 64 cycles per SM quarter, but a 32 x 32 + 64 -> 64 bit
// integer multiply-add (IMAD.WIDE) every 4 (tgf_fma_peak: 2.0 and 31.9 lanes per clock and SM).
// Entries of SU(N) matrices are at most 1, so they need no exponent: an entry is the integer
// v = floor(x 2^58), split as v = hi 2^29 + lo with 0 <= lo < 2^29, and one multiply-add of two
// entries is three IMAD.WIDE (hi hi; hi lo and lo hi, summed apart; lo lo is below the last bit kept):
// 12 cycles instead of 64.
//
// Accuracy.  Operands of 2^-5 and more are exact, smaller ones are cut towards 0 at 2^-58.  Sums are exact: rounding
// enters once per entry and product, when the sum of the cross terms is rounded to 2^-58 (half a unit at most) and
// the 2N products lo lo, each below a unit, are replaced by their mean (0.3 of a unit left each, rms).  In FP64 the same
// entry, a sum of 2N products of size up to 1, carries up to 2N roundings of 2^-54: where the entries are not
// all small (fx_rough), a staple formed here is nearer to its exact value than one formed in FP64.
// No rounding leans to one side, as the observables add millions of sites: with operands and sums cut
// downwards, the lo lo products dropped and cross sums rounded to 2^-55, which costs the same time (a fourth
// fewer instructions, but on the multiply pipe), S and Q of 4x4x12x12 at amplitude 0.15 were off by 1.5 x 2^-53 S and
// 0.5 x 2^-53 on the average of 16 fields; now 0.2 and 0.0.
//
// Range.  Nothing wraps as long as operand entries stay within the bounds noted at each split: with
// 2N <= 8 terms of a link and another operand, hi hi sums stay below 8 x 2^30 x 2^29.01 and cross sums
// below 8 (2^30 2^29 + 2^29.01 2^29), both under 2^63.  The
// fields are arbitrary user data, so every operand is checked as it is taken in: a link entry
// above 1 + 2^-10 in magnitude (also infinities and NaN), a product T above 2, a staple sum above 8, an entry of Omega
// above 32 (the trace adds up to four) set bits in a guard word; a thread that finds them set repeats its link in FP64
// arithmetic, which takes any input.  SU(N) fields never do.  Sums are tested in 64 bits, before a split narrows them:
// entries of size 1 that add up in phase make T as large as 2N sqrt 2, which the 32 bits of hi fold back.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "expm.cuh"
#include "lattice.cuh"
#include "su3.cuh"

namespace tgf {

// (hi 2^29 + lo) in units that depend on the operand: 2^-58 for links and T (SPLIT 0), 2^(SH-58)
// for wider operands split with SH > 0
template <int N>
struct matx {
    int rh[N][N], rl[N][N], ih[N][N], il[N][N];
};
// sums of products
template <int N>
struct matq {
    long long re[N][N], im[N][N];
};

constexpr int kFxBits = 58;


struct fx_guard {
    unsigned top = 0;   // bit 31: an operand outside its bound
    unsigned top2 = 0;  // not 0: a sum outside its bound
    unsigned far = 0;   // bits 26-28: an entry away from 0 and +-1 (fx_rough)
    __device__ __forceinline__ bool rough() const { return (far & 0x1c000000u) != 0; }
    __device__ __forceinline__ bool bad() const { return ((top >> 31) | top2) != 0; }
};

// x 2^58, cut towards 0, split into hi, lo.  The mantissa with its leading bit is aligned at the top of 64 bits and
// shifted right by 1025 - exponent, which leaves |x| 2^61; shifts past 63 bits give 0.  A negative x takes the
// complement, floor(-|x| 2^58) - 1 once it is cut, and that unit back on lo (1 <= lo <= 2^29 then).
// `up` takes x 2^up instead (a matrix of small entries keeps its relative precision), flip = -1 takes -x.
__device__ __forceinline__ void fx_take(double x, int& hi, int& lo, fx_guard& g, unsigned up = 0, int flip = 0) {
    const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
    const unsigned a = h & 0x7fffffffu;
    g.top |= (0x3FF00400u - (up << 20)) - a;  // |x| 2^up <= 1 + 2^-10, else bit 31
    const unsigned s = (1025u - up) - (a >> 20);
    unsigned long long m = ((unsigned long long)(__funnelshift_l(l, h, 11) | 0x80000000u) << 32) | (l << 11);
    asm("shr.b64 %0, %0, %1;" : "+l"(m) : "r"(s));
    const int sg = ((int)h >> 31) ^ flip;
    asm("xor.b32 %0, %1, %2;" : "=r"(hi) : "r"((int)(m >> 32)), "r"(sg));
    asm("{.reg .u32 t; shr.u32 t, %1, 3; sub.s32 %0, t, %2;}" : "=r"(lo) : "r"((unsigned)m ^ (unsigned)sg), "r"(sg));
}

// a sum (units 2^-58) -> operand in units 2^(SH-58); |v| < 2 (SH = 0), 4 (SH = 1) or 8 (SH = 2).  ROUND: to the nearest
// (ties to even, half the values of SH = 1 are ties) for sums that reach an observable, cut downwards otherwise
template <int SH, bool ROUND = false>
__device__ __forceinline__ void fx_split(long long v, int& hi, int& lo) {
    if (ROUND && SH > 0) v += ((1 << SH) / 2 - 1) + (int)(((unsigned)v >> SH) & 1u);
    asm("{.reg .b64 t; shr.s64 t, %1, %2; cvt.u32.u64 %0, t;}" : "=r"(hi) : "l"(v), "n"(29 + SH));
    asm("and.b32 %0, %1, 0x1fffffff;" : "=r"(lo) : "r"((int)(v >> SH)));
}

template <int N>
__device__ __forceinline__ void fx_zero(matq<N>& a) {
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = 0; j < N; ++j) a.re[i][j] = a.im[i][j] = 0;
}

// a wider operand; its bound (2^(SH+1)) must have been checked
template <int N, int SH, bool ROUND = false>
__device__ __forceinline__ void fx_operand_wide(matx<N>& o, const matq<N>& v) {
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = 0; j < N; ++j) {
            fx_split<SH, ROUND>(v.re[i][j], o.rh[i][j], o.rl[i][j]);
            fx_split<SH, ROUND>(v.im[i][j], o.ih[i][j], o.il[i][j]);
        }
}
// |entries| < 2^(B - 26), else the guard's second word (the top word of a sum counts in 2^-26)
template <int N, int B>
__device__ __forceinline__ void fx_check(const matq<N>& v, fx_guard& g) {
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = 0; j < N; ++j)
            g.top2 |= (((unsigned)(int)(v.re[i][j] >> 32) + (1u << B)) | ((unsigned)(int)(v.im[i][j] >> 32) + (1u << B))) &
                      ~((2u << B) - 1u);
}

// c + a b by one IMAD.WIDE.  Written as C++: mad.wide in PTX becomes a product and a separate 64-bit
// addition.  The compiler must not see that lo is never negative nor where hi comes from (their last instruction is
// therefore inline assembly): a zero-extended factor times a sign-extended one would become a full
// 64 x 64 bit product.
__device__ __forceinline__ long long mad_wide(int a, int b, long long c) { return c + (long long)a * b; }
__device__ __forceinline__ int fx_neg(int a) { return (int)(0u - (unsigned)a); }
__device__ __forceinline__ void fx_mad(long long& hh, long long& cr, int ah, int al, int bh, int bl) {
    hh = mad_wide(ah, bh, hh);
    cr = mad_wide(ah, bl, cr);
    cr = mad_wide(al, bh, cr);
}
// start of a cross sum (opaque: an accumulator of the first multiply-add, not an addition of its own): half a unit of
// the hi hi sum, for the rounding, and a quarter of one, the mean of lo lo, for each of TERMS products that add up
// with one sign (those of both signs cancel)
template <int TERMS = 0>
__device__ __forceinline__ long long fx_round() {
    long long r;
    asm("mov.b64 %0, %1;" : "=l"(r) : "n"((1ll << 28) + ((long long)TERMS << 27)));
    return r;
}
// hi hi sum + rounded cross sum: the cross unit is 2^-29 of the hi hi unit
__device__ __forceinline__ long long fx_join(long long hh, long long cr) { return hh + (cr >> 29); }

// Re and Im of c + sum_k a_k w_k, w = b or (CONJ) its complex conjugate; minus signs go to a negated copy of a
// (lo < 2^29, so -lo is exact).
template <int N>
struct vecx {
    int rh[N], rl[N], ih[N], il[N];
};
template <int N, bool CONJ>
__device__ __forceinline__ void fx_dot(long long& re, long long& im, const vecx<N>& a, const vecx<N>& na, const vecx<N>& b) {
    long long rc = fx_round<CONJ ? 2 * N : 0>(), ic = fx_round<CONJ ? 0 : 2 * N>();
#pragma unroll
    for (int k = 0; k < N; ++k) {
        fx_mad(re, rc, a.rh[k], a.rl[k], b.rh[k], b.rl[k]);
        if (CONJ) {
            fx_mad(im, ic, a.ih[k], a.il[k], b.rh[k], b.rl[k]);
            fx_mad(re, rc, a.ih[k], a.il[k], b.ih[k], b.il[k]);
            fx_mad(im, ic, na.rh[k], na.rl[k], b.ih[k], b.il[k]);
        } else {
            fx_mad(im, ic, a.rh[k], a.rl[k], b.ih[k], b.il[k]);
            fx_mad(re, rc, na.ih[k], na.il[k], b.ih[k], b.il[k]);
            fx_mad(im, ic, a.ih[k], a.il[k], b.rh[k], b.rl[k]);
        }
    }
    re = fx_join(re, rc);
    im = fx_join(im, ic);
}
template <int N>
__device__ __forceinline__ vecx<N> fx_negated(const vecx<N>& a) {
    vecx<N> n;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        n.rh[k] = fx_neg(a.rh[k]);
        n.rl[k] = fx_neg(a.rl[k]);
        n.ih[k] = fx_neg(a.ih[k]);
        n.il[k] = fx_neg(a.il[k]);
    }
    return n;
}
template <int N>
__device__ __forceinline__ vecx<N> fx_row(const matx<N>& m, int i) {
    vecx<N> v;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        v.rh[k] = m.rh[i][k];
        v.rl[k] = m.rl[i][k];
        v.ih[k] = m.ih[i][k];
        v.il[k] = m.il[i][k];
    }
    return v;
}
template <int N>
__device__ __forceinline__ vecx<N> fx_col(const matx<N>& m, int j) {
    vecx<N> v;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        v.rh[k] = m.rh[k][j];
        v.rl[k] = m.rl[k][j];
        v.ih[k] = m.ih[k][j];
        v.il[k] = m.il[k][j];
    }
    return v;
}

// c = a b
template <int N>
__device__ __forceinline__ void fx_mul_nn(matq<N>& c, const matx<N>& a, const matx<N>& b) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const vecx<N> r = fx_row(a, i), nr = fx_negated(r);
#pragma unroll
        for (int j = 0; j < N; ++j) {
            c.re[i][j] = c.im[i][j] = 0;
            fx_dot<N, false>(c.re[i][j], c.im[i][j], r, nr, fx_col(b, j));
        }
    }
}

// c *= exp(2 pi i k / 3) or its conjugate (zr + i zi): once in a while, at the twisted corner
template <int N>
__device__ __forceinline__ void fx_scale(matx<N>& m, double zr, double zi) {
    fx_guard g;
    int zrh, zrl, zih, zil;
    fx_take(zr, zrh, zrl, g);
    fx_take(zi, zih, zil, g);
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = 0; j < N; ++j) {
            long long rh = 0, ih = 0, rc = fx_round(), ic = fx_round<2>();
            fx_mad(rh, rc, m.rh[i][j], m.rl[i][j], zrh, zrl);
            fx_mad(rh, rc, fx_neg(m.ih[i][j]), fx_neg(m.il[i][j]), zih, zil);
            fx_mad(ih, ic, m.rh[i][j], m.rl[i][j], zih, zil);
            fx_mad(ih, ic, m.ih[i][j], m.il[i][j], zrh, zrl);
            fx_split<0>(fx_join(rh, rc), m.rh[i][j], m.rl[i][j]);
            fx_split<0>(fx_join(ih, ic), m.ih[i][j], m.il[i][j]);
        }
}

template <int N>
__device__ __forceinline__ void fx_take_entry(matx<N>& o, int i, int j, double re, double im, fx_guard& g, unsigned up = 0) {
    fx_take(re, o.rh[i][j], o.rl[i][j], g, up);
    fx_take(im, o.ih[i][j], o.il[i][j], g, up);
}

// ---- staple sums ------------------------------------------------------------------------------
//
// Both staples of a direction are one computation.  With V, B, C the three links,
//   forward   F = Z*_{mu nu}(n) U_nu(n+mu) U_mu(n+nu)^+ U_nu(n)^+:
//             row i of F = conj-dot of (row i of V, rows of B) with the rows of C,  V = U_nu(n+mu), B = U_mu(n+nu), C = U_nu(n)
//   backward  G = Z_{mu nu}(n-nu) U_nu(n+mu-nu)^+ U_mu(n-nu)^+ U_nu(n-nu):
//             column j of G is the same expression of the transposed links V = U_nu(n-nu), B = U_mu(n-nu), C = U_nu(n+mu-nu)
// so one loop body serves both, reading the backward links transposed (an address choice) and summing onto the
// transposed staple sum, which is transposed in registers between the two.  The body of about 1500
// instructions stays in the instruction cache, where two would not, and only B, C, the sum and one row
// are live, so that 12 warps fit on an SM instead of 8.
//
// SRC: get(dir, site, i, j, tr) loads entry (i, j), transposed if tr (a value uniform over the warp).
// SYNC: a block barrier per iteration (every thread of the block must be here).  The warps of a block then
// fetch the same instructions at the same time: 11 % on the FP64 stage (8.63 instead of 9.74 ms for
// 4 steps of 4 x 8x8x24x24, before its exponential and shared links, which took it to 7.6).
// visit(q, nu, sig): called after the forward (q = 0) and after the backward staple (q = 1) of a direction,
// with the sum in normal orientation.  q0, q1: the part of the six staples (in
// pairs) that this thread sums.
template <int N>
__device__ __forceinline__ void fx_transpose(matq<N>& m) {
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = i + 1; j < N; ++j) {
            const long long r = m.re[i][j], q = m.im[i][j];
            m.re[i][j] = m.re[j][i];
            m.im[i][j] = m.im[j][i];
            m.re[j][i] = r;
            m.im[j][i] = q;
        }
}

// Weak fields.  A resolution of 2^-58 for every entry serves fields whose links are of size 1 all over.  Near the unit matrix
// (or any field of one entry +-1, +-i per row and column) force and clover come from the small entries, which FP64 holds
// to 53 bits and whose products it rounds relative to their own size.  So a link takes the FP64 path if it is weak: if
// every real and imaginary part of it and of the 18 links that its staples read is within 2^-4 of 0 or +-1, or if the links that
// its block shares are.  Error of a link's force relative to its largest entry (rms, SU(3), links exp(i amp omega T);
// of a clover half a quarter more), and how many are weak by themselves:
//    amp          0.3      0.1      0.07     0.05     0.03     0.01     1e-4     1e-8
//    FP64         6.8e-17  6.2e-17  6.2e-17  6.3e-17  6.2e-17  6.4e-17  6.4e-17  6.3e-17
//    fixed point  2.6e-17  3.1e-17  3.5e-17  4.5e-17  6.8e-17  2e-16    2e-14    2e-10
//    weak         0        0        0        4 %      98 %     all      all      all
// A rough field pays up to 1 % for the test of the links that it shares.  A weak one runs at the FP64 pipe's rate: two
// steps of 4 x 8x8x24x24 take 13.6 ms at amp 1e-6, 14.6 at 0.05 where most warps do both, 4.2 at 0.07, 3.7 above.
__device__ __forceinline__ bool fx_rough(double2 x) {
    constexpr unsigned lo = 0x3FB00000u, n = 0x3FEE0000u - lo;  // top words of 2^-4 and 1 - 2^-4
    return ((unsigned)__double2hiint(x.x) & 0x7fffffffu) - lo < n || ((unsigned)__double2hiint(x.y) & 0x7fffffffu) - lo < n;
}

// a link, transposed if `tr`; flip = -1 conjugates it; TEST: its entries go to the guard's far
template <int N, bool TEST = false, class SRC>
__device__ __forceinline__ void fx_take_matrix(matx<N>& o, SRC& src, int dir, int site, bool tr, fx_guard& g, int flip = 0) {
    double2 x[N][N];
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = 0; j < N; ++j) x[i][j] = src.get(dir, site, i, j, tr);
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = 0; j < N; ++j) {
            fx_take(x[i][j].x, o.rh[i][j], o.rl[i][j], g);
            fx_take(x[i][j].y, o.ih[i][j], o.il[i][j], g, 0, flip);
            // hi, in 2^-29, plus 2^25: bits 26-28 are clear within 2^25 of 0 and +-2^29
            if (TEST) g.far |= (unsigned)(o.rh[i][j] + (1 << 25)) | (unsigned)(o.ih[i][j] + (1 << 25));
        }
}

// Links that several warps of a block need, taken as operands once and shared: [dir] U_dir(n) and [4 + dir] U_dir(n - dir)
// of the block's 32 sites, entry by entry (re hi, lo, im hi, lo), and whether each is out of range (bit 0) and rough (bit 26).
template <int N>
struct fx_shared {
    int4 u[8][N * N][32];
    unsigned flags[8][32];
};
template <int N>
__device__ __forceinline__ void fx_share(fx_shared<N>& sh, int m, int lane, const matx<N>& o, const fx_guard& g) {
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = 0; j < N; ++j) sh.u[m][i * N + j][lane] = make_int4(o.rh[i][j], o.rl[i][j], o.ih[i][j], o.il[i][j]);
    sh.flags[m][lane] = (unsigned)g.bad() | (g.rough() ? 1u << 26 : 0u);
}
// The flags of the links at lane's site that the link in direction mu reads, into its guard; whether none of the block's links
// is rough.  All lanes of the warp.
template <int N>
__device__ __forceinline__ bool fx_shared_flags(fx_guard& g, const fx_shared<N>& sh, int mu, int lane) {
    unsigned f = 0;
#pragma unroll
    for (int m = 0; m < 8; ++m) {
        const unsigned v = sh.flags[m][lane];
        f |= v;
        if (m != 4 + mu) g.far |= v;
    }
    g.top2 |= f & 1u;
    return !__any_sync(0xffffffffu, f >> 26);
}
template <int N>
__device__ __forceinline__ void fx_shared_link(matx<N>& o, const fx_shared<N>& sh, int m, int lane) {
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = 0; j < N; ++j) {
            const int4 v = sh.u[m][i * N + j][lane];
            o.rh[i][j] = v.x;
            o.rl[i][j] = v.y;
            o.ih[i][j] = v.z;
            o.il[i][j] = v.w;
        }
}

// sh: the block's shared links (SHARE), filled and followed by a barrier of fx_staples' first iteration
template <int N, bool SYNC, bool SHARE, class SRC, class VISIT>
__device__ __forceinline__ void fx_staples(matq<N>& sig, SRC& src, const fx_shared<N>* sh, int lane, const CfgDesc& c, int s,
                                           int mu, unsigned eb, fx_guard& g, VISIT&& visit, int q0 = 0, int q1 = 6) {
    const int s_mp = fwd(c, eb, s, mu);
    const bool at_mu0 = (eb >> mu) & 1u;  // x_mu = 0: the twisted plaquettes' corner row
#pragma unroll 1
    for (int q = q0; q < q1; ++q) {
        const bool back = q & 1;
        const int nu = (mu + 1 + (q >> 1)) & 3;
        if (SYNC) __syncthreads();
        const int s_nm = bwd(c, eb, s, nu);
        const int sb = back ? s_nm : fwd(c, eb, s, nu);
        const int sv = back ? s_nm : s_mp;
        const int sc = back ? fwd(c, eb, s_nm, mu) : s;  // x_mu(n - nu) = x_mu(n)
        if (back) fx_transpose(sig);
        matx<N> b, d;
        fx_take_matrix<N>(b, src, mu, sb, back, g);
        // the twisted corner's centre factor goes to B: Z* V B^+ = V (Z B)^+
        const int k = c.tw[mu * 4 + nu];
        if (k != 0 && at_mu0 && ((eb >> (back ? 8 + nu : nu)) & 1u)) {
            double zr, zi;
            SRC::centre(k, zr, zi);
            fx_scale(b, zr, back ? -zi : zi);
        }
        if (SHARE && !back) fx_shared_link<N>(d, *sh, nu, lane);
        else fx_take_matrix<N>(d, src, nu, sc, back, g);
        unsigned wide = 0;  // top words of T, in 2^-26, plus 2: 28 bits while |T| < 2
#pragma unroll
        for (int i = 0; i < N; ++i) {
            vecx<N> v, t;
            if (SHARE && back) {
#pragma unroll
                for (int j = 0; j < N; ++j) {
                    const int4 x = sh->u[4 + nu][j * N + i][lane];
                    v.rh[j] = x.x;
                    v.rl[j] = x.y;
                    v.ih[j] = x.z;
                    v.il[j] = x.w;
                }
            } else {
#pragma unroll
                for (int j = 0; j < N; ++j) {
                    const double2 x = src.get(nu, sv, i, j, back);
                    fx_take(x.x, v.rh[j], v.rl[j], g);
                    fx_take(x.y, v.ih[j], v.il[j], g);
                }
            }
            vecx<N> nv = fx_negated(v);
#pragma unroll
            for (int j = 0; j < N; ++j) {
                long long re = 0, im = 0;
                fx_dot<N, true>(re, im, v, nv, fx_row(b, j));
                wide |= (unsigned)((int)(re >> 32) + (1 << 27)) | (unsigned)((int)(im >> 32) + (1 << 27));
                fx_split<0>(re, t.rh[j], t.rl[j]);
                fx_split<0>(im, t.ih[j], t.il[j]);
            }
            nv = fx_negated(t);
#pragma unroll
            for (int j = 0; j < N; ++j) fx_dot<N, true>(sig.re[i][j], sig.im[i][j], t, nv, fx_row(d, j));
        }
        if (back) fx_transpose(sig);
        g.top2 |= wide >> 28;
        fx_check<N, 29>(sig, g);
        visit(q & 1, nu, sig);
    }
}

// FP64 links for fixed.cuh: entry e of a link at base + (e / 2) 4 Vp + 4 s + 2 (e % 2), entry 8 at 16 Vp + 2 s.
// A plane's offset, 12 Vp + 2 doubles at most, exceeds 31 bits from 1.8e8 sites on and stays below 2^32 up to the
// library's limit of 2^28: unsigned, so that choosing between the two orientations stays a 32-bit select.  The base is
// stepped first: with the three offsets summed before it, which lengthens the chain that a small launch waits for, a
// sweep of 8 x 4x4x12x12 takes 3.55 ms instead of 3.41 (3.48 with 64-bit planes).
struct Su3Src {
    const double* base;
    int Vp;
    static __host__ __device__ __forceinline__ unsigned plane(int e, int Vp) { return (e >> 1) * 4u * (unsigned)Vp + (e & 1) * 2u; }
    __device__ __forceinline__ double2 get(int dir, int s, int i, int j, bool tr) const {
        s = checked_site(s, Vp);
        const double* p = base + (size_t)dir * 18 * Vp;
        if (i == 2 && j == 2) return __ldg(reinterpret_cast<const double2*>(p + (size_t)16 * Vp) + s);
        const unsigned oe = plane(3 * i + j, Vp), of = plane(3 * j + i, Vp);
        return __ldg(reinterpret_cast<const double2*>(p + (size_t)(tr ? of : oe) + (size_t)s * 4));
    }
    static __device__ __forceinline__ void centre(int k, double& zr, double& zi) { tgf::centre<double>(k, zr, zi); }
};

// Whether a link, and all links that the staples of U_mu(s) read, are near 0 and +-1
template <int N, class SRC>
__device__ __forceinline__ bool fx_near(const SRC& src, int dir, int s) {
    bool rough = false;
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = 0; j < N; ++j) rough |= fx_rough(src.get(dir, s, i, j, false));
    return !rough;
}
template <int N, class SRC>
__device__ __forceinline__ bool fx_near_staples(const SRC& src, const CfgDesc& c, unsigned eb, int s, int mu) {
#pragma unroll 1
    for (int q = 0; q < 18; ++q) {
        // U_nu at n, n - nu, n + mu, n + mu - nu, U_mu at n + nu, n - nu
        const int nu = (mu + 1 + q % 3) & 3, k = q / 3;
        int t = (k & 1) ? bwd(c, eb, s, nu) : k == 4 ? fwd(c, eb, s, nu) : s;
        if (k == 2 || k == 3) t = fwd(c, eb, t, mu);  // x_mu(n - nu) = x_mu(n)
        if (!fx_near<N>(src, k < 4 ? nu : mu, t)) return false;
    }
    return true;
}

// The largest up <= 40 for which every entry of m, times 2^up, stays below 1 in magnitude.
template <int N>
__device__ __forceinline__ unsigned fx_scale_of(const cx<double> (&m)[N][N]) {
    unsigned a = 0;
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = 0; j < N; ++j) {
            a = max(a, (unsigned)__double2hiint(m[i][j].re) & 0x7fffffffu);
            a = max(a, (unsigned)__double2hiint(m[i][j].im) & 0x7fffffffu);
        }
    return (unsigned)min(max(1022 - (int)(a >> 20), 0), 40);
}
// v 2^-58, the factor taken off the exponent (a whole number but 0 is at least 1 in magnitude)
__device__ __forceinline__ double fx_value(long long v) {
    const double x = (double)v;
    const int h = __double2hiint(x);
    return __hiloint2double(h ? h - (kFxBits << 20) : 0, __double2loint(x));
}
// 2^(-58 - up)
__device__ __forceinline__ double fx_unit(unsigned up) { return __hiloint2double((int)((1023u - kFxBits - up) << 20), 0); }

// ---- exp(X) - 1 of a traceless anti-Hermitian 3x3 matrix ------------------------------------------
//
// For X = iQ with ||Q||_F^2 <= kFxExpMax: exp(iQ) - 1 = f0 + f1 Q + f2 Q^2 (f0 without its 1) with the f as the sums
// over n <= 10 of i^n/n! times the coefficients of Q^n (expm.cuh's recursion, written out as polynomials in
// c1 = tr Q^2 / 2 and c0 = tr Q^3 / 3); the dropped tail is below 0.126^11 / 11! = 3e-18.  Q is scaled by 2^up to the
// size of 1, Q^2, the traces and the assembly run in fixed point, the 6 polynomials in FP64: about 45 FP64
// instructions where the series of expm_su3 takes 210, each of which holds the pipe for 64 cycles and drags four
// empty issue slots behind it.  Result: operands in units 2^(-58 - up); false if ||Q||_F is too large.
constexpr double kFxExpMax = 0.016;

struct fx_num {
    int h, l;
};
__device__ __forceinline__ void fx_mac(long long& hh, long long& cr, const fx_num& a, const fx_num& b) {
    fx_mad(hh, cr, a.h, a.l, b.h, b.l);
}
__device__ __forceinline__ fx_num fx_minus(const fx_num& a) { return {fx_neg(a.h), fx_neg(a.l)}; }
__device__ __forceinline__ fx_num fx_operand(long long v) {
    fx_num o;
    fx_split<0>(v, o.h, o.l);
    return o;
}
__device__ __forceinline__ fx_num fx_number(double x, fx_guard& g, unsigned up, int flip = 0) {
    fx_num o;
    fx_take(x, o.h, o.l, g, up, flip);
    return o;
}
// s + a b + c d
__device__ __forceinline__ long long fx_sum2(long long s, const fx_num& a, const fx_num& b, const fx_num& c, const fx_num& d,
                                             long long half) {
    long long cr = half;
    fx_mac(s, cr, a, b);
    fx_mac(s, cr, c, d);
    return fx_join(s, cr);
}

__device__ __forceinline__ bool fx_exp_su3(matx<3>& o, unsigned& up, const alg8<double>& x) {
    fx_guard g;
    const long long half = fx_round();
    const double x22 = -(x.v[0] + x.v[1]);
    unsigned amax = (unsigned)__double2hiint(x22) & 0x7fffffffu;
#pragma unroll
    for (int i = 0; i < 8; ++i) amax = max(amax, (unsigned)__double2hiint(x.v[i]) & 0x7fffffffu);
    up = (unsigned)min(max(1022 - (int)(amax >> 20), 0), 40);
    // Q = -i X, times 2^up
    const fx_num a[3] = {fx_number(x.v[0], g, up), fx_number(x.v[1], g, up), fx_number(x22, g, up)};
    const fx_num qr[3] = {fx_number(x.v[3], g, up), fx_number(x.v[5], g, up), fx_number(x.v[7], g, up)};  // 01, 02, 12
    const fx_num qi[3] = {fx_number(x.v[2], g, up, -1), fx_number(x.v[4], g, up, -1), fx_number(x.v[6], g, up, -1)};
    // Q^2, times 2^(2 up)
    long long n[3], d[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        n[i] = fx_sum2(0, qr[i], qr[i], qi[i], qi[i], half);
        long long cr = half;
        d[i] = 0;
        fx_mac(d[i], cr, a[i], a[i]);
        d[i] = fx_join(d[i], cr);
    }
    d[0] += n[0] + n[1];
    d[1] += n[0] + n[2];
    d[2] += n[1] + n[2];
    const double two_up = fx_unit(2 * up);
    const double c1 = 0.5 * two_up * (double)(d[0] + d[1] + d[2]);
    // u01 = -a2 q01 + q02 q12^*, u02 = -a1 q02 + q01 q12, u12 = -a0 q12 + q01^* q02
    long long ur[3], ui[3];
    {
        const fx_num ma0 = fx_minus(a[0]), ma1 = fx_minus(a[1]), ma2 = fx_minus(a[2]);
        const fx_num mi12 = fx_minus(qi[2]), mi01 = fx_minus(qi[0]);
        ur[0] = fx_sum2(fx_sum2(0, ma2, qr[0], qr[1], qr[2], half), qi[1], qi[2], {0, 0}, {0, 0}, half);
        ui[0] = fx_sum2(fx_sum2(0, ma2, qi[0], qi[1], qr[2], half), qr[1], mi12, {0, 0}, {0, 0}, half);
        ur[1] = fx_sum2(fx_sum2(0, ma1, qr[1], qr[0], qr[2], half), qi[0], mi12, {0, 0}, {0, 0}, half);
        ui[1] = fx_sum2(fx_sum2(0, ma1, qi[1], qr[0], qi[2], half), qi[0], qr[2], {0, 0}, {0, 0}, half);
        ur[2] = fx_sum2(fx_sum2(0, ma0, qr[2], qr[0], qr[1], half), qi[0], qi[1], {0, 0}, {0, 0}, half);
        ui[2] = fx_sum2(fx_sum2(0, ma0, qi[2], qr[0], qi[1], half), mi01, qr[1], {0, 0}, {0, 0}, half);
    }
    // Q^2 times 2^up as operands, and c0 = tr Q^3 / 3
    fx_num dx[3], vr[3], vi[3];
    long long t = 0, tc = half, t2 = 0, t2c = half;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        dx[i] = fx_operand(d[i] >> up);
        vr[i] = fx_operand(ur[i] >> up);
        vi[i] = fx_operand(ui[i] >> up);
        fx_mac(t, tc, a[i], dx[i]);
        fx_mac(t2, t2c, qr[i], vr[i]);
        fx_mac(t2, t2c, qi[i], vi[i]);
    }
    const double c0 = two_up * (1.0 / 3.0) * (double)(fx_join(t, tc) + 2 * fx_join(t2, t2c));
    const double w = c0 * c0, c2 = c1 * c1;
    const double a3 = fma(c1, c2, w), a4 = fma(c1, a3, 2.0 * w * c1);
    const double f2r = fma(a4, -1.0 / 3628800, fma(a3, 1.0 / 40320, fma(c2, -1.0 / 720, fma(c1, 1.0 / 24, -0.5))));
    const double f2i = c0 * fma(c2, 3.0 / 362880, fma(c1, -2.0 / 5040, 1.0 / 120));
    const double f1i = fma(a4, 1.0 / 362880, fma(a3, -1.0 / 5040, fma(c2, 1.0 / 120, fma(c1, -1.0 / 6, 1.0))));
    const double f1r = c0 * fma(fma(4.0 * c1, c2, w), -1.0 / 3628800, fma(c2, 3.0 / 40320, fma(c1, -2.0 / 720, 1.0 / 24)));
    const double f0r = w * fma(c2, -3.0 / 3628800, fma(c1, 2.0 / 40320, -1.0 / 720));
    const double f0i = c0 * fma(a3, 1.0 / 362880, fma(c2, -1.0 / 5040, fma(c1, 1.0 / 120, -1.0 / 6)));
    const fx_num g1r = fx_number(f1r, g, 0), g1i = fx_number(f1i, g, 0), g2r = fx_number(f2r, g, 0), g2i = fx_number(f2i, g, 0);
    const fx_num g0r = fx_number(f0r, g, up), g0i = fx_number(f0i, g, up);
    const long long f0re = ((long long)g0r.h << 29) + g0r.l, f0im = ((long long)g0i.h << 29) + g0i.l;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        fx_split<0>(fx_sum2(f0re, g1r, a[i], g2r, dx[i], half), o.rh[i][i], o.rl[i][i]);
        fx_split<0>(fx_sum2(f0im, g1i, a[i], g2i, dx[i], half), o.ih[i][i], o.il[i][i]);
        // off-diagonal pair: with A, D = f1 re q + f2 re u and C, B = f1 im q + f2 im u, m_ij = (A - B, D + C),
        // m_ji = (A + B, D - C)
        const int p = i == 2 ? 1 : 0, q = i == 0 ? 1 : 2;
        const long long A = fx_sum2(0, g1r, qr[i], g2r, vr[i], half), D = fx_sum2(0, g1i, qr[i], g2i, vr[i], half);
        const long long C = fx_sum2(0, g1r, qi[i], g2r, vi[i], half), Bv = fx_sum2(0, g1i, qi[i], g2i, vi[i], half);
        fx_split<0>(A - Bv, o.rh[p][q], o.rl[p][q]);
        fx_split<0>(D + C, o.ih[p][q], o.il[p][q]);
        fx_split<0>(A + Bv, o.rh[q][p], o.rl[q][p]);
        fx_split<0>(D - C, o.ih[q][p], o.il[q][p]);
    }
    return !g.bad() && 2.0 * c1 <= kFxExpMax;
}

// exp(X) - 1 as operands in units 2^(-58 - up): the form above, or, for larger X and where the caller needs it in
// FP64 (`general`), the series of expm_su3
__device__ __forceinline__ unsigned fx_exp_m1_su3(matx<3>& o, mat3<double>& e, const alg8<double>& x, bool general, fx_guard& g) {
    unsigned up;
    if (!fx_exp_su3(o, up, x) || general) {
        expm_su3<double, true>(e, x);
        up = fx_scale_of(e.e);
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) fx_take_entry<3>(o, i, j, e.e[i][j].re, e.e[i][j].im, g, up);
    }
    return up;
}

}  // namespace tgf
