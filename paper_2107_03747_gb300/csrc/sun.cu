// sun.cu -- the twisted Wilson flow and its observables for SU(N), N = 2, 3, 4, in FP64.
//
// The paper's coupling is defined for SU(N) on the l x l x (Nl) x (Nl) box with twist
// exp(2 pi i k / N) in the short plane (Sec. 1 and Sec. 3.1); its numbers are for N = 3, and its
// outlook (Sec. 5) is larger N.  This file is the generic-N form of the flow: the same
// definitions as the SU(3) kernels (twisted staples, Z = -P_ta(U Sigma) with the 1/N trace,
// Luscher's low-storage RK3, W' = exp(X) W, the clover G = -(i/8)(C - C^+), E, q and the twisted
// plaquette), written for N x N matrices in registers.  The exponential is a Taylor polynomial of
// degree 7-11 after scaling by 2^-s, evaluated with few products, then squared s times (SU(2):
// closed form; SU(3): the Cayley-Hamilton form of the SU(3) kernels).  Matrix products run in fixed point
// on the integer pipe (fixed.cuh); the FP64 forms of the products and of the exponential serve links outside
// its range.
//
// Storage per configuration and direction: N^2 double2 planes (matrix entries, row-major) of
// Vp sites; the RK3 accumulator X holds N^2 reals per link: the imaginary parts of the N
// diagonal entries, then real and imaginary parts of the entries above the diagonal.
#include <cuda_runtime.h>
#include <math_constants.h>
#include <stdint.h>

#include "expm.cuh"
#include "fixed.cuh"
#include "lattice.cuh"

namespace tgf {

namespace {

constexpr int kSunSites = 128;  // sites (threads) per block of the measurement

template <int N>
struct matN {
    cx<double> e[N][N];
};

template <int N>
__device__ __forceinline__ void zeroN(matN<N>& a) {
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = 0; j < N; ++j) a.e[i][j] = {0.0, 0.0};
}

// c (+)= a b, a b^+, a^+ b
template <int N, bool ACC>
__device__ __forceinline__ void nnN(matN<N>& c, const matN<N>& a, const matN<N>& b) {
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = 0; j < N; ++j) {
            double re = ACC ? c.e[i][j].re : 0.0, im = ACC ? c.e[i][j].im : 0.0;
#pragma unroll
            for (int k = 0; k < N; ++k) {
                re = fma(a.e[i][k].re, b.e[k][j].re, re);
                re = fma(-a.e[i][k].im, b.e[k][j].im, re);
                im = fma(a.e[i][k].re, b.e[k][j].im, im);
                im = fma(a.e[i][k].im, b.e[k][j].re, im);
            }
            c.e[i][j] = {re, im};
        }
}
template <int N, bool ACC>
__device__ __forceinline__ void ndN(matN<N>& c, const matN<N>& a, const matN<N>& b) {
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = 0; j < N; ++j) {
            double re = ACC ? c.e[i][j].re : 0.0, im = ACC ? c.e[i][j].im : 0.0;
#pragma unroll
            for (int k = 0; k < N; ++k) {
                re = fma(a.e[i][k].re, b.e[j][k].re, re);
                re = fma(a.e[i][k].im, b.e[j][k].im, re);
                im = fma(a.e[i][k].im, b.e[j][k].re, im);
                im = fma(-a.e[i][k].re, b.e[j][k].im, im);
            }
            c.e[i][j] = {re, im};
        }
}
template <int N, bool ACC>
__device__ __forceinline__ void dnN(matN<N>& c, const matN<N>& a, const matN<N>& b) {
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = 0; j < N; ++j) {
            double re = ACC ? c.e[i][j].re : 0.0, im = ACC ? c.e[i][j].im : 0.0;
#pragma unroll
            for (int k = 0; k < N; ++k) {
                re = fma(a.e[k][i].re, b.e[k][j].re, re);
                re = fma(a.e[k][i].im, b.e[k][j].im, re);
                im = fma(a.e[k][i].re, b.e[k][j].im, im);
                im = fma(-a.e[k][i].im, b.e[k][j].re, im);
            }
            c.e[i][j] = {re, im};
        }
}

template <int N>
__device__ __forceinline__ void scaleN(matN<N>& a, double zr, double zi) {
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = 0; j < N; ++j) {
            const double r = a.e[i][j].re, m = a.e[i][j].im;
            a.e[i][j] = {r * zr - m * zi, r * zi + m * zr};
        }
}

template <int N>
__device__ __forceinline__ void addN(matN<N>& a, const matN<N>& b) {
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = 0; j < N; ++j) {
            a.e[i][j].re += b.e[i][j].re;
            a.e[i][j].im += b.e[i][j].im;
        }
}

template <int N>
__device__ __forceinline__ void loadN(const double* __restrict__ base, int Vp, int dir, int s, matN<N>& u) {
    s = checked_site(s, Vp);
    const double2* q = reinterpret_cast<const double2*>(base) + (size_t)dir * N * N * Vp;
#pragma unroll
    for (int k = 0; k < N * N; ++k) {
        const double2 v = __ldg(q + (size_t)k * Vp + s);
        u.e[k / N][k % N] = {v.x, v.y};
    }
}
template <int N>
__device__ __forceinline__ void storeN(double* __restrict__ base, int Vp, int dir, int s, const matN<N>& u) {
    s = checked_site(s, Vp);
    double2* q = reinterpret_cast<double2*>(base) + (size_t)dir * N * N * Vp;
#pragma unroll
    for (int k = 0; k < N * N; ++k) q[(size_t)k * Vp + s] = make_double2(u.e[k / N][k % N].re, u.e[k / N][k % N].im);
}

// exp(2 pi i k / N)
template <int N>
__device__ __forceinline__ void centreN(int k, double& zr, double& zi) {
    sincospi(2.0 * k / N, &zi, &zr);
}

// exp(X) for anti-Hermitian X: X is scaled by 2^-s to ||Y||_F <= 1/5 and exp(Y) is replaced by
// its Taylor polynomial T_d of degree d, evaluated by Paterson and Stockmeyer's scheme (SIAM J.
// Comput. 2 (1973) 60) in blocks of B terms: with M = Y^B, T_d(Y) = B_0 + M (B_1 + M (B_2 + ...)),
// B_j = sum_{i<B} Y^i / (Bj+i)!, d = B NB - 1 for NB blocks.  B = 3 (Y^2, Y^3, then NB - 1 Horner
// products) for N <= 3; B = 2 (Y^2, then NB - 1 Horner products) for N = 4, which keeps one
// matrix fewer live.  The dropped tail is at most ||Y||^{d+1}/(d+1)! e^{||Y||}, so NB follows the
// norm: the smallest degree whose bound stays under 1.1e-17 (far below FP64 rounding of the
// unitary result):
//   B = 3:  d = 8 for ||Y|| <= 0.05,  d = 11 up to 0.2;
//   B = 2:  d = 7 for ||Y|| <= 0.028, d = 9 for <= 0.088, d = 11 up to 0.2.
// A flow step of eps = 0.01 has ||X||_F of a few 0.01, so it takes 4 matrix products where the
// plain series takes one per term (7-9); the result is then squared s times.
template <int N>
__device__ void expN(matN<N>& out, const matN<N>& X) {
    constexpr int B = N >= 4 ? 2 : 3;
    double n2 = 0.0;
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = 0; j < N; ++j) n2 += X.e[i][j].re * X.e[i][j].re + X.e[i][j].im * X.e[i][j].im;
    int s = 0;
    double sc = 1.0;
    while (n2 * sc * sc > 0.04 && s < 60) {
        sc *= 0.5;
        ++s;
    }
    n2 *= sc * sc;
    // blocks and 1/d!
    int NB;
    double ctop;
    if (B == 3) {
        if (n2 <= 0.05 * 0.05) { NB = 3; ctop = 1.0 / 40320.0; }
        else { NB = 4; ctop = 1.0 / 39916800.0; }
    } else {
        if (n2 <= 0.028 * 0.028) { NB = 4; ctop = 1.0 / 5040.0; }
        else if (n2 <= 0.088 * 0.088) { NB = 5; ctop = 1.0 / 362880.0; }
        else { NB = 6; ctop = 1.0 / 39916800.0; }
    }
    matN<N> Y, Y2, Y3, t;
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = 0; j < N; ++j) Y.e[i][j] = {X.e[i][j].re * sc, X.e[i][j].im * sc};
    nnN<N, false>(Y2, Y, Y);
    if constexpr (B == 3) nnN<N, false>(Y3, Y2, Y);
    const matN<N>& M = B == 3 ? Y3 : Y2;
    // dst = B_j, given ctop = 1/(Bj+B-1)!; returns 1/(Bj)!
    auto block = [&](matN<N>& dst, int jb, double ct) {
        double c0 = ct * double(B * jb + B - 1), c1 = ct, c2 = 0.0;
        if constexpr (B == 3) {
            c2 = ct;
            c1 = c0;
            c0 = c1 * double(B * jb + 1);
        }
#pragma unroll
        for (int i = 0; i < N; ++i)
#pragma unroll
            for (int j = 0; j < N; ++j) {
                cx<double> v = {c1 * Y.e[i][j].re + (i == j ? c0 : 0.0), c1 * Y.e[i][j].im};
                if constexpr (B == 3) {
                    v.re += c2 * Y2.e[i][j].re;
                    v.im += c2 * Y2.e[i][j].im;
                }
                dst.e[i][j] = v;
            }
        return c0;
    };
    // top block, then 1/(Bj-1)! = Bj / (Bj)! going down; each Horner step forms B_j first and
    // accumulates the product M (B_{j+1} + ...) onto it in the product's own FMAs
    ctop = block(out, NB - 1, ctop) * double(B * (NB - 1));
#pragma unroll 1
    for (int jb = NB - 2; jb >= 0; --jb) {
        ctop = block(t, jb, ctop) * double(B * jb);
        nnN<N, true>(t, M, out);
        out = t;
    }
#pragma unroll 1
    for (int k = 0; k < s; ++k) {
        t = out;
        nnN<N, false>(out, t, t);
    }
}

// SU(2): closed form.  X = i tau 1 + X0 with X0 traceless anti-Hermitian, X0^2 = -theta^2 1
// (theta^2 = a^2 + |b|^2 for X0 = [[i a, b], [-b*, -i a]]), so
// exp(X) = e^{i tau} (cos theta 1 + (sin theta / theta) X0).
template <>
__device__ void expN<2>(matN<2>& out, const matN<2>& X) {
    const double tau = 0.5 * (X.e[0][0].im + X.e[1][1].im);
    const double a = X.e[0][0].im - tau;
    const double br = X.e[0][1].re, bi = X.e[0][1].im;
    const double th = sqrt(a * a + br * br + bi * bi);
    const double c = cos(th), sn = th > 1e-30 ? sin(th) / th : 1.0;
    double er, ei;
    sincos(tau, &ei, &er);
    // M = c 1 + sn X0;  out = e^{i tau} M
    const cx<double> m00 = {c, sn * a}, m11 = {c, -sn * a};
    const cx<double> m01 = {sn * br, sn * bi}, m10 = {-sn * br, sn * bi};
    out.e[0][0] = {er * m00.re - ei * m00.im, er * m00.im + ei * m00.re};
    out.e[0][1] = {er * m01.re - ei * m01.im, er * m01.im + ei * m01.re};
    out.e[1][0] = {er * m10.re - ei * m10.im, er * m10.im + ei * m10.re};
    out.e[1][1] = {er * m11.re - ei * m11.im, er * m11.im + ei * m11.re};
}

// SU(3): the Cayley-Hamilton exponential of the SU(3) kernels (expm.cuh) on the 8 parameters of
// the traceless X (the stage builds X traceless; a trace at rounding level is dropped): a few
// dozen scalar operations instead of the polynomial's 4 matrix products.
template <>
__device__ void expN<3>(matN<3>& out, const matN<3>& X) {
    alg8<double> x;
    x.v[0] = X.e[0][0].im;
    x.v[1] = X.e[1][1].im;
    x.v[2] = X.e[0][1].re;
    x.v[3] = X.e[0][1].im;
    x.v[4] = X.e[0][2].re;
    x.v[5] = X.e[0][2].im;
    x.v[6] = X.e[1][2].re;
    x.v[7] = X.e[1][2].im;
    mat3<double> m;
    expm_su3<double, false>(m, x);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) out.e[i][j] = m.e[i][j];
}

// links for fixed.cuh: entry planes of double2
template <int N>
struct SunSrc {
    const double2* q;
    int Vp;
    __device__ __forceinline__ double2 get(int dir, int s, int i, int j, bool tr) const {
        s = checked_site(s, Vp);
        return __ldg(q + ((size_t)dir * N * N + (tr ? j * N + i : i * N + j)) * Vp + s);
    }
    static __device__ __forceinline__ void centre(int k, double& zr, double& zi) { centreN<N>(k, zr, zi); }
};

// Omega = U Sigma in FP64, for links whose staples leave the range of fixed.cuh and for weak ones (fx_rough)
template <int N>
__device__ __forceinline__ void native_omegaN(matN<N>& om, const CfgDesc& c, const double* __restrict__ base, int s, int mu,
                                              unsigned eb) {
    const int Vp = c.Vp;
    const int s_mp = fwd(c, eb, s, mu);
    const bool at_mu0 = (eb >> mu) & 1u;
    matN<N> sig, a, b, t;
    zeroN(sig);
#pragma unroll 1
    for (int dn = 1; dn < 4; ++dn) {
        const int nu = (mu + dn) & 3;
        const int s_nm = bwd(c, eb, s, nu);
        const int k = c.tw[mu * 4 + nu];
        double zr = 1.0, zi = 0.0;
        if (k != 0) centreN<N>(k, zr, zi);
        // forward staple Z*_{mu nu}(n) U_nu(n+mu) U_mu(n+nu)^+ U_nu(n)^+
        loadN<N>(base, Vp, nu, s_mp, a);
        loadN<N>(base, Vp, mu, fwd(c, eb, s, nu), b);
        ndN<N, false>(t, a, b);
        if (k != 0 && at_mu0 && ((eb >> nu) & 1u)) scaleN(t, zr, -zi);
        loadN<N>(base, Vp, nu, s, a);
        ndN<N, true>(sig, t, a);
        // backward staple Z_{mu nu}(n-nu) U_nu(n+mu-nu)^+ U_mu(n-nu)^+ U_nu(n-nu)
        loadN<N>(base, Vp, mu, s_nm, a);
        loadN<N>(base, Vp, nu, fwd(c, eb, s_nm, mu), b);
        nnN<N, false>(t, a, b);
        if (k != 0 && at_mu0 && ((eb >> (8 + nu)) & 1u)) scaleN(t, zr, -zi);
        loadN<N>(base, Vp, nu, s_nm, a);
        dnN<N, true>(sig, t, a);
    }
    loadN<N>(base, Vp, mu, s, a);
    nnN<N, false>(om, a, sig);
}

// exp(X) - 1 as an operand in units 2^(-58 - up), X traceless anti-Hermitian.  SU(3): fx_exp_m1_su3; SU(2):
// X^2 = -z 1, so exp(X) - 1 = (cos sqrt z - 1) + (sin sqrt z / sqrt z) X, the two
// functions by their power series in z up to z = 1/4 (the tail of the eighth term is below 1e-18).
template <int N>
__device__ __forceinline__ unsigned fx_exp_m1(matx<N>& o, const matN<N>& X, fx_guard& g) {
    if constexpr (N == 3) {
        const alg8<double> x = {{X.e[0][0].im, X.e[1][1].im, X.e[0][1].re, X.e[0][1].im, X.e[0][2].re, X.e[0][2].im,
                                 X.e[1][2].re, X.e[1][2].im}};
        mat3<double> e;
        return fx_exp_m1_su3(o, e, x, false, g);
    }
    matN<N> m;
    if constexpr (N == 2) {
        const double a = 0.5 * (X.e[0][0].im - X.e[1][1].im), br = X.e[0][1].re, bi = X.e[0][1].im;
        const double z = a * a + br * br + bi * bi;
        double cm1, sc;
        if (z <= 0.25) {
            // 1/k! for k = 2, 4, ... and 1, 3, ...
            constexpr double f[17] = {1.0, 1.0, 1.0 / 2, 1.0 / 6, 1.0 / 24, 1.0 / 120, 1.0 / 720, 1.0 / 5040, 1.0 / 40320,
                                      1.0 / 362880, 1.0 / 3628800, 1.0 / 39916800, 1.0 / 479001600, 1.0 / 6227020800.0,
                                      1.0 / 87178291200.0, 1.0 / 1307674368000.0, 1.0 / 20922789888000.0};
            cm1 = f[16];
            sc = f[15];
#pragma unroll
            for (int k = 7; k >= 1; --k) {
                cm1 = fma(-z, cm1, f[2 * k]);
                sc = fma(-z, sc, f[2 * k - 1]);
            }
            cm1 *= -z;
        } else {
            const double th = sqrt(z);
            double sn, cs;
            sincos(th, &sn, &cs);
            cm1 = cs - 1.0;
            sc = sn / th;
        }
        m.e[0][0] = {cm1, sc * a};
        m.e[1][1] = {cm1, -sc * a};
        m.e[0][1] = {sc * br, sc * bi};
        m.e[1][0] = {-sc * br, sc * bi};
    }
    const unsigned up = fx_scale_of(m.e);
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = 0; j < N; ++j) fx_take_entry<N>(o, i, j, m.e[i][j].re, m.e[i][j].im, g, up);
    return up;
}

// 1/k! in units 2^-58
__constant__ long long c_inv_fact[12] = {1ll << 58, 1ll << 58, (1ll << 58) / 2, (1ll << 58) / 6, (1ll << 58) / 24,
                                         (1ll << 58) / 120, (1ll << 58) / 720, (1ll << 58) / 5040, (1ll << 58) / 40320,
                                         (1ll << 58) / 362880, (1ll << 58) / 3628800, (1ll << 58) / 39916800};

// SU(4): the Taylor polynomial of expN (same degrees), in fixed point: Y and Y' = 2^up Y as operands, M = Y^2,
// T = B_1 + M (B_2 + ...) with B_j = 1/(2j)! + Y/(2j+1)!, then exp(Y) - 1 = Y + M T and, s times,
// exp(2Y) - 1 = 2 (exp(Y) - 1) + (exp(Y) - 1)^2.  M, the last product and the Y that is added to it carry the factor
// 2^up, so that the small matrix keeps its relative precision.
template <>
__device__ __forceinline__ unsigned fx_exp_m1<4>(matx<4>& o, const matN<4>& X, fx_guard& g) {
    constexpr int N = 4;
    double n2 = 0.0;
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = i; j < N; ++j) n2 += (i == j ? 1.0 : 2.0) * (X.e[i][j].re * X.e[i][j].re + X.e[i][j].im * X.e[i][j].im);
    int s = 0;
    while (n2 > 0.04 && s < 30) {
        n2 *= 0.25;
        ++s;
    }
    const int nb = n2 <= 0.028 * 0.028 ? 4 : n2 <= 0.088 * 0.088 ? 5 : 6;
    const double sc = __hiloint2double((1023 - s) << 20, 0);
    matN<N> Y;
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = 0; j < N; ++j) Y.e[i][j] = {X.e[i][j].re * sc, X.e[i][j].im * sc};
    const unsigned up = s > 0 ? 0u : fx_scale_of(Y.e);
    matx<N> y, m, t;
    matq<N> q;
    const long long half = fx_round();
    {
        matx<N> yu;
#pragma unroll
        for (int i = 0; i < N; ++i)
#pragma unroll
            for (int j = 0; j < N; ++j) {
                fx_take_entry<N>(y, i, j, Y.e[i][j].re, Y.e[i][j].im, g);
                fx_take_entry<N>(yu, i, j, Y.e[i][j].re, Y.e[i][j].im, g, up);
            }
        fx_mul_nn<N>(q, y, yu);
    }
    // q = 2^up Y^2; m = Y^2
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = 0; j < N; ++j) {
            fx_split<0>(q.re[i][j] >> up, m.rh[i][j], m.rl[i][j]);
            fx_split<0>(q.im[i][j] >> up, m.ih[i][j], m.il[i][j]);
        }
    matq<N> h;
    fx_zero(h);
#pragma unroll 1
    for (int jb = nb - 1; jb >= 1; --jb) {
        // h = B_jb + M t (t = 0 for the top block)
        const long long c0 = c_inv_fact[2 * jb], c1 = c_inv_fact[2 * jb + 1];
        int c1h, c1l;
        fx_split<0>(c1, c1h, c1l);
        const bool top = jb == nb - 1;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const vecx<N> r = fx_row(m, i), nr = fx_negated(r);
#pragma unroll
            for (int j = 0; j < N; ++j) {
                long long re = i == j ? c0 : 0, im = 0, rc = half, ic = half;
                fx_mad(re, rc, y.rh[i][j], y.rl[i][j], c1h, c1l);
                fx_mad(im, ic, y.ih[i][j], y.il[i][j], c1h, c1l);
                re = fx_join(re, rc);
                im = fx_join(im, ic);
                if (!top) fx_dot<N, false>(re, im, r, nr, fx_col(t, j));
                h.re[i][j] = re;
                h.im[i][j] = im;
            }
        }
        fx_operand_wide<N, 0>(t, h);
    }
    // exp(Y) - 1 = Y + M T in units 2^(-58 - up)
    matx<N> mu_;
    fx_operand_wide<N, 0>(mu_, q);
    fx_mul_nn<N>(h, mu_, t);
    if (up > 0) {  // Y = X, taken once more with the bits that up keeps
#pragma unroll
        for (int i = 0; i < N; ++i)
#pragma unroll
            for (int j = 0; j < N; ++j) fx_take_entry<N>(y, i, j, X.e[i][j].re, X.e[i][j].im, g, up);
    }
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = 0; j < N; ++j) {
            h.re[i][j] += ((long long)y.rh[i][j] << 29) + y.rl[i][j];
            h.im[i][j] += ((long long)y.ih[i][j] << 29) + y.il[i][j];
        }
    fx_operand_wide<N, 0>(o, h);
#pragma unroll 1
    for (int k = 0; k < s; ++k) {
        fx_mul_nn<N>(q, o, o);
#pragma unroll
        for (int i = 0; i < N; ++i)
#pragma unroll
            for (int j = 0; j < N; ++j) {
                h.re[i][j] = 2 * h.re[i][j] + q.re[i][j];
                h.im[i][j] = 2 * h.im[i][j] + q.im[i][j];
            }
        fx_operand_wide<N, 0>(o, h);
    }
    fx_check<N, 27>(h, g);
    return up;
}

// Whether the block's warps share operands: splitting a link costs 14 instructions per real entry, a shared one a
// 16-byte load per entry.  SU(3) 3 % and SU(4) 8 % faster (1103 -> 1065 us, 4.83 -> 4.44 ms for the case below),
// SU(2) 0.6 % slower.
template <int N>
constexpr bool kSunShares = N > 2;

// one RK3 stage for SU(N); block = 4 warps (one per direction) x 32 sites.  Matrix products in fixed point
// on the integer pipe (fixed.cuh), scalars in FP64, as the SU(3) kernels of stage64.cuh; all of it in FP64 kept
// that pipe 90-96 % busy.  Two steps and a measurement of 8 x 8x8x16x16 in SU(2): 4.08 ms before, 1.46 now; one
// step and a measurement of 4 x 6x6x24x24 in SU(4): 12.9 ms before, 4.16 now.
template <int N, int STAGE, int CAP>
__global__ void __launch_bounds__(128, N == 4 ? 2 : 3)
k_sun_stage(const __grid_constant__ BatchT<CAP> B, const double* __restrict__ w_in, double* __restrict__ w_out,
            double* __restrict__ acc) {
    const int mu = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int blk = blockIdx.x;
    if (blk >= B.nblk) return;
    const int ci = find_cfg(B, blk);
    const CfgDesc& c = B.c[ci];
    int s = (blk - c.blk0) * 32 + lane;
    const bool valid = s < c.V;  // the others take part in the barriers and store nothing
    if (!valid) s = 0;
    int xc[4];
    site_coords(c, s, xc);
    const unsigned eb = edge_bits(c, xc);
    const int Vp = c.Vp;
    const double* base = w_in + c.w_off;
    fx_guard g;
    SunSrc<N> src{reinterpret_cast<const double2*>(base), Vp};
    // the links at n and one step back in each direction, shared by the block's warps (kSunShares)
    constexpr bool SHARE = kSunShares<N>;
    extern __shared__ __align__(16) unsigned char s_links[];
    fx_shared<N>& links = *reinterpret_cast<fx_shared<N>*>(s_links);
    matx<N> u;
    bool all_near = false;
    if (SHARE) {
        bool rough = false;
#pragma unroll 1
        for (int m = mu; m < 8; m += 4) {
            fx_guard gl;
            fx_take_matrix<N, true>(u, src, mu, m < 4 ? s : bwd(c, eb, s, mu), false, gl);
            fx_share<N>(links, m, lane, u, gl);
            rough |= gl.rough();
        }
        all_near = !__syncthreads_or(rough);  // a block of weak links needs no fixed-point staples
    }
    auto own_link = [&]() {
        if (SHARE) fx_shared_link<N>(u, links, mu, lane);
        else fx_take_matrix<N, true>(u, src, mu, s, false, g);
    };
    matN<N> X;
    double x[N * N];  // Z, then X: diagonal imaginary parts, then (re, im) above the diagonal
    if (!all_near) {
        matq<N> sig, om;
        fx_zero(sig);
        fx_staples<N, true, SHARE>(sig, src, &links, lane, c, s, mu, eb, g, [](int, int, const matq<N>&) {});
        // Omega = U Sigma (units 2^-56); Z = -P_ta(Omega) = -(Omega - Omega^+)/2 + tr(Omega - Omega^+)/(2N)
        matx<N> sx;
        fx_operand_wide<N, 2>(sx, sig);
        own_link();
        fx_mul_nn<N>(om, u, sx);
        fx_check<N, 29>(om, g);
        long long tr = 0;
#pragma unroll
        for (int i = 0; i < N; ++i) tr += om.im[i][i];
        const double trim = (double)tr * (1.0 / N);
        int r = 0;
#pragma unroll
        for (int i = 0; i < N; ++i) x[r++] = 0x1p-56 * (trim - (double)om.im[i][i]);
#pragma unroll
        for (int i = 0; i < N; ++i)
#pragma unroll
            for (int j = i + 1; j < N; ++j) {
                x[r++] = 0x1p-57 * (double)(om.re[j][i] - om.re[i][j]);
                x[r++] = -0x1p-57 * (double)(om.im[i][j] + om.im[j][i]);
            }
    }
    if (SHARE) fx_shared_flags<N>(g, links, mu, lane);
    if (!valid) return;
    if (g.bad() || all_near || (!g.rough() && fx_near_staples<N>(src, c, eb, s, mu))) {
        g.top2 = 1;
        matN<N> t;
        native_omegaN<N>(t, c, base, s, mu, eb);
        double trim = 0.0;
#pragma unroll
        for (int i = 0; i < N; ++i) trim += t.e[i][i].im;
        trim /= N;
        int r = 0;
#pragma unroll
        for (int i = 0; i < N; ++i) x[r++] = -(t.e[i][i].im - trim);
#pragma unroll
        for (int i = 0; i < N; ++i)
#pragma unroll
            for (int j = i + 1; j < N; ++j) {
                x[r++] = -0.5 * (t.e[i][j].re - t.e[j][i].re);
                x[r++] = -0.5 * (t.e[i][j].im + t.e[j][i].im);
            }
    }
    const double h = c.h;
    double* xb = acc + c.x_off + (size_t)mu * N * N * Vp;
#pragma unroll
    for (int q = 0; q < N * N; ++q) {
        double v;
        if (STAGE == 1) v = 0.25 * h * x[q];
        else if (STAGE == 2) v = (8.0 / 9.0) * h * x[q] - (17.0 / 9.0) * xb[(size_t)q * Vp + s];
        else v = 0.75 * h * x[q] - xb[(size_t)q * Vp + s];
        x[q] = v;
        if (STAGE != 3) xb[(size_t)q * Vp + s] = v;
    }
    int r = 0;
#pragma unroll
    for (int i = 0; i < N; ++i) X.e[i][i] = {0.0, x[r++]};
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = i + 1; j < N; ++j) {
            X.e[i][j] = {x[r], x[r + 1]};
            X.e[j][i] = {-x[r], x[r + 1]};
            r += 2;
        }
    matx<N> ex;
    // (left out where FP64 follows only for SU(4): its six products; the branch costs SU(3) 7 % and SU(2) 3 %)
    const unsigned up = N == 4 && g.bad() ? 0u : fx_exp_m1<N>(ex, X, g);
    matN<N> w;
    loadN<N>(base, Vp, mu, s, w);
    if (g.bad()) {
        matN<N> e, a = w;
        expN<N>(e, X);
        nnN<N, false>(w, e, a);
    } else {
        // W' = W + (exp(X) - 1) W, rounded once onto W
        matq<N> d;
        if (SHARE) own_link();
        fx_mul_nn<N>(d, ex, u);
        const double unit = fx_unit(up);
#pragma unroll
        for (int i = 0; i < N; ++i)
#pragma unroll
            for (int j = 0; j < N; ++j) {
                w.e[i][j].re = fma((double)d.re[i][j], unit, w.e[i][j].re);
                w.e[i][j].im = fma((double)d.im[i][j], unit, w.e[i][j].im);
            }
    }
    storeN<N>(w_out + c.w_off, Vp, mu, s, w);
}

// C = sum of the four twisted leaves of the plane (mu, nu) at site s (Sec. 3.1, eq. gmunu), and
// Re Tr[Z* P_{mu nu}(n)], the first leaf's trace.  Leaf by leaf, a product of four links from the left,
// each read as it is or as its adjoint, so that one product in a loop serves all twelve:
//   L1 = Z*(n)       U_mu(n)      U_nu(n+mu)       U_mu(n+nu)^+    U_nu(n)^+
//   L2 = Z*(n-nu)    U_nu(n-nu)^+ U_mu(n-nu)       U_nu(n-nu+mu)   U_mu(n)^+
//   L3 = Z*(n-mu)    U_nu(n)      U_mu(n-mu+nu)^+  U_nu(n-mu)^+    U_mu(n-mu)
//   L4 = Z*(n-mu-nu) U_mu(n-mu)^+ U_nu(n-mu-nu)^+  U_mu(n-mu-nu)   U_nu(n-nu)
// In bytes of a word, link k of the leaf: bit 0 the direction (0 mu, 1 nu), bit 1 adjoint, bits 2-5 the site of
// the table below.
constexpr unsigned leaf_link(int dir, int adj, int site) { return (unsigned)(dir | adj << 1 | site << 2); }
constexpr unsigned leaf_word(unsigned a, unsigned b, unsigned c, unsigned d) { return a | b << 8 | c << 16 | d << 24; }
// sites: 0 n, 1 n+mu, 2 n+nu, 3 n-nu, 4 n-nu+mu, 5 n-mu, 6 n-mu+nu, 7 n-mu-nu
static __constant__ unsigned c_leaf[4] = {
    leaf_word(leaf_link(0, 0, 0), leaf_link(1, 0, 1), leaf_link(0, 1, 2), leaf_link(1, 1, 0)),
    leaf_word(leaf_link(1, 1, 3), leaf_link(0, 0, 3), leaf_link(1, 0, 4), leaf_link(0, 1, 0)),
    leaf_word(leaf_link(1, 0, 0), leaf_link(0, 1, 6), leaf_link(1, 1, 5), leaf_link(0, 0, 5)),
    leaf_word(leaf_link(0, 1, 5), leaf_link(1, 1, 7), leaf_link(0, 0, 7), leaf_link(1, 0, 3))};

// where the corner of leaf l touches the twisted corner (bits of edge_bits: x = 0 at n, x = 1 one step back)
__device__ __forceinline__ bool leaf_twisted(unsigned eb, int mu, int nu, int leaf) {
    return ((eb >> ((leaf & 2 ? 8 : 0) + mu)) & 1u) && ((eb >> ((leaf & 1 ? 8 : 0) + nu)) & 1u);
}
__device__ __forceinline__ int leaf_site(const CfgDesc& c, unsigned eb, int s, int mu, int nu, unsigned w) {
    const int k = (int)(w >> 2) & 15;
    if (k == 1 || k == 4) s = fwd(c, eb, s, mu);
    if (k >= 5) s = bwd(c, eb, s, mu);
    if (k == 2 || k == 6) s = fwd(c, eb, s, nu);
    if (k == 3 || k == 4 || k == 7) s = bwd(c, eb, s, nu);
    return s;
}

template <int N>
__device__ __forceinline__ void native_leaves(matN<N>& C, double& retr, const double* __restrict__ base, const CfgDesc& c, int s,
                                              unsigned eb, int mu, int nu) {
    zeroN(C);
    retr = 0.0;
    const int k = c.tw[mu * 4 + nu];
#pragma unroll 1
    for (int leaf = 0; leaf < 4; ++leaf) {
        unsigned w = c_leaf[leaf];
        matN<N> t, b, q;
        auto take = [&](matN<N>& o) {
            loadN<N>(base, c.Vp, w & 1 ? nu : mu, leaf_site(c, eb, s, mu, nu, w & 0xffu), q);
            const bool adj = w & 2;
#pragma unroll
            for (int i = 0; i < N; ++i)
#pragma unroll
                for (int j = 0; j < N; ++j)
                    o.e[i][j] = adj ? cx<double>{q.e[j][i].re, -q.e[j][i].im} : q.e[i][j];
        };
        take(t);
        if (k != 0 && leaf_twisted(eb, mu, nu, leaf)) {
            double zr, zi;
            centreN<N>(k, zr, zi);
            scaleN(t, zr, -zi);
        }
#pragma unroll 1
        for (int m = 1; m < 4; ++m) {
            w >>= 8;
            take(b);
            nnN<N, false>(q, t, b);
            t = q;
        }
        if (leaf == 0)
#pragma unroll
            for (int i = 0; i < N; ++i) retr += t.e[i][i].re;
        addN(C, t);
    }
}

// The same in fixed point, two leaves at a time: with F, B the staples of U_mu in the plane, L1 + L2^+ goes with
// U_mu(n) (F - B) and L3 + L4^+ with (F - B) U_mu at n - mu (C - C^+ needs no more), so that a plane takes 10 products
// instead of 12 and four instead of sixteen links more than once.  Both halves are one loop body: the first
// is formed transposed.  ah: C - C^+ in units 2^-58, diagonal imaginary parts, then (re, im) above the diagonal; retr: Re
// Tr[Z* P(n)], up to 4 N^2, in units 2^(kTraceShift<N> - 58).  |F| and |F - B| are below 2 and |D| below 4 or the guard is
// set.  Every thread of the block takes part.
template <int N>
constexpr int kTraceShift = N - 2;  // 2 N^2 products of a link and F in these units stay below 2^62.2
template <int N>
__device__ __forceinline__ void fx_clover(long long (&ah)[N * N], long long& retr, const SunSrc<N>& src, const CfgDesc& c, int s,
                                          unsigned eb, int mu, int nu, fx_guard& g) {
    const int q0 = 2 * ((nu - mu - 1) & 3);
#pragma unroll
    for (int r = 0; r < N * N; ++r) ah[r] = 0;
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
        const int n = h ? bwd(c, eb, s, mu) : s;
        int xc[4];
        site_coords(c, n, xc);
        matq<N> k;
        fx_zero(k);
        fx_staples<N, true, false>(k, src, nullptr, 0, c, n, mu, edge_bits(c, xc), g, [&](int back, int, matq<N>& sum) {
            if (back) return;
            fx_check<N, 27>(sum, g);
            if (h == 0) {
                long long hh = 0;
#pragma unroll
                for (int i = 0; i < N; ++i) {
                    long long cr = fx_round<2 * N>();
#pragma unroll
                    for (int j = 0; j < N; ++j) {
                        int rh, rl, ih, il, fh, fl;
                        const double2 x = src.get(mu, n, i, j, false);
                        fx_take(x.x, rh, rl, g);
                        fx_take(x.y, ih, il, g, 0, -1);
                        fx_split<kTraceShift<N>, true>(sum.re[j][i], fh, fl);
                        fx_mad(hh, cr, rh, rl, fh, fl);
                        fx_split<kTraceShift<N>, true>(sum.im[j][i], fh, fl);
                        fx_mad(hh, cr, ih, il, fh, fl);
                    }
                    hh = fx_join(hh, cr);
                }
                retr = hh;
            }
#pragma unroll
            for (int i = 0; i < N; ++i)
#pragma unroll
                for (int j = 0; j < N; ++j) {
                    sum.re[i][j] = -sum.re[i][j];
                    sum.im[i][j] = -sum.im[i][j];
                }
        }, q0, q0 + 2);
        // k = B - F; d = (B - F) U at n - mu, the transpose of U (B - F) at n
        fx_check<N, 27>(k, g);
        if (h == 0) fx_transpose(k);
        matx<N> kx, u;
        matq<N> d;
        fx_operand_wide<N, 0>(kx, k);
        fx_take_matrix<N, true>(u, src, mu, n, h == 0, g);
        fx_mul_nn<N>(d, kx, u);
        fx_check<N, 28>(d, g);
        int r = 0;
#pragma unroll
        for (int i = 0; i < N; ++i) ah[r++] -= 2 * d.im[i][i];
#pragma unroll
        for (int i = 0; i < N; ++i)
#pragma unroll
            for (int j = i + 1; j < N; ++j) {
                const long long re = d.re[i][j] - d.re[j][i];
                ah[r++] += h ? -re : re;
                ah[r++] -= d.im[i][j] + d.im[j][i];
            }
    }
}

// Whether the 12 links of a plane's leaves are near 0 and +-1 (fx_rough): its clover is formed in FP64 then (Re Tr[Z* P],
// of the size of N, stays as it is).
template <int N>
__device__ __forceinline__ bool weak_plane(const SunSrc<N>& src, const CfgDesc& c, unsigned eb, int s, int mu, int nu) {
#pragma unroll 1
    for (int q = 0; q < 12; ++q) {
        // direction a at n and n - a, each at 0, + and - one step of the other one
        const int a = q & 1 ? nu : mu, b = q & 1 ? mu : nu, k = q >> 2;
        int t = k == 1 ? fwd(c, eb, s, b) : k == 2 ? bwd(c, eb, s, b) : s;
        if (q & 2) t = bwd(c, eb, t, a);
        if (!fx_near<N>(src, a, t)) return false;
    }
    return true;
}

// Re Tr[A B] for Hermitian A, B
template <int N>
__device__ __forceinline__ double retr_prod(const matN<N>& A, const matN<N>& B) {
    double v = 0.0;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        v += A.e[i][i].re * B.e[i][i].re;
#pragma unroll
        for (int k = i + 1; k < N; ++k) v += 2.0 * (A.e[i][k].re * B.e[i][k].re + A.e[i][k].im * B.e[i][k].im);
    }
    return v;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// per-site E, q, p, s summed over each block of kSunSites sites (fixed order).  Bound by the integer pipe and latency: SU(2)
// fits 4 blocks on an SM (two steps and a measurement of 8 x 8x8x16x16 1.49 -> 1.45 ms), SU(3) 3
// (1.02 -> 0.99 for one step and a measurement of 4 x 6x6x18x18), SU(4) 2 (3 spill: 4.30 -> 4.54 ms on 6x6x24x24).  With the
// leaves multiplied out one by one, 12 products a plane, these took 1.51, 1.07 and 4.41.
template <int N, int CAP>
__global__ void __launch_bounds__(kSunSites, N == 2 ? 4 : N == 3 ? 3 : 2)
k_sun_measure(const __grid_constant__ BatchT<CAP> B, const double* __restrict__ w, double* __restrict__ partial,
              int traceless) {
    __shared__ double red[kSunSites / 32][4];
    const int blk = blockIdx.x;
    if (blk >= B.nblk) return;
    const int ci = find_cfg(B, blk);
    const CfgDesc& c = B.c[ci];
    const int blk_site = (blk - c.blk0) * kSunSites + threadIdx.x;
    double e = 0.0, q = 0.0, p = 0.0, sa = 0.0;
    {
        const bool inside = blk_site < c.V;  // the others take part in the barriers
        const int s = inside ? blk_site : 0;
        int xc[4];
        site_coords(c, s, xc);
        const unsigned eb = edge_bits(c, xc);
        const double* base = w + c.w_off;
        const SunSrc<N> src{reinterpret_cast<const double2*>(base), c.Vp};
        matN<N> G0;  // the first plane of a pair
#pragma unroll 1
        for (int pl = 0; pl < 6; ++pl) {
            // planes in pairs (01, 23), (02, 13), (03, 12) with the signs of eq. qlatt
            const int mu = (int)(0x020101u >> (4 * (5 - pl))) & 3, nu = (int)(0x132332u >> (4 * (5 - pl))) & 3;
            fx_guard g;
            matN<N> G;
            double retr, dev;
            {
                long long ah[N * N], tr;
                fx_clover<N>(ah, tr, src, c, s, eb, mu, nu, g);
                constexpr double unit = 0x1p-58 * (1 << kTraceShift<N>);
                retr = (double)tr * unit;
                dev = (double)(((long long)N << (kFxBits - kTraceShift<N>)) - tr) * unit;
                // G = -(i/8)(C - C^+): G_jk = -(i/8)(C_jk - conj(C_kj))
                int r = 0;
#pragma unroll
                for (int i = 0; i < N; ++i) G.e[i][i] = {(double)ah[r++] * 0x1p-61, 0.0};
#pragma unroll
                for (int i = 0; i < N; ++i)
#pragma unroll
                    for (int j = i + 1; j < N; ++j) {
                        G.e[i][j] = {(double)ah[r + 1] * 0x1p-61, -(double)ah[r] * 0x1p-61};
                        r += 2;
                    }
            }
            if (g.bad() || (!g.rough() && weak_plane<N>(src, c, eb, s, mu, nu))) {
                matN<N> C;
                double rt;
                native_leaves<N>(C, rt, base, c, s, eb, mu, nu);
                if (g.bad()) {
                    retr = rt;
                    dev = N - rt;
                }
#pragma unroll
                for (int i = 0; i < N; ++i)
#pragma unroll
                    for (int j = i; j < N; ++j)
                        G.e[i][j] = {(C.e[i][j].im + C.e[j][i].im) / 8.0, -(C.e[i][j].re - C.e[j][i].re) / 8.0};
            }
            if (traceless) {
                double tr = 0.0;
#pragma unroll
                for (int i = 0; i < N; ++i) tr += G.e[i][i].re;
                tr /= N;
#pragma unroll
                for (int i = 0; i < N; ++i) G.e[i][i].re -= tr;
            }
            e += retr_prod(G, G);
            if (pl & 1) q += (pl == 3 ? -1.0 : 1.0) * retr_prod(G0, G);
            else G0 = G;
            p += retr / N;
            sa += dev;
        }
        q *= 1.0 / (4.0 * CUDART_PI * CUDART_PI);
        if (!inside) e = q = p = sa = 0.0;
    }
    e = warp_sum(e);
    q = warp_sum(q);
    p = warp_sum(p);
    sa = warp_sum(sa);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) {
        red[warp][0] = e;
        red[warp][1] = q;
        red[warp][2] = p;
        red[warp][3] = sa;
    }
    __syncthreads();
    if (threadIdx.x < 4) {
        double v = 0.0;
        for (int i = 0; i < kSunSites / 32; ++i) v += red[i][threadIdx.x];
        partial[(size_t)blk * 4 + threadIdx.x] = v;
    }
}

// per configuration: sum of its block partials in block order -> {t, E, Q, P, S}
template <int CAP>
__global__ void __launch_bounds__(256) k_sun_reduce(const __grid_constant__ BatchT<CAP> B, const double* __restrict__ partial,
                                                    double* __restrict__ obs) {
    __shared__ double red[4][256];
    const CfgDesc& c = B.c[blockIdx.x];
    const int nb = (c.V + kSunSites - 1) / kSunSites;
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    for (int i = threadIdx.x; i < nb; i += 256)
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] += partial[(size_t)(c.blk0 + i) * 4 + k];
#pragma unroll
    for (int k = 0; k < 4; ++k) red[k][threadIdx.x] = v[k];
    __syncthreads();
    for (int wdt = 128; wdt > 0; wdt >>= 1) {
        if (threadIdx.x < wdt)
#pragma unroll
            for (int k = 0; k < 4; ++k) red[k][threadIdx.x] += red[k][threadIdx.x + wdt];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        double* o = obs + (size_t)c.o_off * 5;
        o[0] = c.h;
        o[1] = red[0][0] / c.V;
        o[2] = red[1][0];
        o[3] = red[2][0] / (6.0 * c.V);
        o[4] = red[3][0];
    }
}

// canonical [site][mu][N][N] complex <-> storage planes
template <int N, int CAP, bool TO_STORAGE>
__global__ void k_sun_layout(const __grid_constant__ BatchT<CAP> B, double* __restrict__ canon, double* __restrict__ w) {
    const int blk = blockIdx.x;
    if (blk >= B.nblk) return;
    const int ci = find_cfg(B, blk);
    const CfgDesc& c = B.c[ci];
    const int s = (blk - c.blk0) * 128 + threadIdx.x;
    if (s >= c.V) return;
    double2* q = reinterpret_cast<double2*>(w + c.w_off);
    double2* cn = reinterpret_cast<double2*>(canon + c.m_off) + (size_t)s * 4 * N * N;
#pragma unroll
    for (int mu = 0; mu < 4; ++mu)
#pragma unroll
        for (int k = 0; k < N * N; ++k) {
            if (TO_STORAGE) q[((size_t)mu * N * N + k) * c.Vp + s] = cn[mu * N * N + k];
            else cn[mu * N * N + k] = q[((size_t)mu * N * N + k) * c.Vp + s];
        }
}

template <int CAP>
BatchT<CAP> shrink(const Batch& B) {
    BatchT<CAP> b;
    b.ncfg = B.ncfg;
    b.nblk = B.nblk;
    for (int i = 0; i < B.ncfg; ++i) b.c[i] = B.c[i];
    return b;
}

template <int N, int CAP>
void sun_stage_cap(int stage, const Batch& B, const double* w_in, double* w_out, double* acc, cudaStream_t st) {
    const BatchT<CAP> b = shrink<CAP>(B);
    auto launch = [&](auto kernel) {
        constexpr int bytes = kSunShares<N> ? (int)sizeof(fx_shared<N>) : 0;
        // a failure is the launch's to report
        if (bytes > 48 * 1024) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        kernel<<<B.nblk, 128, bytes, st>>>(b, w_in, w_out, acc);
    };
    if (stage == 1) launch(k_sun_stage<N, 1, CAP>);
    else if (stage == 2) launch(k_sun_stage<N, 2, CAP>);
    else launch(k_sun_stage<N, 3, CAP>);
}

template <int N, int CAP>
void sun_measure_cap(const Batch& Bm, const Batch& Br, const double* w, double* partial, double* obs, int traceless,
                     cudaStream_t st) {
    const BatchT<CAP> bm = shrink<CAP>(Bm), br = shrink<CAP>(Br);
    k_sun_measure<N, CAP><<<Bm.nblk, kSunSites, 0, st>>>(bm, w, partial, traceless);
    k_sun_reduce<CAP><<<Br.ncfg, 256, 0, st>>>(br, partial, obs);
}

template <int N, int CAP>
void sun_layout_cap(bool to_storage, const Batch& B, double* canon, double* w, cudaStream_t st) {
    const BatchT<CAP> b = shrink<CAP>(B);
    if (to_storage) k_sun_layout<N, CAP, true><<<B.nblk, 128, 0, st>>>(b, canon, w);
    else k_sun_layout<N, CAP, false><<<B.nblk, 128, 0, st>>>(b, canon, w);
}

template <int N>
void sun_dispatch(int op, int stage, bool to_storage, const Batch& B, const Batch& B2, const double* a, double* b,
                  double* c, double* d, int flag, cudaStream_t st) {
    const bool small = B.ncfg <= kSmallCap;
    if (op == 0) {
        if (small) sun_stage_cap<N, kSmallCap>(stage, B, a, b, c, st);
        else sun_stage_cap<N, kMaxCfg>(stage, B, a, b, c, st);
    } else if (op == 1) {
        if (small) sun_measure_cap<N, kSmallCap>(B, B2, a, c, d, flag, st);
        else sun_measure_cap<N, kMaxCfg>(B, B2, a, c, d, flag, st);
    } else {
        if (small) sun_layout_cap<N, kSmallCap>(to_storage, B, c, b, st);
        else sun_layout_cap<N, kMaxCfg>(to_storage, B, c, b, st);
    }
}

void sun_any(int N, int op, int stage, bool to_storage, const Batch& B, const Batch& B2, const double* a, double* b,
             double* c, double* d, int flag, cudaStream_t st) {
    if (N == 2) sun_dispatch<2>(op, stage, to_storage, B, B2, a, b, c, d, flag, st);
    else if (N == 3) sun_dispatch<3>(op, stage, to_storage, B, B2, a, b, c, d, flag, st);
    else sun_dispatch<4>(op, stage, to_storage, B, B2, a, b, c, d, flag, st);
}

}  // namespace

void launch_sun_stage(int N, int stage, const Batch& B, const double* w_in, double* w_out, double* acc,
                      cudaStream_t st) {
    sun_any(N, 0, stage, false, B, B, w_in, w_out, acc, nullptr, 0, st);
}

void launch_sun_measure(int N, const Batch& Bm, const Batch& Br, const double* w, double* partial, double* obs,
                        int traceless, cudaStream_t st) {
    sun_any(N, 1, 0, false, Bm, Br, w, nullptr, partial, obs, traceless, st);
}

void launch_sun_layout(int N, bool to_storage, const Batch& B, double* canon, double* w, cudaStream_t st) {
    sun_any(N, 2, 0, to_storage, B, B, nullptr, w, canon, nullptr, 0, st);
}

TGF_CHECK_WORD(sun)

}  // namespace tgf
