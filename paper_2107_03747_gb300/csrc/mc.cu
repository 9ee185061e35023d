// mc.cu -- twisted hybrid Monte Carlo update of FP64 link fields: Cabibbo-Marinari heat-bath
// and over-relaxation in the three SU(2) subgroups, one checkerboard pass per launch.
//
// Ensembles of the twisted Wilson action S_W = 3b sum_n sum_{mu!=nu} Tr[1 - Z* P] (Sec. 3.1) are
// generated with one heat-bath sweep followed by L~ over-relaxation sweeps (the hybrid
// algorithm the paper cites).  With beta = 18 b the weight of one link U = U_mu(n) is
// exp((beta/3) Re Tr[U Sigma]), Sigma its twisted staple sum.  For the SU(2) block (i, j) of
// W = U Sigma, with SU(2)-proportional part k v (v in SU(2)):
//   heat-bath        R = X v^+, X drawn with density exp(alpha X0) dHaar, alpha = 2 beta k / 3
//   over-relaxation  R = (v^+)^2                      (keeps Re Tr[U Sigma])
// and U <- R U.  X0 comes from Kennedy-Pendleton's sampler (alpha > 2) or Creutz's (otherwise).
//
// Thread mapping: one thread per link (n, mu) of one parity; a launch updates every link of
// direction mu on the sites with x0+x1+x2+x3 = parity (mod 2).  Their staples contain only links
// of the other directions or of the other parity, so the in-place update is race-free and equal
// to any sequential order inside the pass.
//
// Random numbers are counter-based: draw = SplitMix64 output function of
// key + (counter + 1) * 0x9E3779B97F4A7C15, u = ((x >> 11) + 1) 2^-53 in (0, 1], with
// key = the same hash of (seed, configuration index) and counter
// (((sweep * 4 + mu) * V + site) * 3 + subgroup) * 260 + slot; slots 4a..4a+3 serve rejection
// attempt a < 64, slots 256 and 257 the direction of X.  A subgroup whose 64 attempts are all
// rejected is left unchanged.
#include <cuda_runtime.h>
#include <stdint.h>

#include "fixed.cuh"
#include "lattice.cuh"

namespace tgf {

namespace {

constexpr uint64_t kGolden = 0x9E3779B97F4A7C15ull;
constexpr int kSlots = 260;
constexpr int kAttempts = 64;
constexpr int kMcThreads = 128;

__device__ __forceinline__ uint64_t mix64(uint64_t z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
__device__ __forceinline__ uint64_t hash64(uint64_t key, uint64_t counter) { return mix64(key + (counter + 1) * kGolden); }
__device__ __forceinline__ double draw(uint64_t key, uint64_t counter) {
    return (double)((hash64(key, counter) >> 11) + 1) * 0x1.0p-53;  // at most 2^53: exact
}

struct quat {
    double a0, a1, a2, a3;
};
__device__ __forceinline__ quat qmul(const quat& a, const quat& b) {
    // (a0 + i a.s)(b0 + i b.s) = a0 b0 - a.b + i (a0 b + b0 a - a x b).s
    return {a.a0 * b.a0 - (a.a1 * b.a1 + a.a2 * b.a2 + a.a3 * b.a3),
            a.a0 * b.a1 + b.a0 * a.a1 - (a.a2 * b.a3 - a.a3 * b.a2),
            a.a0 * b.a2 + b.a0 * a.a2 - (a.a3 * b.a1 - a.a1 * b.a3),
            a.a0 * b.a3 + b.a0 * a.a3 - (a.a1 * b.a2 - a.a2 * b.a1)};
}
__device__ __forceinline__ quat qconj(const quat& a) { return {a.a0, -a.a1, -a.a2, -a.a3}; }

// X0 with density sqrt(1 - X0^2) exp(alpha X0) on [-1, 1]; false when every attempt is rejected
__device__ bool sample_x0(double alpha, uint64_t key, uint64_t c0, double& x0) {
    const bool kp = alpha > 2.0;
    const double e2a = kp ? 0.0 : exp(-2.0 * alpha);
    const double inv = 0.5 / alpha;
#pragma unroll 1
    for (int a = 0; a < kAttempts; ++a) {
        const uint64_t c = c0 + 4 * a;
        const double r1 = draw(key, c), r2 = draw(key, c + 1);
        if (kp) {
            // Kennedy-Pendleton: lambda^2 = -(ln r1 + cos^2(2 pi r2) ln r3) / (2 alpha)
            const double r3 = draw(key, c + 2), r4 = draw(key, c + 3);
            const double cs = cospi(2.0 * r2);
            const double lam2 = -__dadd_rn(log(r1), __dmul_rn(__dmul_rn(cs, cs), log(r3))) * inv;
            if (__dmul_rn(r4, r4) <= 1.0 - lam2) {
                x0 = 1.0 - 2.0 * lam2;
                return true;
            }
        } else {
            // Creutz: X0 = 1 + ln(e^{-2 alpha} + (1 - e^{-2 alpha}) r1) / alpha, kept with probability sqrt(1 - X0^2)
            const double xc = alpha < 1e-8 ? 2.0 * r1 - 1.0
                                           : 1.0 + log(__dadd_rn(e2a, __dmul_rn(1.0 - e2a, r1))) / alpha;
            if (__dmul_rn(r2, r2) <= 1.0 - __dmul_rn(xc, xc)) {
                x0 = xc;
                return true;
            }
        }
    }
    return false;
}

// Omega = U_mu(n) Sigma_mu(n) in FP64, for links whose staples leave the range of fixed.cuh.  Weak links (fx_rough) stay in
// fixed point here: every call begins with a heat-bath pass, whose sqrt(1 - x0^2) has a relative error of 2^-53 / amp^2
// in FP64 on links of amplitude amp, more than the fixed-point staples' 2^-58 / amp at any amp.
__device__ __forceinline__ void native_omega(mat3<double>& om, const double* __restrict__ base, int Vp, const CfgDesc& c, int s,
                                             unsigned eb, int mu) {
    auto link = [&](int dir, int site, mat3<double>& u) { Store<P64>::load(base + (size_t)dir * 18 * Vp, Vp, site, u); };
    mat3<double> sig, a, b, t, f;
    set_zero(sig);
    const int s_mp = fwd(c, eb, s, mu);
    const bool at_mu0 = (eb >> mu) & 1u;
#pragma unroll 1
    for (int dn = 1; dn < 4; ++dn) {
        const int nu = (mu + dn) & 3;
        const int s_nm = bwd(c, eb, s, nu);
        const int k = c.tw[mu * 4 + nu];
        double zr = 1.0, zi = 0.0;
        if (k != 0) centre<double>(k, zr, zi);
        // forward: Z*_{mu nu}(n) U_nu(n+mu) U_mu(n+nu)^+ U_nu(n)^+
        link(nu, s_mp, a);
        link(mu, fwd(c, eb, s, nu), b);
        mul_nd(t, a, b);
        link(nu, s, a);
        mul_nd(f, t, a);
        if (k != 0 && at_mu0 && ((eb >> nu) & 1u)) scale_cx(f, zr, -zi);
        add_to(sig, f);
        // backward: Z_{mu nu}(n-nu) U_nu(n+mu-nu)^+ U_mu(n-nu)^+ U_nu(n-nu)
        link(mu, s_nm, a);
        link(nu, fwd(c, eb, s_nm, mu), b);
        mul_nn(t, a, b);
        link(nu, s_nm, a);
        mul_dn(f, t, a);
        if (k != 0 && at_mu0 && ((eb >> (8 + nu)) & 1u)) scale_cx(f, zr, zi);
        add_to(sig, f);
    }
    link(mu, s, a);
    mul_nn(om, a, sig);
}

// R as a 2x2 matrix [[r00, r01], [-r01^*, r00^*]] with r00 = R0 + i R3, r01 = R2 + i R1, acting on rows i, j
struct rot2 {
    cx<double> a, b;  // r00, r01
};
__device__ __forceinline__ cx<double> rot_i(const rot2& R, const cx<double>& p, const cx<double>& q) {
    return {R.a.re * p.re - R.a.im * p.im + (R.b.re * q.re - R.b.im * q.im),
            R.a.re * p.im + R.a.im * p.re + (R.b.re * q.im + R.b.im * q.re)};
}
__device__ __forceinline__ cx<double> rot_j(const rot2& R, const cx<double>& p, const cx<double>& q) {
    return {-R.b.re * p.re - R.b.im * p.im + (R.a.re * q.re + R.a.im * q.im),
            -R.b.re * p.im + R.b.im * p.re + (R.a.re * q.im - R.a.im * q.re)};
}

// The update of the SU(2) block x (twice its SU(2)-proportional part): over-relaxation R = (v^+)^2 or a
// heat-bath draw R = X v^+, x = |x| v.
template <int OVERRELAX>
__device__ __forceinline__ rot2 draw_rotation(const quat& x, double unit, double beta, uint64_t key, uint64_t c0) {
    const double n2 = x.a0 * x.a0 + x.a1 * x.a1 + x.a2 * x.a2 + x.a3 * x.a3;
    const bool live = n2 > 1e-290;
    quat R = {1.0, 0.0, 0.0, 0.0};
    if (OVERRELAX) {
        // (v^+)^2 = (2 x0^2 / n2 - 1, -2 x0 x_i / n2)
        if (live) {
            const double y = 2.0 * x.a0 / n2;
            R = {fma(y, x.a0, -1.0), -y * x.a1, -y * x.a2, -y * x.a3};
        }
    } else {
        const double k2 = sqrt(n2);  // 2 k
        double x0;
        if (sample_x0(beta * (k2 * unit) / 3.0, key, c0, x0)) {
            const double cth = 2.0 * draw(key, c0 + 256) - 1.0;
            double sphi, cphi;
            sincospi(2.0 * draw(key, c0 + 257), &sphi, &cphi);
            const double sth = sqrt(fmax(0.0, 1.0 - cth * cth));
            const double rr = sqrt(fmax(0.0, 1.0 - x0 * x0));
            const quat X = {x0, rr * sth * cphi, rr * sth * sphi, rr * cth};
            const quat v = live ? quat{x.a0 / k2, x.a1 / k2, x.a2 / k2, x.a3 / k2} : quat{1.0, 0.0, 0.0, 0.0};
            R = qmul(X, qconj(v));
        }
    }
    return {{R.a0, R.a3}, {R.a2, R.a1}};
}

__device__ __forceinline__ quat su2_block(const mat3<double>& w, int i, int j) {
    return {w.e[i][i].re + w.e[j][j].re, w.e[i][j].im + w.e[j][i].im, w.e[i][j].re - w.e[j][i].re,
            w.e[i][i].im - w.e[j][j].im};
}

// R as operands: rows (r00, r01) and (-r01^*, r00^*) and their negatives.  |R| = 1 to FP64 rounding, as x is
// finite where this is used, so no entry needs a check.
struct rot_fx {
    vecx<2> i, ni, j, nj;
};
__device__ __forceinline__ void take_rotation(rot_fx& o, const rot2& R) {
    fx_guard g;
    fx_take(R.a.re, o.i.rh[0], o.i.rl[0], g);
    fx_take(R.a.im, o.i.ih[0], o.i.il[0], g);
    fx_take(R.b.re, o.i.rh[1], o.i.rl[1], g);
    fx_take(R.b.im, o.i.ih[1], o.i.il[1], g);
    o.ni = fx_negated(o.i);
    o.j.rh[0] = o.ni.rh[1]; o.j.rl[0] = o.ni.rl[1]; o.j.ih[0] = o.i.ih[1]; o.j.il[0] = o.i.il[1];
    o.j.rh[1] = o.i.rh[0]; o.j.rl[1] = o.i.rl[0]; o.j.ih[1] = o.ni.ih[0]; o.j.il[1] = o.ni.il[0];
    o.nj = fx_negated(o.j);
}

// rows i, j of the link by R, in fixed point: rows that a later rotation reads are taken back as
// operands, finished rows stay as sums
template <bool KEEP_I, bool KEEP_J>
__device__ __forceinline__ void fx_rotate(matq<3>& out, matx<3>& u, int i, int j, const rot_fx& R) {
#pragma unroll
    for (int col = 0; col < 3; ++col) {
        vecx<2> p;
        p.rh[0] = u.rh[i][col]; p.rl[0] = u.rl[i][col]; p.ih[0] = u.ih[i][col]; p.il[0] = u.il[i][col];
        p.rh[1] = u.rh[j][col]; p.rl[1] = u.rl[j][col]; p.ih[1] = u.ih[j][col]; p.il[1] = u.il[j][col];
        long long re = 0, im = 0;
        fx_dot<2, false>(re, im, R.i, R.ni, p);
        if (KEEP_I) {
            fx_split<0>(re, u.rh[i][col], u.rl[i][col]);
            fx_split<0>(im, u.ih[i][col], u.il[i][col]);
        } else {
            out.re[i][col] = re;
            out.im[i][col] = im;
        }
        re = im = 0;
        fx_dot<2, false>(re, im, R.j, R.nj, p);
        if (KEEP_J) {
            fx_split<0>(re, u.rh[j][col], u.rl[j][col]);
            fx_split<0>(im, u.ih[j][col], u.il[j][col]);
        } else {
            out.re[j][col] = re;
            out.im[j][col] = im;
        }
    }
}

// entry (i, col) and/or (j, col) of W by R.  W's parts are checked to be below kWideW (six unitary matrices sum to
// 6 at most); the rotations keep the norm of the three entries of a column, so a part stays below
// sqrt(6) 6.25 = 15.4, hi below 2^31 and the sums of fx_dot below 2^62.4.
constexpr int kWideW = 25 << 22;  // 6.25 in the top word of a sum in units 2^-56
template <bool I, bool J>
__device__ __forceinline__ void fx_rotate_entry(matq<3>& w, int i, int j, int col, const rot_fx& R) {
    vecx<2> p;
    fx_split<0>(w.re[i][col], p.rh[0], p.rl[0]);
    fx_split<0>(w.im[i][col], p.ih[0], p.il[0]);
    fx_split<0>(w.re[j][col], p.rh[1], p.rl[1]);
    fx_split<0>(w.im[j][col], p.ih[1], p.il[1]);
    if (I) {
        w.re[i][col] = w.im[i][col] = 0;
        fx_dot<2, false>(w.re[i][col], w.im[i][col], R.i, R.ni, p);
    }
    if (J) {
        w.re[j][col] = w.im[j][col] = 0;
        fx_dot<2, false>(w.re[j][col], w.im[j][col], R.j, R.nj, p);
    }
}

// the block of W, a sum before it is rounded to FP64
__device__ __forceinline__ quat su2_block(const matq<3>& w, int i, int j) {
    return {(double)(w.re[i][i] + w.re[j][j]), (double)(w.im[i][j] + w.im[j][i]), (double)(w.re[i][j] - w.re[j][i]),
            (double)(w.im[i][i] - w.im[j][j])};
}

// The whole update in FP64, for links whose staples leave the range of fixed.cuh
template <int OVERRELAX>
__device__ __forceinline__ void native_update(double* __restrict__ base, int Vp, const CfgDesc& c, int s, unsigned eb, int mu,
                                              double beta, uint64_t key, uint64_t c0) {
    mat3<double> wm, un;
    native_omega(wm, base, Vp, c, s, eb, mu);
    Store<P64>::load(base + (size_t)mu * 18 * Vp, Vp, s, un);
#pragma unroll 1
    for (int sub = 0; sub < 3; ++sub) {
        const int i = sub >> 1, j = sub == 0 ? 1 : 2;
        const rot2 R = draw_rotation<OVERRELAX>(su2_block(wm, i, j), 1.0, beta, key, c0 + sub * kSlots);
        for (int col = 0; col < 3; ++col) {
            cx<double> p = wm.e[i][col], q = wm.e[j][col];
            wm.e[i][col] = rot_i(R, p, q);
            wm.e[j][col] = rot_j(R, p, q);
            p = un.e[i][col], q = un.e[j][col];
            un.e[i][col] = rot_i(R, p, q);
            un.e[j][col] = rot_j(R, p, q);
        }
    }
    Store<P64>::store(base + (size_t)mu * 18 * Vp, Vp, s, un);
}

// Staples, W and the rotations of W and U run in fixed point on the integer pipe (fixed.cuh); FP64 keeps the
// SU(2) blocks' direction (an over-relaxation takes (v^+)^2 from x with one division), the heat-bath's draws and the
// conversion of the result: about 130 FP64 instructions instead of 2,200, which kept the FP64 pipe 94 % busy.
// W rotated in FP64 put 210 there, in three chains that nothing overlaps.
// One hybrid sweep (1 heat-bath, 12 over-relaxation) of 256 x 4x4x12x12: 114.9 ms in FP64, 33.2 with W rotated in
// FP64, 31.7 in fixed point, 31.4 now; of 60 such fields 9.93 -> 9.06 -> 9.01, of 8 3.76 -> 3.47 -> 3.41.
// The integer multiply pipe is about 63 % busy; with 168 registers an SM holds
// 12 warps, and 4 blocks of it spill (35.8 ms).
template <int OVERRELAX, int CAP>
__global__ void __launch_bounds__(kMcThreads, 3) k_mc(const __grid_constant__ BatchT<CAP> B, double* __restrict__ w,
                                                      int mu, int parity, double beta, uint64_t seed, uint64_t sweep) {
    const int blk = blockIdx.x;
    if (blk >= B.nblk) return;
    const int ci = find_cfg(B, blk);
    const CfgDesc& c = B.c[ci];
    int t = (blk - c.blk0) * kMcThreads + threadIdx.x;
    const bool valid = t < c.V / 2;  // the others take part in the barriers and store nothing
    if (!valid) t = 0;
    // t -> the t-th site of this parity (every extent even): x0 = 2j + ((x1 + x2 + x3 + parity) & 1)
    int x[4];
    const int h0 = c.L[0] / 2;
    int r = t / h0;
    const int j = t - r * h0;
    x[1] = r % c.L[1];
    r /= c.L[1];
    x[2] = r % c.L[2];
    x[3] = r / c.L[2];
    x[0] = 2 * j + ((x[1] + x[2] + x[3] + parity) & 1);
    const int s = x[0] + c.st[1] * x[1] + c.st[2] * x[2] + c.st[3] * x[3];
    const unsigned eb = edge_bits(c, x);
    const int Vp = c.Vp;
    double* base = w + c.w_off;

    fx_guard g;
    Su3Src src{base, Vp};
    matq<3> om;  // W, in units 2^-56: the rotations depend on its direction only, but for the heat-bath's alpha
    {
        matq<3> sig;
        fx_zero(sig);
        fx_staples<3, true, false>(sig, src, nullptr, 0, c, s, mu, eb, g, [](int, int, const matq<3>&) {});
        if (!valid) return;
        matx<3> u, sx;
        fx_operand_wide<3, 2>(sx, sig);
        fx_take_matrix<3>(u, src, mu, s, false, g);
        fx_mul_nn<3>(om, u, sx);
    }
    unsigned wide = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            wide = max(wide, (unsigned)((int)(om.re[i][k] >> 32) + kWideW));
            wide = max(wide, (unsigned)((int)(om.im[i][k] >> 32) + kWideW));
        }
    const uint64_t key = hash64(seed, (uint64_t)ci);
    const uint64_t c0 = (((uint64_t)sweep * 4 + (uint64_t)mu) * (uint64_t)c.V + (uint64_t)s) * 3 * kSlots;
    if (g.bad() || wide >= 2u * kWideW) {
        native_update<OVERRELAX>(base, Vp, c, s, eb, mu, beta, key, c0);
        return;
    }
    // the three subgroups (0,1), (0,2), (1,2), each on W after the ones before it; only the entries
    // that a later block reads are rotated
    constexpr double kUnit = 0x1p-56;
    matx<3> u;
    matq<3> out;
    rot_fx R;
    take_rotation(R, draw_rotation<OVERRELAX>(su2_block(om, 0, 1), kUnit, beta, key, c0));
    fx_rotate_entry<true, false>(om, 0, 1, 0, R);
    fx_rotate_entry<true, true>(om, 0, 1, 1, R);
    fx_rotate_entry<true, true>(om, 0, 1, 2, R);
    // U is taken in a second time rather than held over the first draw (36 registers: 31.8 instead of 31.7 ms for
    // the sweep below, 3.53 instead of 3.37 for 8 fields); the opaque copy keeps the compiler from merging the two
    int dir = mu;
    asm volatile("" : "+r"(dir));
    fx_take_matrix<3>(u, src, dir, s, false, g);
    fx_rotate<true, true>(out, u, 0, 1, R);
    take_rotation(R, draw_rotation<OVERRELAX>(su2_block(om, 0, 2), kUnit, beta, key, c0 + kSlots));
    fx_rotate_entry<false, true>(om, 0, 2, 1, R);
    fx_rotate_entry<false, true>(om, 0, 2, 2, R);
    fx_rotate<false, true>(out, u, 0, 2, R);
    take_rotation(R, draw_rotation<OVERRELAX>(su2_block(om, 1, 2), kUnit, beta, key, c0 + 2 * kSlots));
    fx_rotate<false, false>(out, u, 1, 2, R);

    mat3<double> un;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int k = 0; k < 3; ++k) un.e[i][k] = {fx_value(out.re[i][k]), fx_value(out.im[i][k])};
    Store<P64>::store(base + (size_t)mu * 18 * Vp, Vp, s, un);
}

template <int OVERRELAX, int CAP>
void launch_cap(const Batch& B, double* w, int mu, int parity, double beta, uint64_t seed, uint64_t sweep,
                cudaStream_t st) {
    if constexpr (CAP == kMaxCfg) {
        k_mc<OVERRELAX, kMaxCfg><<<B.nblk, kMcThreads, 0, st>>>(B, w, mu, parity, beta, seed, sweep);
    } else {
        BatchT<CAP> b;
        b.ncfg = B.ncfg;
        b.nblk = B.nblk;
        for (int i = 0; i < B.ncfg; ++i) b.c[i] = B.c[i];
        k_mc<OVERRELAX, CAP><<<B.nblk, kMcThreads, 0, st>>>(b, w, mu, parity, beta, seed, sweep);
    }
}

}  // namespace

void launch_mc(int overrelax, const Batch& B, double* w, int mu, int parity, double beta, uint64_t seed,
               uint64_t sweep, cudaStream_t st) {
    if (B.ncfg <= kSmallCap) {
        if (overrelax) launch_cap<1, kSmallCap>(B, w, mu, parity, beta, seed, sweep, st);
        else launch_cap<0, kSmallCap>(B, w, mu, parity, beta, seed, sweep, st);
    } else {
        if (overrelax) launch_cap<1, kMaxCfg>(B, w, mu, parity, beta, seed, sweep, st);
        else launch_cap<0, kMaxCfg>(B, w, mu, parity, beta, seed, sweep, st);
    }
}

TGF_CHECK_WORD(mc)

}  // namespace tgf
