// stage64.cuh -- one RK3 stage, the clover halves, or both, in double precision: links, the accumulator
// X and scalars in FP64, the matrix products and the exponential's assembly in 58-bit fixed point on the
// integer pipe (fixed.cuh).
//
// With everything in FP64 the stage kept the FP64 pipe 94-97 % busy (107,000 cycles per warp and SM
// quarter), and nothing else of the chip was in use.  Here that pipe carries about 115 instructions (7,200
// cycles) and the integer pipe 13 products (4,500 IMAD.WIDE of 4 cycles) and the splitting of the operands:
// 34,000 cycles, the multiply pipe 53 % busy.  4 steps of 4 x 8x8x24x24, measured each step: 23.8 ms before,
// 8.6 with the products in fixed point, 7.8 with the exponential (fx_exp_su3) as well, 7.6 with the block's
// links taken in once and shared, and 7.6 with the unbiased sums and the checks that it has now; one measurement of
// 4 x 7x7x21x21: 693 us before, 271 now; 3 steps of 4x4x12x12 (latency): 696 us before, 281 now.
#pragma once

#include <cuda_runtime.h>

#include "expm.cuh"
#include "fixed.cuh"
#include "lattice.cuh"
#include "planes.cuh"

namespace tgf {

// the anti-Hermitian part D - D^+ of a product (units `unit`), as store_ah
__device__ __forceinline__ void fx_store_ah(double* __restrict__ p, int Vp, int s, const matq<3>& d, double unit) {
    const double v[9] = {2 * unit * (double)d.im[0][0],          2 * unit * (double)d.im[1][1],
                         2 * unit * (double)d.im[2][2],          unit * (double)(d.re[0][1] - d.re[1][0]),
                         unit * (double)(d.im[0][1] + d.im[1][0]), unit * (double)(d.re[0][2] - d.re[2][0]),
                         unit * (double)(d.im[0][2] + d.im[2][0]), unit * (double)(d.re[1][2] - d.re[2][1]),
                         unit * (double)(d.im[1][2] + d.im[2][1])};
    AhStore<double>::store(p, Vp, s, v);
}

// X of stage STAGE from the force z, with the accumulator read and written where the stage does.
template <int STAGE>
__device__ __forceinline__ void rk3_x(alg8<double>& x, const alg8<double>& z, double h, double* xb, int Vp, int s) {
    if (STAGE == 1) {
#pragma unroll
        for (int i = 0; i < 8; ++i) x.v[i] = 0.25 * h * z.v[i];
    } else {
        AccStore<double>::load(xb, Vp, s, x);
#pragma unroll
        for (int i = 0; i < 8; ++i)
            x.v[i] = STAGE == 2 ? (8.0 / 9.0) * h * z.v[i] - (17.0 / 9.0) * x.v[i] : 0.75 * h * z.v[i] - x.v[i];
    }
    if (STAGE != 3) AccStore<double>::store(xb, Vp, s, x);
}

// The force (and the clover halves) in FP64 throughout, for links whose fields leave the range of
// fixed.cuh (entries above 1 + 2^-10, infinities, NaN) and for weak ones (fx_rough): any input, at the FP64 pipe's rate.
// trace: also the plaquette deviations 3 - Re Tr(U F), which fixed point has to 2^-57 where it is in range.
template <int MODE>
__device__ __forceinline__ void native_force64(alg8<double>& z, const CfgDesc& c, const double* __restrict__ base,
                                               double* __restrict__ cb, int s, int mu, unsigned eb, bool trace, int dn0 = 1,
                                               int dn1 = 4) {
    const int Vp = c.Vp;
    auto link = [&](int dir, int site, mat3<double>& u) { Store<P64>::load(base + (size_t)dir * 18 * Vp, Vp, site, u); };
    mat3<double> sig, a, b, t, f;
    set_zero(sig);
    const int s_mp = fwd(c, eb, s, mu);
    const bool at_mu0 = (eb >> mu) & 1u;
#pragma unroll 1
    for (int dn = dn0; dn < dn1; ++dn) {
        const int nu = (mu + dn) & 3;
        const bool clover = MODE != 0 && c_clover_owner[mu][nu];
        const int s_nm = bwd(c, eb, s, nu);
        const int k = c.tw[mu * 4 + nu];
        double zr = 1.0, zi = 0.0;
        if (k != 0) centre<double>(k, zr, zi);
        link(nu, s_mp, a);
        link(mu, fwd(c, eb, s, nu), b);
        mul_nd(t, a, b);
        link(nu, s, a);
        mul_nd(f, t, a);
        if (k != 0 && at_mu0 && ((eb >> nu) & 1u)) scale_cx(f, zr, -zi);
        add_to(sig, f);
        link(mu, s_nm, a);
        link(nu, fwd(c, eb, s_nm, mu), b);
        mul_nn(t, a, b);
        link(nu, s_nm, a);
        mul_dn(b, t, a);
        if (k != 0 && at_mu0 && ((eb >> (8 + nu)) & 1u)) scale_cx(b, zr, zi);
        add_to(sig, b);
        if (clover) {
            const int pl = c_plane_of[mu < nu ? mu : nu][mu < nu ? nu : mu];
            link(mu, s, a);
            double rt = 0.0;
            const double sg = nu > mu ? 1.0 : -1.0;
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int j = 0; j < 3; ++j)
                    rt = fma(a.e[i][j].re, f.e[j][i].re, fma(-a.e[i][j].im, f.e[j][i].im, rt));
            if (trace) cb[(size_t)(108 + pl) * Vp + s] = 3.0 - rt;
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    f.e[i][j].re = sg * (f.e[i][j].re - b.e[i][j].re);
                    f.e[i][j].im = sg * (f.e[i][j].im - b.e[i][j].im);
                }
            mul_nn(t, a, f);
            store_ah(cb + (size_t)(pl * 2 + 0) * 9 * Vp, Vp, s, t);
            mul_nn(t, f, a);
            store_ah(cb + (size_t)(pl * 2 + 1) * 9 * Vp, Vp, s_mp, t);
        }
    }
    if (MODE == 2) return;
    link(mu, s, a);
    mul_nn(t, a, sig);
    minus_proj_ta(z, t);
}

// One thread per link; a block covers 32 sites x 4 directions, warps grouped by mu.  MODE as in k_stage:
// 0 the stage, 1 the stage and the clover halves of the input field, 2 the halves only (three warps with two planes
// each, c_half; WIDE: six with one).
//
// WIDE: three threads per link, one for each direction nu, whose staple sums meet in shared memory (whole numbers:
// the result is the same to the bit) before the first goes on with the link.  For launches that leave most of
// the chip idle (launch_m in stage64.cu).
constexpr int stage64_threads(int mode, bool wide) { return mode == 2 ? (wide ? 192 : 96) : wide ? 384 : 128; }
template <int STAGE, int MODE, int CAP, bool WIDE>
__global__ void __launch_bounds__(stage64_threads(MODE, WIDE), WIDE ? 1 : MODE == 0 ? 3 : MODE == 1 ? 2 : 4)
k_stage64(const __grid_constant__ BatchT<CAP> B, const double* __restrict__ w_in, double* __restrict__ w_out,
          double* __restrict__ acc, double* __restrict__ clov) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int mu = warp & 3;
    const int part = MODE == 2 ? 0 : warp >> 2;
    // the links shared by the block's warps; WIDE: then the staple sums of its second and third part
    __shared__ union {
        fx_shared<3> links;
        struct {
            long long v[2][18][128];
            unsigned bad[2][128];
        } sum;
    } sm;
    for (int blk = blockIdx.x; blk < B.nblk; blk += gridDim.x) {
        const int ci = find_cfg(B, blk);
        const CfgDesc& c = B.c[ci];
        if (MODE != 0) clear_counter(c, blk);
        int s = (blk - c.blk0) * 32 + lane;
        const bool valid = s < c.V;  // lanes past the end take part in the barriers on site 0 and store nothing
        if (!valid) s = 0;
        int xc[4];
        site_coords(c, s, xc);
        const unsigned eb = edge_bits(c, xc);
        const int Vp = c.Vp;
        const double* base = w_in + c.w_off;
        double* xb = acc + c.x_off + (size_t)mu * 8 * Vp;
        double* cb = clov + c.m_off;
        fx_guard g;
        matq<3> sig, kk;  // kk: F - B of a clover plane, from the staple sum before, between and after
        matx<3> u;
        Su3Src src{base, Vp};
        fx_zero(sig);
        if (MODE != 0) fx_zero(kk);
        __syncthreads();  // the block before is done with the shared memory
        bool rough = false;
#pragma unroll 1
        for (int m = warp; m < 8; m += (int)blockDim.x >> 5) {
            fx_guard gl;
            fx_take_matrix<3, true>(u, src, m & 3, m < 4 ? s : bwd(c, eb, s, m & 3), false, gl);
            fx_share<3>(sm.links, m, lane, u, gl);
            rough |= gl.rough();
        }
        // a block of weak links needs no fixed-point staples (but for the plaquette deviations of a measured stage)
        const bool skip = MODE == 0 && !__syncthreads_or(rough);
        auto weak = [&]() { return !g.rough() && fx_near_staples<3>(src, c, eb, s, mu); };
#pragma unroll 1
        for (int it = skip ? 1 : 0; it < (MODE == 2 && !WIDE ? 2 : 1); ++it) {
            int q0 = WIDE ? 2 * part : 0, q1 = WIDE ? 2 * part + 2 : 6;
            if (MODE == 2) {
                const int e = WIDE ? warp : 2 * warp + it;
                mu = c_half[e][0];
                q0 = 2 * ((c_half[e][1] - mu - 1) & 3);
                q1 = q0 + 2;
                fx_zero(sig);
                fx_zero(kk);
                g = fx_guard{};
            }
            fx_staples<3, true, true>(sig, src, &sm.links, lane, c, s, mu, eb, g, [&](int back, int nu, const matq<3>& sum) {
                if (!valid || MODE == 0) return;
                if (MODE == 1 && !c_clover_owner[mu][nu]) {
                    if (back) kk = sum;
                    return;
                }
                const int pl = c_plane_of[mu < nu ? mu : nu][mu < nu ? nu : mu];
                fx_shared_link<3>(u, sm.links, mu, lane);
                if (!back) {
                    // 3 - Re Tr(U F), the deviation of the twisted plaquette from the unit matrix.  With entries of F below
                    // 2, the 18 hi hi products stay below 2^62.2 and the cross sum of a row below 2^61.6.
#pragma unroll
                    for (int i = 0; i < 3; ++i)
#pragma unroll
                        for (int j = 0; j < 3; ++j) {
                            kk.re[i][j] = sum.re[i][j] - kk.re[i][j];
                            kk.im[i][j] = sum.im[i][j] - kk.im[i][j];
                        }
                    fx_check<3, 27>(kk, g);
                    long long hh = 0;
#pragma unroll
                    for (int i = 0; i < 3; ++i) {
                        long long cr = fx_round();
#pragma unroll
                        for (int j = 0; j < 3; ++j) {
                            int rh, rl, ih, il;
                            fx_split<1, true>(kk.re[j][i], rh, rl);
                            fx_split<1, true>(kk.im[j][i], ih, il);
                            fx_mad(hh, cr, u.rh[i][j], u.rl[i][j], rh, rl);
                            fx_mad(hh, cr, fx_neg(u.ih[i][j]), fx_neg(u.il[i][j]), ih, il);
                        }
                        hh = fx_join(hh, cr);
                    }
                    cb[(size_t)(108 + pl) * Vp + s] = (double)((3ll << 57) - hh) * 0x1p-57;
#pragma unroll
                    for (int i = 0; i < 3; ++i)
#pragma unroll
                        for (int j = 0; j < 3; ++j) {
                            kk.re[i][j] += sum.re[i][j];
                            kk.im[i][j] += sum.im[i][j];
                        }
                    return;
                }
                // K = F - B; D1 = U K (site n), D2 = K U (site n + mu).  A plane built through its second
                // direction (nu < mu) takes the other sign: its leaves are the conjugates of (mu, nu)'s.
#pragma unroll
                for (int i = 0; i < 3; ++i)
#pragma unroll
                    for (int j = 0; j < 3; ++j) {
                        kk.re[i][j] -= sum.re[i][j];
                        kk.im[i][j] -= sum.im[i][j];
                    }
                fx_check<3, 28>(kk, g);
                matx<3> kx;
                matq<3> t;
                fx_operand_wide<3, 1, true>(kx, kk);
                const double unit = nu > mu ? 0x1p-57 : -0x1p-57;
                fx_mul_nn<3>(t, u, kx);
                fx_store_ah(cb + (size_t)(pl * 2 + 0) * 9 * Vp, Vp, s, t, unit);
                fx_mul_nn<3>(t, kx, u);
                fx_store_ah(cb + (size_t)(pl * 2 + 1) * 9 * Vp, Vp, fwd(c, eb, s, mu), t, unit);
                kk = sum;
            }, q0, q1);
            if (MODE == 2) {
                const bool all_near = fx_shared_flags<3>(g, sm.links, mu, lane);
                alg8<double> z;
                if (valid && (g.bad() || all_near || weak()))
                    native_force64<MODE>(z, c, base, cb, s, mu, eb, g.bad(), q0 / 2 + 1, q0 / 2 + 2);
            }
        }
        if (MODE == 2) continue;
        const bool all_near = fx_shared_flags<3>(g, sm.links, mu, lane);
        fx_shared_link<3>(u, sm.links, mu, lane);
        if constexpr (WIDE && MODE != 2) {
            const int lt = threadIdx.x & 127;
            __syncthreads();  // the links have been read: their place takes the sums
            if (part) {
                sm.sum.bad[part - 1][lt] = g.bad();
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    sm.sum.v[part - 1][i][lt] = sig.re[i / 3][i % 3];
                    sm.sum.v[part - 1][9 + i][lt] = sig.im[i / 3][i % 3];
                }
            }
            __syncthreads();
            if (part) continue;
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                g.top2 |= sm.sum.bad[p][lt];
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    sig.re[i / 3][i % 3] += sm.sum.v[p][i][lt];
                    sig.im[i / 3][i % 3] += sm.sum.v[p][9 + i][lt];
                }
            }
            fx_check<3, 29>(sig, g);
        }
        if (!valid) continue;
        // Omega = U_mu(n) Sigma (units 2^-56), Z = -P_ta(Omega)
        alg8<double> x, z;
        {
            matx<3> sx;
            matq<3> om;
            fx_operand_wide<3, 2>(sx, sig);
            fx_mul_nn<3>(om, u, sx);
            fx_check<3, 29>(om, g);
            const double tr = (double)(om.im[0][0] + om.im[1][1] + om.im[2][2]) * (1.0 / 3.0);
            z.v[0] = 0x1p-56 * (tr - (double)om.im[0][0]);
            z.v[1] = 0x1p-56 * (tr - (double)om.im[1][1]);
            z.v[2] = 0x1p-57 * (double)(om.re[1][0] - om.re[0][1]);
            z.v[3] = -0x1p-57 * (double)(om.im[0][1] + om.im[1][0]);
            z.v[4] = 0x1p-57 * (double)(om.re[2][0] - om.re[0][2]);
            z.v[5] = -0x1p-57 * (double)(om.im[0][2] + om.im[2][0]);
            z.v[6] = 0x1p-57 * (double)(om.re[2][1] - om.re[1][2]);
            z.v[7] = -0x1p-57 * (double)(om.im[1][2] + om.im[2][1]);
        }
        if (g.bad() || all_near || weak()) {
            native_force64<MODE>(z, c, base, cb, s, mu, eb, g.bad());
            g.top2 = 1;
        }
        rk3_x<STAGE>(x, z, c.h, xb, Vp, s);
        mat3<double> e, w;
        matx<3> ex;
        const unsigned up = fx_exp_m1_su3(ex, e, x, g.bad(), g);
        Store<P64>::load(base + (size_t)mu * 18 * Vp, Vp, s, w);
        // W' = W + (exp(X) - 1) W, the product in fixed point (unless a factor is out of its range),
        // rounded once onto W
        if (g.bad()) {
            mat3<double> d;
            mul_nn(d, e, w);
            add_to(w, d);
        } else {
            matq<3> d;
            if (!WIDE) fx_shared_link<3>(u, sm.links, mu, lane);
            fx_mul_nn<3>(d, ex, u);
            const double unit = fx_unit(up);
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    w.e[i][j].re = fma((double)d.re[i][j], unit, w.e[i][j].re);
                    w.e[i][j].im = fma((double)d.im[i][j], unit, w.e[i][j].im);
                }
        }
        Store<P64>::store(w_out + c.w_off + (size_t)mu * 18 * Vp, Vp, s, w);
    }
}

}  // namespace tgf
