// lb_pair.cuh -- the fluctuating collision of two nodes side by side, for the TMA-staged step
// kernels of FP32 storage (single lattice, batched ensemble, server).
//
// What bounds a step.  At 72 bytes a node the 4096^2 step cannot take less than 178 us (copy
// bandwidth 6790 GB/s); with one node per arithmetic instruction it took 212 us, because a node
// cost 341 issued instructions at 68 % issue.  So this file spends fewer instructions per node:
//   * a thread's nodes are pairs (x, x + 1), x even, and the FP32 arithmetic is on packed pairs
//     (add, mul, fma .f32x2: one issue slot for two nodes; the FMA pipe runs them at the same
//     128 operations a clock per SM as scalar ones, measured 120, and 80 when all three operands
//     are register pairs, so two-operand forms are preferred and coefficients are scalars from
//     the constant bank, which cost nothing as a broadcast operand);
//   * rows of a thread's pairs are adjacent, so the density rows of its stencils are loaded once
//     (12 shared loads for 2 x 2 nodes instead of 36) and their sums over x are shared;
//   * planes with c_x = 0, the density and all stores move 8 bytes at a time;
//   * the relaxation and noise factors carry the 1/N_a of the back-transform (host side, PairCoef),
//     and the stencil weights 1/6 and 1/12 are folded into kappa;
//   * log2, sine and cosine are the flush-to-zero forms (their arguments are never subnormal),
//     sqrt(2 ln 2) and the sign of the Box-Muller angle's shift are in the noise factors, and
//     -log2 u1 needs no clamp: u1 <= 1 - 2^-21, so log2 u1 <= -6.8e-7, further from zero than
//     the approximation's error there (2^-22 = 2.4e-7).
#pragma once

#include "lb_internal.cuh"
#include "lb_tma.cuh"

namespace lbf {

// --- packed FP32 pairs ---------------------------------------------------------------------

using F2 = float2;

__device__ __forceinline__ F2 bc(float v) { return make_float2(v, v); }
__device__ __forceinline__ F2 add2(F2 a, F2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ F2 mul2(F2 a, F2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ F2 sub2(F2 a, F2 b) {
    F2 r;
    asm("{\n\t.reg .b64 p, q, s;\n\t"
        "mov.b64 p, {%2, %3};\n\tmov.b64 q, {%4, %5};\n\t"
        "sub.rn.f32x2 s, p, q;\n\t"
        "mov.b64 {%0, %1}, s;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ F2 max0(F2 a) { return make_float2(fmaxf(a.x, 0.f), fmaxf(a.y, 0.f)); }
__device__ __forceinline__ F2 sqrt2(F2 a) { return make_float2(sqrt_approx(a.x), sqrt_approx(a.y)); }
__device__ __forceinline__ F2 rcp2(F2 a) { return make_float2(rcp_approx(a.x), rcp_approx(a.y)); }

__device__ __forceinline__ float lg2_ftz(float x) {
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float cos_ftz(float x) {
    float y;
    asm("cos.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float sin_ftz(float x) {
    float y;
    asm("sin.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// The Box-Muller pairs of two Philox words (gauss_pair of lb_internal.cuh) over
// GAUSS_SCALE = -sqrt(2 ln 2), which is left to the factors that multiply the normals: the sign of
// the angle's shift by pi, and the 2 ln 2 of -2 ln u = 2 ln 2 (-log2 u).  The approximations make the
// normals 1.22e-7 of themselves too small on average (2^31 draws against the FP64 pair), more than half of
// their error of 2.1e-7; the factors give it back.  Error of a step against FP64, 512^2 real-space noise:
// 1.84e-7 without this, 1.55e-7 with it (1.74e-7 with scalar nodes).
constexpr double GAUSS_SCALE = -1.17741002251547469101 * (1.0 + 1.22e-7);
__device__ __forceinline__ void gauss2(uint32_t wa, uint32_t wb, F2* n0, F2* n1) {
    const F2 u = add2(make_float2(__uint_as_float(((wa >> 9) & 0x7ffff8u) | 0x3f800004u),
                                  __uint_as_float(((wb >> 9) & 0x7ffff8u) | 0x3f800004u)), bc(-1.0f));
    const F2 v = add2(make_float2(__uint_as_float(((wa << 11) & 0x7ff800u) | 0x3f800400u),
                                  __uint_as_float(((wb << 11) & 0x7ff800u) | 0x3f800400u)), bc(-1.5f));
    const F2 r = make_float2(sqrt_approx(-lg2_ftz(u.x)), sqrt_approx(-lg2_ftz(u.y)));
    const F2 th = mul2(v, bc(6.2831853071795865f));
    *n0 = mul2(r, make_float2(cos_ftz(th.x), cos_ftz(th.y)));
    *n1 = mul2(r, make_float2(sin_ftz(th.x), sin_ftz(th.y)));
}

// --- coefficients ----------------------------------------------------------------------------

// One lattice's coefficients as collide_pair takes them: a mode's rate and noise factors carry the
// 1 / N_a of its increment in the back-transform (collide_node's d4..d9), noise factors GAUSS_SCALE as
// well (G below).  The weights w_i stay out of them, so that a rate of -1 is exact: with 1/36 in it a
// ghost mode kept 3e-8 of itself, and a two-phase run was 6 % further from FP64.
struct PairCoef {
    float rho0, cs2m;
    float kl, kg;                    // -kappa / 6 and kappa / 144
    float lb, ls5, ls6, lq, le;      // lambda_b / 4, 9 lambda_s / 4, 9 lambda_s, 3 lambda_q / 2, lambda_e / 16
    float L44, L49, L94, L99;        // G (L44, L49) / 4 and G (L94, L99) / 16
    float s5, s6, s7;                // G (9 s5 / 4, 9 s6, 3 s7 / 2)
};

// the double well's pressure and the noise at the local density (single lattices)
struct PairLocal {
    float e2, e3, e4;
    float cq[4];
    float lu[9];                     // of x44 / 16, x49 / 64, x99 / 256 per unit density, then
                                     // G (9 / 4, 9, 3 / 2) times the roots of x55, x66, x77
};

// real-space correlated noise: G / 4 and G / 16 times the factors / 4 of Xi at k^2 = 0, 4, 16/3
struct PairStencil {
    float sL[3][4];
};

template <typename S>
__host__ inline void pair_coef(double rho0, double cs2m, double kappa, double lb, double ls, double lq, double le,
                               const S L[4], const S s[3], PairCoef* o) {
    o->rho0 = (float)rho0;
    o->cs2m = (float)cs2m;
    o->kl = (float)(-kappa / 6.0);
    o->kg = (float)(kappa / 144.0);
    o->lb = (float)(lb / 4.0);
    o->ls5 = (float)(ls * 2.25);
    o->ls6 = (float)(ls * 9.0);
    o->lq = (float)(lq * 1.5);
    o->le = (float)(le / 16.0);
    const double G = GAUSS_SCALE;
    o->L44 = (float)(G * L[0] / 4.0);
    o->L49 = (float)(G * L[1] / 4.0);
    o->L94 = (float)(G * L[2] / 16.0);
    o->L99 = (float)(G * L[3] / 16.0);
    o->s5 = (float)(G * s[0] * 2.25);
    o->s6 = (float)(G * s[1] * 9.0);
    o->s7 = (float)(G * s[2] * 1.5);
}

template <typename S>
__host__ inline void pair_stencil(const S sL[3][4], PairStencil* o) {
    const double G = GAUSS_SCALE;
    for (int j = 0; j < 3; ++j) {
        o->sL[j][0] = (float)(G * sL[j][0] / 4.0);
        o->sL[j][1] = (float)(G * sL[j][1] / 4.0);
        o->sL[j][2] = (float)(G * sL[j][2] / 16.0);
        o->sL[j][3] = (float)(G * sL[j][3] / 16.0);
    }
}

template <typename S>
__host__ inline void pair_local(double e2, double e3, double e4, const S cq[4], const S lu[9], PairLocal* o) {
    o->e2 = (float)e2;
    o->e3 = (float)e3;
    o->e4 = (float)e4;
    for (int q = 0; q < 4; ++q) o->cq[q] = (float)cq[q];
    const double f[9] = {1 / 16.0, 1 / 16.0, 1 / 64.0, 1 / 64.0, 1 / 256.0, 1 / 256.0,
                         GAUSS_SCALE * 2.25, GAUSS_SCALE * 9.0, GAUSS_SCALE * 1.5};
    for (int q = 0; q < 9; ++q) o->lu[q] = (float)(f[q] * lu[q]);
}

// --- one pair --------------------------------------------------------------------------------

// density deviation of a pair from its pulled values (one order of summation, for a node and for
// the ring: drho_of of lb_collide.cuh is the scalar counterpart)
__device__ __forceinline__ F2 drho_pair(const F2 f[Q]) {
    const F2 sa = add2(add2(f[1], f[3]), add2(f[2], f[4]));
    const F2 sd = add2(add2(f[5], f[7]), add2(f[6], f[8]));
    return add2(add2(f[0], sa), sd);
}

// The stencil of a pair: 6 lap rho, 12 d_x rho, 12 d_y rho (Appendix B and the isotropic
// gradient), from the rows below (m), of (c) and above (p) the pair: C the pair's columns,
// s = E + W and d = E - W.
struct RhoRow {
    F2 C, s, d;
};

__device__ __forceinline__ RhoRow rho_row(const float* R) {
    // R at the pair's first column (8-byte aligned)
    RhoRow r;
    r.C = *reinterpret_cast<const F2*>(R);
    const float l = R[-1], e = R[2];
    r.s = make_float2(l + r.C.y, r.C.x + e);
    r.d = make_float2(r.C.y - l, e - r.C.x);
    return r;
}

// MODE as in collide_node (lb_collide.cuh).  rho: density deviations of the pair; lap6, gx12, gy12:
// its stencil; node: the first node's index (the second's is node + 1); z4, z9: the scaled
// (xi_4, xi_9) of modes 2 and 3; a: coefficients (PairCoef, the round keys rk and the time t_lo,
// t_hi); loc: POLY and MODE 4.  Writes the nine post-collision values of both nodes.
template <int MODE, bool POLY, typename Args>
__device__ __forceinline__ void collide_pair(const Args& a, const PairLocal* loc, const F2 f[Q], F2 rho, F2 lap6,
                                             F2 gx12, F2 gy12, uint32_t node, F2 z4, F2 z9, F2 o[Q]) {
    // moments of the deviations (rows of T, Eq. Tmat); ux of opposite pairs first
    const F2 g0 = f[0];
    const F2 sa = add2(add2(f[1], f[3]), add2(f[2], f[4]));
    const F2 sd = add2(add2(f[5], f[7]), add2(f[6], f[8]));
    const F2 nax = sub2(f[3], f[1]), nay = sub2(f[4], f[2]);             // minus the axis momenta
    const F2 d57 = sub2(f[5], f[7]), d86 = sub2(f[8], f[6]);
    const F2 dx = add2(d57, d86), dy = sub2(d57, d86);
    const F2 m5 = sub2(add2(f[1], f[3]), add2(f[2], f[4]));
    const F2 m6 = sub2(add2(f[5], f[7]), add2(f[6], f[8]));
    const F2 jx = sub2(dx, nax), jy = sub2(dy, nay);
    const F2 m4 = fma2(sd, bc(4.0f), fma2(g0, bc(-2.0f), sa));
    const F2 m9 = fma2(sd, bc(8.0f), fma2(sa, bc(-4.0f), add2(g0, g0)));
    const F2 m7 = fma2(bc(2.0f), dx, nax), m8 = fma2(bc(2.0f), dy, nay);

    // equilibrium deviations, Table II
    const F2 dens = add2(rho, bc(a.rho0));
    const F2 inv = rcp2(dens);
    const F2 ux = mul2(jx, inv), uy = mul2(jy, inv);
    const F2 hx = mul2(gx12, bc(a.kg)), hy = mul2(gy12, bc(a.kg));
    const F2 jxx = mul2(jx, ux), jyy = mul2(jy, uy), gxx = mul2(hx, gx12), gyy = mul2(hy, gy12);
    const F2 klap = mul2(mul2(dens, bc(a.kl)), lap6);                    // -kappa rho lap rho
    F2 iso;
    if constexpr (POLY) {
        const F2 dp = fma2(rho, fma2(rho, fma2(rho, bc(loc->e4), bc(loc->e3)), bc(loc->e2)), bc(a.cs2m));
        iso = fma2(dp, rho, klap);
    } else {
        iso = fma2(rho, bc(a.cs2m), klap);
    }
    // m - m^eq with the equilibrium summed first (it is small beside the moment, so one rounding at the
    // moment's size)
    const F2 iso6 = mul2(iso, bc(6.0f));
    const F2 x4 = sub2(m4, fma2(add2(jxx, jyy), bc(3.0f), iso6));
    const F2 x5 = sub2(m5, add2(sub2(jxx, jyy), sub2(gxx, gyy)));
    const F2 x6 = sub2(m6, fma2(hx, gy12, mul2(jx, uy)));
    const F2 x9 = add2(m9, fma2(add2(gxx, gyy), bc(3.0f), iso6));

    // noise (Sec. IV) and relaxation, as increments in the units of PairCoef
    F2 d4, d5, d6, d7, d8, d9;
    if constexpr (MODE == 0) {
        d4 = mul2(x4, bc(a.lb));
        d5 = mul2(x5, bc(a.ls5));
        d6 = mul2(x6, bc(a.ls6));
        d7 = mul2(m7, bc(a.lq));
        d8 = mul2(m8, bc(a.lq));
        d9 = mul2(x9, bc(a.le));
    } else {
        const uint4 ra = philox4x32_10(make_uint4(node, a.t_lo, a.t_hi, TAG_NODE), a.rk);
        const uint4 rb = philox4x32_10(make_uint4(node + 1u, a.t_lo, a.t_hi, TAG_NODE), a.rk);
        F2 n0, n1, k5, k6, k7;
        if constexpr (MODE == 4) {
            // Xi(0) at the node's own density and sound speed (lb_collide.cuh), factored here
            const F2 cs = fma2(rho, fma2(rho, fma2(rho, bc(loc->cq[3]), bc(loc->cq[2])), bc(loc->cq[1])), bc(loc->cq[0]));
            const F2 y44 = mul2(dens, fma2(cs, bc(loc->lu[1]), bc(loc->lu[0])));
            const F2 y49 = mul2(dens, fma2(cs, bc(loc->lu[3]), bc(loc->lu[2])));
            const F2 y99 = mul2(dens, fma2(cs, bc(loc->lu[5]), bc(loc->lu[4])));
            const F2 sr = sqrt2(max0(dens));
            k5 = mul2(sr, bc(loc->lu[6]));
            k6 = mul2(sr, bc(loc->lu[7]));
            k7 = mul2(sr, bc(loc->lu[8]));
            const F2 l44 = sqrt2(max0(y44));
            F2 l94 = mul2(y49, rcp2(l44));
            l94 = make_float2(l44.x > 0.f ? l94.x : 0.f, l44.y > 0.f ? l94.y : 0.f);
            const F2 l99 = sqrt2(max0(sub2(y99, mul2(l94, l94))));
            gauss2(ra.z, rb.z, &n0, &n1);
            z4 = mul2(mul2(l44, bc((float)GAUSS_SCALE)), n0);
            z9 = mul2(fma2(l94, n0, mul2(l99, n1)), bc((float)GAUSS_SCALE));
        } else {
            k5 = bc(a.s5);
            k6 = bc(a.s6);
            k7 = bc(a.s7);
        }
        if constexpr (MODE == 1) {
            gauss2(ra.z, rb.z, &n0, &n1);
            z4 = fma2(n0, bc(a.L44), mul2(n1, bc(a.L49)));
            z9 = fma2(n0, bc(a.L94), mul2(n1, bc(a.L99)));
        }
        d4 = fma2(x4, bc(a.lb), z4);
        d9 = fma2(x9, bc(a.le), z9);
        gauss2(ra.x, rb.x, &n0, &n1);
        d5 = fma2(n0, k5, mul2(x5, bc(a.ls5)));
        d6 = fma2(n1, k6, mul2(x6, bc(a.ls6)));
        gauss2(ra.y, rb.y, &n0, &n1);
        d7 = fma2(n0, k7, mul2(m7, bc(a.lq)));
        d8 = fma2(n1, k7, mul2(m8, bc(a.lq)));
    }

    // back to populations (Sec. III A)
    const F2 A = fma2(d9, bc(-4.0f), d4);
    const F2 A1 = add2(A, d5), A2 = sub2(A, d5);
    const F2 e4 = mul2(fma2(d9, bc(2.0f), d4), bc(4.0f));
    const F2 D1 = add2(e4, d6), D2 = sub2(e4, d6);
    const F2 p = add2(d7, d8), m = sub2(d7, d8);
    const F2 u0 = bc(8.0f / 9.0f), u1 = bc(1.0f / 9.0f), u5 = bc(1.0f / 36.0f);
    o[5] = fma2(fma2(p, bc(2.0f), D1), u5, f[5]);
    o[7] = fma2(fma2(p, bc(-2.0f), D1), u5, f[7]);
    o[6] = fma2(fma2(m, bc(-2.0f), D2), u5, f[6]);
    o[8] = fma2(fma2(m, bc(2.0f), D2), u5, f[8]);
    o[0] = fma2(sub2(d9, d4), u0, f[0]);
    o[1] = fma2(sub2(A1, d7), u1, f[1]);
    o[2] = fma2(sub2(A2, d8), u1, f[2]);
    o[3] = fma2(add2(A1, d7), u1, f[3]);
    o[4] = fma2(add2(A2, d8), u1, f[4]);
}

// --- a staged tile ------------------------------------------------------------------------------

// Thread t < ACTIVE of a TX x TY tile on NT threads owns the 2 x RPT nodes at column
// 2 (t mod TX/2), row RPT (t div TX/2); threads past ACTIVE (tiles with fewer pairs than threads)
// only form ring and halo nodes.
template <int TX, int TY, int NT>
struct PairMap {
    static constexpr int PX = TX / 2;
    static constexpr int RPT = TX * TY / (2 * NT) > 1 ? TX * TY / (2 * NT) : 1;
    static constexpr int ACTIVE = PX * (TY / RPT);
    static_assert(ACTIVE <= NT && TY % RPT == 0, "2 x RPT nodes per thread must cover the tile");
};

// Resident CTAs per SM that the register budget of a step kernel on TX x TY tiles and NT threads is
// set for: 128 registers a thread with two rows of pairs each, 64 with one (80 with the
// contributions of the real-space correlated noise).
template <int TX, int TY, int NT, bool RS>
constexpr int pair_min_blocks() {
    return (PairMap<TX, TY, NT>::RPT > 1 ? 512 : (RS ? 768 : 1024)) / NT;
}

// The pulled values of the pair whose unshifted box index is b (even): plane i at b - cx_i, the
// y shift already in the box origin.
template <int PS>
__device__ __forceinline__ void pull_pair(const float* S, int b, F2 f[Q]) {
    auto even = [&](int i, int k) -> F2 { return *reinterpret_cast<const F2*>(S + i * PS + k); };
    auto odd = [&](int i, int k) -> F2 { return make_float2(S[i * PS + k], S[i * PS + k + 1]); };
    f[0] = even(0, b);
    f[1] = odd(1, b - 1);
    f[2] = even(2, b);
    f[3] = odd(3, b + 1);
    f[4] = even(4, b);
    f[5] = odd(5, b - 1);
    f[6] = odd(6, b + 1);
    f[7] = odd(7, b + 1);
    f[8] = odd(8, b - 1);
}

// Pulls a thread's pairs from the staged tile S into registers and writes the density deviations
// of the tile and of its one-node ring to R (tile node (lx, ly) at R[(ly + 1) RW + lx + 2]).  The
// ring's rows go as pairs to the last threads and its columns, corners included, to the ones
// before them, a warp-aligned block each (one list of single nodes over the last threads cost 60
// instructions on 6 of 16 warps of a 64 x 16 tile, this one 30 on 4); FIRST puts them on the first
// threads instead, where the last form the noise contributions of the halo.  Nodes beyond a ragged
// edge take part (their values are never used).
template <int TX, int TY, int NT, bool FIRST>
__device__ __forceinline__ void tile_pull(const float* S, float* R, F2 (&fr)[PairMap<TX, TY, NT>::RPT][Q]) {
    using TT = TmaTile<TX, TY>;
    using M = PairMap<TX, TY, NT>;
    const int tid = threadIdx.x;
    const int lx = 2 * (tid % M::PX), ly = (tid / M::PX) * M::RPT;
    if (M::ACTIVE == NT || tid < M::ACTIVE) {
#pragma unroll
        for (int j = 0; j < M::RPT; ++j) {
            pull_pair<TT::PS>(S, (ly + j + 1) * TT::BW + lx + TT::XO, fr[j]);
            *reinterpret_cast<F2*>(R + (ly + j + 1) * TT::RW + lx + 2) = drho_pair(fr[j]);
        }
    }
    constexpr int NR = TX, NC = 2 * (TY + 2);          // row pairs (below, then above); column nodes
    for (int j = FIRST ? tid : NT - 1 - tid; j < NR + NC; j += NT) {
        if (j < NR) {
            const int p = 2 * (j % M::PX), ry = j < M::PX ? 0 : TY + 1;
            F2 f[Q];
            pull_pair<TT::PS>(S, ry * TT::BW + p + TT::XO, f);
            *reinterpret_cast<F2*>(R + ry * TT::RW + p + 2) = drho_pair(f);
        } else {
            const int u = j - NR, ry = u >> 1, rx = (u & 1) ? TX : -1;
            const int b = ry * TT::BW + rx + TT::XO;
            auto at = [&](int i, int k) -> float { return S[i * TT::PS + k]; };
            const float sa = (at(1, b - 1) + at(3, b + 1)) + (at(2, b) + at(4, b));
            const float sd = (at(5, b - 1) + at(7, b + 1)) + (at(6, b + 1) + at(8, b - 1));
            R[ry * TT::RW + rx + 2] = (at(0, b) + sa) + sd;
        }
    }
}

// Real-space correlated noise (LB_NOISE_FULL_RS, stencil_h of lb_internal.cuh): the contributions
// h_d of two nodes na, nb to themselves (d = 0), the node to the right (1), above (2) and above
// right (3), scaled: h4 and h9 are the xi_4 and xi_9 parts.
template <typename Args>
__device__ __forceinline__ void stencil_pair(const Args& a, uint32_t na, uint32_t nb, F2 h4[4], F2 h9[4]) {
    const uint4 wa = philox4x32_10(make_uint4(na, a.t_lo, a.t_hi, TAG_STENCIL), a.rk);
    const uint4 wb = philox4x32_10(make_uint4(nb, a.t_lo, a.t_hi, TAG_STENCIL), a.rk);
    F2 g4[4], g9[4];
    const uint32_t va[4] = {wa.x, wa.y, wa.z, wa.w}, vb[4] = {wb.x, wb.y, wb.z, wb.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        F2 n0, n1;
        gauss2(va[k], vb[k], &n0, &n1);
        const int c = k == 0 ? 0 : (k == 3 ? 2 : 1);
        g4[k] = fma2(n0, bc(a.sL[c][0]), mul2(n1, bc(a.sL[c][1])));
        g9[k] = fma2(n0, bc(a.sL[c][2]), mul2(n1, bc(a.sL[c][3])));
    }
    auto hadamard = [](const F2 g[4], F2 h[4]) {
        const F2 u = add2(g[0], g[1]), v = sub2(g[0], g[1]), w = add2(g[2], g[3]), z = sub2(g[2], g[3]);
        h[0] = add2(u, w);
        h[1] = sub2(u, w);
        h[2] = add2(v, z);
        h[3] = sub2(v, z);
    };
    hadamard(g4, h4);
    hadamard(g9, h9);
}

// Exchange of the contributions that cross a thread's block of 2 x RPT nodes, in shared memory:
//   to the right: er[y][p + 1] = h1 of the pair p's second node in row y, ed[y + 1][p + 1] = its h3
//     (for row y + 1), with column 0 from the halo column x0 - 1;
//   upwards: up[r][p] = (xi_4 pair, xi_9 pair) that block row r's first row receives from below:
//     h2 of both nodes and the first node's h3 for the second.
template <int TX, int TY, int NT>
struct StencilTile {
    using M = PairMap<TX, TY, NT>;
    static constexpr int W = M::PX + 1;
    static constexpr int NR = TY / M::RPT;
    static constexpr int ER = 0;                         // float2 [TY][W]
    static constexpr int ED = ER + TY * W * 8;           // float2 [TY + 1][W]
    static constexpr int UP = ((ED + (TY + 1) * W * 8 + 15) / 16) * 16;    // float4 [NR + 1][PX]
    static constexpr int BYTES = UP + (NR + 1) * M::PX * 16;
};

// Before the tile's barrier: the contributions of the thread's own nodes, their in-block sums in
// (z4, z9)[row], the rest into the exchange x; then the halo below and left of the tile (periodic),
// on the last threads.  Nodes past a ragged edge send only to nodes past it.
template <int TX, int TY, int NT, typename Args>
__device__ __forceinline__ void stencil_tile(const Args& a, unsigned char* x, int x0, int y0, int nx, int ny,
                                             F2 (&z4)[PairMap<TX, TY, NT>::RPT], F2 (&z9)[PairMap<TX, TY, NT>::RPT]) {
    using M = PairMap<TX, TY, NT>;
    using ST = StencilTile<TX, TY, NT>;
    F2* er = reinterpret_cast<F2*>(x + ST::ER);
    F2* ed = reinterpret_cast<F2*>(x + ST::ED);
    float4* up = reinterpret_cast<float4*>(x + ST::UP);
    const int tid = threadIdx.x;
    const int p = tid % M::PX, rb = tid / M::PX, ly = rb * M::RPT;
    if (M::ACTIVE == NT || tid < M::ACTIVE) {
        F2 c4 = bc(0.f), c9 = bc(0.f);             // carried to the row above
#pragma unroll
        for (int j = 0; j < M::RPT; ++j) {
            const int y = ly + j;
            const uint32_t node = (uint32_t)(y0 + y) * (uint32_t)nx + (uint32_t)(x0 + 2 * p);
            F2 h4[4], h9[4];
            stencil_pair(a, node, node + 1u, h4, h9);
            z4[j] = make_float2(h4[0].x, h4[0].y + h4[1].x);
            z9[j] = make_float2(h9[0].x, h9[0].y + h9[1].x);
            if (j > 0) {
                z4[j] = add2(z4[j], c4);
                z9[j] = add2(z9[j], c9);
            }
            c4 = make_float2(h4[2].x, h4[2].y + h4[3].x);
            c9 = make_float2(h9[2].x, h9[2].y + h9[3].x);
            er[y * ST::W + p + 1] = make_float2(h4[1].y, h9[1].y);
            ed[(y + 1) * ST::W + p + 1] = make_float2(h4[3].y, h9[3].y);
        }
        up[(rb + 1) * M::PX + p] = make_float4(c4.x, c4.y, c9.x, c9.y);
    }
    // the halo: PX pairs of the row below, then the column to the left two rows at a time
    for (int j = NT - 1 - tid; j < M::PX + TY / 2 + 1; j += NT) {
        const bool below = j < M::PX;
        const int y = below ? -1 : 2 * (j - M::PX) - 1;          // row of the first node
        int gx = below ? x0 + 2 * j : x0 - 1, ga = y0 + y, gb = below ? ga : ga + 1;
        if (gx < 0) gx += nx;
        if (ga < 0) ga += ny;
        if (gb < 0) gb += ny;
        const uint32_t na = (uint32_t)ga * (uint32_t)nx + (uint32_t)gx;
        const uint32_t nb = below ? na + 1u : (uint32_t)gb * (uint32_t)nx + (uint32_t)gx;
        F2 h4[4], h9[4];
        stencil_pair(a, na, nb, h4, h9);
        if (below) {
            up[j] = make_float4(h4[2].x, h4[2].y + h4[3].x, h9[2].x, h9[2].y + h9[3].x);
            ed[j + 1] = make_float2(h4[3].y, h9[3].y);
        } else {
            if (y >= 0) er[y * ST::W] = make_float2(h4[1].x, h9[1].x);
            ed[(y + 1) * ST::W] = make_float2(h4[3].x, h9[3].x);
            if (y + 1 < TY) {
                er[(y + 1) * ST::W] = make_float2(h4[1].y, h9[1].y);
                ed[(y + 2) * ST::W] = make_float2(h4[3].y, h9[3].y);
            }
        }
    }
}

// Whether the tile at x0 is stored by its threads instead of its TMA box: a box is clipped at the
// lattice's last column in units of 16 bytes, so a row that ends inside such a unit would lose its
// first ghost columns to the tile's unused ones.
template <int TX>
__device__ __forceinline__ bool tile_direct(const Grid& g, int x0) {
    return x0 + TX > g.nx && g.nx % Elem<float>::XO != 0;
}

// a pair, at an even column
__device__ __forceinline__ void put_pair(float* q, F2 v) { *reinterpret_cast<F2*>(q) = v; }

// the nodes of the pair at (x, y) themselves (a tile that tile_direct names); the second only if
// x + 1 < nx
__device__ __forceinline__ void store_pair(float* dst, long long P, const Grid& g, int x, int y, const F2 o[Q]) {
    float* p = dst + g.at(x, y);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        if (x + 1 < g.nx) put_pair(p + i * P, o[i]);
        else p[i * P] = o[i].x;
    }
}

// Periodic ghost copies of the pair at (x, y), x even, of a tile near an edge (store9 of
// lb_internal.cuh); the nodes themselves leave with the tile.  Where nx is even and no node feeds
// more than one ghost column and row, both nodes of a pair feed the same ones and the copies are
// pairs; else each node is written with all its copies.
__device__ __forceinline__ void ghost_pair(float* dst, long long P, const Grid& g, int x, int y, const F2 o[Q]) {
    constexpr int GW = Elem<float>::GW;
    if (!(x < GW || x + 1 >= g.nx - GW || y < 2 || y >= g.ny - 2)) return;
    if ((g.nx & 1) == 0 && g.nx >= 2 * GW && g.ny >= 4) {
        float* p = dst + g.at(x, y);
        const bool hx = x < GW || x >= g.nx - GW, hy = y < 2 || y >= g.ny - 2;
        const long long dx = x < GW ? (long long)g.nx : -(long long)g.nx;
        const long long dy = (y < 2 ? (long long)g.ny : -(long long)g.ny) * g.pitch;
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            float* q = p + i * P;
            if (hx) put_pair(q + dx, o[i]);
            if (hy) put_pair(q + dy, o[i]);
            if (hx & hy) put_pair(q + dx + dy, o[i]);
        }
    } else {
        float v[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) v[i] = o[i].x;
        store9<float, float>(dst, P, g, x, y, v);
        if (x + 1 < g.nx) {
#pragma unroll
            for (int i = 0; i < Q; ++i) v[i] = o[i].y;
            store9<float, float>(dst, P, g, x + 1, y, v);
        }
    }
}

// After the tile's barrier: collide the thread's nodes from the pulled values fr and the density
// tile R into the outgoing tile `out` (one TMA store per tile takes it away: nine 8-byte shared
// stores at fixed offsets from one address in place of nine global ones with an address each), and
// write the ghost copies of a tile near an edge to dst.  xi49: the (xi_4, xi_9) field of MODE 2 (nx even
// there); z4, z9 and xch: the in-block sums and the exchange of MODE 3.
template <int MODE, bool POLY, int TX, int TY, int NT, typename Args>
__device__ __forceinline__ void tile_collide(const Args& a, const PairLocal* loc,
                                             const F2 (&fr)[PairMap<TX, TY, NT>::RPT][Q], const float* R,
                                             const Grid& g, int x0, int y0, float* out, float* dst, const float2* __restrict__ xi49,
                                             const F2 (&z4)[PairMap<TX, TY, NT>::RPT],
                                             const F2 (&z9)[PairMap<TX, TY, NT>::RPT], const unsigned char* xch) {
    using TT = TmaTile<TX, TY>;
    using M = PairMap<TX, TY, NT>;
    using ST = StencilTile<TX, TY, NT>;
    const int tid = threadIdx.x;
    const int p = tid % M::PX, rb = tid / M::PX;
    const int lx = 2 * p, ly = rb * M::RPT;
    const int x = x0 + lx;
    if ((M::ACTIVE < NT && tid >= M::ACTIVE) || x >= g.nx || y0 + ly >= g.ny) return;
    const bool edge = x0 < Elem<float>::GW || x0 + TX > g.nx - Elem<float>::GW || y0 < 2 || y0 + TY > g.ny - 2;
    const float* r0 = R + (ly + 1) * TT::RW + lx + 2;
    float* po = out + ly * TX + lx;
    RhoRow m = rho_row(r0 - TT::RW), c = rho_row(r0);
#pragma unroll
    for (int j = 0; j < M::RPT; ++j) {
        const int y = y0 + ly + j;
        const RhoRow n = rho_row(r0 + (j + 1) * TT::RW);
        if (j > 0 && y >= g.ny) return;
        const F2 lap6 = fma2(c.C, bc(-20.0f), fma2(add2(c.s, add2(n.C, m.C)), bc(4.0f), add2(n.s, m.s)));
        const F2 gx12 = fma2(c.d, bc(4.0f), add2(n.d, m.d));
        const F2 gy12 = fma2(sub2(n.C, m.C), bc(4.0f), sub2(n.s, m.s));
        const uint32_t node = (uint32_t)y * (uint32_t)g.nx + (uint32_t)x;
        F2 v4 = bc(0.f), v9 = bc(0.f);
        if constexpr (MODE == 2) {
            const float4 v = *reinterpret_cast<const float4*>(xi49 + (long long)y * g.nx + x);
            v4 = mul2(make_float2(v.x, v.z), bc(0.25f));
            v9 = mul2(make_float2(v.y, v.w), bc(0.0625f));
        }
        if constexpr (MODE == 3) {
            const F2 e = reinterpret_cast<const F2*>(xch + ST::ER)[(ly + j) * ST::W + p];
            const F2 q = reinterpret_cast<const F2*>(xch + ST::ED)[(ly + j) * ST::W + p];
            v4 = z4[j];
            v9 = z9[j];
            if (j == 0) {
                const float4 u = reinterpret_cast<const float4*>(xch + ST::UP)[rb * M::PX + p];
                v4 = add2(v4, make_float2(u.x, u.y));
                v9 = add2(v9, make_float2(u.z, u.w));
            }
            v4.x += e.x + q.x;
            v9.x += e.y + q.y;
        }
        F2 o[Q];
        collide_pair<MODE, POLY>(a, loc, fr[j], c.C, lap6, gx12, gy12, node, v4, v9, o);
#pragma unroll
        for (int i = 0; i < Q; ++i) put_pair(po + (i * TY + j) * TX, o[i]);
        if (edge && tile_direct<TX>(g, x0)) store_pair(dst, g.plane, g, x, y, o);
        if (edge) ghost_pair(dst, g.plane, g, x, y, o);
        m = c;
        c = n;
    }
}

}  // namespace lbf
