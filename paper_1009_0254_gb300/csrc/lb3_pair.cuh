// lb3_pair.cuh -- packed FP32 (add, mul, fma .f32x2) in the FP32 step kernels of lb3d_kernel.cuh: the
// D3Q27 collision and the normals of both lattices; FP64 keeps collide27.
//
// The arithmetic of one node is packed where its structure gives pairs:
//   * sum and difference of two values are one instruction, (a + b, a - b) = b (1, -1) + (a, a);
//   * the z = +1, -1 values of a D3Q27 column are one pair through the x and y transforms;
//   * a Box-Muller evaluation takes two Philox words (gauss2 of lb_pair.cuh);
//   * the 1/6 of each axis of the D3Q27 back-transform is in the rates and noise factors (host side).
// D3Q27 1,564 -> 1,321 instructions a node.  The D3Q19 collision is packed in the correlated-noise kernel
// only: elsewhere 1,082 -> 1,005 instructions left the step time where it was (616 us at 256^3), and the
// mass of a noiseless run drifted three times as fast (rounding of the reordered increments).
#pragma once

#include "lb27_collide.cuh"
#include "lb3_collide.cuh"
#include "lb_pair.cuh"

namespace lbf3 {

using lbf::F2;
using lbf::add2;
using lbf::bc;
using lbf::fma2;
using lbf::mul2;
using lbf::sub2;

// (a + b, a - b)
__device__ __forceinline__ F2 sum_diff(float a, float b) { return fma2(bc(b), make_float2(1.f, -1.f), bc(a)); }

// D3Q27 density deviation: the pairs (+, -) along z of the nine columns, then their rest values
__device__ __forceinline__ float drho27_pairs(const float* f) {
    F2 t = make_float2(f[1], f[2]);
    float a = f[0];
#pragma unroll
    for (int j = 1; j < 9; ++j) {
        t = add2(t, make_float2(f[3 * j + 1], f[3 * j + 2]));
        a += f[3 * j];
    }
    return a + (t.x + t.y);
}

// D3Q19 in the correlated-noise kernel, collide19 with sums and differences of opposite velocities in
// one instruction.  A mode's increment D_a enters the back-transform times scale19(a) (collide19's factor
// over 36); rates and noise coefficients are given times it.
__host__ __device__ constexpr double scale19(int a) {
    return (a == 4 ? 1.5 : a == 5 ? 0.75 : a == 6 ? 2.25 : a <= 9 ? 9.0 : a <= 12 ? 1.5 : a <= 15 ? 4.5 : a == 16 ? 0.5
            : a == 17 ? 0.75 : 2.25) / 36.0;
}

// the relaxation rates of the modes times scale19
struct Lam19 {
    float l4, l5, l6, l7, l10, l13, l16, l17, l18;
};

// collide19 for xi[a] already times scale19 (a = 4..18)
__device__ __forceinline__ void collide19_f(const Coef3<float>& a, const Lam19& L, const float f[Q3], const Rho3<float>& r,
                                            const float xi[Q3], float o[Q3]) {
    const float c3 = 1.f / 3.f, c6 = 1.f / 6.f, c12 = 1.f / 12.f;
    const F2 rx = sum_diff(r.xp, r.xm), ry = sum_diff(r.yp, r.ym), rz = sum_diff(r.zp, r.zm);
    const F2 ra = sum_diff(r.ap, r.am), rb = sum_diff(r.bp, r.bm), rc = sum_diff(r.cp, r.cm);
    const F2 rd = sum_diff(r.dp, r.dm), re = sum_diff(r.ep, r.em), rf = sum_diff(r.fp, r.fm);
    const float sfc = (rx.x + ry.x) + rz.x;
    const float sed = ((ra.x + rb.x) + (rc.x + rd.x)) + (re.x + rf.x);
    const float lap = sfc * c3 + sed * c6 - 4.f * r.c;
    const float gx = rx.y * c6 + ((ra.y + rb.y) + (re.y - rf.y)) * c12;
    const float gy = ry.y * c6 + ((ra.y - rb.y) + (rc.y + rd.y)) * c12;
    const float gz = rz.y * c6 + ((rc.y - rd.y) + (re.y + rf.y)) * c12;

    const F2 X = sum_diff(f[1], f[2]), Y = sum_diff(f[3], f[4]), Z = sum_diff(f[5], f[6]);
    const F2 A = sum_diff(f[7], f[10]), B = sum_diff(f[8], f[9]), C = sum_diff(f[11], f[14]);
    const F2 D = sum_diff(f[12], f[13]), E = sum_diff(f[15], f[18]), F = sum_diff(f[16], f[17]);
    const float sAB = A.x + B.x, sCD = C.x + D.x, sEF = E.x + F.x;
    const float sedge = (sAB + sCD) + sEF, sface = (X.x + Y.x) + Z.x;
    const float drho = f[0] + (sface + sedge);
    const float qab = A.y + B.y, qef = E.y - F.y, qa_b = A.y - B.y, qcd = C.y + D.y, qc_d = C.y - D.y, qe_f = E.y + F.y;
    const float ex = qab + qef, ey = qa_b + qcd, ez = qc_d + qe_f;      // edge momenta
    const float jx = X.y + ex, jy = Y.y + ey, jz = Z.y + ez;
    const float m4 = sedge - f[0];
    const float t5 = (sAB + sEF) - 2.f * sCD, t6 = sAB - sEF;
    const float m5 = ((2.f * X.x - Y.x) - Z.x) + t5;
    const float m6 = (Y.x - Z.x) + t6;
    const float m16 = f[0] - 2.f * sface + sedge;
    const float m17 = ((Y.x + Z.x) - 2.f * X.x) + t5;
    const float m18 = (Z.x - Y.x) + t6;

    const float rho = a.rho0 + drho;
    const float inv = recip19(rho);
    const float ux = jx * inv, uy = jy * inv, uz = jz * inv;
    const float kx = a.kappa * gx, ky = a.kappa * gy, kz = a.kappa * gz;
    const float jxx = jx * ux, jyy = jy * uy, jzz = jz * uz;
    const float pxx = jxx + kx * gx, pyy = jyy + ky * gy, pzz = jzz + kz * gz;
    const float kg2 = (kx * gx + ky * gy) + kz * gz;
    const float klap = a.kappa * rho * lap;
    const float dd = pressure_slope(a, drho);
    const float iso = dd * drho - 3.f * klap;
    const float e4 = (iso + ((jxx + jyy) + jzz)) - 0.5f * kg2;
    const float e16 = -iso - 4.5f * kg2;

    // h_a / 36 with h_a of collide19
    const float h4 = L.l4 * (m4 - e4) + xi[4];
    const float h5 = L.l5 * (m5 - ((2.f * pxx - pyy) - pzz)) + xi[5];
    const float h6 = L.l6 * (m6 - (pyy - pzz)) + xi[6];
    const float h7 = L.l7 * ((A.x - B.x) - (jx * uy + kx * gy)) + xi[7];
    const float h8 = L.l7 * ((C.x - D.x) - (jy * uz + ky * gz)) + xi[8];
    const float h9 = L.l7 * ((E.x - F.x) - (jz * ux + kz * gx)) + xi[9];
    const float h10 = L.l10 * (ex - 2.f * X.y) + xi[10];
    const float h11 = L.l10 * (ey - 2.f * Y.y) + xi[11];
    const float h12 = L.l10 * (ez - 2.f * Z.y) + xi[12];
    const float h13 = L.l13 * (qab - qef) + xi[13];
    const float h14 = L.l13 * (qcd - qa_b) + xi[14];
    const float h15 = L.l13 * (qe_f - qc_d) + xi[15];
    const float h16 = L.l16 * (m16 - e16) + xi[16];
    const float h17 = L.l17 * m17 + xi[17];
    const float h18 = L.l18 * m18 + xi[18];

    // back: a pair's even part and its odd part, faces twice the edges
    auto pair = [&](int i, int k, float ev, float od) {
        const F2 v = add2(make_float2(f[i], f[k]), sum_diff(ev, od));
        o[i] = v.x;
        o[k] = v.y;
    };
    o[0] = f[0] + 12.f * (h16 - h4);
    const float s57 = h5 + h17, d57 = h17 - h5, s68 = h6 + h18, d68 = h6 - h18;
    pair(1, 2, -4.f * (h16 + d57), -4.f * h10);
    pair(3, 4, 2.f * ((d57 + d68) - 2.f * h16), -4.f * h11);
    pair(5, 6, 2.f * ((d57 - d68) - 2.f * h16), -4.f * h12);
    const float h416 = h4 + h16, e1 = h416 + s57;
    const float exy = e1 + s68, ezx = e1 - s68, eyz = h416 - 2.f * s57;
    const float p1 = h10 + h11, n1 = h10 - h11, p2 = h11 + h12, n2 = h11 - h12, p3 = h10 + h12, n3 = h12 - h10;
    const float b1 = h13 - h14, b2 = h13 + h14, b3 = h14 - h15, b4 = h14 + h15, b5 = h15 - h13, b6 = h13 + h15;
    pair(7, 10, exy + h7, p1 + b1);
    pair(8, 9, exy - h7, n1 + b2);
    pair(11, 14, eyz + h8, p2 + b3);
    pair(12, 13, eyz - h8, n2 + b4);
    pair(15, 18, ezx + h9, p3 + b5);
    pair(16, 17, ezx - h9, n3 + b6);
}

// D3Q27 FP32: modes with p_2 on an odd number of axes are carried with their sign flipped (x0 - 2 s is
// one packed fma, 2 s - x0 two instructions), increments over 216 = 6^3
__host__ __device__ constexpr double sign27(int k) {
    return ((k / 9 == 2) + ((k / 3) % 3 == 2) + (k % 3 == 2)) % 2 ? -1.0 : 1.0;
}
constexpr double SCALE27 = 1.0 / 216.0;

// collide27 for xi[k] already times sign27(k) SCALE27; co's rates times SCALE27
template <bool NOISE>
__device__ __forceinline__ void collide27_f(const Coef3<float>& a, const float f[Q27], const float nb[Q27],
                                            const float xi[Q27], float o[Q27]) {
    // Appendix B's stencils: 4 t0 + (t+ + t-) and t+ - t- along z, y, x (216 and 216 times the weighted
    // sums; a.kappa's products take the powers of 72)
    float gx, gy, gz, lap;
    {
        F2 zz[9];                                // (weighted sum, difference) along z of column 3 ix + iy
#pragma unroll
        for (int j = 0; j < 9; ++j) {
            const F2 sd = sum_diff(nb[3 * j + 1], nb[3 * j + 2]);
            zz[j] = make_float2(4.f * nb[3 * j] + sd.x, sd.y);
        }
        F2 yy[3];
        float wy[3];
#pragma unroll
        for (int ix = 0; ix < 3; ++ix) {
            yy[ix] = fma2(zz[3 * ix], bc(4.f), add2(zz[3 * ix + 1], zz[3 * ix + 2]));
            wy[ix] = zz[3 * ix + 1].x - zz[3 * ix + 2].x;
        }
        const F2 t = fma2(yy[0], bc(4.f), add2(yy[1], yy[2]));
        lap = t.x * (1.f / 36.f) - 6.f * nb[0];
        gz = t.y * (1.f / 72.f);
        gx = (yy[1].x - yy[2].x) * (1.f / 72.f);
        gy = (4.f * wy[0] + (wy[1] + wy[2])) * (1.f / 72.f);
    }

    // moments, z then y then x; a_[j]: the column's p_0 part, b_[j]: its (p_1, -p_2) parts
    float A[9];
    F2 B[9];
#pragma unroll
    for (int j = 0; j < 9; ++j) {
        const F2 sd = sum_diff(f[3 * j + 1], f[3 * j + 2]);
        A[j] = f[3 * j] + sd.x;
        B[j] = make_float2(sd.y, f[3 * j] - 2.f * sd.x);
    }
    auto fwd1 = [](float& x0, float& x1, float& x2) {
        const float s = x1 + x2, d = x1 - x2, m2 = x0 - 2.f * s;
        x0 = x0 + s;
        x1 = d;
        x2 = m2;
    };
    auto fwd2 = [](F2& x0, F2& x1, F2& x2) {
        const F2 s = add2(x1, x2), d = sub2(x1, x2), m2 = fma2(s, bc(-2.f), x0);
        x0 = add2(x0, s);
        x1 = d;
        x2 = m2;
    };
#pragma unroll
    for (int ix = 0; ix < 3; ++ix) {
        fwd1(A[3 * ix], A[3 * ix + 1], A[3 * ix + 2]);
        fwd2(B[3 * ix], B[3 * ix + 1], B[3 * ix + 2]);
    }
#pragma unroll
    for (int iy = 0; iy < 3; ++iy) {
        fwd1(A[iy], A[3 + iy], A[6 + iy]);
        fwd2(B[iy], B[3 + iy], B[6 + iy]);
    }
    // mode 9 a + 3 b + c is A[3 a + b] for c = 0, B[3 a + b].x and .y for c = 1, 2
    const float drho = A[0], jx = A[3], jy = A[1], jz = B[0].x;
    const float rho = a.rho0 + drho;
    const float inv = recip19(rho);
    const float ux = jx * inv, uy = jy * inv, uz = jz * inv;
    const float kx = a.kappa * gx, ky = a.kappa * gy, kz = a.kappa * gz;
    const float kg2 = (kx * gx + ky * gy) + kz * gz;
    const float klap = a.kappa * rho * lap;
    const float dd = pressure_slope(a, drho);
    const float iso = dd * drho - 3.f * klap;
    const float base2 = iso - 1.5f * kg2;
    const float e18 = base2 + 3.f * (jx * ux + kx * gx), e6 = base2 + 3.f * (jy * uy + ky * gy);
    const float e2 = base2 + 3.f * (jz * uz + kz * gz);
    const float e12 = jx * uy + kx * gy, e4 = jy * uz + ky * gz, e10 = jx * uz + kx * gz;
    const float e44 = -iso - 1.5f * kg2;
    // m - m^eq of the modes with an equilibrium (signs as carried: 2, 6, 18, 26 flipped)
    A[4] -= e12;
    B[1].x -= e4;
    B[3].x -= e10;
    A[8] -= e44;
    B[2].y -= e44;
    B[6].y -= e44;
    B[8].y += base2;
    const float dx2 = A[6] + e18, dy2 = A[2] + e6, dz2 = B[0].y + e2;
    const float bulk = (a.lb - a.ls) * (((dx2 + dy2) + dz2) * (1.f / 3.f));
    // increments over 216
    auto inc = [&](float l, float d, int k) { return NOISE ? l * d + xi[k] : l * d; };
    const float d12 = inc(a.ls, A[4], 12), d4 = inc(a.ls, B[1].x, 4), d10 = inc(a.ls, B[3].x, 10);
    const float d18 = inc(a.ls, dx2, 18) + bulk, d6 = inc(a.ls, dy2, 6) + bulk, d2 = inc(a.ls, dz2, 2) + bulk;
#pragma unroll
    for (int j = 0; j < 9; ++j) {
        A[j] = inc(a.lg, A[j], 3 * j);
        if constexpr (NOISE) B[j] = fma2(B[j], bc(a.lg), make_float2(xi[3 * j + 1], xi[3 * j + 2]));
        else B[j] = mul2(B[j], bc(a.lg));
    }
    A[0] = 0.f;
    A[1] = 0.f;
    A[3] = 0.f;
    A[4] = d12;
    A[6] = d18;
    A[2] = d6;
    B[0] = make_float2(0.f, d2);
    B[1].x = d4;
    B[3].x = d10;

    // back, x then y then z: 6 g(0) = 4 h0 - 2 h2, 6 g(+-) = (h0 + h2) +- 3 h1, with -h2 as carried
    auto bwd1 = [](float& h0, float& h1, float& h2) {
        const float g0 = 4.f * h0 + 2.f * h2, e = h0 - h2;
        h2 = e - 3.f * h1;
        h1 = e + 3.f * h1;
        h0 = g0;
    };
    auto bwd2 = [](F2& h0, F2& h1, F2& h2) {
        const F2 g0 = fma2(h0, bc(4.f), add2(h2, h2)), e = sub2(h0, h2);
        h2 = fma2(h1, bc(-3.f), e);
        h1 = fma2(h1, bc(3.f), e);
        h0 = g0;
    };
#pragma unroll
    for (int iy = 0; iy < 3; ++iy) {
        bwd1(A[iy], A[3 + iy], A[6 + iy]);
        bwd2(B[iy], B[3 + iy], B[6 + iy]);
    }
#pragma unroll
    for (int ix = 0; ix < 3; ++ix) {
        bwd1(A[3 * ix], A[3 * ix + 1], A[3 * ix + 2]);
        bwd2(B[3 * ix], B[3 * ix + 1], B[3 * ix + 2]);
    }
#pragma unroll
    for (int j = 0; j < 9; ++j) {
        const float h1 = B[j].x, h2 = B[j].y, e = A[j] - h2;
        o[3 * j] = f[3 * j] + (4.f * A[j] + 2.f * h2);
        const F2 v = add2(make_float2(f[3 * j + 1], f[3 * j + 2]), fma2(bc(h1), make_float2(3.f, -3.f), bc(e)));
        o[3 * j + 1] = v.x;
        o[3 * j + 2] = v.y;
    }
}

// the normals (over GAUSS_SCALE) of the four words of one Philox draw, in word order
__device__ __forceinline__ void normals8(const uint4& r, float n[8]) {
    F2 a, b;
    lbf::gauss2(r.x, r.y, &a, &b);
    n[0] = a.x; n[1] = b.x; n[2] = a.y; n[3] = b.y;
    lbf::gauss2(r.z, r.w, &a, &b);
    n[4] = a.x; n[5] = b.x; n[6] = a.y; n[7] = b.y;
}

}  // namespace lbf3
