// btrt_sweep3.cuh -- device side of the fused B-TriRT sweep on the D3Q19 lattice.
//
// Same scheme as the D2Q9 sweep in three dimensions (the appendix's D3Q19
// relaxation matrix S_f = diag(k0, K1, k2 I_6, k0 I_9) with a 3x3 first-order
// block K1 = (3 A^ + I/2)^-1 from Eq. 30, k2 from Eq. 62 at the mean rate
// 1/k1_eff = tr(K1^-1)/3, the correction of Eq. 11 and scheme-2 sources).  One
// thread owns one node; the sweep pulls f_i(x) = f_i^+(x - c_i), replaces links
// that cross bounce-back faces (one face, or two at an edge: mean of their
// values) by -f_opp^+(x) + wall term, collides in moment space and writes f^+
// and phi to the other buffers.  Lattice units (c = 1, cs^2 = 1/3).
//
// Velocity order (columns of Eq. 86): 0 rest; 1, 2 = +-x; 3, 4 = +-y; 5, 6 = +-z;
// 7 (1,1,0) 8 (-1,1,0) 9 (1,-1,0) 10 (-1,-1,0); 11 (1,0,1) 12 (-1,0,1)
// 13 (1,0,-1) 14 (-1,0,-1); 15 (0,1,1) 16 (0,-1,1) 17 (0,1,-1) 18 (0,-1,-1).
// Weights 1/3, 1/18, 1/36.  Populations are stored in the forms of the D2Q9
// sweep (unshifted FP64, or FP32/FP16/BF16 shifted by w_i phi_ref or by w_i phi
// of the writing node).
#pragma once

#include "btrt_sweep.cuh"

namespace btrt {

__host__ __device__ constexpr int cx3(int i) {
    return (i == 1 || i == 7 || i == 9 || i == 11 || i == 13) ? 1
           : (i == 2 || i == 8 || i == 10 || i == 12 || i == 14) ? -1 : 0;
}
__host__ __device__ constexpr int cy3(int i) {
    return (i == 3 || i == 7 || i == 8 || i == 15 || i == 17) ? 1
           : (i == 4 || i == 9 || i == 10 || i == 16 || i == 18) ? -1 : 0;
}
__host__ __device__ constexpr int cz3(int i) {
    return (i == 5 || i == 11 || i == 12 || i == 15 || i == 16) ? 1
           : (i == 6 || i == 13 || i == 14 || i == 17 || i == 18) ? -1 : 0;
}
// opposite directions (checked against cx3/cy3/cz3 by a static assertion below)
__host__ __device__ constexpr int opposite3(int i) {
    constexpr int o[19] = {0, 2, 1, 4, 3, 6, 5, 10, 9, 8, 7, 14, 13, 12, 11, 18, 17, 16, 15};
    return o[i];
}
__host__ __device__ constexpr bool opposites_ok() {
    for (int i = 0; i < 19; ++i) {
        const int o = opposite3(i);
        if (cx3(o) != -cx3(i) || cy3(o) != -cy3(i) || cz3(o) != -cz3(i)) return false;
    }
    return true;
}
static_assert(opposites_ok(), "D3Q19 opposite table");

template <typename Real> __device__ __forceinline__ Real wgt3(int i) {
    return i == 0 ? cst<Real>(1, 3) : (i <= 6 ? cst<Real>(1, 18) : cst<Real>(1, 36));
}

// Constants of the integer collision: FP64 lattices only.
template <typename Real> struct FxPart3 {};
template <> struct FxPart3<double> {
    FxFold3 fx;
};

template <typename Real>
struct Sweep3Params : FxPart3<Real> {
    const void *fin;       // post-collision populations of the previous step: 19 planes, `plane` apart
    void *fout;
    const Real *phi_in;    // phi of the nodes that wrote fin
    Real *phi_out;
    int nx, ny, nz;
    int pitch;             // elements between rows
    int slab;              // elements between z layers (pitch * ny)
    int plane;             // elements between population planes; 19 * plane < 2^31
    int hbb_x, hbb_y, hbb_z;
    Real wall[6];          // wall value per face (x-, x+, y-, y+, z-, z+), times wall_fac
    Real wall_fac;
    Real wref[3];          // w phi_ref for |c|^2 = 0, 1, 2 (reference shift)
    Real phi_ref;

    Real ux, uy, uz;       // B = u phi + bg phi^q
    Real bgx, bgy, bgz, bq;
    int bq2;
    int bq_n, bq_h;        // q = bq_n + bq_h / 2 when bq_n >= 0 (products and a square root)
    Real c3;               // C = phi + c3 phi^3
    Real A0[6];            // xx, xy, xz, yy, yz, zz (lattice units)
    Real a2;
    Real k0, om;           // k0, 1 - k0
    int nonlin;            // 1: A depends on phi (K1, k2 per node) or B, C nonlinear
    int k2_hbb;
    Real k2c;
    Real K1[6];            // constant K1 (symmetric) and k2 when A is constant
    Real k2;
    Real Q[3];             // diagonal of K1 - k0 I (constant K1)
    Real ka[3];            // w_i kap, kap = (9/2)(k2 - k0), for |c|^2 = 0, 1, 2 (constant k2)
    Real kak[3];           // -(3/2) k0, -k0/4, -k0/8: w_i kap = (3/2, 1/4, 1/8) k2 + kak (k2 per node)
    Real a2x3, k0x15;      // 3 a2, (3/2) k0
    int k0_one;            // 1: k0 == 1
    Real Ku[3];            // constant-coefficient fold: K1 u (B = u phi)
    Real gu[3];            //   and (I - K1/2) u
    Real cond_limit;       // FP32: tr^3 > cond_limit det -> build and invert the block in FP64
    double A0d[6], a2d;    // A0^ and a2 in FP64 for that path

    int src_kind;          // 0 none, 1 const, 3 per-node field, 4 reaction
    Real src_val;          // dt S (const), dt (3 T_n - T_{n-1}) / 2 (field), dt (reaction)
    const Real *srcF;      // field: F(x) per node (pitched)
    Real react_rate, react_exp;
    int react2;
    int re_n, re_h;

    int first;
    int *flags;            // bit 0: non-finite phi
};

template <typename Real>
__device__ __forceinline__ Real wall3_term(const Sweep3Params<Real> &p, int n2, Real phi_w) {
    // 2 x even part of f^eq at phi_w: 2 w [phi_w + (C - phi_w)(3/2)(|c|^2 - 1)]
    const Real w = n2 == 0 ? cst<Real>(1, 3) : (n2 == 1 ? cst<Real>(1, 18) : cst<Real>(1, 36));
    const Real dC = p.c3 * phi_w * phi_w * phi_w;
    return Real(2) * w * fma(dC, Real(1.5) * Real(n2 - 1), phi_w);
}

// Shifted equilibrium (Eq. 7, D = C I) for the initialising collision.
template <typename Real, int SH>
__device__ __forceinline__ void equilibrium3(const Sweep3Params<Real> &p, Real phi, Real (&f)[19]) {
    const Real g = p.bq2 ? phi * phi : pow_half(phi, p.bq, p.bq_n, p.bq_h);
    const Real Bx = Real(3) * fma(p.ux, phi, p.bgx * g);
    const Real By = Real(3) * fma(p.uy, phi, p.bgy * g);
    const Real Bz = Real(3) * fma(p.uz, phi, p.bgz * g);
    const Real Cm = Real(1.5) * p.c3 * phi * phi * phi;   // (3/2)(C - phi)
#pragma unroll
    for (int i = 0; i < 19; ++i) {
        const int n2 = cx3(i) * cx3(i) + cy3(i) * cy3(i) + cz3(i) * cz3(i);
        Real v = fma(Cm, Real(n2 - 1), phi);
        v = v + Real(cx3(i)) * Bx + Real(cy3(i)) * By + Real(cz3(i)) * Bz;
        f[i] = wgt3<Real>(i) * v;
        if constexpr (SH == kShiftRef) f[i] = f[i] - p.wref[n2];
        if constexpr (SH == kShiftLocal) f[i] = fma(-wgt3<Real>(i), phi, f[i]);
    }
}

// K1 = (3 A^ + I/2)^-1 (Eq. 30) for A^ = (1 + a2 phi^2) A0^ (xx, xy, xz, yy, yz,
// zz), built and inverted in FP64 by cofactors and rounded to FP32: the FP32
// sweep's path for ill-conditioned blocks, not inlined so that well-conditioned
// nodes issue none of its FP64 instructions.
struct K1f3 {
    float v[6];
};
static __device__ __noinline__ K1f3 k1_fp64_3(double phi, double a2, const double *A0) {
    const double s3d = 3.0 + 3.0 * a2 * phi * phi;
    const double dxx = s3d * A0[0] + 0.5, dxy = s3d * A0[1], dxz = s3d * A0[2];
    const double dyy = s3d * A0[3] + 0.5, dyz = s3d * A0[4], dzz = s3d * A0[5] + 0.5;
    const double ex = dyy * dzz - dyz * dyz, exy = dxz * dyz - dxy * dzz, exz = dxy * dyz - dxz * dyy;
    const double ey = dxx * dzz - dxz * dxz, eyz = dxy * dxz - dxx * dyz, ez = dxx * dyy - dxy * dxy;
    const double id = 1.0 / (dxx * ex + dxy * exy + dxz * exz);
    return K1f3{{(float)(ex * id), (float)(exy * id), (float)(exz * id), (float)(ey * id), (float)(eyz * id),
                 (float)(ez * id)}};
}

// Moment-space collision of one node in shifted form d_i = f_i - w_i rs
// (rs = 0, phi_ref or phi^{n-1} of the node):
//   d_i^+ = (1 - k0) d_i + w_i [a + cC_i + 3 c_i.V - kap H_i],
//   a = k0 (phi - rs) + source, cC_i = (3/2) k0 (C - phi)(|c_i|^2 - 1),
//   V = k0 B - (K1 - k0 I)(M1) + (I - K1/2) dB, M1 = j - B,
//   H_i = c_i c_i : M2 - tr(M2)/3, M2 = Pi - (C - rs)/3 I, kap = (9/2)(k2 - k0).
// Returns phi; phid = phi - rs.
template <typename Real, int MODE, int SRC, int SH>
__device__ __forceinline__ Real collide3(const Sweep3Params<Real> &p, Real (&d)[19], Real rs, Real phi_prev,
                                         Real srcv, bool first, Real &phid_out) {
    // moments of the shifted populations
    const Real ax = d[1] + d[2], ay = d[3] + d[4], az = d[5] + d[6];
    const Real sxy = (d[7] + d[8]) + (d[9] + d[10]);
    const Real sxz = (d[11] + d[12]) + (d[13] + d[14]);
    const Real syz = (d[15] + d[16]) + (d[17] + d[18]);
    const Real phid = ((d[0] + (ax + ay)) + (az + sxy)) + (sxz + syz);
    phid_out = phid;
    Real phi = phid;
    if constexpr (SH != kShiftNone) phi = phid + rs;
    const Real jx = (d[1] - d[2]) + ((d[7] - d[8]) + (d[9] - d[10])) + ((d[11] - d[12]) + (d[13] - d[14]));
    const Real jy = (d[3] - d[4]) + ((d[7] + d[8]) - (d[9] + d[10])) + ((d[15] - d[16]) + (d[17] - d[18]));
    const Real jz = (d[5] - d[6]) + ((d[11] + d[12]) - (d[13] + d[14])) + ((d[15] + d[16]) - (d[17] + d[18]));
    const Real Pxx = (ax + sxy) + sxz, Pyy = (ay + sxy) + syz, Pzz = (az + sxz) + syz;
    const Real Pxy = (d[7] - d[8]) - (d[9] - d[10]);
    const Real Pxz = (d[11] - d[12]) - (d[13] - d[14]);
    const Real Pyz = (d[15] - d[16]) - (d[17] - d[18]);
    const Real dphi = first ? Real(0) : (SH == kShiftLocal ? phid : phi - phi_prev);

    // coefficients
    Real Bx, By, Bz, dBx, dBy, dBz, Cm = Real(0);
    Real Kxx, Kxy, Kxz, Kyy, Kyz, Kzz, k2 = Real(0);
    if constexpr (MODE == kGeneral) {
        const Real p2 = phi * phi;
        if (p.bq2) {
            Bx = fma(p.ux, phi, p.bgx * p2);
            By = fma(p.uy, phi, p.bgy * p2);
            Bz = fma(p.uz, phi, p.bgz * p2);
            const Real sp = phi + phi_prev;
            dBx = fma(p.bgx, sp, p.ux) * dphi;
            dBy = fma(p.bgy, sp, p.uy) * dphi;
            dBz = fma(p.bgz, sp, p.uz) * dphi;
        } else {
            const Real gq = pow_half(phi, p.bq, p.bq_n, p.bq_h);
            const Real dg = first ? Real(0) : gq - pow_half(phi_prev, p.bq, p.bq_n, p.bq_h);
            Bx = fma(p.ux, phi, p.bgx * gq);
            By = fma(p.uy, phi, p.bgy * gq);
            Bz = fma(p.uz, phi, p.bgz * gq);
            dBx = fma(p.ux, dphi, p.bgx * dg);
            dBy = fma(p.uy, dphi, p.bgy * dg);
            dBz = fma(p.uz, dphi, p.bgz * dg);
        }
        Cm = p.c3 * p2 * phi;
        // K1 = (3 A^ + I/2)^-1, A^ = (1 + a2 phi^2) A0^ (Eq. 30), symmetric 3x3 by cofactors
        const Real s3 = fma(p.a2x3, p2, Real(3));
        const Real mxx = fma(s3, p.A0[0], Real(0.5)), mxy = s3 * p.A0[1], mxz = s3 * p.A0[2];
        const Real myy = fma(s3, p.A0[3], Real(0.5)), myz = s3 * p.A0[4];
        const Real mzz = fma(s3, p.A0[5], Real(0.5));
        const Real cxx = fma(myy, mzz, -(myz * myz));
        const Real cxy = fma(mxz, myz, -(mxy * mzz));
        const Real cxz = fma(mxy, myz, -(mxz * myy));
        const Real cyy = fma(mxx, mzz, -(mxz * mxz));
        const Real cyz = fma(mxy, mxz, -(mxx * myz));
        const Real czz = fma(mxx, myy, -(mxy * mxy));
        const Real det = fma(mxx, cxx, fma(mxy, cxy, mxz * cxz));
        const Real tr = (mxx + myy) + mzz;
        bool ill = false;
        if constexpr (sizeof(Real) == 4) ill = tr * tr * tr > p.cond_limit * det;
        if (ill) {
            // ill-conditioned FP32 block: rebuilt from FP64 coefficients (FP32-rounded
            // entries carry errors the condition number amplifies), inverted in FP64
            const K1f3 k = k1_fp64_3(static_cast<double>(phi), p.a2d, p.A0d);
            Kxx = (Real)k.v[0]; Kxy = (Real)k.v[1]; Kxz = (Real)k.v[2];
            Kyy = (Real)k.v[3]; Kyz = (Real)k.v[4]; Kzz = (Real)k.v[5];
        } else {
            const Real id = quot(Real(1), det);
            Kxx = cxx * id; Kxy = cxy * id; Kxz = cxz * id;
            Kyy = cyy * id; Kyz = cyz * id; Kzz = czz * id;
        }
        // Eq. 62 at k1_eff = 3/tr:  k2 = (8/3)(2 tr - 3) / (4 tr - 3)
        k2 = p.k2_hbb ? quot(cst<Real>(8, 3) * fma(Real(2), tr, Real(-3)), fma(Real(4), tr, Real(-3))) : p.k2c;
    } else {
        Bx = By = Bz = dBx = dBy = dBz = Real(0);   // folded into Ku, gu below
        Kxx = p.K1[0]; Kxy = p.K1[1]; Kxz = p.K1[2]; Kyy = p.K1[3]; Kyz = p.K1[4]; Kzz = p.K1[5];
    }
    // V = k0 B - (K1 - k0 I)(j - B) + (I - K1/2) dB = K1 (B - j - dB/2) + k0 j + dB,
    // dB = B^n - B^{n-1} (its first form takes 36 operations, the second 18); for
    // B = u phi it is K1 u phi - (K1 - k0 I) j + (I - K1/2) u dphi
    Real Vx, Vy, Vz;
    if constexpr (MODE == kGeneral) {
        const Real ex = fma(Real(-0.5), dBx, Bx - jx);
        const Real ey = fma(Real(-0.5), dBy, By - jy);
        const Real ez = fma(Real(-0.5), dBz, Bz - jz);
        Vx = fma(Kxx, ex, fma(Kxy, ey, fma(Kxz, ez, fma(p.k0, jx, dBx))));
        Vy = fma(Kxy, ex, fma(Kyy, ey, fma(Kyz, ez, fma(p.k0, jy, dBy))));
        Vz = fma(Kxz, ex, fma(Kyz, ey, fma(Kzz, ez, fma(p.k0, jz, dBz))));
    } else {
        (void)Bx; (void)By; (void)Bz; (void)dBx; (void)dBy; (void)dBz;
        const Real qx = fma(p.Q[0], jx, fma(Kxy, jy, Kxz * jz));
        const Real qy = fma(Kxy, jx, fma(p.Q[1], jy, Kyz * jz));
        const Real qz = fma(Kxz, jx, fma(Kyz, jy, p.Q[2] * jz));
        Vx = fma(p.gu[0], dphi, fma(p.Ku[0], phi, -qx));
        Vy = fma(p.gu[1], dphi, fma(p.Ku[1], phi, -qy));
        Vz = fma(p.gu[2], dphi, fma(p.Ku[2], phi, -qz));
    }

    // second-order non-equilibrium moments M2 = Pi - (C - rs)/3 I: the deviatoric
    // parts h_a = Pi_aa - tr(Pi)/3 (C and the shift cancel from them) and
    // t3 = tr(M2)/3; H_i = c_i c_i : M2 - t3 is then h_a (axis a), t3 - h_c (the
    // face diagonals normal to axis c, from h_x + h_y + h_z = 0) +- 2 M_ab
    const Real third = cst<Real>(1, 3);
    const Real tP3 = third * ((Pxx + Pyy) + Pzz);
    const Real hx = Pxx - tP3, hy = Pyy - tP3, hz = Pzz - tP3;
    const Real cmid = MODE == kGeneral ? phid + Cm : phid;       // C - rs
    const Real t3 = fma(-third, cmid, tP3);
    // w_i kap for the three speeds, kap = (9/2)(k2 - k0)
    Real ka0, ka1, ka2;
    if constexpr (MODE == kGeneral) {
        ka0 = fma(Real(1.5), k2, p.kak[0]);
        ka1 = fma(Real(0.25), k2, p.kak[1]);
        ka2 = fma(Real(0.125), k2, p.kak[2]);
    } else {
        ka0 = p.ka[0];
        ka1 = p.ka[1];
        ka2 = p.ka[2];
    }

    Real a = MODE == kLinearK0One ? phid : p.k0 * phid;
    if constexpr (SRC == kSrcReaction || SRC == kSrcRuntime) {
        if (SRC == kSrcReaction || p.src_kind == kSrcReaction) {
            const Real Sn =
                p.react_rate * phi * (Real(1) - (p.react2 ? phi * phi : pow_half(phi, p.react_exp, p.re_n, p.re_h)));
            const Real Sp = first ? Sn
                                  : p.react_rate * phi_prev *
                                        (Real(1) - (p.react2 ? phi_prev * phi_prev
                                                             : pow_half(phi_prev, p.react_exp, p.re_n, p.re_h)));
            srcv = fma(Real(1.5), Sn, Real(-0.5) * Sp);
        }
    }
    if constexpr (SRC != kSrcNone) a = fma(p.src_val, srcv, a);
    const Real cC = MODE == kGeneral ? p.k0x15 * Cm : Real(0);   // (3/2) k0 (C - phi)

    const Real w0 = cst<Real>(1, 3), w1 = cst<Real>(1, 18), w2 = cst<Real>(1, 36);
    const Real v1 = cst<Real>(1, 6), v2 = cst<Real>(1, 12);      // 3 w1, 3 w2
    Real r[19];
    r[0] = fma(ka0, t3, w0 * (MODE == kGeneral ? a - cC : a));
    // axis directions: w1 (a - kap h_a) +- 3 w1 V_a
    const Real w1a = w1 * a;
    const Real bx = fma(-ka1, hx, w1a), by = fma(-ka1, hy, w1a), bz = fma(-ka1, hz, w1a);
    r[1] = fma(v1, Vx, bx); r[2] = fma(-v1, Vx, bx);
    r[3] = fma(v1, Vy, by); r[4] = fma(-v1, Vy, by);
    r[5] = fma(v1, Vz, bz); r[6] = fma(-v1, Vz, bz);
    // face diagonals: w2 (a + cC - kap (t3 - h_c)) -+ 2 w2 kap M_ab (2 w2 = w1) + 3 w2 c_i . V
    const Real G = fma(-ka2, t3, w2 * (MODE == kGeneral ? a + cC : a));
    const Real bxy = fma(ka2, hz, G), bxz = fma(ka2, hy, G), byz = fma(ka2, hx, G);
    const Real bxym = fma(-ka1, Pxy, bxy), bxyp = fma(ka1, Pxy, bxy);
    const Real bxzm = fma(-ka1, Pxz, bxz), bxzp = fma(ka1, Pxz, bxz);
    const Real byzm = fma(-ka1, Pyz, byz), byzp = fma(ka1, Pyz, byz);
    const Real sxyp = Vx + Vy, sxym = Vx - Vy;
    const Real sxzp = Vx + Vz, sxzm = Vx - Vz;
    const Real syzp = Vy + Vz, syzm = Vy - Vz;
    r[7] = fma(v2, sxyp, bxym);  r[10] = fma(-v2, sxyp, bxym);
    r[8] = fma(-v2, sxym, bxyp); r[9] = fma(v2, sxym, bxyp);
    r[11] = fma(v2, sxzp, bxzm); r[14] = fma(-v2, sxzp, bxzm);
    r[12] = fma(-v2, sxzm, bxzp); r[13] = fma(v2, sxzm, bxzp);
    r[15] = fma(v2, syzp, byzm); r[18] = fma(-v2, syzp, byzm);
    r[16] = fma(-v2, syzm, byzp); r[17] = fma(v2, syzm, byzp);
    // k0 = 1 (bitwise the same as (1 - k0) d_i + r_i); constant coefficients have their own variant
    if (MODE == kLinearK0One || (MODE == kGeneral && p.k0_one)) {
#pragma unroll
        for (int i = 0; i < 19; ++i) d[i] = r[i];
    } else {
#pragma unroll
        for (int i = 0; i < 19; ++i) d[i] = fma(p.om, d[i], r[i]);
    }
    return phi;
}

// ---------------------------------------------------------------- the FP64 collision on the integer pipes
// As in two dimensions (btrt_fx.cuh, collide_f64): the FP64 forms out of line for
// the nodes the integer form does not take.  FP64 alone takes 113 operations per node
// and ran at 0.83 of the FP64 pipe, 4.3 GLUPS at 128^3; with the integer form 15.5.
template <int MODE, int SRC>
static __device__ __noinline__ double collide3_f64_slow(const Sweep3Params<double> &p, double *t, double phi_prev,
                                                        double srcv) {
    double d[19], phid;
#pragma unroll
    for (int i = 0; i < 19; ++i) d[i] = t[i];
    if (fx_all_zero(d, phi_prev, SRC == kSrcNone || SRC == kSrcReaction ? 0.0 : srcv)) return 0.0;
    const double phi = collide3<double, MODE, SRC, kShiftNone>(p, d, 0.0, phi_prev, srcv, false, phid);
#pragma unroll
    for (int i = 0; i < 19; ++i) t[i] = d[i];
    return phi;
}
static __device__ __noinline__ void init3_f64_slow(const Sweep3Params<double> &p, double *t, double phi, double src) {
    double d[19];
    equilibrium3<double, kShiftNone>(p, phi, d);
#pragma unroll
    for (int i = 0; i < 19; ++i) t[i] = fma(wgt3<double>(i), src, d[i]);
}

BTRT_HD double reaction3(const Sweep3Params<double> &p, double phi) {
    return p.react_rate * phi * (1.0 - (p.react2 ? phi * phi : pow_half(phi, p.react_exp, p.re_n, p.re_h)));
}

// Per-node coefficients or a reaction source: integer moments and populations, FP64
// coefficients and V.
template <int MODE, int SRC>
BTRT_HD bool fx_collide_general3(const Sweep3Params<double> &p, double (&d)[19], double phi_prev,
                                                    double srcv, double &phi_out) {
    unsigned int em;
    const bool in = fx_common_exp(d, em);
    if (!in || fx_exp(phi_prev) > em + (2u << 20))
        return !in && fx_out_of_range<false>(d, phi_prev, SRC == kSrcNone || SRC == kSrcReaction ? 0.0 : srcv, phi_out);
    fx D[19];
#pragma unroll
    for (int i = 0; i < 19; ++i) D[i] = fx_from<kFxTop3>(d[i], em);
    FxMoments3 m = fx_moments3(D);
    const double phi = fx_to<kFxTop3>(m.phi, em);
    // k0 phi + source stays in its word below 15 2^58 units for every k0 below 2
    const bool k0_one = MODE == kLinearK0One || p.k0_one, fits = k0_one || fx_below<15 << 26>(m.phi);
    fx X, Y, Z, z = 0;
    FxConst d12, d24, d4;
    if constexpr (MODE == kGeneral) {
        const double jx = fx_to<kFxTop3>(m.jx, em), jy = fx_to<kFxTop3>(m.jy, em), jz = fx_to<kFxTop3>(m.jz, em);
        const double dphi = phi - phi_prev, p2 = phi * phi;
        double Bx, By, Bz, dBx, dBy, dBz;
        if (p.bq2) {
            Bx = fma(p.ux, phi, p.bgx * p2);
            By = fma(p.uy, phi, p.bgy * p2);
            Bz = fma(p.uz, phi, p.bgz * p2);
            const double sp = phi + phi_prev;
            dBx = fma(p.bgx, sp, p.ux) * dphi;
            dBy = fma(p.bgy, sp, p.uy) * dphi;
            dBz = fma(p.bgz, sp, p.uz) * dphi;
        } else {
            const double gq = pow_half(phi, p.bq, p.bq_n, p.bq_h);
            const double dg = gq - pow_half(phi_prev, p.bq, p.bq_n, p.bq_h);
            Bx = fma(p.ux, phi, p.bgx * gq);
            By = fma(p.uy, phi, p.bgy * gq);
            Bz = fma(p.uz, phi, p.bgz * gq);
            dBx = fma(p.ux, dphi, p.bgx * dg);
            dBy = fma(p.uy, dphi, p.bgy * dg);
            dBz = fma(p.uz, dphi, p.bgz * dg);
        }
        if (p.c3 != 0.0) {
            // C(phi) - phi: in 3 t3, and k0 (C - phi) / 24 on the diagonals
            const double Cm = p.c3 * p2 * phi;
            if (fx_exp(Cm) > em + (1u << 20)) return false;
            m.t3 -= fx_from<kFxTop3>(Cm, em);
            z = fx_from<kFxTop3>(p.k0 * cst<double>(1, 24) * Cm, em);
        }
        const double s3 = fma(p.a2x3, p2, 3.0);
        const double mxx = fma(s3, p.A0[0], 0.5), mxy = s3 * p.A0[1], mxz = s3 * p.A0[2];
        const double myy = fma(s3, p.A0[3], 0.5), myz = s3 * p.A0[4], mzz = fma(s3, p.A0[5], 0.5);
        const double cxx = fma(myy, mzz, -(myz * myz)), cxy = fma(mxz, myz, -(mxy * mzz));
        const double cxz = fma(mxy, myz, -(mxz * myy)), cyy = fma(mxx, mzz, -(mxz * mxz));
        const double cyz = fma(mxy, mxz, -(mxx * myz)), czz = fma(mxx, myy, -(mxy * mxy));
        const double det = fma(mxx, cxx, fma(mxy, cxy, mxz * cxz));
        const double tr = (mxx + myy) + mzz;
        double id, k2;
        if (p.k2_hbb) {
            const double q2 = fma(4.0, tr, -3.0);
            const double rc = recip_f64(det * q2);
            id = rc * q2;
            k2 = (fma(cst<double>(16, 3), tr, -8.0) * det) * rc;
        } else {
            id = recip_f64(det);
            k2 = p.k2c;
        }
        const double dk = k2 - p.k0;
        // K1 e with the cofactors, divided by the determinant once per component
        const double ex = id * fma(-0.5, dBx, Bx - jx), ey = id * fma(-0.5, dBy, By - jy), ez = id * fma(-0.5, dBz, Bz - jz);
        const double Vx = fma(cxx, ex, fma(cxy, ey, fma(cxz, ez, fma(p.k0, jx, dBx))));
        const double Vy = fma(cxy, ex, fma(cyy, ey, fma(cyz, ez, fma(p.k0, jy, dBy))));
        const double Vz = fma(cxz, ex, fma(cyz, ey, fma(czz, ez, fma(p.k0, jz, dBz))));
        const unsigned int far = em + (2u << 20);
        // id 0: the reciprocal underflowed (and k2 with it)
        if (fx_exp(dk) > (1023u << 20) || fx_exp(Vx) > far || fx_exp(Vy) > far || fx_exp(Vz) > far || fx_exp(id) == 0 || !fits)
            return false;
        const FxConst sixth = {0x2aaaaaab, (int)0xaaaaaaab};   // 2^64 / 6
        X = fx_mul(fx_arg(fx_from<kFxTop3>(Vx, em)), sixth);
        Y = fx_mul(fx_arg(fx_from<kFxTop3>(Vy, em)), sixth);
        Z = fx_mul(fx_arg(fx_from<kFxTop3>(Vz, em)), sixth);
        const FxArg c = fx_arg(fx_from(dk, 1019u << 20));      // dk / 4 in units of 2^-64
        d4.hi = c.h;
        d4.lo = c.l;
        d12 = d24 = d4;
        // (k2 - k0)/12 and /24 as (k2 - k0)/4 of a third and a sixth of the moment
        m.hx = 2 * fx_mul(fx_arg(m.hx), sixth);
        m.hy = 2 * fx_mul(fx_arg(m.hy), sixth);
        m.t3 = fx_mul(fx_arg(m.t3), sixth);
    } else {
        const FxArg jx = fx_arg(m.jx), jy = fx_arg(m.jy), jz = fx_arg(m.jz), ph = fx_arg(m.phi);
        const FxArg pp = fx_arg(fx_from<kFxTop3>(phi_prev, em));
        FxSum s[3] = {fx_sum(), fx_sum(), fx_sum()};
        constexpr int at[3][3] = {{0, 1, 2}, {1, 3, 4}, {2, 4, 5}};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            fx_add(s[a], jx, p.fx.Q[at[a][0]]);
            fx_add(s[a], jy, p.fx.Q[at[a][1]]);
            fx_add(s[a], jz, p.fx.Q[at[a][2]]);
            fx_add(s[a], ph, p.fx.P[a]);
            fx_add(s[a], pp, p.fx.g[a]);
        }
        X = fx_value(s[0]);
        Y = fx_value(s[1]);
        Z = fx_value(s[2]);
        d12 = p.fx.d12;
        d24 = p.fx.d24;
        d4 = p.fx.d4;
    }
    double src = 0.0;
    if constexpr (SRC == kSrcReaction) srcv = fma(1.5, reaction3(p, phi), -0.5 * reaction3(p, phi_prev));
    if constexpr (SRC != kSrcNone) src = p.src_val * srcv;
    if (SRC != kSrcNone && fx_exp(src) > em + (1u << 20)) return false;
    if (MODE != kGeneral && !fits) return false;
    fx a = m.phi, r[19];
    if (!k0_one) a -= 2 * fx_mul(fx_arg(m.phi), p.fx.om2);
    if (SRC != kSrcNone) a += fx_from<kFxTop3>(src, em);
    fx_expand3(a, z, X, Y, Z, fx_mul(fx_arg(m.hx), d12), fx_mul(fx_arg(m.hy), d12), fx_mul(fx_arg(m.t3), d24),
               fx_mul(fx_arg(m.pxy), d4), fx_mul(fx_arg(m.pxz), d4), fx_mul(fx_arg(m.pyz), d4), r);
    if (k0_one) fx_store<true, 0, kFxTop3>(D, r, p.fx.om2, em, d);
    else fx_store<false, 0, kFxTop3>(D, r, p.fx.om2, em, d);
    phi_out = phi;
    return true;
}

// The initialising collision: f^eq + w S (init_f64 in three dimensions).
template <int MODE, int SRC>
__device__ __forceinline__ void init3_f64(const Sweep3Params<double> &p, double (&d)[19], double phi, double src) {
    double Bx = p.ux * phi, By = p.uy * phi, Bz = p.uz * phi, Cm = 0.0;
    if constexpr (MODE == kGeneral) {
        const double g = p.bq2 ? phi * phi : pow_half(phi, p.bq, p.bq_n, p.bq_h);
        Bx = fma(p.bgx, g, Bx);
        By = fma(p.bgy, g, By);
        Bz = fma(p.bgz, g, Bz);
        Cm = p.c3 * phi * phi * phi;
    }
    unsigned int em = fx_exp(phi);
    const bool tiny = em < kFxExpMin && ((fx_bits(phi) | fx_bits(src)) << 1) != 0;
    em = em > kFxExpMin ? em : kFxExpMin;
    const unsigned int far = em + (1u << 20);
    if (tiny || em > kFxExpMax || fx_exp(Bx) > far || fx_exp(By) > far || fx_exp(Bz) > far || fx_exp(src) > far ||
        fx_exp(Cm) > far) {
        double t[19];
        init3_f64_slow(p, t, phi, src);
#pragma unroll
        for (int i = 0; i < 19; ++i) d[i] = t[i];
        return;
    }
    const FxConst sixth = {0x2aaaaaab, (int)0xaaaaaaab};   // 2^64 / 6
    fx a = fx_from<kFxTop3>(phi, em), z = 0, r[19];
    if (SRC != kSrcNone) a += fx_from<kFxTop3>(src, em);
    if (MODE == kGeneral) z = fx_from<kFxTop3>(cst<double>(1, 24) * Cm, em);
    fx_expand3(a, z, fx_mul(fx_arg(fx_from<kFxTop3>(Bx, em)), sixth),
               fx_mul(fx_arg(fx_from<kFxTop3>(By, em)), sixth),
               fx_mul(fx_arg(fx_from<kFxTop3>(Bz, em)), sixth), 0, 0, 0, 0, 0, 0, r);
    fx_store<true, BTRT_FX_NADD3, kFxTop3>(r, r, p.fx.om2, em, d);
}

template <int MODE, int SRC>
__device__ __forceinline__ double collide3_f64(const Sweep3Params<double> &p, double (&d)[19], double phi_prev,
                                               double srcv) {
    if (p.first) {
        init3_f64<MODE, SRC>(p, d, phi_prev, SRC == kSrcReaction ? p.src_val * reaction3(p, phi_prev)
                                             : SRC != kSrcNone   ? p.src_val * srcv
                                                                 : 0.0);
        return phi_prev;
    }
    double phi;
    bool done = false;
    if (p.fx.ok & (MODE == kGeneral ? kFxOkGeneral : kFxOkLinear)) {
        if constexpr (MODE == kGeneral || SRC == kSrcReaction)
            done = fx_collide_general3<MODE, SRC>(p, d, phi_prev, srcv, phi);
        else
            done = fx_collide_linear3<MODE == kLinearK0One, SRC != kSrcNone>(
                p.fx, d, phi_prev, SRC != kSrcNone ? p.src_val * srcv : 0.0, phi);
    }
    if (!done) {
        double t[19];
#pragma unroll
        for (int i = 0; i < 19; ++i) t[i] = d[i];
        phi = collide3_f64_slow<MODE, SRC>(p, t, phi_prev, srcv);
#pragma unroll
        for (int i = 0; i < 19; ++i) d[i] = t[i];
    }
    return phi;
}

// Element `at` of population plane i.  BASE: the plane's base is uniform over the
// launch and the byte offset in it fits 32 bits (19 planes hold fewer than 2^31
// values), so one 32-bit offset per neighbour serves every plane.
template <bool BASE, typename Real, typename S>
__device__ __forceinline__ const S *plane3_at(const Sweep3Params<Real> &p, const S *f, int i, int at) {
#ifndef BTRT_DEBUG_BOUNDS
    if constexpr (BASE)
        return reinterpret_cast<const S *>(reinterpret_cast<const char *>(f + (size_t)i * p.plane) +
                                           (unsigned int)at * (unsigned int)sizeof(S));
#endif
    return f + BTRT_IX(p.flags, i * p.plane + at, 19 * p.plane);
}
// FP64 only: FP32 and 16-bit storage measured within 3 % either way.
template <typename S> struct Base3 { static constexpr bool value = std::is_same<S, double>::value; };

// Index distances to the six neighbours of a node, wrapped on the domain's far side:
// a node that touches no bounce-back wall pulls through them whatever its place, so
// the warps that hold a row's two ends run no second path (with the boundary pull
// there, two warps of every row ran both): 256^3 hill, FP16 local shift, 20 steps
// 8.26 -> 6.56 ms, 64^3 917 -> 440 us, 128^3 FP64 3.27 -> 2.56 ms.
struct Near3 {
    int xm, xp, ym, yp, zm, zp;
};
template <typename Real>
__device__ __forceinline__ Near3 near3(const Sweep3Params<Real> &p, int x, int y, int z) {
    Near3 n;
    n.xm = x == 0 ? p.nx - 1 : -1;
    n.xp = x == p.nx - 1 ? 1 - p.nx : 1;
    n.ym = y == 0 ? (p.ny - 1) * p.pitch : -p.pitch;
    n.yp = y == p.ny - 1 ? (1 - p.ny) * p.pitch : p.pitch;
    n.zm = z == 0 ? (p.nz - 1) * p.slab : -p.slab;
    n.zp = z == p.nz - 1 ? (1 - p.nz) * p.slab : p.slab;
    return n;
}
// Distance to the node that population i comes from, x - c_i.
__device__ __forceinline__ int from3(const Near3 &n, int i) {
    return (cz3(i) == 1 ? n.zm : cz3(i) == -1 ? n.zp : 0) + (cy3(i) == 1 ? n.ym : cy3(i) == -1 ? n.yp : 0) +
           (cx3(i) == 1 ? n.xm : cx3(i) == -1 ? n.xp : 0);
}
template <typename Real>
__device__ __forceinline__ bool touches_wall3(const Sweep3Params<Real> &p, int x, int y, int z) {
    return (p.hbb_x && (x == 0 || x == p.nx - 1)) || (p.hbb_y && (y == 0 || y == p.ny - 1)) ||
           (p.hbb_z && (z == 0 || z == p.nz - 1));
}

// Resident blocks per SM asked of the compiler (0: its choice).
// FP64, 128^3 hill, 20 steps: three blocks (80 registers) 3.27 ms, two 3.72, four 3.31,
// five 4.09; per-node coefficients three (80 registers, spilling) 8.14 against 8.44 with
// two (128) and 11.5 with one.
#ifndef BTRT3_MINBLOCKS_F64
#define BTRT3_MINBLOCKS_F64 3
#endif
#ifndef BTRT3_MINBLOCKS_F64_GEN
#define BTRT3_MINBLOCKS_F64_GEN 3
#endif
// 16-bit storage, per-node coefficients (250 x 131 x 200, 40 steps): five (48 registers)
// 6.56 ms, the compiler's 64 registers 6.76, six 7.66.
#ifndef BTRT3_MINBLOCKS_S16_GEN
#define BTRT3_MINBLOCKS_S16_GEN 5
#endif
template <typename Real, typename S, int MODE, int SRC> struct MinBlocks3 {
    static constexpr int value = MODE == kGeneral ? BTRT3_MINBLOCKS_S16_GEN : 0;
};
template <int MODE, int SRC> struct MinBlocks3<float, float, MODE, SRC> { static constexpr int value = 0; };
template <int MODE, int SRC> struct MinBlocks3<double, double, MODE, SRC> {
    static constexpr int value = MODE == kLinearK0One && SRC != kSrcReaction ? BTRT3_MINBLOCKS_F64 : BTRT3_MINBLOCKS_F64_GEN;
};

// Pull of a node with at least one neighbour across the domain boundary.
template <typename Real, typename S, int SH>
__device__ __forceinline__ void pull3_boundary(const Sweep3Params<Real> &p, const S *__restrict__ fin, int x, int y,
                                               int z, int node, Real phi_prev, Real (&d)[19]) {
#pragma unroll
    for (int i = 0; i < 19; ++i) {
        int sx = x - cx3(i), sy = y - cy3(i), sz = z - cz3(i);
        Real wsum = Real(0);
        int crossed = 0;
        if (sx < 0) { if (p.hbb_x) { wsum += p.wall[0]; ++crossed; } else sx += p.nx; }
        if (sx >= p.nx) { if (p.hbb_x) { wsum += p.wall[1]; ++crossed; } else sx -= p.nx; }
        if (sy < 0) { if (p.hbb_y) { wsum += p.wall[2]; ++crossed; } else sy += p.ny; }
        if (sy >= p.ny) { if (p.hbb_y) { wsum += p.wall[3]; ++crossed; } else sy -= p.ny; }
        if (sz < 0) { if (p.hbb_z) { wsum += p.wall[4]; ++crossed; } else sz += p.nz; }
        if (sz >= p.nz) { if (p.hbb_z) { wsum += p.wall[5]; ++crossed; } else sz -= p.nz; }
        if (!crossed) {
            const int src = sz * p.slab + sy * p.pitch + sx;
            d[i] = Storage<S>::load(fin[BTRT_IX(p.flags, i * p.plane + src, 19 * p.plane)]);
            if constexpr (SH == kShiftLocal)
                if (i != 0) d[i] = fma(wgt3<Real>(i), p.phi_in[BTRT_IX(p.flags, src, p.plane)] - phi_prev, d[i]);
        } else {
            const int o = opposite3(i);
            const int n2 = cx3(i) * cx3(i) + cy3(i) * cy3(i) + cz3(i) * cz3(i);
            const Real phi_w = (crossed == 1 ? wsum : Real(0.5) * wsum) * p.wall_fac;
            const Real dout = Storage<S>::load(fin[BTRT_IX(p.flags, o * p.plane + node, 19 * p.plane)]);
            Real wt = wall3_term(p, n2, phi_w);
            if constexpr (SH == kShiftRef) wt = wt - Real(2) * p.wref[n2];
            if constexpr (SH == kShiftLocal) wt = fma(Real(-2) * wgt3<Real>(i), phi_prev, wt);
            d[i] = wt - dout;
        }
    }
}

// One node: pull, collision, write-back.
template <typename Real, typename S, int SH, int MODE, int SRC>
__device__ __forceinline__ void sweep3_node(const Sweep3Params<Real> &p, int x, int y, int z) {
    const S *__restrict__ fin = static_cast<const S *>(p.fin);
    S *__restrict__ fout = static_cast<S *>(p.fout);
    const int node = z * p.slab + y * p.pitch + x;
    const Real phi_prev = p.phi_in[BTRT_IX(p.flags, node, p.plane)];
    Real d[19];
    if (p.first) {   // FP64: formed in the collision (init3_f64)
        if constexpr (!std::is_same<Real, double>::value) equilibrium3<Real, SH>(p, phi_prev, d);
    } else if (!touches_wall3(p, x, y, z)) {
        const Near3 nb = near3(p, x, y, z);
#pragma unroll
        for (int i = 0; i < 19; ++i)
            d[i] = Storage<S>::load(*plane3_at<Base3<S>::value, Real, S>(p, fin, i, node + from3(nb, i)));
        if constexpr (SH == kShiftLocal) {
#pragma unroll
            for (int i = 1; i < 19; ++i)
                d[i] = fma(wgt3<Real>(i), p.phi_in[BTRT_IX(p.flags, node + from3(nb, i), p.plane)] - phi_prev, d[i]);
        }
    } else {
        pull3_boundary<Real, S, SH>(p, fin, x, y, z, node, phi_prev, d);
    }
    Real srcv = Real(0);
    if constexpr (SRC == kSrcConst) srcv = Real(1);
    if constexpr (SRC == kSrcField) srcv = p.srcF[BTRT_IX(p.flags, node, p.plane)];
    const Real rs = SH == kShiftLocal ? phi_prev : p.phi_ref;
    Real phid, phi;
    if constexpr (std::is_same<Real, double>::value) {
        phi = collide3_f64<MODE, SRC>(p, d, phi_prev, srcv);
        phid = phi;
    } else {
        phi = collide3<Real, MODE, SRC, SH>(p, d, rs, phi_prev, srcv, p.first != 0, phid);
    }
#pragma unroll
    for (int i = 0; i < 19; ++i) {
        Real v = d[i];
        if constexpr (SH == kShiftLocal) v = fma(-wgt3<Real>(i), phid, v);
        *const_cast<S *>(plane3_at<Base3<S>::value, Real, S>(p, fout, i, node)) = Storage<S>::pack(v);
    }
    p.phi_out[BTRT_IX(p.flags, node, p.plane)] = phi;
    if (not_finite(phi)) atomicOr(p.flags, 1);
}

template <typename Real, typename S, int SH, int MODE, int SRC>
__global__ void __launch_bounds__(256, MinBlocks3<Real, S, MODE, SRC>::value)
    sweep3_kernel(const __grid_constant__ Sweep3Params<Real> p) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x < p.nx && y < p.ny) sweep3_node<Real, S, SH, MODE, SRC>(p, x, y, blockIdx.z);
}

// ---------------------------------------------------------------- two nodes per thread, 16-bit storage
// The scalar sweep of 16-bit storage is bound by instruction issue: 19 16-bit loads,
// 18 of phi, 20 stores and their addresses per node.  Here a thread owns the nodes
// x0, x0 + 1 (x0 even) of one row: per plane one 32-bit load brings the pair of the
// source row (rows are padded to 64 elements, so it is aligned) and, for the ten
// directions with c_x != 0, one 16-bit load the value beyond the pair; nine rows of
// phi arrive as pairs, five of them with two values more; the results leave as 32-bit
// stores (256^3 hill, FP16 local shift, 20 steps: 6.56 -> 5.36 ms, 63 GLUPS, 0.79 of
// HBM).  The nodes' arithmetic and its order are the scalar sweep's, so the results
// are equal bitwise.  Pairs that touch a bounce-back wall, or the half pair
// at the end of an odd row, take the scalar path.
template <typename S> __device__ __forceinline__ float pair_get(unsigned int w, int k);
template <> __device__ __forceinline__ float pair_get<__half>(unsigned int w, int k) {
    return __half2float(__ushort_as_half((unsigned short)(k ? w >> 16 : w & 0xffffu)));
}
template <> __device__ __forceinline__ float pair_get<__nv_bfloat16>(unsigned int w, int k) {
    return __uint_as_float(k ? w & 0xffff0000u : w << 16);
}
template <typename S> __device__ __forceinline__ unsigned int pair_put(float a, float b);
template <> __device__ __forceinline__ unsigned int pair_put<__half>(float a, float b) {
    const __half2 h = __floats2half2_rn(a, b);
    unsigned int w;
    memcpy(&w, &h, 4);
    return w;
}
template <> __device__ __forceinline__ unsigned int pair_put<__nv_bfloat16>(float a, float b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    unsigned int w;
    memcpy(&w, &h, 4);
    return w;
}

// Four blocks per SM (64 registers): 5.36 ms on that hill, three 5.55, five 6.37.
#ifndef BTRT3_VEC_MINBLOCKS
#define BTRT3_VEC_MINBLOCKS 4
#endif
template <typename S, int SH, int MODE, int SRC>
__global__ void __launch_bounds__(256, BTRT3_VEC_MINBLOCKS) sweep3_vec_kernel(const __grid_constant__ Sweep3Params<float> p) {
    const int x0 = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
    const int y = blockIdx.y * blockDim.y + threadIdx.y, z = blockIdx.z;
    if (x0 >= p.nx || y >= p.ny) return;
    if (x0 + 1 >= p.nx || touches_wall3(p, x0, y, z) || touches_wall3(p, x0 + 1, y, z)) {
#pragma unroll 1
        for (int v = 0; v < 2 && x0 + v < p.nx; ++v) sweep3_node<float, S, SH, MODE, SRC>(p, x0 + v, y, z);
        return;
    }
    const S *__restrict__ fin = static_cast<const S *>(p.fin);
    S *__restrict__ fout = static_cast<S *>(p.fout);
    const int node = z * p.slab + y * p.pitch + x0;
    Near3 nb = near3(p, x0, y, z);
    nb.xp = x0 + 2 == p.nx ? 2 - p.nx : 2;   // beyond the pair
    // distance of the source row of direction i (c_y, c_z)
    auto row = [&](int i) {
        return (cz3(i) == 1 ? nb.zm : cz3(i) == -1 ? nb.zp : 0) + (cy3(i) == 1 ? nb.ym : cy3(i) == -1 ? nb.yp : 0);
    };
    unsigned int raw[19];
    S edge[19];
#pragma unroll
    for (int i = 0; i < 19; ++i) {
        const int at = node + row(i);
        raw[i] = *reinterpret_cast<const unsigned int *>(plane3_at<true, float, S>(p, fin, i, at));
        if (cx3(i) == 1) edge[i] = *plane3_at<true, float, S>(p, fin, i, at + nb.xm);
        if (cx3(i) == -1) edge[i] = *plane3_at<true, float, S>(p, fin, i, at + nb.xp);
    }
    // phi of the node's row (directions 1, 2) and, for the local shift, of the source
    // rows: [row][x0 - 1 .. x0 + 2], rows named by one direction that comes from them
    constexpr int kRowDir[9] = {0, 3, 4, 5, 6, 15, 16, 17, 18};
    float ph[9][4];
#pragma unroll
    for (int r = 0; r < (SH == kShiftLocal ? 9 : 1); ++r) {
        const int at = node + row(kRowDir[r]);
        const float2 m = *reinterpret_cast<const float2 *>(p.phi_in + BTRT_IX(p.flags, at, p.plane));
        ph[r][1] = m.x;
        ph[r][2] = m.y;
        if (SH == kShiftLocal && r < 5) {
            ph[r][0] = p.phi_in[BTRT_IX(p.flags, at + nb.xm, p.plane)];
            ph[r][3] = p.phi_in[BTRT_IX(p.flags, at + nb.xp, p.plane)];
        }
    }
    bool bad = false;
    float out[19], phi_o[2];
#pragma unroll
    for (int v = 0; v < 2; ++v) {
        const float phi_prev = ph[0][1 + v];
        float d[19];
#pragma unroll
        for (int i = 0; i < 19; ++i) {
            const int k = v - cx3(i);   // 0, 1: of the pair; -1, 2: the value beyond it
            d[i] = k < 0 || k > 1 ? Storage<S>::load(edge[i]) : pair_get<S>(raw[i], k);
        }
        if constexpr (SH == kShiftLocal) {
#pragma unroll
            for (int i = 1; i < 19; ++i) {
                constexpr int kRow[3][3] = {{8, 4, 7}, {2, 0, 1}, {6, 3, 5}};   // [1 + c_z][1 + c_y]
                d[i] = fma(wgt3<float>(i), ph[kRow[1 + cz3(i)][1 + cy3(i)]][1 + v - cx3(i)] - phi_prev, d[i]);
            }
        }
        float srcv = 0.f;
        if constexpr (SRC == kSrcConst) srcv = 1.f;
        if constexpr (SRC == kSrcField) srcv = p.srcF[BTRT_IX(p.flags, node + v, p.plane)];
        const float rs = SH == kShiftLocal ? phi_prev : p.phi_ref;
        float phid;
        phi_o[v] = collide3<float, MODE, SRC, SH>(p, d, rs, phi_prev, srcv, false, phid);
        bad |= not_finite(phi_o[v]);
#pragma unroll
        for (int i = 0; i < 19; ++i) {
            const float t = SH == kShiftLocal ? fma(-wgt3<float>(i), phid, d[i]) : d[i];
            if (v == 0) out[i] = t;
            else *reinterpret_cast<unsigned int *>(const_cast<S *>(plane3_at<true, float, S>(p, fout, i, node))) =
                     pair_put<S>(out[i], t);
        }
    }
    *reinterpret_cast<float2 *>(p.phi_out + BTRT_IX(p.flags, node, p.plane)) = make_float2(phi_o[0], phi_o[1]);
    if (bad) atomicOr(p.flags, 1);
}

}  // namespace btrt
