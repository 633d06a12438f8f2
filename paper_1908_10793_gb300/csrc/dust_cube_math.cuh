// Single-precision arithmetic of the three-dimensional slab kernels
// (dust_cube.cuh): weights, drifts, kick and impulse of a grain relative to its
// key zone.  The formulas are those of dust_device.cuh; here every product and
// sum is rounded as written (no contraction is left to the compiler), so that
// the results do not depend on how the surrounding kernel is arranged, on its
// register budget or on the compiler's choice of what to fuse.
#pragma once

#include "dust_device.cuh"

namespace dust {

__device__ __forceinline__ float fm(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fa(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float fs(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float ff(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float fd(float a, float b) { return __fdiv_rn(a, b); }

// ---- weights (Sec. 3.4, App. C); d, nu as in dust_device.cuh

__device__ __forceinline__ void cube_w_cart(int tsc, float d, float w[3])
{
    if (tsc) {
        const float a = fs(0.5f, d), b = fa(0.5f, d);
        w[0] = fm(fm(0.5f, a), a);
        w[1] = ff(-d, d, 0.75f);
        w[2] = fm(fm(0.5f, b), b);
    } else {
        w[0] = d < 0.f ? -d : 0.f;
        w[2] = d > 0.f ? d : 0.f;
        w[1] = fs(fs(1.f, w[0]), w[2]);
    }
}

__device__ __forceinline__ void cube_w_cyl(int tsc, float d, float nu, float w[3])
{
    if (tsc) {
        const float inv = fd(1.f, fm(3.f, fa(d, nu)));
        const float base = ff(3.f, nu, d);
        const float a = fs(0.5f, d), b = fa(0.5f, d);
        w[0] = fm(fm(fm(fm(fs(base, 2.f), inv), 0.5f), a), a);
        w[2] = fm(fm(fm(fm(fa(base, 2.f), inv), 0.5f), b), b);
        w[1] = fm(fm(base, inv), ff(-d, d, 0.75f));
    } else {
        const float inv = fd(1.f, fm(2.f, fa(d, nu)));
        const float base = ff(2.f, nu, d);  // the doubling is exact
        const float ad = fabsf(d);
        w[0] = fm(fm(fm(fs(base, 1.f), inv), 0.5f), fs(ad, d));
        w[2] = fm(fm(fm(fa(base, 1.f), inv), 0.5f), fa(ad, d));
        w[1] = fm(fm(base, inv), fs(1.f, ad));
    }
}

// EXACT: the path of grains outside their key zone, which fuses other products of
// some sums (as the per-grain kernel does)
template <bool EXACT>
__device__ __forceinline__ void cube_w_sphr(int tsc, float d, float nu, float w[3])
{
    const float s = fa(d, nu);
    if (tsc) {
        const float inv = fd(1.f, ff(fm(6.f, s), s, 1.f));
        const float a = fs(0.5f, d), b = fa(0.5f, d);
        const float c0 = ff(fm(4.f, nu), d, ff(d, d, ff(fm(6.f, nu), nu, 2.75f)));
        const float odd = EXACT ? ff(3.f, d, fm(8.f, nu)) : ff(8.f, nu, fm(3.f, d));
        w[0] = fm(fm(fm(fm(fs(c0, odd), inv), 0.5f), a), a);
        w[2] = fm(fm(fm(fm(fa(c0, odd), inv), 0.5f), b), b);
        const float t = ff(2.f, nu, d);  // the doubling is exact
        const float n2 = fm(2.f, nu);
        const float x = fa(ff(n2, nu, fm(t, t)), 0.75f);
        w[1] = fm(ff(x, ff(-d, d, 0.75f), -0.25f), inv);
    } else {
        const float inv = fd(1.f, ff(fm(12.f, s), s, 1.f));
        const float ad = fabsf(d);
        const float base = EXACT ? ff(2.f, d, fm(3.f, nu)) : ff(3.f, nu, fm(2.f, d));
        const float p = fa(base, 1.5f), m = fs(base, 1.5f);
        const float np_ = fa(nu, 0.5f), nm = fs(nu, 0.5f);
        const float t = ff(2.f, nu, d), u = fs(ad, 1.f);
        const float m3 = fm(3.f, nm), p3 = fm(3.f, np_), t3 = fm(3.f, t);
        w[0] = fm(fm(fm(ff(m3, nm, fm(m, m)), inv), 0.5f), fs(ad, d));
        w[2] = fm(fm(fm(ff(p3, np_, fm(p, p)), inv), 0.5f), fa(ad, d));
        w[1] = fm(fm(EXACT ? ff(u, u, fm(t3, t)) : ff(t3, t, fm(u, u)), inv), fs(1.f, ad));
    }
}

// e - sin(e), without cancellation for small e (Taylor series, |e| < 0.5)
__device__ __forceinline__ float cube_e_minus_sin(float e)
{
    const float s = fm(e, e);
    if (fabsf(e) < 0.5f) {
        const float i3 = ff(-s, 1.f / 72.f, 1.f);
        const float i2 = ff(-fm(s, 1.f / 42.f), i3, 1.f);
        const float i1 = ff(-fm(s, 1.f / 20.f), i2, 1.f);
        return fm(fm(fm(e, s), 1.f / 6.f), i1);
    }
    return fs(e, sinf(e));
}

__device__ __forceinline__ void cube_w_theta(int tsc, float th, float lo, float hi, float dr, float hw, float w[3])
{
    const float sh = sinf(hw);
    if (tsc) {
        const float N = fm(fm(fm(4.f, sinf(th)), sh), sh);
        const float ep = fa(hw, dr), em = fs(hw, dr);
        const float sp = sinf(fm(0.5f, ep)), sm = sinf(fm(0.5f, em));
        const float ap = fm(fm(2.f, sp), sp), am = fm(fm(2.f, sm), sm);
        const float sph = sinf(hi), sml = sinf(lo), ch = cosf(hi), cl = cosf(lo);
        const float xp = cube_e_minus_sin(ep), xm = cube_e_minus_sin(em);
        w[2] = fd(ff(ap, sph, fm(ch, xp)), N);
        w[0] = fd(ff(-cl, xm, fm(am, sml)), N);
    } else {
        const float D = fm(fm(2.f, sinf(th)), sh);
        const float s2 = sinf(fm(0.5f, dr));
        w[2] = dr > 0.f ? fd(fm(fm(2.f, sinf(ff(0.5f, dr, hi))), s2), D) : 0.f;
        w[0] = dr < 0.f ? fd(fm(fm(-2.f, sinf(ff(0.5f, dr, lo))), s2), D) : 0.f;
    }
    w[1] = fs(fs(1.f, w[0]), w[2]);
}

// Eq. CIC_vol relative to the host zone's centre c, for a coordinate x = c + u
// inside the zone: the shell volume between c and x (written so that it stays
// accurate for small u) times the inverse shell volume between c and the
// neighbouring node on that side (ivl, ivh, from vol_shell and vol_node in
// double precision).  d = 0: the radius (cylindrical R^2, spherical r^3); d = 1:
// the spherical polar angle.
template <int GEOM>
__device__ __forceinline__ void cube_w_vol(int d, float u, float c, float ivl, float ivh, float w[3])
{
    float num;
    if (GEOM == GEOM_SPH && d == 1) {
        num = fm(fm(2.f, sinf(ff(0.5f, u, c))), sinf(fm(0.5f, fabsf(u))));
    } else if (GEOM == GEOM_SPH) {
        const float c3 = fm(3.f, c);
        num = fm(fabsf(u), ff(u, u, ff(c3, c, fm(c3, u))));
    } else {
        num = fm(fabsf(u), ff(2.f, c, u));
    }
    w[0] = u < 0.f ? fm(num, ivl) : 0.f;
    w[2] = u > 0.f ? fm(num, ivh) : 0.f;
    w[1] = fs(fs(1.f, w[0]), w[2]);
}

// ---- drifts

// First half drift of the offsets u from the zone's centre zcf (Eq.
// exp_midpoint; Eq. drift1_cylindrical; spherical r, theta, phi in turn);
// inc: the increments.
template <int GEOM>
__device__ __forceinline__ void cube_drift1(const PhysDev &ph, float h, const float zcf[3], const float p[3],
                                            float u[3], float inc[3])
{
    inc[0] = fm(h, p[0]);
    u[0] = (GEOM == GEOM_SPH) ? ff(h, p[0], u[0]) : fa(u[0], inc[0]);
    const float x = fa(zcf[0], u[0]);
    if (GEOM == GEOM_CYL || GEOM == GEOM_SPH) inc[1] = fd(fm(h, p[1]), fm(x, x));
    else inc[1] = fm(h, (GEOM == GEOM_SB && ph.fargo) ? ff(-ph.q_om_f, x, p[1]) : p[1]);
    u[1] = fa(u[1], inc[1]);
    if (GEOM == GEOM_SPH) {
        const float st = sinf(fa(zcf[1], u[1]));
        inc[2] = fd(fm(h, p[2]), fm(fm(fm(x, x), st), st));
    } else {
        inc[2] = fm(h, p[2]);
    }
    u[2] = fa(u[2], inc[2]);
}

// The first half drift of the next step from the end offsets u, for the key
// prediction (the linear increments are fused into their sums).
template <int GEOM>
__device__ __forceinline__ void cube_drift_key(const PhysDev &ph, float h, const float zcf[3], const float p[3], float u[3])
{
    u[0] = ff(h, p[0], u[0]);
    const float x = fa(zcf[0], u[0]);
    if (GEOM == GEOM_CYL || GEOM == GEOM_SPH) u[1] = fa(u[1], fd(fm(h, p[1]), fm(x, x)));
    else u[1] = ff(h, (GEOM == GEOM_SB && ph.fargo) ? ff(-ph.q_om_f, x, p[1]) : p[1], u[1]);
    if (GEOM == GEOM_SPH) {
        const float st = sinf(fa(zcf[1], u[1]));
        u[2] = fa(u[2], fd(fm(h, p[2]), fm(fm(fm(x, x), st), st)));
    } else {
        u[2] = ff(h, p[2], u[2]);
    }
}

// Increments of the second half drift (metric factors of the half step,
// coordinates qf).
template <int GEOM>
__device__ __forceinline__ void cube_drift2(const PhysDev &ph, float h, const float qf[3], const float p[3], float inc[3])
{
    inc[0] = fm(h, p[0]);
    if (GEOM == GEOM_CYL || GEOM == GEOM_SPH) inc[1] = fd(fm(h, p[1]), fm(qf[0], qf[0]));
    else inc[1] = fm(h, (GEOM == GEOM_SB && ph.fargo) ? ff(-ph.q_om_f, qf[0], p[1]) : p[1]);
    if (GEOM == GEOM_SPH) {
        const float st = sinf(qf[1]);
        inc[2] = fd(fm(h, p[2]), fm(fm(fm(qf[0], qf[0]), st), st));
    } else {
        inc[2] = fm(h, p[2]);
    }
}

// ---- kick (Eq. kick_modified; App. B.1, B.2; see kick_any) and the impulse
// D = -mq (dp - dt a), its energy D[3] = sum D_c dH/dp_c

__device__ __forceinline__ float cube_exp3(float E, float p, float h1, float a, float cg, float v)
{
    return ff(cg, v, ff(E, p, fm(h1, a)));
}

// Semi-implicit kick (see kick_si; Cartesian and shearing box)
template <int GEOM>
__device__ __forceinline__ void cube_kick_si(const PhysDev &ph, const float qm[3], const float pn[3], const float vg[3],
                                             float it, float dt, float pp[3], float a[3], float dH[3])
{
    const float l00 = ff(fm(0.5f, dt), it, 1.f);
    float at[3] = {0.f, 0.f, 0.f};
    float l01 = 0.f, l10 = 0.f, Om = 0.f, q = 0.f, az = 0.f;
    if (GEOM == GEOM_SB) {
        Om = ph.omega_f;
        q = ph.qshear_f;
        az = ph.vgrav ? fm(fm(-Om, Om), qm[2]) : 0.f;
        l10 = ph.fargo ? fm(fm(ff(-0.5f, q, 1.f), Om), dt) : fm(Om, dt);
        l01 = fm(-Om, dt);
        at[2] = az;
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const float dv = fs(vg[d], pn[d]);
        if (GEOM == GEOM_SB && d < 2) {
            const float c = d == 0 ? fm(2.f, Om) : (ph.fargo ? fm(fs(q, 2.f), Om) : fm(-2.f, Om));
            const float x = d == 1 ? pn[0] : (ph.fargo ? pn[1] : ff(fm(q, Om), qm[0], pn[1]));
            at[d] = ff(c, x, fm(dv, it));
        } else {
            at[d] = ff(dv, it, at[d]);
        }
    }
    const float det = ff(-l01, l10, fm(l00, l00));
    const float r0 = fm(dt, at[0]), r1 = fm(dt, at[1]);
    pp[0] = fa(pn[0], fd(ff(l00, r0, -fm(l01, r1)), det));
    pp[1] = fa(pn[1], fd(ff(l00, r1, -fm(l10, r0)), det));
    pp[2] = fa(pn[2], fd(fm(dt, at[2]), l00));
    const float vx = fm(0.5f, fa(pn[0], pp[0])), vy = fm(0.5f, fa(pn[1], pp[1]));
    if (GEOM == GEOM_SB) {
        if (ph.fargo) {
            a[0] = fm(fm(2.f, Om), vy);
            a[1] = fm(fm(fs(q, 2.f), Om), vx);
        } else {
            a[0] = fm(fm(2.f, Om), ff(fm(q, Om), qm[0], vy));
            a[1] = fm(fm(-2.f, Om), vx);
        }
        a[2] = az;
    }
    dH[0] = vx;
    dH[1] = vy;
    dH[2] = fm(0.5f, fa(pn[2], pp[2]));
}

template <int GEOM>
__device__ __forceinline__ void cube_kick(const PhysDev &ph, float mq, const float qm[3], const float pn[3],
                                          const float vg[3], float tau, float dt, float E, float cg, float h1,
                                          float pp[3], float D[4])
{
    float a[3] = {0.f, 0.f, 0.f}, dH[3], dp[3];
    if ((GEOM == GEOM_CART || GEOM == GEOM_SB) && ph.pusher == DUST_PUSHER_SEMI_IMPLICIT) {
        cube_kick_si<GEOM>(ph, qm, pn, vg, fd(1.f, tau), dt, pp, a, dH);
#pragma unroll
        for (int c = 0; c < 3; ++c) dp[c] = fs(pp[c], pn[c]);
    } else if (GEOM == GEOM_SB) {
        const float Om = ph.omega_f, q = ph.qshear_f;
        const float az = ph.vgrav ? fm(fm(-Om, Om), qm[2]) : 0.f;
        const float Om1 = fm(Om, h1);
        float G0, G1;
        if (ph.fargo) {
            G0 = fm(Om, pn[1]);
            G1 = fm(fm(fm(0.5f, fs(q, 2.f)), Om), pn[0]);
        } else {
            G0 = ff(Om, pn[1], fm(fm(fm(fm(2.f, q), Om), Om), qm[0]));
            G1 = fm(-Om, pn[0]);
        }
        const float r0 = cube_exp3(E, pn[0], h1, G0, cg, vg[0]);
        const float r1 = cube_exp3(E, pn[1], h1, G1, cg, vg[1]);
        pp[2] = ff(cg, vg[2], ff(h1, az, fm(E, pn[2])));
        const float Om2 = ph.fargo ? fm(Om1, ff(-0.5f, q, 1.f)) : Om1;
        const float inv = fd(1.f, ff(Om1, Om2, 1.f));
        const float x0 = ff(Om1, r1, r0), x1 = ff(-Om2, r0, r1);
        pp[0] = fm(inv, x0);
        pp[1] = fm(inv, x1);
        const float vx = fm(0.5f, fa(pn[0], pp[0]));
        const float vy = fm(0.5f, fa(pn[1], pp[1]));
        if (ph.fargo) {
            a[0] = fm(fm(2.f, Om), vy);
            a[1] = fm(fm(fs(q, 2.f), Om), vx);
        } else {
            a[0] = fm(fm(2.f, Om), fa(vy, fm(fm(q, Om), qm[0])));
            a[1] = fm(fm(-2.f, Om), vx);
        }
        a[2] = az;
        dH[0] = vx;
        dH[1] = vy;
        dH[2] = fm(0.5f, fa(pn[2], pp[2]));
        dp[0] = fs(pp[0], pn[0]);
        dp[1] = fs(pp[1], pn[1]);
        dp[2] = fs(pp[2], pn[2]);
    } else if (GEOM == GEOM_CYL) {
        const float R = qm[0], R2 = fm(R, R);
        float gR = 0.f, gz = 0.f;
        if (ph.gm != 0.0) {
            if (ph.vgrav) {
                const float z = qm[2];
                const float r2 = ff(R, R, fm(z, z));
                const float ir3 = fd(1.f, fm(r2, sqrtf(r2)));
                gR = fm(fm(-ph.gm_f, R), ir3);
                gz = fm(fm(-ph.gm_f, z), ir3);
            } else {
                gR = fd(-ph.gm_f, R2);
            }
        }
        pp[2] = ff(cg, vg[2], ff(h1, gz, fm(E, pn[2])));
        pp[1] = ff(cg, vg[1], fm(E, pn[1]));
        const float l2 = fm(0.5f, ff(pn[1], pn[1], fm(pp[1], pp[1])));
        a[0] = fa(fd(l2, fm(R2, R)), gR);
        a[2] = gz;
        pp[0] = cube_exp3(E, pn[0], h1, a[0], cg, vg[0]);
        dH[0] = fm(0.5f, fa(pn[0], pp[0]));
        dH[1] = fd(fm(0.5f, fa(pn[1], pp[1])), R2);
        dH[2] = fm(0.5f, fa(pn[2], pp[2]));
#pragma unroll
        for (int c = 0; c < 3; ++c) dp[c] = fs(pp[c], pn[c]);
    } else if (GEOM == GEOM_SPH) {
        const float r = qm[0], r2 = fm(r, r);
        const float st = sinf(qm[1]), ct = cosf(qm[1]);
        const float gr = ph.gm != 0.0 ? fd(-ph.gm_f, r2) : 0.f;
        pp[2] = ff(cg, vg[2], fm(E, pn[2]));
        const float lp2 = fm(0.5f, ff(pn[2], pn[2], fm(pp[2], pp[2])));
        a[1] = fd(fm(lp2, ct), fm(fm(fm(r2, st), st), st));
        pp[1] = cube_exp3(E, pn[1], h1, a[1], cg, vg[1]);
        const float lt = ff(pn[1], pn[1], fm(pp[1], pp[1]));
        const float lq = fd(lp2, fm(st, st));
        a[0] = fa(fd(ff(0.5f, lt, lq), fm(r2, r)), gr);
        pp[0] = cube_exp3(E, pn[0], h1, a[0], cg, vg[0]);
        dH[0] = fm(0.5f, fa(pn[0], pp[0]));
        dH[1] = fd(fm(0.5f, fa(pn[1], pp[1])), r2);
        dH[2] = fd(fm(0.5f, fa(pn[2], pp[2])), fm(fm(r2, st), st));
#pragma unroll
        for (int c = 0; c < 3; ++c) dp[c] = fs(pp[c], pn[c]);
    } else {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            pp[c] = ff(E, pn[c], fm(cg, vg[c]));
            dH[c] = fm(0.5f, fa(pn[c], pp[c]));
            dp[c] = fs(pp[c], pn[c]);
        }
    }
    D[3] = 0.f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        D[c] = fm(-mq, ff(-dt, a[c], dp[c]));
        D[3] = ff(D[c], dH[c], D[3]);
    }
}

}  // namespace dust
