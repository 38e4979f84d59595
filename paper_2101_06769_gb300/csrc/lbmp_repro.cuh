// lbmp_repro.cuh -- the per-cell arithmetic of the steps whose results must be
// reproduced to the last bit: shifted 16-bit storage, and D2Q9 with a symmetry
// x axis.
//
// The update is that of lbmp_common.cuh in the form in which it was first
// written: opposite pairs of directions as the lanes of the paired arithmetic,
// post-collision central moments taken back to populations axis by axis, the
// stencil over all neighbours of a cell.  The other FP32 steps have moved to a
// form with 30 % fewer instructions that rounds differently in the last bit
// (and is no further from 64 bits); their runs stay within 1e-5 of the earlier
// ones for as long as they were compared (80 steps).  Two kinds of run do not:
//   * a 16-bit step rounds every output to a code by a threshold drawn per
//     code, so a last-bit change turns some codes over, and these change the
//     next step's phi and references: after 20 to 40 steps 40 % of the FP16
//     codes differ by an ulp and the references by 3e-5 of their norm (BF16:
//     2e-4);
//   * the droplet impacts that the symmetry axis is for (density ratio 1000)
//     amplify a last-bit change: 1e-5 after 21 steps, 1e-3 after 42, 4e-3 (of
//     the largest population) after 80, about as far as both forms are from
//     64 bits.
// Those are equally good states, but stored runs would not be continued on the
// same trajectory; so these kernels, and their reference pair, keep these
// functions.
#pragma once

#include "lbmp_common.cuh"

namespace lbmp {
namespace repro {

template <int D, class Get>
__device__ __forceinline__ void phi_sum(const Get& get, float& hi, float& lo)
{
    constexpr int Q = Lat<D>::Q;
    constexpr int C = Q / 2;
    float2 h = f2(get(C), 0.f), l = f2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < C; ++k) {
        const int a = by_weight<D>(k);
        const float2 v = f2(get(a), get(Q - 1 - a));
        const float2 s = add2(h, v);
        l = add2(l, add2(v, neg2(add2(s, neg2(h)))));
        h = s;
    }
    // join the lanes exactly, then renormalise (|lo| <= ulp(hi)/2)
    const float t = h.x + h.y;
    const float bb = t - h.x;
    const float e = (h.x - (t - bb)) + (h.y - bb);
    const float lsum = (l.x + l.y) + e;
    hi = t + lsum;
    lo = lsum - (hi - t);
}

template <int D, bool PR, class Get>
__device__ __forceinline__ void phi_sum_phase(const Get& get, float& hi, float& lo)
{
    if constexpr (PR)
        phi_sum_red<D>(get, hi, lo);
    else
        repro::phi_sum<D>(get, hi, lo);
}

// Isotropic differences (Sec. 2.2) from the Q neighbour values
// phi(x + c_a) = nh[a] + nl[a]: grad_i = 3 sum w c_i phi(x+c),
// lap = 6 sum w (phi(x+c) - phi(x)).  Opposite neighbours are taken as a
// pair: the gradient from the difference of their deviations from the
// centre (exactly zero on a uniform field), the Laplacian from their sum.
// nb(a) returns the pair (hi, lo) of phi(x + c_a); centre = nb(C).
template <int D, class NB>
__device__ __forceinline__ void stencil_from(const NB& nb, float2 centre, float grad[3], float& lap)
{
    constexpr int Q = Lat<D>::Q;
    constexpr int C = Q / 2;
    float gx = 0.f, gy = 0.f, gz = 0.f;
    float2 ls = f2(0.f, 0.f);
#pragma unroll
    for (int a = 0; a < C; ++a) {
        const int b = Q - 1 - a;
        const float w = Lat<D>::w(a);
        // phi(x + c) - phi(x) and phi(x - c) - phi(x), hi and lo parts differenced first
        const float2 dd = f2(pair_diff(nb(a), centre), pair_diff(nb(b), centre));
        ls = fma2(f2(w, w), dd, ls);
        const float d = w * (dd.x - dd.y);
        if (Lat<D>::cx(a)) gx += Lat<D>::cx(a) * d;
        if (Lat<D>::cy(a)) gy += Lat<D>::cy(a) * d;
        if (Lat<D>::cz(a)) gz += Lat<D>::cz(a) * d;
    }
    grad[0] = 3.f * gx;
    grad[1] = 3.f * gy;
    grad[2] = (D == 3) ? 3.f * gz : 0.f;
    lap = 6.f * (ls.x + ls.y);
}

template <int D>
__device__ __forceinline__ void stencil_from_nb(const float* nh, const float* nl, float grad[3], float& lap)
{
    constexpr int C = Lat<D>::Q / 2;
    stencil_from<D>([&](int a) { return f2(nh[a], nl[a]); }, f2(nh[C], nl[C]), grad, lap);
}

// Moments of the pre-collision f': P, J, and the second moments Pi_ij.
struct FlowMoments {
    float P, J[3];
    float Pxx, Pyy, Pzz, Pxy, Pxz, Pyz;
};

// Moments of the Q pre-collision values f[a].  J is summed over opposite
// pairs, c_a (f_a - f_opp(a)): the O(w p_h) part common to both members of a
// pair cancels exactly before the sum, so the small momentum of a light phase
// (density ratio up to 1000) is not buried under the pressure in FP32.
template <int D>
__device__ __forceinline__ void flow_moments(FlowMoments& m, const float* f)
{
    constexpr int Q = Lat<D>::Q;
    constexpr int C = Q / 2;
    m.P = f[C];
    m.J[0] = m.J[1] = m.J[2] = 0.f;
    m.Pxx = m.Pyy = m.Pzz = m.Pxy = m.Pxz = m.Pyz = 0.f;
#pragma unroll
    for (int a = 0; a < C; ++a) {
        const int cx = Lat<D>::cx(a), cy = Lat<D>::cy(a), cz = Lat<D>::cz(a);
        const float2 sd = fma2(f2(1.f, -1.f), f2(f[Q - 1 - a], f[Q - 1 - a]), f2(f[a], f[a]));
        const float s = sd.x, d = sd.y;  // f_a + f_opp, f_a - f_opp
        m.P += s;
        if (cx) m.J[0] += cx * d;
        if (cy) m.J[1] += cy * d;
        if (cz) m.J[2] += cz * d;
        if (cx) m.Pxx += s;
        if (cy) m.Pyy += s;
        if (cz) m.Pzz += s;
        if (cx * cy) m.Pxy += (cx * cy) * s;
        if (cx * cz) m.Pxz += (cx * cz) * s;
        if (cy * cz) m.Pyz += (cy * cz) * s;
    }
}

// Per-cell results of the collision set-up that the output loops need.
struct CellState {
    float u[3];        // velocity
    float n[3];        // interface normal
    float rcs2;        // rho cs2
    float ph;          // p_h = P + sum(Xi)/2
    float F[3], uF;    // force density F = F_s + F_b
    float G[3], uG;    // G = cs2 grad(rho)
    float uu;          // |u|^2
    float ew[3][3];    // per-axis product-equilibrium deviation e_d(c) - w1(c), [axis][c+1]
    float phi, sharp;  // phi and lambda_phi 4 phi (1-phi)/W
};

// Local closure (Sec. 2.1/2.3; readings A1, A2, A7, A12, A13, A15): density,
// interface normal, chemical potential, force, velocity and p_h of one cell
// into s (every field but ew); returns rho.  Also the observables use it.
template <int D>
__device__ __forceinline__ float flow_closure(const DevParams& p, float phi, const float grad[3], float lap,
                                              const FlowMoments& m, CellState& s, float& inv_rho, float& nu)
{
    const float rho = p.rho_l + p.drho * phi;
    inv_rho = recip(rho);
    if (p.flags & kFlagDynamicVisc)
        nu = (p.eta_l + (p.eta_h - p.eta_l) * phi) * inv_rho;
    else
        nu = p.nu_h + (p.nu_l - p.nu_h) * (1.0f - phi);
    // interface normal, chemical potential, force
    const float g2 = grad[0] * grad[0] + grad[1] * grad[1] + (D == 3 ? grad[2] * grad[2] : 0.f);
    const float inv_g = recip(fmaxf(root(fmaxf(g2, 1e-12f)), 1e-4f));
    const float mu = p.beta2 * phi * (phi - 1.0f) * (2.0f * phi - 1.0f) - p.kappa * lap;
    float F[3];
    F[0] = mu * grad[0];
    F[1] = mu * grad[1];
    F[2] = (D == 3) ? mu * grad[2] : 0.f;
    if (p.flags & kFlagUniformForce)
        F[0] += p.force_x;
    else
        F[D - 1] -= (rho - p.rho_bar) * p.g_accel;

    // u = J/(rho cs2) + F/(2 rho)
    for (int i = 0; i < 3; ++i) {
        s.u[i] = (D == 2 && i == 2) ? 0.f : (3.0f * m.J[i] + 0.5f * F[i]) * inv_rho;
        s.n[i] = (D == 2 && i == 2) ? 0.f : grad[i] * inv_g;
        s.G[i] = (D == 2 && i == 2) ? 0.f : third(__fmul_rn(p.drho, grad[i]));
        s.F[i] = F[i];
    }
    const float ux = s.u[0], uy = s.u[1], uz = s.u[2];
    s.uG = ux * s.G[0] + uy * s.G[1] + uz * s.G[2];
    s.uF = ux * F[0] + uy * F[1] + uz * F[2];
    s.uu = ux * ux + uy * uy + uz * uz;
    s.rcs2 = third(rho);
    s.ph = m.P + 0.5f * s.uG;
    s.phi = phi;
    s.sharp = p.lam_sharp * phi * (1.0f - phi);
    return rho;
}

// The relaxation of the flow collision, after the closure (inv_rho and nu
// from flow_closure): the relaxed second-order deviations and the per-axis
// product equilibrium (s.ew).  Produces the 27-entry Kronecker inverse of the
// post-collision moment differences in dh[] (h* - E(u)).
template <int D>
__device__ __forceinline__ void flow_relax(const FlowMoments& m, CellState& s, float inv_rho, float nu, float dh[27])
{
    const float omega = recip(3.0f * nu + 0.5f);
    const float om1 = 1.0f - omega;
    const float ux = s.u[0], uy = s.u[1], uz = s.u[2];
    float V[3];
    for (int i = 0; i < 3; ++i) V[i] = s.G[i] + s.F[i];
    const float uV = s.uG + s.uF;

    // second moments of f^p minus theta cs2 delta, i.e. with 1/cs2 = 3:
    // [3 Pi_ij - P delta_ij + (u_i V_j + u_j V_i)/2 - 3 u_i u_j u.V/2] / rho - u_i u_j
    // (cs2 itself never enters as a rounded constant)
    const float hV3 = 1.5f * uV;
    float dxx = (3.0f * m.Pxx - m.P + ux * V[0] - ux * ux * hV3) * inv_rho - ux * ux;
    float dyy = (3.0f * m.Pyy - m.P + uy * V[1] - uy * uy * hV3) * inv_rho - uy * uy;
    float dxy = (3.0f * m.Pxy + 0.5f * (ux * V[1] + uy * V[0]) - ux * uy * hV3) * inv_rho - ux * uy;
    float dzz = 0.f, dxz = 0.f, dyz = 0.f;
    if (D == 3) {
        dzz = (3.0f * m.Pzz - m.P + uz * V[2] - uz * uz * hV3) * inv_rho - uz * uz;
        dxz = (3.0f * m.Pxz + 0.5f * (ux * V[2] + uz * V[0]) - ux * uz * hV3) * inv_rho - ux * uz;
        dyz = (3.0f * m.Pyz + 0.5f * (uy * V[2] + uz * V[1]) - uy * uz * hV3) * inv_rho - uy * uz;
    }
    // cumulant relaxation: shear rate on off-diagonal and deviatoric parts,
    // trace to D cs2 (rate one), every higher cumulant to zero (rate one)
    const float tr = (D == 3) ? (dxx + dyy + dzz) * (1.0f / 3.0f) : (dxx + dyy) * 0.5f;
    const float a = om1 * (dxx - tr), b = om1 * (dyy - tr), c = (D == 3) ? om1 * (dzz - tr) : 0.f;
    const float pq = om1 * dxy, qq = om1 * dxz, rr = om1 * dyz;

    // per-axis product equilibrium and its deviation from w1
    for (int i = 0; i < 3; ++i) {
        const float ui = s.u[i], u2 = ui * ui;
        s.ew[i][0] = 0.5f * (u2 - ui);
        s.ew[i][1] = -u2;
        s.ew[i][2] = 0.5f * (u2 + ui);
    }

    // post-collision central-moment differences (Gaussian closure minus the
    // Gaussian of cs2 I), index ia + 3 ib + 9 ic
    float k[27];
#pragma unroll
    for (int i = 0; i < 27; ++i) k[i] = 0.f;
    const float cs2 = kCs2;
    k[2] = a;            // 200
    k[6] = b;            // 020
    k[4] = pq;           // 110
    k[8] = cs2 * (a + b) + a * b + 2.f * pq * pq;  // 220
    if (D == 3) {
        k[18] = c;       // 002
        k[10] = qq;      // 101
        k[12] = rr;      // 011
        k[20] = cs2 * (a + c) + a * c + 2.f * qq * qq;           // 202
        k[24] = cs2 * (b + c) + b * c + 2.f * rr * rr;           // 022
        k[14] = (cs2 + a) * rr + 2.f * pq * qq;                  // 211
        k[16] = (cs2 + b) * qq + 2.f * pq * rr;                  // 121
        k[22] = (cs2 + c) * pq + 2.f * qq * rr;                  // 112
        k[26] = cs2 * cs2 * (a + b + c) + cs2 * (a * b + b * c + c * a) + a * b * c +
                2.f * ((cs2 + a) * rr * rr + (cs2 + b) * qq * qq + (cs2 + c) * pq * pq) + 8.f * pq * qq * rr;  // 222
    }
    // Kronecker inverse about u: per axis (k0,k1,k2) -> (c=-1, 0, +1)
    // m1 = k1 + u k0, m2 = k2 + 2u k1 + u^2 k0; f(0) = k0 - m2, f(+-1) = (m2 +- m1)/2
    constexpr int NZ = (D == 3) ? 3 : 1;
    // (along x first: a line holds k2 alone, k1 alone, or k0 and k2)
#pragma unroll
    for (int ic = 0; ic < NZ; ++ic)
#pragma unroll
        for (int ib = 0; ib < 3; ++ib) {
            const int o = 3 * ib + 9 * ic;
            if (ib == 0 && ic == 0) {
                const float k2 = k[o + 2];
                k[o] = k[o + 2] = 0.5f * k2;
                k[o + 1] = -k2;
            } else if (((ib + ic) & 1) != 0) {
                const float m1 = k[o + 1], m2 = __fmul_rn(2.f * ux, m1);
                k[o] = 0.5f * (m2 - m1);
                k[o + 1] = -m2;
                k[o + 2] = 0.5f * (m2 + m1);
            } else {
                const float k0 = k[o], m1 = __fmul_rn(ux, k0), m2 = fmaf(__fmul_rn(ux, ux), k0, k[o + 2]);
                k[o] = 0.5f * (m2 - m1);
                k[o + 1] = k0 - m2;
                k[o + 2] = 0.5f * (m2 + m1);
            }
        }
#pragma unroll
    for (int ic = 0; ic < NZ; ++ic)
#pragma unroll
        for (int ia = 0; ia < 3; ++ia) {
            const int o = ia + 9 * ic;
            const float k0 = k[o], k1 = k[o + 3], k2 = k[o + 6];
            const float m1 = k1 + uy * k0, m2 = k2 + 2.f * uy * k1 + uy * uy * k0;
            k[o] = 0.5f * (m2 - m1);
            k[o + 3] = k0 - m2;
            k[o + 6] = 0.5f * (m2 + m1);
        }
    if (D == 3) {
#pragma unroll
        for (int ib = 0; ib < 3; ++ib)
#pragma unroll
            for (int ia = 0; ia < 3; ++ia) {
                const int o = ia + 3 * ib;
                const float k0 = k[o], k1 = k[o + 9], k2 = k[o + 18];
                const float m1 = k1 + uz * k0, m2 = k2 + 2.f * uz * k1 + uz * uz * k0;
                k[o] = 0.5f * (m2 - m1);
                k[o + 9] = k0 - m2;
                k[o + 18] = 0.5f * (m2 + m1);
            }
    }
#pragma unroll
    for (int i = 0; i < 27; ++i) dh[i] = k[i];
}

// Deviation of the second-order Hermite equilibrium f_eq/rho (App. A) from
// its rest value: Gamma_a - w_a = w_a [c.u/cs2 + ((c.u)^2 - cs2 u^2)/(2 cs4)].
template <int D>
__device__ __forceinline__ float gamma_dev(const CellState& s, int a)
{
    const int cx = Lat<D>::cx(a), cy = Lat<D>::cy(a), cz = Lat<D>::cz(a);
    const float cu = cx * s.u[0] + cy * s.u[1] + cz * s.u[2];
    return Lat<D>::w(a) * (3.0f * cu + 4.5f * cu * cu - 1.5f * s.uu);
}

// Post-collision f'*_a = rho cs2 (h*_a - w_a) + w_a p_h + Xi_a/2 with
// h* - w = (E(u) - w) + dh and the source (Sec. 2.3, reading A6)
//   Xi_a = cs2 (Gamma_a - w_a)(c_a - u).grad(rho) + Gamma_a (c_a - u).F,
// both terms formed from small factors (no O(w |grad rho|) cancellation).
template <int D>
__device__ __forceinline__ float flow_post(const CellState& s, const float dh[27], int a, float gdev)
{
    const int cx = Lat<D>::cx(a), cy = Lat<D>::cy(a), cz = Lat<D>::cz(a);
    const float w = Lat<D>::w(a);
    const float cG = cx * s.G[0] + cy * s.G[1] + cz * s.G[2] - s.uG;
    const float cF = cx * s.F[0] + cy * s.F[1] + cz * s.F[2] - s.uF;
    const float xi = gdev * cG + (w + gdev) * cF;
    // telescoped E - w = e_x e_y e_z - w_x w_y w_z
    const float wy = (float)w1d(cy), wz = (float)w1d(cz);
    const float ex = (float)w1d(cx) + s.ew[0][cx + 1], ey = wy + s.ew[1][cy + 1];
    float ew;
    if (D == 3)
        ew = s.ew[0][cx + 1] * wy * wz + ex * s.ew[1][cy + 1] * wz + ex * ey * s.ew[2][cz + 1];
    else
        ew = s.ew[0][cx + 1] * wy + ex * s.ew[1][cy + 1];
    return s.rcs2 * (ew + dh[a]) + w * s.ph + 0.5f * xi;
}

// Phase-field BGK with the sharpening source (Sec. 2.2, readings A3-A5):
// g* = g + (phi Gamma - g)/tau + lambda w (c.n) 4 phi (1-phi)/W
template <int D>
__device__ __forceinline__ float phase_post(const DevParams& p, const CellState& s, int a, float g, float gdev)
{
    const int cx = Lat<D>::cx(a), cy = Lat<D>::cy(a), cz = Lat<D>::cz(a);
    const float w = Lat<D>::w(a);
    const float cn = cx * s.n[0] + cy * s.n[1] + cz * s.n[2];
    return g + p.inv_tau_phi * (s.phi * (w + gdev) - g) + w * cn * s.sharp;
}

// Offsets S v_C/W_C of the shifted encoders: the rest populations of f' and
// g from their formulas (the rest value emitted last equals them to within
// rounding).
template <int D, class St, class GSrc>
__device__ __forceinline__ void rest_offsets(const DevParams& p, const CellState& s, const float dh[27],
                                             const GSrc& gin, float& off_f, float& off_g)
{
    constexpr int C = Lat<D>::Q / 2;
    const float gd = gamma_dev<D>(s, C);
    const float k = St::S / wint<D>(C);
    off_f = k * flow_post<D>(s, dh, C, gd);
    off_g = k * phase_post<D>(p, s, C, gin(C), gd);
}

// The outputs are formed for each direction a together with its opposite
// (c -> -c, same weight): (a, opp(a)) are the two lanes of the paired FP32
// arithmetic, and the shared factors (c.u, (c.u)^2, c.G, c.F, c.n) are
// computed once per pair.
// dh source: the register array of flow_relax
struct DhArray {
    const float* v;
    __device__ __forceinline__ float operator[](int a) const { return v[a]; }
};

// Per-pair pieces of the outputs.  Direction a < Q/2 and its opposite
// b = Q-1-a are the two lanes (c, -c) of the paired arithmetic.
//
// pair_gamma: the equilibrium deviation Gamma - w = w [3 c.u + 4.5 (c.u)^2 -
// 1.5 u^2] (gd) and Gamma itself (wgd = w + gd); m15uu = -1.5 |u|^2.
template <int D>
__device__ __forceinline__ void pair_gamma(const CellState& s, int a, float m15uu, float2& gd, float2& wgd)
{
    const int cx = Lat<D>::cx(a), cy = Lat<D>::cy(a), cz = Lat<D>::cz(a);
    const float w = Lat<D>::w(a);
    const float2 w2 = f2(w, w);
    const float cu = cx * s.u[0] + cy * s.u[1] + cz * s.u[2];
    const float X = fmaf(4.5f * cu, cu, m15uu);
    gd = mul2(w2, fma2(f2(3.f, -3.f), f2(cu, cu), f2(X, X)));
    wgd = add2(w2, gd);
}

// pair_flow: f'* = rho cs2 (E - w + dh) + w p_h + Xi/2 of the pair, with
// Xi = (Gamma - w)(c - u).G + Gamma (c - u).F and E(u) - w telescoped over
// the axes; dab = (dh[a], dh[b]).
template <int D>
__device__ __forceinline__ float2 pair_flow(const CellState& s, int a, float2 gd, float2 wgd, float2 dab)
{
    const int cx = Lat<D>::cx(a), cy = Lat<D>::cy(a), cz = Lat<D>::cz(a);
    const float w = Lat<D>::w(a);
    const float2 pm1 = f2(1.f, -1.f);
    const float cG0 = cx * s.G[0] + cy * s.G[1] + cz * s.G[2];
    const float cF0 = cx * s.F[0] + cy * s.F[1] + cz * s.F[2];
    const float2 cG = fma2(pm1, f2(cG0, cG0), f2(-s.uG, -s.uG));
    const float2 cF = fma2(pm1, f2(cF0, cF0), f2(-s.uF, -s.uF));
    float2 xi = fma2(gd, cG, mul2(wgd, cF));
    const float2 exs = f2(s.ew[0][cx + 1], s.ew[0][1 - cx]);
    const float2 eys = f2(s.ew[1][cy + 1], s.ew[1][1 - cy]);
    const float wx = (float)w1d(cx), wy = (float)w1d(cy), wz = (float)w1d(cz);
    const float2 ex = add2(f2(wx, wx), exs);
    float2 ew;
    if (D == 3) {
        const float2 ezs = f2(s.ew[2][cz + 1], s.ew[2][1 - cz]);
        const float2 ey = add2(f2(wy, wy), eys);
        ew = fma2(mul2(ex, ey), ezs, fma2(mul2(ex, eys), f2(wz, wz), mul2(exs, f2(wy * wz, wy * wz))));
    } else {
        ew = fma2(ex, eys, mul2(exs, f2(wy, wy)));
    }
    const float wph = w * s.ph;
    return fma2(f2(s.rcs2, s.rcs2), add2(ew, dab), fma2(f2(0.5f, 0.5f), xi, f2(wph, wph)));
}

// pair_phase: g* = g + (phi Gamma - g)/tau + w (c.n) lambda 4 phi (1-phi)/W
// of the pair (flow lattice), gi = (g_a, g_b) pre-collision
template <int D>
__device__ __forceinline__ float2 pair_phase(const DevParams& p, const CellState& s, int a, float2 wgd, float2 gi)
{
    const int cx = Lat<D>::cx(a), cy = Lat<D>::cy(a), cz = Lat<D>::cz(a);
    const float w = Lat<D>::w(a);
    const float2 pm1 = f2(1.f, -1.f);
    const float cn0 = cx * s.n[0] + cy * s.n[1] + cz * s.n[2];
    const float ws = w * s.sharp;
    const float2 itau = f2(p.inv_tau_phi, p.inv_tau_phi);
    return fma2(f2(ws, ws), mul2(pm1, f2(cn0, cn0)), fma2(itau, fma2(f2(s.phi, s.phi), wgd, neg2(gi)), gi));
}

// d/dt(phi u) for collide_outputs, with the previous value at prev[k * stride]
// (staged, or the stored array itself)
// (prev[k * stride]); the new value goes to the stored array
template <int D>
struct PhiUStaged {
    const DevParams& p;
    float* phiu;
    long long i;
    const float* prev;
    int stride;
    __device__ __forceinline__ void operator()(const CellState& s, float d[3]) const
    {
#pragma unroll
        for (int k = 0; k < D; ++k) {
            const float v = s.phi * s.u[k];
            d[k] = v - prev[k * stride];
            phiu[k * p.N + i] = v;
        }
        if (D == 2) d[2] = 0.f;
    }
};
// The rest populations from the conservation identities (see below): the
// flow total P + u.G less the moving outputs fs,
// the phase-field total (gsum_hi, gsum_lo) less the compensated moving
// outputs (gs, gl); or a shifted encoder takes the totals themselves.
template <class Out>
__device__ __forceinline__ void flow_rest(const CellState& s, const FlowMoments& m, float2 fs, const Out& fout,
                                          int C)
{
    if constexpr (Out::kTotal)
        fout.finish(m.P, s.uG);
    else
        fout(C, (m.P + s.uG) - (fs.x + fs.y));
}
template <class Out>
__device__ __forceinline__ void phase_rest(float gsum_hi, float gsum_lo, float2 gs, float2 gl, const Out& gout, int GC)
{
    if constexpr (Out::kTotal) {
        gout.finish(gsum_hi, gsum_lo);
    } else {
        float t = gs.x + gs.y;  // combine the lanes exactly
        const float bb = t - gs.x;
        const float e = (gs.x - (t - bb)) + (gs.y - bb);
        gout(GC, (gsum_hi - t) + (gsum_lo - (gl.x + gl.y + e)));
    }
}

// The phase-field update on the reduced lattice: g* = g + (g_eq - g)/tau +
// w c.(lambda 4 phi(1-phi)/W n + lambda/cs2 d/dt(phi u)) with the
// first-order equilibrium g_eq = w phi (1 + c.u/cs2), the sharpening source
// and the correction term (Sec. 2.2), lanes (r, opposite); the rest slot
// from the conserved total.
template <int D, class GSrc, class Out, class DPhiU>
__device__ __forceinline__ void phase_outputs_reduced(const DevParams& p, const CellState& s, const GSrc& gin,
                                                      float gsum_hi, float gsum_lo, const Out& gout,
                                                      const DPhiU& dphiu_fn, float2 gs, float2 gl)
{
    constexpr int GC = PhaseLat<D, true>::C;
    constexpr float ics = PhaseLat<D, true>::inv_cs2;
    const float2 itau = f2(p.inv_tau_phi, p.inv_tau_phi);
    const float2 pm1 = f2(1.f, -1.f);
    float qv[3];
    dphiu_fn(s, qv);
#pragma unroll
    for (int i = 0; i < 3; ++i) qv[i] = fmaf(p.lam_corr, qv[i], s.sharp * s.n[i]);
#pragma unroll
    for (int r = 0; r < GC; ++r) {
        const int a = PhaseLat<D, true>::full(r);
        const int cx = Lat<D>::cx(a), cy = Lat<D>::cy(a), cz = Lat<D>::cz(a);
        const float w = PhaseLat<D, true>::w(r);
        const float cu = cx * s.u[0] + cy * s.u[1] + cz * s.u[2];
        const float cq = cx * qv[0] + cy * qv[1] + cz * qv[2];
        const float wphi = w * s.phi;
        const float t = wphi * ics * cu;
        const float2 geq = fma2(pm1, f2(t, t), f2(wphi, wphi));
        const float2 gi = f2(gin(r), gin(2 * GC - r));
        const float2 go = fma2(f2(w, w), mul2(pm1, f2(cq, cq)), fma2(itau, add2(geq, neg2(gi)), gi));
        gout(r, go.x);
        gout(2 * GC - r, go.y);
        two_sum2(gs, gl, go);
    }
    phase_rest(gsum_hi, gsum_lo, gs, gl, gout, GC);
}

// PR: g on the reduced phase lattice (gin / gout index its slots), with
// dphiu(s, d) giving d/dt(phi u) of the cell for the correction term.
template <int D, bool PR = false, class GSrc, class Out, class DH, class DPhiU = NoPhiU>
__device__ __forceinline__ void collide_outputs(const DevParams& p, const CellState& s, const DH& dh,
                                                const FlowMoments& m, const GSrc& gin, float gsum_hi,
                                                float gsum_lo, const Out& fout, const Out& gout,
                                                const DPhiU& dphiu_fn = DPhiU{})
{
    static_assert(!(PR && Out::kTotal), "the reduced phase lattice is stored in FP32 only");
    constexpr int Q = Lat<D>::Q;
    constexpr int C = Q / 2;
    const float m15uu = -1.5f * s.uu;
    float2 fs = f2(0.f, 0.f), gs = f2(0.f, 0.f), gl = f2(0.f, 0.f);
#pragma unroll
    for (int a = 0; a < C; ++a) {
        const int b = Q - 1 - a;
        float2 gd, wgd;
        pair_gamma<D>(s, a, m15uu, gd, wgd);
        const float2 fo = pair_flow<D>(s, a, gd, wgd, f2(dh[a], dh[b]));
        out_pair<Q>(fout, a, fo);
        fs = add2(fs, fo);
        if constexpr (!PR) {
            const float2 go = pair_phase<D>(p, s, a, wgd, f2(gin(a), gin(b)));
            out_pair<Q>(gout, a, go);
            two_sum2(gs, gl, go);
        }
        out_pair_done();
    }
    // target totals: P + u.G (flow) and the incoming sum (phase field); the
    // rest populations take the difference (conservation identities above),
    // or a shifted encoder takes the totals themselves
    flow_rest(s, m, fs, fout, C);
    if constexpr (PR)
        phase_outputs_reduced<D>(p, s, gin, gsum_hi, gsum_lo, gout, dphiu_fn, gs, gl);
    else
        phase_rest(gsum_hi, gsum_lo, gs, gl, gout, C);
}

}  // namespace repro
}  // namespace lbmp
