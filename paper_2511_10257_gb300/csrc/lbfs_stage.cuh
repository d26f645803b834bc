// lbfs_stage.cuh -- one Runge-Kutta stage of the LBFS finite-volume update in one kernel:
// the cell quantities (Eq. 8 inversion, Eq. 11 mixture, velocity, mu_c, |H|^2), every face
// flux by the LBFS reconstruction (Eqs. 44, 45, 20, 28, 29, 22, 32, 33, 43), the sources
// (Eq. 41), R(W) (Eq. 42) and the SSP-RK3 combination.  Stage 1 also forms the lagged
// dF_s/dt of the step; the last stage applies the step-end rest condition of the solid,
// writes the potential coefficient mu_m for the next solve, and reduces the diagnostics.
#pragma once
#include <type_traits>

#include "lbfs_internal.cuh"
#include "lbfs_kernels.h"

namespace lbfs {

// ---- pairs of values, one per axis ---------------------------------------------------
// Lane x belongs to the cell's x-normal face, lane y to its y-normal face.  In FP32 a pair
// is one operand of the packed instructions (FADD2 / FMUL2 / FFMA2), so both faces of a
// cell advance in one instruction stream.
template <class R>
struct PairOf;
template <>
struct PairOf<float> {
    using T = float2;
};
template <>
struct PairOf<double> {
    using T = double2;
};
__device__ __forceinline__ float2 mk(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ double2 mk(double a, double b) { return make_double2(a, b); }
__device__ __forceinline__ float2 sp(float a) { return make_float2(a, a); }
__device__ __forceinline__ double2 sp(double a) { return make_double2(a, a); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 vsub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
// Scalars, with every rounding written out: the compiler must not contract products and sums
// differently in the kernel's variants, which have to give the same bits.
__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float vsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double vadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double vsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double vmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double vfma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ double2 vadd(double2 a, double2 b) { return make_double2(vadd(a.x, b.x), vadd(a.y, b.y)); }
__device__ __forceinline__ double2 vsub(double2 a, double2 b) { return make_double2(vsub(a.x, b.x), vsub(a.y, b.y)); }
__device__ __forceinline__ double2 vmul(double2 a, double2 b) { return make_double2(vmul(a.x, b.x), vmul(a.y, b.y)); }
__device__ __forceinline__ double2 vfma(double2 a, double2 b, double2 c) {
    return make_double2(vfma(a.x, b.x, c.x), vfma(a.y, b.y, c.y));
}
// Eq. 11 from a property's gas value and its differences
template <class R>
__device__ __forceinline__ R vmix(R Fs, R C, R gs, R glg, R gg) {
    const R liq = vfma(C, glg, gg);
    return vfma(Fs, vsub(gs, liq), liq);
}

template <class R>
__device__ __forceinline__ R up(R v) { return __shfl_up_sync(0xffffffffu, v, 1); }
template <class R>
__device__ __forceinline__ R dn(R v) { return __shfl_down_sync(0xffffffffu, v, 1); }

// ---- the case's coefficients ------------------------------------------------------------
// UNI: one case's StageCase is a kernel argument, and its coefficients are operands of the
// constant bank.  Otherwise (a batch of cases) each block keeps its case's StageCase in shared
// memory; reads are volatile there, so that the loop does not hold several dozen coefficients
// in registers, and the face fluxes read them from a copy that stores each twice, one 64-bit
// load for both axes.
template <bool UNI, class R>
__device__ __forceinline__ R cf(const R& x) {
    if constexpr (UNI) return x;
    else return *const_cast<const volatile R*>(&x);
}
template <class R>
struct Coefs {
    const PhysT<R>& Q;
    const float2* twice;   // FP32, not UNI: PhysT's members, each stored twice
};
template <bool UNI>
__device__ __forceinline__ float2 c2(const Coefs<float>& k, const float& x) {
    if constexpr (UNI) {
        return sp(x);
    } else {
        const float2* p = k.twice + (&x - reinterpret_cast<const float*>(&k.Q));
        float2 r;
        asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(r.x), "=f"(r.y) : "r"((unsigned)__cvta_generic_to_shared(p)));
        return r;
    }
}
template <bool UNI>
__device__ __forceinline__ double2 c2(const Coefs<double>& k, const double& x) {
    return sp(cf<UNI>(x));
}

// ---- the surrounding-point equilibria of one cell -------------------------------------
// A cell serves two faces on each axis: its upper face as cell A (points with e_a.n = +1)
// and its lower face as cell B (e_a.n = -1).  The three points are c, c + G (e_a.t = +1)
// and c - G (e_a.t = -1) along the tangent, G = -dts times the tangential slope, and with
// s = e_a.n = +-1 the polynomial Gamma_a(u)/3 at a point splits into an even part E and an
// odd part s O:
//   c:      E0 = u^2 - v^2/2,                O0 = u
//   c +- G: E = a + a^2 + u^2,               O = u (1 + 3 a),  a = e_t v at that point,
// u and v the normal and tangential velocity there.  Written as mean and half-difference
// over the two tangential points (Eb, dE; Ob, dO), every sum over the three points of
// products of linear quantities (rho, C_p, T, C are linear along the tangent at the cell's
// F_s) is a few multiply-adds, formed once per cell and used by both its faces.
// e[], o[]: even and odd parts, in units of 1/18 (F, dF) and 1/6 (the others), of
//   0 F = sum w f_eq,  1 g = sum g_eq,  2 h = sum h_eq,  3 b = sum w Gamma,
//   4 dF = sum e_t w f_eq (even in s),  5 dG: s e_t w Gamma (its even part is dO).
// Inputs: p3 = 3 p, u, v, C, C3 = 3 C, m3 = 3 mu_c Q_g, T, rho, k = C_p, kT = C_p T,
// cT = C_p,ref T, r1 and k1 the slopes of rho and C_p in C, G[] of p, u, v, C, mu_c, T.
template <class V>
__device__ __forceinline__ void side_sums(V p3, V u, V v, V C, V C3, V m3, V T, V rho, V k, V kT, V cT, V r1, V k1,
                                          const V G[6], V e[6], V o[6]) {
    using S = decltype(p3.x);
    const V Gu = G[1], Gv = G[2], GC = G[3], GT = G[5];
    const V z = vfma(Gu, Gu, vmul(Gv, vadd(Gv, sp(S(1)))));
    const V s = vmul(u, u);
    const V X = vfma(sp(S(3)), s, z);                        // 2 E0 + Eb
    const V Eb = vfma(v, v, vadd(s, z));
    const V dE = vfma(sp(S(2)), vfma(u, Gu, vmul(v, Gv)), v);
    const V b = vfma(sp(S(3)), Gv, sp(S(1))), c = vmul(sp(S(3)), v);
    const V Ob = vfma(Gu, c, vmul(u, b)), dO = vfma(Gu, b, vmul(u, c));
    const V Y = vfma(sp(S(2)), u, Ob);                       // 2 O0 + Ob
    const V dr = vmul(r1, GC), dk = vmul(k1, GC);
    e[0] = vfma(rho, X, vfma(dr, dE, p3));
    o[0] = vfma(rho, Y, vmul(dr, dO));
    e[1] = vfma(C, Gv, vfma(GC, v, m3));
    o[1] = vfma(GC, Gu, vmul(C3, u));
    const V ep = vmul(dk, GT), dkT = vfma(k, GT, vmul(dk, T));
    e[2] = vfma(kT, X, vfma(ep, Eb, vfma(dkT, dE, cT)));
    o[2] = vfma(kT, Y, vfma(ep, Ob, vmul(dkT, dO)));
    e[3] = X;
    o[3] = Y;
    e[4] = vfma(rho, dE, vfma(dr, Eb, G[0]));
    o[4] = vfma(rho, dO, vmul(dr, Ob));
    e[5] = dO;
    o[5] = dE;
}

// What a face needs of its lower/left cell A (held by the neighbouring lane, or by this
// lane from the row before): the six sums with s = +1, the half-weighted reconstructions of
// the seven quantities at the face, G of six quantities, p at the centre point, and F_s.
enum { A_SUM = 0, A_REC = 6, A_G = 13, A_P = 19, A_FS = 20, NA = 21 };

// The fluxes of an x face (lane x) and a y face (lane y) from A's values a[], B's sums with
// s = -1 bs[], B's reconstructions br[], slopes G[], centre p and F_s.  The points with
// e_a.n = 0 sit at the face centre, on the mean of both cells' reconstructions.
// F: H_e, p, normal and tangential momentum, C.
template <bool UNI, class R, class V>
__device__ __forceinline__ void face_flux(const Coefs<R>& k_, const V a[NA], const V bs[6], const V br[7],
                                          const V bG[6], V bp, R bFs, V F[5]) {
    const PhysT<R>& Q = k_.Q;
    const V fsm = vmul(sp(R(0.5)), vadd(a[A_FS], sp(bFs)));
    const V om = vsub(sp(R(1)), fsm);
    const V r0 = vfma(fsm, c2<UNI>(k_, Q.rho_sg), c2<UNI>(k_, Q.rho_g)), r1 = vmul(om, c2<UNI>(k_, Q.rho_lg));
    const V k0 = vfma(fsm, c2<UNI>(k_, Q.cp_sg), c2<UNI>(k_, Q.cp_g)), k1 = vmul(om, c2<UNI>(k_, Q.cp_lg));
    V m[7], G[6];
#pragma unroll
    for (int q = 0; q < 7; ++q) m[q] = vadd(a[A_REC + q], br[q]);
#pragma unroll
    for (int q = 0; q < 6; ++q)
        if (q != 4) G[q] = vmul(sp(R(0.5)), vadd(a[A_G + q], bG[q]));
    const V p = m[0], u = m[1], v = m[2], C = m[3], T = m[5];
    const V Gu = G[1], Gv = G[2], GC = G[3], GT = G[5];
    // e_a.n = 0: E = a + a^2 - u^2/2 at the tangential points, E0 = -(u^2 + v^2)/2 at rest
    const V t = vmul(sp(R(-0.5)), Gu);
    const V z = vfma(t, Gu, vmul(Gv, vadd(Gv, sp(R(1)))));
    const V s = vmul(u, u);
    const V X = vfma(sp(R(-1.5)), s, z);
    const V Eb = vfma(v, v, vfma(sp(R(-0.5)), s, z));
    const V dE = vfma(sp(R(2)), vfma(u, t, vmul(v, Gv)), v);
    const V rho = vfma(r1, C, r0), k = vfma(k1, C, k0);
    const V dr = vmul(r1, GC), dk = vmul(k1, GC);
    const V kT = vmul(k, T), ep = vmul(dk, GT), dkT = vfma(k, GT, vmul(dk, T));
    const V Fm = vfma(rho, X, vfma(dr, dE, vmul(sp(R(3)), p)));
    const V Jm = vfma(rho, dE, vfma(dr, Eb, G[0]));
    const V hm = vfma(kT, X, vfma(ep, Eb, vmul(dkT, dE)));
    const V gm = vfma(C, Gv, vmul(GC, v));
    // Eq. 45: interface values
    const V w18 = sp(R(1.0 / 18.0)), w6 = sp(R(1.0 / 6.0));
    const V pf = vfma(w18, vadd(a[0], bs[0]), vmul(sp(R(2.0 / 9.0)), Fm));
    const V jn = vmul(w18, vsub(a[0], bs[0]));
    const V jt = vfma(w18, vadd(a[4], bs[4]), vmul(sp(R(2.0 / 9.0)), Jm));
    const V Cf = vfma(w6, vadd(a[1], bs[1]), vfma(sp(R(2.0 / 3.0)), gm, vfma(c2<UNI>(k_, Q.m_Qg), m[4], C)));
    const V Hf = vfma(w6, vadd(a[2], bs[2]), vfma(sp(R(2.0 / 3.0)), hm, vfma(c2<UNI>(k_, Q.m_cp_ref3), T, m[6])));
    const V Ag = vmul(w6, vsub(a[1], bs[1])), Ah = vmul(w6, vsub(a[2], bs[2]));
    const V Bn = vmul(w18, vadd(a[3], bs[3])), Bt = vmul(w18, vadd(a[5], bs[5]));   // thirds of sum e_n e w Gamma
    const V rhof = vfma(r1, Cf, r0), cpf = vfma(k1, Cf, k0);
    const V lamf = vfma(vmul(om, c2<UNI>(k_, Q.lam_lg)), Cf, vfma(fsm, c2<UNI>(k_, Q.lam_sg), c2<UNI>(k_, Q.lam_g)));
    const V muf = vfma(vmul(om, c2<UNI>(k_, Q.mu_lg)), Cf, vfma(fsm, c2<UNI>(k_, Q.mu_sg), c2<UNI>(k_, Q.mu_g)));
    // 1/rho_f and 1/C_p,L(C_f) from one reciprocal per face
    const V cpL = vfma(c2<UNI>(k_, Q.cp_lg), Cf, c2<UNI>(k_, Q.cp_g));
    const V den = vmul(rhof, cpL);
    const V rc = mk(fdiv(R(1), den.x), fdiv(R(1), den.y));
    const V irc = vmul(sp(R(3)), vmul(rc, cpL));             // 1 / (rho_f c_s^2)
    const V icp = vmul(rc, rhof);
    const V un = vmul(jn, irc), ut = vmul(jt, irc);
    // Eq. 8 at the face (T only)
    const V Tm = c2<UNI>(k_, Q.T_m);
    const V dl = vsub(Hf, vfma(cpL, Tm, c2<UNI>(k_, Q.L))), ds = vsub(Hf, c2<UNI>(k_, Q.Hes_hi));
    const V Tl = vfma(dl, icp, Tm), Ts = vfma(ds, c2<UNI>(k_, Q.inv_cps), Tm);
    V Tf;
    Tf.x = Cf.x < R(0.5) ? Tl.x : (ds.x < R(0) ? Ts.x : (dl.x <= R(0) ? Tm.x : Tl.x));
    Tf.y = Cf.y < R(0.5) ? Tl.y : (ds.y < R(0) ? Ts.y : (dl.y <= R(0) ? Tm.y : Tl.y));
    // tau - 1/2 = x, so X* = (1 - x) X_eq(x_f) + x X_eq(x - e_a dts)
    const V xf = vmul(vmul(muf, irc), c2<UNI>(k_, Q.inv_dts)), xh = vmul(vmul(lamf, irc), c2<UNI>(k_, Q.inv_cpref_dts));
    F[0] = vfma(xh, Ah, vmul(vsub(sp(R(1)), xh), vmul(vmul(cpf, Tf), un)));
    F[1] = jn;
    const V x3 = vmul(sp(R(1.0 / 3.0)), vsub(sp(R(1)), xf));
    const V ru = vmul(rhof, un);
    const V Bpn = vmul(w6, vadd(a[A_P], bp)), Bpt = vmul(w18, vsub(a[A_G], bG[0]));
    F[2] = vfma(x3, vfma(ru, un, pf), vmul(xf, vfma(rhof, Bn, Bpn)));
    F[3] = vfma(x3, vmul(ru, ut), vmul(xf, vfma(rhof, Bt, Bpt)));
    F[4] = vfma(c2<UNI>(k_, Q.x_g), Ag, vmul(vmul(c2<UNI>(k_, Q.om_x_g), Cf), un));
}

// Eq. 8 on the stored enthalpy without divergent branches: one quotient serves the solid
// and liquid temperature and the mushy liquid fraction.  Thresholds in FP64, or in FP32
// pairs in mixed precision (the high parts of two nearby values subtract exactly).
template <bool UNI, class R>
__device__ __forceinline__ void invert_cell(const PhysT<R>& Q, typename HeStore<R>::T He, R C, R& T, R& Fl, R& He_r) {
    const R cpL = vfma(C, cf<UNI>(Q.cp_lg), cf<UNI>(Q.cp_g));
    R ds, dl;
    if constexpr (sizeof(R) == 8) {
        ds = vsub(He, cf<UNI>(Q.Hes_hi));
        dl = vsub(He, vfma(cpL, cf<UNI>(Q.T_m), cf<UNI>(Q.L)));
        He_r = He;
    } else if (cf<UNI>(Q.T_m) == R(0)) {   // H_es = 0 and H_el = L
        ds = __fadd_rn(He.x, He.y);
        dl = __fadd_rn(__fsub_rn(He.x, cf<UNI>(Q.L_hi)), __fsub_rn(He.y, cf<UNI>(Q.L_lo)));
        He_r = ds;
    } else {
        const float2 Hel = pair_add_f(make_float2(cf<UNI>(Q.L_hi), cf<UNI>(Q.L_lo)), vmul(cpL, cf<UNI>(Q.T_m)));
        ds = __fadd_rn(__fsub_rn(He.x, cf<UNI>(Q.Hes_hi)), __fsub_rn(He.y, cf<UNI>(Q.Hes_lo)));
        dl = __fadd_rn(__fsub_rn(He.x, Hel.x), __fsub_rn(He.y, Hel.y));
        He_r = ds + cf<UNI>(Q.Hes_hi);
    }
    const bool gas = C < R(0.5), solid = !gas && ds < R(0), band = !gas && !solid && dl <= R(0);
    const R q = fdiv(solid || band ? ds : dl, solid ? cf<UNI>(Q.cp_s) : (band ? ds - dl : cpL));
    T = band ? cf<UNI>(Q.T_m) : cf<UNI>(Q.T_m) + q;
    Fl = band ? q : (solid ? R(0) : R(1));
}

// H_e's Runge-Kutta update: stage 1 W + dt R(W); later stages W^n + b ((W + dt R) - W^n)
// (a W^n + b X with a + b = 1 exactly).  FP64 in the FP64 mode.  In mixed precision the
// stage increment is small next to H_e and is formed in FP32 from the pairs'
// difference (their high parts subtract exactly when close), then added to the pair.
__device__ __forceinline__ double he_rk(int stage, double Hek, double He0, double dt, double Rw, double b) {
    const double x = vfma(dt, Rw, Hek);
    return stage == 0 ? x : vfma(b, vsub(x, He0), He0);
}
__device__ __forceinline__ float2 he_rk(int stage, float2 Hek, float2 He0, float dt, float Rw, float b) {
    if (stage == 0) return pair_add_f(Hek, __fmul_rn(dt, Rw));
    const float d = __fadd_rn(__fsub_rn(Hek.x, He0.x), __fsub_rn(Hek.y, He0.y));
    return pair_add_f(He0, __fmul_rn(b, __fmaf_rn(dt, Rw, d)));
}
__device__ __forceinline__ bool he_finite(double h) { return isfinite(h); }
__device__ __forceinline__ bool he_finite(float2 h) { return isfinite(h.x) && isfinite(h.y); }

// Wall face (no-slip, no-flux): momentum flux c_s^2 (p n - mu du_t/dn) with the wall
// half a cell from the inner centre; enthalpy flux -(lambda/rho) dT/dn on Dirichlet
// walls, zero on adiabatic ones; no mass or phase-field flux.  F: H_e, p, normal and
// tangential momentum, C; ut the inner cell's tangential velocity.
template <class R>
__device__ __noinline__ void wall_flux(const PhysT<R>& Q, int dirichlet, int wall, R Fs, R C, R rho, R p, R ut, R T,
                                       R F[5]) {
    const R mu = mix(Fs, C, Q.mu_s, Q.mu_l, Q.mu_g);
    const R lam = mix(Fs, C, Q.lam_s, Q.lam_l, Q.lam_g);
    const R side = (wall == 0 || wall == 2) ? R(2) : R(-2);
    const R c3 = R(1.0 / 3.0);
    F[0] = dirichlet ? -fdiv(lam, rho) * (side * (T - Q.wall_T[wall])) : R(0);
    F[1] = R(0);
    F[2] = c3 * p;
    F[3] = c3 * (-mu * (side * ut));
    F[4] = R(0);
}

// Twice the far field -H0 (x cos a + y sin a) at a wall face, rounded to R.  ix, iy: the face's
// whole coordinates; half: the half cell of its centre belongs to x (0) or y (1).  In mixed
// precision by FP32 pairs (FP64 instructions would cost a strip at a wall most of its time)
// while the coordinates are exact in FP32.
template <class R>
__device__ __forceinline__ R far_field_twice(const StageCase<R>& S, int ix, int iy, int half) {
    if constexpr (sizeof(R) == 4) {
        if (max(S.nx, S.ny) < (1 << 22)) {
            const float wx = (float)ix + (half == 0 ? 0.5f : 0.0f), wy = (float)iy + (half == 1 ? 0.5f : 0.0f);
            float p, e, q, f, s, t;
            two_prod(S.far_h[0], wx, p, e);
            two_prod(S.far_h[1], wy, q, f);
            e = __fmaf_rn(S.far_l[0], wx, e);
            f = __fmaf_rn(S.far_l[1], wy, f);
            two_sum(p, q, s, t);
            return __fadd_rn(s, __fadd_rn(t, __fadd_rn(e, f)));
        }
    }
    const double wx = ix + (half == 0 ? 0.5 : 0.0), wy = iy + (half == 1 ? 0.5 : 0.0);
    return R(vfma(wx, S.far_x, vmul(wy, S.far_y)));
}

// Asynchronous copy of one element from global to shared memory (cp.async), the end of a
// group of copies, and the wait until at most N groups are in flight.
template <class T>
__device__ __forceinline__ void cp_async(T* smem, const T* gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    if constexpr (sizeof(T) == 4) {
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(sa), "l"(gmem) : "memory");
    } else if constexpr (sizeof(T) == 8) {
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(sa), "l"(gmem) : "memory");
    } else {
        asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(gmem) : "memory");
        if constexpr (sizeof(T) == 32)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(sa + 16),
                         "l"(reinterpret_cast<const char*>(gmem) + 16)
                         : "memory");
    }
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// One warp's rows in flight: the stage input from row c-1 up to kAhead rows ahead of the one
// being read, and the operands of the update (W^n, H_e^n) and of the sources (F_s of the
// previous step or dF_s/dt).  Each lane copies and reads only its own column.
constexpr int kAhead = 4;   // rows c-1 = L-3 to L+4 fill the eight slots
template <class R>
struct StripBuf {
    typename Quad<R>::T w[8][32], w0[8][32];
    typename HeStore<R>::T he[8][32], he0[8][32];
    R phi[8][32], sd[8][32];
};

template <class R, bool UNI>
struct StageSmem {
    StripBuf<R> buf;
};
template <class R>
struct StageSmem<R, false> {
    StripBuf<R> buf;
    StageCase<R> c;
    float2 twice[sizeof(R) == 4 ? sizeof(PhysT<R>) / sizeof(R) : 1];
};

// Step end (Eq. 51): the strip's sums go to its slot, and the warp that finishes a group of
// 64 strips (512 where one group holds them all) last (an atomic ticket, no waiting) sums the group, the one that finishes the
// last group sums the groups and updates the case's statistics.  Both sums run in a fixed
// order, so the result does not depend on which warp is last.  (A kernel of its own for this
// took 10 us a step on the 128x64 case and 14 us on the 4096x2048 one.)

template <class R>
__device__ __forceinline__ void sum_slots(const typename DSum<R>::Slot* s, int n, int lane, DSum<R> a[kRedN]) {
#pragma unroll
    for (int q = 0; q < kRedN; ++q) a[q] = DSum<R>::zero();
#pragma unroll 2
    for (int t = lane; t < n; t += 32)
#pragma unroll
        for (int q = 0; q < kRedN; ++q) a[q].add(DSum<R>::of(ld_cg(&s[(size_t)t * kRedN + q])));
    // a butterfly: every lane ends with the same sums
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int q = 0; q < kRedN; ++q) a[q].shfl_xor_add(o);
}
template <class R>
__device__ __noinline__ void finish_strip(const StageCase<R>& S, int strips, int slot, int lane, DSum<R> sumC, DSum<R> sumH,
                                          DSum<R> sumF, int nDrop, int nBad) {
    using Slot = typename DSum<R>::Slot;
    Slot* red = static_cast<Slot*>(S.red);
    Slot* groups = static_cast<Slot*>(S.red_groups);
    if (lane == 0) {
        Slot* r = red + (size_t)slot * kRedN;
        DSum<R> sol = DSum<R>::count(nDrop);   // the droplet's solid sum: its cells minus its liquid sum
        sol.sub(sumF);
        r[0] = sumC.slot();
        r[1] = sumH.slot();
        r[2] = sumF.slot();
        r[3] = DSum<R>::count(nDrop).slot();
        r[4] = sol.slot();
        r[5] = DSum<R>::count(nBad).slot();
    }
    const int size = strips <= 512 ? 512 : kStageGroup;
    const int g = slot / size, ng = (strips + size - 1) / size;
    const int n = min(size, strips - g * size);
    if (!last_of(&S.tickets[1 + g], n, lane)) return;
    DSum<R> a[kRedN];
    sum_slots<R>(red + (size_t)g * size * kRedN, n, lane, a);
    if (ng > 1) {
        if (lane == 0)
            for (int q = 0; q < kRedN; ++q) groups[(size_t)g * kRedN + q] = a[q].slot();
        if (!last_of(&S.tickets[0], ng, lane)) return;
        sum_slots<R>(groups, ng, lane, a);
    }
    // one statistics slot per lane: FP64 instructions are slow, so each runs once for all slots
    double* st = S.stats;
    const double old = lane < kStatN ? st[lane] : 0.0;
    DSum<R> pick = a[0];
    if (lane == ST_SUM_HE) pick = a[1];
    if (lane == ST_SUM_FL_DROP) pick = a[2];
    if (lane == ST_N_DROP) pick = a[3];
    if (lane == ST_Q_L || lane == ST_QL_PREV) pick = a[4];
    if (lane == ST_NONFINITE) pick = a[5];
    double v = pick.value();
    const double drop = __shfl_sync(0xffffffffu, v, ST_N_DROP);
    const double QL = drop > 0.0 ? __shfl_sync(0xffffffffu, v, ST_Q_L) / drop : 0.0;
    const double t1 = __shfl_sync(0xffffffffu, old, ST_T) + S.dt, q0 = __shfl_sync(0xffffffffu, old, ST_QL_PREV);
    const double resid = __shfl_sync(0xffffffffu, old, ST_POT_RESID), cycles = __shfl_sync(0xffffffffu, old, ST_POT_CYCLES);
    bool put = lane <= ST_N_DROP;
    if (lane == ST_Q_L || lane == ST_QL_PREV) v = QL, put = true;
    if (lane == ST_NONFINITE) put = v > 0.0, v = 1.0;
    if (lane == ST_T) v = t1, put = true;
    if (lane == ST_STEP || lane == ST_STEPS_CALL) v = old + 1.0, put = true;
    // freezing time: first t with Q_L >= 0.99, linear between steps
    if (lane == ST_T_FREEZE && old < 0.0 && QL >= 0.99) v = (t1 - S.dt) + S.dt * (0.99 - q0) / (QL - q0), put = true;
    if (S.solve_potential) {
        if (lane == ST_POT_RESID_MAX) v = fmax(old, resid), put = true;
        if (lane == ST_POT_CYCLES_SUM) v = old + cycles, put = true;
    }
    if (put) st[lane] = v;
}

// Derived quantities of one row.
template <class R>
struct RowQ {
    R p, u, v, C, T, H, Fs, rho;
};

// One warp advances a strip of kStripW columns and `rows` rows, one lane per column with three
// halo columns on each side, marching up in y: C and phi of row L are read, row L-1 is derived
// and gets its mu_c and |H|^2, the slopes and face fluxes follow for row c = L-2 (x face to the
// left, y face below), and row c-1 is completed and stored.  What a row's neighbours in y need
// stays in registers; neighbours in x come by warp shuffles.  There is no block barrier.
//
// Bound by instruction issue and the latency of one row's chain (FP32: 59 % of the issue slots
// busy, 44 % of the FMA pipe; HBM at a third), in FP64 by the FP64 pipe.  A marching strip derives
// each cell (rows + 4)/rows x 32/26 times, 1.44 with 24 rows (6.2 with one), instead of a 32 x 8
// tile's 2.08, forms a cell's side sums once for both its faces instead of once per face, and
// reads a face's operands from registers and shuffles instead of 54 shared-memory loads:
// 4096x2048, mixed, 1637 -> 851 thread instructions per cell and 0.52 -> 0.28 ms a launch; FP64
// 18.6 -> 11.3 ms; 1024x512, mixed, 64 -> 33 us.  At 168 registers 12 warps an SM; 16 warps (128
// registers) spill and take 0.50 ms, two columns per lane (255 registers, 8 warps) 0.37-0.43 ms.
// Strips away from walls and wraps run without any of their logic (0.35 -> 0.30 ms),
// coefficients from the constant bank save 4 %, copies four rows ahead 7 %.
template <class R, int STAGE, bool HALF, bool UNI>
__global__ void __launch_bounds__(32, sizeof(R) == 4 ? 12 : 4)
stage_kernel(const StageCase<R>* __restrict__ cases, const TileRef* __restrict__ tiles, int rows,
             const __grid_constant__ StageCase<R> arg) {
    using V = typename PairOf<R>::T;
    using HR = typename HeStore<R>::T;
    using R4 = typename Quad<R>::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    StageSmem<R, UNI>& sm = *reinterpret_cast<StageSmem<R, UNI>*>(smem_raw);
    const int lane = threadIdx.x;
    TileRef tr;
    if constexpr (UNI) {
        const int nsx = (arg.nx + kStripW - 1) / kStripW;
        tr.slot = blockIdx.x;
        tr.x0 = (tr.slot % nsx) * kStripW;
        tr.y0 = (tr.slot / nsx) * rows;
    } else {
        tr = tiles[blockIdx.x];
        const int* src = reinterpret_cast<const int*>(cases + tr.case_id);
        int* dst = reinterpret_cast<int*>(&sm.c);
        for (int i = lane; i < (int)(sizeof(StageCase<R>) / sizeof(int)); i += 32) dst[i] = src[i];
        __syncwarp();
        if constexpr (sizeof(R) == 4) {
            const float* q = reinterpret_cast<const float*>(&sm.c.Q);
            for (int i = lane; i < (int)(sizeof(PhysT<R>) / sizeof(R)); i += 32) sm.twice[i] = make_float2(q[i], q[i]);
            __syncwarp();
        }
    }
    const StageCase<R>* cs;
    if constexpr (UNI) cs = &arg;
    else cs = &sm.c;
    const StageCase<R>& S = *cs;
    const PhysT<R>& Q = S.Q;
    const float2* twice = nullptr;
    if constexpr (!UNI && sizeof(R) == 4) twice = sm.twice;
    const Coefs<R> kc{Q, twice};
    constexpr int in = STAGE, out = STAGE == 2 ? 0 : STAGE + 1;
    StripBuf<R>& B = sm.buf;
    const int nx = S.nx, ny = S.ny, pitch = S.pitch;
    const bool per_x = S.periodic_x != 0, per_y = S.periodic_y != 0;
    const int x0 = tr.x0, y0 = tr.y0, yend = min(y0 + rows, ny);
    const int gx = x0 - 3 + lane;
    // source column and, at a ghost column, its wall
    int sx = gx, wallx = -1;
    if (per_x) {
        sx = gx < 0 ? gx + nx : (gx >= nx ? gx - nx : gx);
    } else {
        if (gx == -1) wallx = 0;
        if (gx == nx) wallx = 1;
    }
    sx = min(max(sx, 0), nx - 1);
    const bool edge_x = !per_x && (x0 == 0 || x0 + 28 >= nx);   // a wall ghost column lies in the strip
    const bool active = lane >= 3 && lane < 3 + kStripW && gx < nx;

    auto march = [&](auto edge_tag) {
    constexpr bool EDGE = decltype(edge_tag)::value;
    auto src_row = [&](int L) {
        if (!EDGE) return L;
        int s = L;
        if (per_y) s = L < 0 ? L + ny : (L >= ny ? L - ny : L);
        return min(max(s, 0), ny - 1);
    };
    auto fetch_row = [&](int L) {
        const unsigned i = (unsigned)src_row(L) * (unsigned)pitch + (unsigned)sx;
        const int q = L & 7;
        cp_async(&B.he[q][lane], static_cast<const HR*>(S.He[in]) + i);
        cp_async(&B.w[q][lane], static_cast<const R4*>(S.W[in]) + i);
        cp_async(&B.phi[q][lane], static_cast<const R*>(S.phi) + i);
    };
    auto wall_row = [&](int L) { return !EDGE || per_y ? -1 : (L == -1 ? 2 : (L == ny ? 3 : -1)); };
    // T, F_l and the reconstruction H_e by Eq. 8, rho by Eq. 11, u = m / (rho / 3); at a wall
    // ghost the mirror rules
    auto derive = [&](int L) {
        RowQ<R> q;
        const R4 w = B.w[L & 7][lane];
        R Fl;
        const R C = w.w;
        invert_cell<UNI, R>(Q, B.he[L & 7][lane], C, q.T, Fl, q.H);
        q.Fs = R(1) - Fl;
        q.rho = vmix(q.Fs, C, cf<UNI>(Q.rho_s), cf<UNI>(Q.rho_lg), cf<UNI>(Q.rho_g));
        const R ri = fdiv(R(3), q.rho);
        q.p = w.x;
        q.u = vmul(w.y, ri);
        q.v = vmul(w.z, ri);
        q.C = C;
        const int wally = wall_row(L);
        if (EDGE && (edge_x || wally >= 0)) {
            const int wall = wally >= 0 ? wally : wallx;
            if (wall >= 0) {
                q.u = -q.u;
                q.v = -q.v;
                if (S.thermal_dir[wall]) q.T = vfma(R(2), Q.wall_T[wall], -q.T);
                q.H = vfma(vmix(q.Fs, C, cf<UNI>(Q.cp_s), cf<UNI>(Q.cp_lg), cf<UNI>(Q.cp_g)), q.T, vmul(cf<UNI>(Q.L), R(1) - q.Fs));
                // a wall ghost's C follows the wetting rule (unchanged at 90 degrees, wet = 0)
                q.C = vfma(vmul(cf<UNI>(Q.wet), C), R(1) - C, C);
            }
        }
        return q;
    };
    // C and phi of row L, with their ghost rules (the wetting rule; the far field mirrored)
    auto load_cphi = [&](int L, R& C, R& phi) {
        C = B.w[L & 7][lane].w;
        phi = B.phi[L & 7][lane];
        const int wally = wall_row(L);
        if (EDGE && (edge_x || wally >= 0)) {
            const int wall = wally >= 0 ? wally : wallx;
            if (wall >= 0) {
                C = vfma(vmul(cf<UNI>(Q.wet), C), R(1) - C, C);
                if (S.mag_dir[wall])
                    phi = far_field_twice(S, wall == 0 ? 0 : (wall == 1 ? nx : sx), wall == 2 ? 0 : (wall == 3 ? ny : src_row(L)),
                                          wall < 2 ? 1 : 0) - phi;
            }
        }
    };

    RowQ<R> qm = {}, q0 = {};               // rows c-1, c
    R mum = 0, mu0 = 0, h2m = 0, h20 = 0;   // mu_c and |H|^2 of rows c-1, c
    R ph0 = 0, ph1 = 0;                     // phi of rows L-2, L-1
    R dxC = 0;                              // C(i+1) - C(i-1) of row c
    R ca[NA];                               // this row's A values for the y face above
    R xs[5];                                // row c-1: R(W) but for its upper y flux
#pragma unroll
    for (int i = 0; i < NA; ++i) ca[i] = 0;
#pragma unroll
    for (int i = 0; i < 5; ++i) xs[i] = 0;
    // step-end sums of this lane's cells (last stage)
    DSum<R> sumC = DSum<R>::zero(), sumH = DSum<R>::zero(), sumF = DSum<R>::zero();
    int nDrop = 0, nBad = 0;
    const R c3 = R(1.0 / 3.0);
    const R b = STAGE == 0 ? R(1) : (STAGE == 1 ? R(0.25) : R(2.0 / 3.0));

    // Copies run kAhead iterations ahead of their use: iteration L reads C and phi of row L, uses
    // the source operand of row L-2 and W^n of row L-3.  Rows y0-3 and y0-2 enter only through
    // C and phi.
    const auto fetch_ops = [&](int rs, int rw) {
        if (!active) return;
        if (rs >= y0 && rs < yend)
            cp_async(&B.sd[rs & 7][lane], static_cast<const R*>(STAGE == 0 ? S.Fs_prev : S.Sdot) +
                                              ((unsigned)rs * (unsigned)pitch + (unsigned)gx));
        if (STAGE > 0 && rw >= y0 && rw < yend) {
            const unsigned i = (unsigned)rw * (unsigned)pitch + (unsigned)gx;
            cp_async(&B.he0[rw & 7][lane], static_cast<const HR*>(S.He[0]) + i);
            cp_async(&B.w0[rw & 7][lane], static_cast<const R4*>(S.W[0]) + i);
        }
    };
    fetch_row(y0 - 3);
#pragma unroll
    for (int i = 0; i <= kAhead; ++i) {
        fetch_row(y0 - 2 + i);
        if (i == kAhead) fetch_ops(y0, y0 - 1);
        cp_commit();
    }
    cp_wait<kAhead>();
    {
        R unused;
        load_cphi(y0 - 3, q0.C, ph0);
        load_cphi(y0 - 2, unused, ph1);
    }
    for (int L = y0 - 1; L <= yend + 2; ++L) {
        const int c = L - 2;
        if (L + kAhead <= yend + 2) fetch_row(L + kAhead);
        fetch_ops(L + 2, L + 1);
        cp_commit();
        cp_wait<kAhead>();
        R ph, Cn;
        load_cphi(L, Cn, ph);
        const RowQ<R> q1 = derive(L - 1);   // row c+1 (of row y0-4, before the first, nothing is used)
        // ---- mu_c and |H|^2 of row L-1
        const R cl = up(q1.C), cr = dn(q1.C), pl = up(ph1), pr = dn(ph1);
        const R lap = vfma(R(-4), q1.C, (cr + cl) + (Cn + q0.C));
        R mu1 = vfma(vmul(vmul(cf<UNI>(Q.beta2), q1.C), q1.C - R(1)), vfma(R(2), q1.C, R(-1)), -vmul(cf<UNI>(Q.kappa), lap));
        const R hx = vmul(R(0.5), pr - pl), hy = vmul(R(0.5), ph - ph0);
        R h21 = vfma(hx, hx, vmul(hy, hy));
        if (EDGE && edge_x) {   // a wall ghost takes its inner cell's values
            const R ml = up(mu1), mr = dn(mu1), hl = up(h21), hr = dn(h21);
            mu1 = wallx == 0 ? mr : (wallx == 1 ? ml : mu1);
            h21 = wallx == 0 ? hr : (wallx == 1 ? hl : h21);
        }
        const R dxC1 = cr - cl;
        if (EDGE && !per_y) {
            if (c == 0) {
                mum = mu0;
                h2m = h20;
            }
            if (c == ny - 1) {
                mu1 = mu0;
                h21 = h20;
            }
        }
        if (c >= y0 - 1) {
            // ---- row c: central differences (twice the slopes) along x and y
            const R dx[7] = {dn(q0.p) - up(q0.p), dn(q0.u) - up(q0.u), dn(q0.v) - up(q0.v), dxC,
                             dn(mu0) - up(mu0), dn(q0.T) - up(q0.T), dn(q0.H) - up(q0.H)};
            const R dy[7] = {q1.p - qm.p, q1.u - qm.u, q1.v - qm.v, q1.C - qm.C, mu1 - mum, q1.T - qm.T, q1.H - qm.H};
            // G: minus dts times the tangential slope; N: normal difference; n and t swap
            // between the axes for the velocity
            V G[6], N[7], c7[7];
            const V mhd = c2<UNI>(kc, Q.mhd);
            G[0] = vmul(mhd, mk(dy[0], dx[0]));
            G[1] = vmul(mhd, mk(dy[1], dx[2]));
            G[2] = vmul(mhd, mk(dy[2], dx[1]));
            G[3] = vmul(mhd, mk(dy[3], dx[3]));
            G[4] = sp(R(0));
            G[5] = vmul(mhd, mk(dy[5], dx[5]));
            N[0] = mk(dx[0], dy[0]);
            N[1] = mk(dx[1], dy[2]);
            N[2] = mk(dx[2], dy[1]);
#pragma unroll
            for (int q = 3; q < 7; ++q) N[q] = mk(dx[q], dy[q]);
            c7[0] = sp(q0.p);
            c7[1] = mk(q0.u, q0.v);
            c7[2] = mk(q0.v, q0.u);
            c7[3] = sp(q0.C);
            c7[4] = sp(mu0);
            c7[5] = sp(q0.T);
            c7[6] = sp(q0.H);
            const R cp0 = vmix(q0.Fs, q0.C, cf<UNI>(Q.cp_s), cf<UNI>(Q.cp_lg), cf<UNI>(Q.cp_g));
            const R om = R(1) - q0.Fs;
            const V r1 = sp(om * cf<UNI>(Q.rho_lg)), k1 = sp(om * cf<UNI>(Q.cp_lg));
            V sa[6], sb[6], pa, pb;
            if (HALF) {
                // the centre point is the cell centre: one set of even and odd parts serves
                // both faces of an axis
                V e[6], o[6];
                side_sums<V>(sp(R(3) * q0.p), c7[1], c7[2], c7[3], sp(R(3) * q0.C), sp(cf<UNI>(Q.Qg3) * mu0), c7[5], sp(q0.rho), sp(cp0),
                             sp(cp0 * q0.T), sp(cf<UNI>(Q.cp_ref) * q0.T), r1, k1, G, e, o);
#pragma unroll
                for (int q = 0; q < 6; ++q) {
                    sa[q] = vadd(e[q], o[q]);
                    sb[q] = vsub(e[q], o[q]);
                }
                pa = pb = c7[0];
            } else {
                // the centre points move along the normal by (1/2 - dts) cells
                const V rg = sp(vfma(q0.Fs, cf<UNI>(Q.rho_sg), cf<UNI>(Q.rho_g))), kg = sp(vfma(q0.Fs, cf<UNI>(Q.cp_sg), cf<UNI>(Q.cp_g)));
#pragma unroll
                for (int side = 0; side < 2; ++side) {
                    const V sh = sp(side == 0 ? cf<UNI>(Q.off) : -cf<UNI>(Q.off));
                    V d[6], e[6], o[6];
#pragma unroll
                    for (int q = 0; q < 6; ++q) d[q] = vfma(sh, N[q], c7[q]);
                    const V rho = vfma(r1, d[3], rg), k = vfma(k1, d[3], kg);
                    side_sums<V>(vmul(sp(R(3)), d[0]), d[1], d[2], d[3], vmul(sp(R(3)), d[3]), vmul(sp(cf<UNI>(Q.Qg3)), d[4]), d[5],
                                 rho, k, vmul(k, d[5]), vmul(sp(cf<UNI>(Q.cp_ref)), d[5]), r1, k1, G, e, o);
#pragma unroll
                    for (int q = 0; q < 6; ++q) {
                        if (side == 0) sa[q] = vadd(e[q], o[q]);
                        else sb[q] = vsub(e[q], o[q]);
                    }
                    if (side == 0) pa = d[0];
                    else pb = d[0];
                }
            }
            // ---- A's values of both faces: x from the lane to the left, y from the row below
            V a[NA], br[7];
#pragma unroll
            for (int q = 0; q < 6; ++q) {
                a[A_SUM + q] = mk(up(sa[q].x), ca[A_SUM + q]);
                ca[A_SUM + q] = sa[q].y;
            }
#pragma unroll
            for (int q = 0; q < 7; ++q) {
                const V h = vmul(sp(R(0.5)), c7[q]);
                const V rp = vfma(sp(R(0.125)), N[q], h);
                br[q] = vfma(sp(R(-0.125)), N[q], h);
                a[A_REC + q] = mk(up(rp.x), ca[A_REC + q]);
                ca[A_REC + q] = rp.y;
            }
#pragma unroll
            for (int q = 0; q < 6; ++q)
                if (q != 4) {
                    a[A_G + q] = mk(up(G[q].x), ca[A_G + q]);
                    ca[A_G + q] = G[q].y;
                }
            a[A_P] = mk(up(pa.x), ca[A_P]);
            ca[A_P] = pa.y;
            const R fs_below = ca[A_FS];
            a[A_FS] = mk(up(q0.Fs), fs_below);
            ca[A_FS] = q0.Fs;
            if (c >= y0) {
                V F[5];
                face_flux<UNI, R, V>(kc, a, sb, br, G, pb, q0.Fs, F);
                // order: H_e, p, m_x, m_y, C
                R fl[5] = {F[0].x, F[1].x, F[2].x, F[3].x, F[4].x};
                R fy[5] = {F[0].y, F[1].y, F[3].y, F[2].y, F[4].y};
                if (EDGE && edge_x) {
                    if (gx == 0) wall_flux<R>(Q, S.thermal_dir[0], 0, q0.Fs, q0.C, q0.rho, q0.p, q0.v, q0.T, fl);
                }
                R fr[5];
#pragma unroll
                for (int q = 0; q < 5; ++q) fr[q] = dn(fl[q]);
                if (EDGE && edge_x) {
                    if (gx == nx - 1) wall_flux<R>(Q, S.thermal_dir[1], 1, q0.Fs, q0.C, q0.rho, q0.p, q0.v, q0.T, fr);
                }
                if (EDGE && !per_y && (c == 0 || c == ny)) {
                    R w[5];
                    if (c == 0) wall_flux<R>(Q, S.thermal_dir[2], 2, q0.Fs, q0.C, q0.rho, q0.p, q0.u, q0.T, w);
                    else wall_flux<R>(Q, S.thermal_dir[3], 3, fs_below, qm.C, qm.rho, qm.p, qm.u, qm.T, w);
                    fy[0] = w[0];
                    fy[1] = w[1];
                    fy[2] = w[3];
                    fy[3] = w[2];
                    fy[4] = w[4];
                }
                // ---- row c-1: R(W), Runge-Kutta combination, store
                if (active && c > y0) {
                    const unsigned io = (unsigned)(c - 1) * (unsigned)pitch + (unsigned)gx;
                    const HR Hek = B.he[(c - 1) & 7][lane];
                    const R4 wk = B.w[(c - 1) & 7][lane];
                    HR He0 = Hek;
                    R4 w0 = wk;
                    if (STAGE > 0) {
                        He0 = B.he0[(c - 1) & 7][lane];
                        w0 = B.w0[(c - 1) & 7][lane];
                    }
                    R Rw[5];
#pragma unroll
                    for (int q = 0; q < 5; ++q) Rw[q] = xs[q] - fy[q];
                    const R dt = cf<UNI>(Q.dt);
                    HR Hen = he_rk(STAGE, Hek, He0, dt, Rw[0], b);
                    R4 wn;
                    // a W^n + b X written as W^n + b (X - W^n): a + b = 1 holds exactly, so a
                    // steady state stays steady in FP32 (1/3 and 2/3 both round up in FP32)
                    auto rk = [&](R n0, R nk, R rw) {
                        const R x = vfma(dt, rw, nk);
                        return STAGE == 0 ? x : vfma(b, vsub(x, n0), n0);
                    };
                    wn.x = rk(w0.x, wk.x, Rw[1]);
                    wn.y = rk(w0.y, wk.y, Rw[2]);
                    wn.z = rk(w0.z, wk.z, Rw[3]);
                    wn.w = rk(w0.w, wk.w, Rw[4]);
                    if (STAGE == 2) {
                        // step end: solid held at rest, (rho u) <- (1 - F_s)(rho u)
                        R Tn, Fln, Hr;
                        invert_cell<UNI, R>(Q, Hen, wn.w, Tn, Fln, Hr);
                        wn.y = vmul(wn.y, Fln);
                        wn.z = vmul(wn.z, Fln);
                        // (the fine multigrid level has the fields' pitch)
                        static_cast<R*>(S.mu)[io] = R(1) + vmix(R(1) - Fln, wn.w, cf<UNI>(Q.chi_s), cf<UNI>(Q.chi_lg), cf<UNI>(Q.chi_g));
                        sumC.add(wn.w);
                        sumH.add(Hen);
                        if (wn.w >= R(0.5)) {
                            sumF.add(Fln);
                            nDrop += 1;
                        }
                        if (!(he_finite(Hen) && isfinite(wn.x) && isfinite(wn.y) && isfinite(wn.z) && isfinite(wn.w))) nBad += 1;
                    }
                    static_cast<HR*>(S.He[out])[io] = Hen;
                    static_cast<R4*>(S.W[out])[io] = wn;
                }
                // ---- row c: sources (Eq. 41) and the x-flux difference
                const R C = q0.C, rho = q0.rho, vr = cf<UNI>(Q.vol_ratio);
                R Sd = B.sd[c & 7][lane];
                if (STAGE == 0) {
                    // lagged dF_s/dt from F_s^n (this stage's input) and the previous step's
                    // F_s, which is then replaced by F_s^n
                    Sd = (q0.Fs - Sd) * cf<UNI>(Q.inv_dt);
                    if (active && c < yend) {
                        const unsigned ic = (unsigned)c * (unsigned)pitch + (unsigned)gx;
                        static_cast<R*>(S.Fs_prev)[ic] = q0.Fs;
                        static_cast<R*>(S.Sdot)[ic] = Sd;
                    }
                }
                const R chi = vmul(vmix(q0.Fs, C, cf<UNI>(Q.chi_s), cf<UNI>(Q.chi_lg), cf<UNI>(Q.chi_g)), R(0.25));
                const R drx = dn(q0.rho) - up(q0.rho), dry = q1.rho - qm.rho;
                const R dhx = dn(h20) - up(h20), dhy = h21 - h2m;
                const R hC = vmul(R(-0.5), C), rs = vmul(rho, Sd);
                xs[0] = vfma(vmul(cp0, q0.T), vmul(R(0.5), dx[1] + dy[2]), -(fr[0] - fl[0]));
                xs[1] = vfma(c3, vfma(R(0.5), vfma(q0.u, drx, vmul(q0.v, dry)), vmul(vr, rs)), -(fr[1] - fl[1]));
                xs[2] = vfma(c3, vfma(-q0.u, rs, vfma(hC, dx[4], vmul(chi, dhx))), -(fr[2] - fl[2]));
                xs[3] = vfma(c3, vfma(-q0.v, rs, vfma(rho, cf<UNI>(Q.gravity), vfma(hC, dy[4], vmul(chi, dhy)))),
                             -(fr[3] - fl[3]));
                xs[4] = vfma(C, vmul(vr, Sd), -(fr[4] - fl[4]));
#pragma unroll
                for (int q = 0; q < 5; ++q) xs[q] += fy[q];
            }
        }
        qm = q0;
        q0 = q1;
        mum = mu0;
        mu0 = mu1;
        h2m = h20;
        h20 = h21;
        ph0 = ph1;
        ph1 = ph;
        dxC = dxC1;
    }
    if (STAGE == 2) {
        // the strip's sums in a fixed order: each lane over its rows, then the lanes
        nDrop = __reduce_add_sync(0xffffffffu, nDrop);
        nBad = __reduce_add_sync(0xffffffffu, nBad);
        for (int o = 16; o > 0; o >>= 1) {
            sumC.shfl_add(o);
            sumH.shfl_add(o);
            sumF.shfl_add(o);
        }
        finish_strip<R>(S, UNI ? (int)gridDim.x : S.strips, tr.slot, lane, sumC, sumH, sumF, nDrop, nBad);
    }
    };
    if (x0 >= 3 && x0 + 28 < nx && y0 >= 3 && yend + 2 < ny) march(std::false_type{});
    else march(std::true_type{});
}

// One stage of every strip; `one`: the case of a UNI launch.
template <class R, bool HALF, bool UNI>
cudaError_t stage_launch(const StageCase<R>& one, const StageCase<R>* cases, const TileRef* tiles, int ntiles, int rows,
                         int stage, cudaStream_t st)
#ifdef LBFS_STAGE_DEFINE
{
    constexpr size_t sm = sizeof(StageSmem<R, UNI>);
    static_assert(sm <= 48 * 1024, "within the default shared memory of a block");
    if (stage == 0) stage_kernel<R, 0, HALF, UNI><<<ntiles, 32, sm, st>>>(cases, tiles, rows, one);
    else if (stage == 1) stage_kernel<R, 1, HALF, UNI><<<ntiles, 32, sm, st>>>(cases, tiles, rows, one);
    else stage_kernel<R, 2, HALF, UNI><<<ntiles, 32, sm, st>>>(cases, tiles, rows, one);
    return cudaGetLastError();
}
#else
    ;
#endif

}  // namespace lbfs
