// lbfs_internal.cuh -- device-side data layout and the per-point physics of the
// LBFS step shared by the stage, potential and reduction kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace lbfs {

constexpr int kMaxLevels = 16;
constexpr int kRedN = 6;        // partial sums of a strip in the step-end reduction
constexpr int kFinChunks = 32;  // blocks per case that sum a stored state's statistics
constexpr int kStatN = 20;      // per-case device statistics slots

// statistics slots (FP64, per case).  ST_POT_RESID_MAX, ST_POT_CYCLES_SUM and
// ST_STEPS_CALL accumulate over the steps of one lbfs_step call.
enum StatSlot {
    ST_SUM_C = 0, ST_SUM_HE, ST_SUM_FL_DROP, ST_N_DROP, ST_Q_L, ST_T, ST_T_FREEZE,
    ST_POT_RESID, ST_POT_CYCLES, ST_NONFINITE, ST_QL_PREV, ST_POT_DONE, ST_B2, ST_STEP,
    ST_POT_FAIL, ST_POT_RESID_MAX, ST_POT_CYCLES_SUM, ST_STEPS_CALL, ST_EXTRAP, ST_SCALE
};

// Physical and numerical parameters of one case, resolved on the host in FP64.
struct CaseParams {
    int nx, ny, pitch;          // cells and row pitch (elements)
    int periodic_x, periodic_y;
    int thermal_dir[4];         // 1: Dirichlet temperature wall
    int mag_dir[4];             // 1: Dirichlet potential wall
    int solve_potential;        // 0: chi == 0 or no Dirichlet wall -> phi fixed
    double wall_T[4];
    double rho_l, rho_g, rho_s, mu_l, mu_g, mu_s, cp_l, cp_g, cp_s;
    double lam_l, lam_g, lam_s, chi_l, chi_g, chi_s;
    double beta, kappa, mobility, Q_g, gravity, T_m, L;
    double dt, dts, cp_ref, vol_ratio, H0, cos_t, sin_t;
    double wet;                 // 4 cos(theta_w)/xi of the wetting ghost rule (0 at 90 deg)
};

// The per-point coefficients in the working precision R, converted once on the host
// so that no kernel converts FP64 parameters inside its inner loops.
template <class R>
struct PhysT {
    R rho_s, rho_g, mu_s, mu_l, mu_g, lam_s, lam_l, lam_g;
    R cp_s, cp_g, chi_s, chi_g;
    R kappa, cp_ref, inv_dts, inv_cpref_dts, dt, vol_ratio, gravity, T_m, L;
    R wall_T[4];
    R wet;
    // the thresholds H_es = C_p,s T_m and L of Eq. 8 as (hi, lo) pairs of R: the exact
    // FP64 value is hi + lo to FP32-pair accuracy (lo = 0 in FP64)
    R Hes_hi, Hes_lo, L_hi, L_lo;
    // formed once: property differences g_s - g_g and g_l - g_g, -Q_g, -C_p,ref/3, 1/C_p,s,
    // tau_g - 1/2 and one minus it, 2 beta, 3 Q_g, -dts/2, (1/2 - dts)/2, 1/dt
    R rho_sg, rho_lg, cp_sg, cp_lg, mu_sg, mu_lg, lam_sg, lam_lg, chi_lg;
    R m_Qg, m_cp_ref3, om_x_g, inv_cps, x_g, beta2, Qg3, mhd, off, inv_dt;
};

// p, rho c_s^2 u, rho c_s^2 v and C of one cell: one vector load or store
struct alignas(32) Quad64 {
    double x, y, z, w;
};
template <class R>
struct Quad;
template <>
struct Quad<float> {
    using T = float4;
};
template <>
struct Quad<double> {
    using T = Quad64;
};

struct MGLevel {
    int nx, ny, pitch;
    // Coarse levels halve the cell count with the size rounded up, so the last column
    // (row) of a level may cover fewer fine cells than the others: wlx (wly) is its
    // width (height) relative to the level's other cells, 1 when the level is regular.
    float wlx, wly;
    int ragged;  // wlx < 1 or wly < 1
    void* mu;   // cell coefficient mu_m (FP32; FP64 on the fine level of the FP64 mode)
    void* e;    // correction (FP32), pre-smoothed
    void* eu;   // the finished correction of a coarse level: an array of its own where a kernel leg writes it
                // (tiles read their neighbours' e), e where one block holds the whole level
    void* r;    // right-hand side / residual (as mu)
};

// Everything the kernels need to know about one case.
struct DevCase {
    CaseParams P;
    // state sets: 0 = W^n (and W^{n+1}), 1 and 2 = Runge-Kutta stage buffers
    void* He[3];      // HR precision (FP64 in both modes)
    void* W[3];       // Quad<R>: p, rho c_s^2 u, rho c_s^2 v, C
    void* phi;        // potential read by the stage kernel (R); FP64 mode: the master
    double* phi64;    // FP64 mode: the master potential (== phi); mixed: unused
    double* phi_prev64;  // FP64 mode: the potentials of the last step and of the one before it; mixed: unused
    float* phi_lo;    // mixed: low word of the master potential phi + phi_lo (FP32 pair)
    void* Fs_prev;    // R: F_s of the previous step, replaced by F_s^n in stage 1
    void* Sdot;       // R: lagged dF_s/dt of the current step, written by stage 1
    int nlev;
    MGLevel lev[kMaxLevels];
    void* red;        // stage-strip partial sums, kRedN 8-byte DSum slots per strip
    void* red_groups; // the same per group of strips
    unsigned* red_tickets;
    int tail;         // level from which the V-cycle runs in one kernel (nlev - 1: the coarsest alone)
    void* mg_red;     // potential residual partial sums, 2 DSum slots per residual strip
    void* mg_groups;  // the same per group of strips
    unsigned* mg_tickets;   // [0] groups, [1 + g] strips of group g that have finished
    int mg_strips;
    float far_h[2], far_l[2];   // the far field's slopes -H0 (cos, sin) as FP32 pairs
    void* chunk;      // kFinChunks x kRedN DSum slots: per-chunk sums of the set-up statistics
    unsigned* tickets;  // set-up statistics: chunks done (the last one finalises)
    double* stats;    // kStatN FP64 slots
};

// What the stage kernel needs of one case.
template <class R>
struct StageCase {
    PhysT<R> Q;
    void* He[3];
    void* W[3];
    void* phi;
    void* Fs_prev;
    void* Sdot;
    void* mu;         // the potential's fine-level coefficient (the fields' pitch)
    void* red;          // per strip, kRedN DSum slots of its step-end sums
    void* red_groups;   // the same per group of strips
    unsigned* tickets;  // [0] groups, [1 + g] strips of group g that have finished
    double* stats;
    double dt;
    double far_x, far_y;   // -2 H0 (cos, sin): twice the far field's slopes
    float far_h[2], far_l[2];   // the same as FP32 pairs
    int nx, ny, pitch, periodic_x, periodic_y;
    int thermal_dir[4], mag_dir[4];
    int solve_potential;
    int strips;         // strips of the case (batch launches)
    int pad_;
};

// One block's work: the tile at (x0, y0) of a case; slot numbers the case's
// partial-sum entries.
struct TileRef {
    int case_id, x0, y0, slot;
};

// Eq. 11 mixture: F_s g_s + (1 - F_s) C g_l + (1 - F_s)(1 - C) g_g
template <class R>
__device__ __forceinline__ R mixture(R Fs, R C, double gs, double gl, double gg) {
    R liq = R(gg) + C * (R(gl) - R(gg));
    return liq + Fs * (R(gs) - liq);
}

// Eq. 8 with T_s = T_l = T_m, H_es = C_p,s T_m, H_el = C_p,L(C) T_m + L, phase change
// only where C >= 1/2.  The differences against the thresholds are formed in the
// enthalpy's storage precision HR (FP64), the rest in R.
template <class R, class HR>
__device__ __forceinline__ void invert_enthalpy(const CaseParams& P, HR He, R C, R& T, R& Fl) {
    R cpL = R(P.cp_g) + C * (R(P.cp_l) - R(P.cp_g));
    HR Hes = HR(P.cp_s) * HR(P.T_m);
    HR Hel = HR(cpL) * HR(P.T_m) + HR(P.L);
    if (C < R(0.5)) {
        Fl = R(1);
        T = R(P.T_m) + R(He - Hel) / cpL;
    } else if (He < Hes) {
        Fl = R(0);
        T = R(He) / R(P.cp_s);
    } else if (He <= Hel) {
        Fl = R(He - Hes) / R(Hel - Hes);
        T = R(P.T_m);
    } else {
        Fl = R(1);
        T = R(P.T_m) + R(He - Hel) / cpL;
    }
}

// a / b: exact in FP64; in FP32 the fast reciprocal-multiply (within 2 ulp), which
// is below the rounding of the FP32 fluxes it feeds
template <class R>
__device__ __forceinline__ R fdiv(R a, R b) {
    return a / b;
}
template <>
__device__ __forceinline__ float fdiv<float>(float a, float b) {
    return __fdividef(a, b);
}

template <class R>
__device__ __forceinline__ R mix(R Fs, R C, R gs, R gl, R gg) {
    const R liq = gg + C * (gl - gg);
    return liq + Fs * (gs - liq);
}

// ---- FP64-accurate arithmetic on FP32 pairs (hi + lo, |lo| <= ulp(hi)/2) ---------
// Error-free transformations: two_sum (Knuth), two_prod (FMA).  Explicit round-to-
// nearest intrinsics keep the compiler from contracting or reordering them.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
__device__ __forceinline__ void two_prod(float a, float b, float& p, float& e) {
    p = __fmul_rn(a, b);
    e = __fmaf_rn(a, b, -p);
}
// (sh, sl) += (ph, pl), renormalised
__device__ __forceinline__ void pair_add(float& sh, float& sl, float ph, float pl) {
    float s, e;
    two_sum(sh, ph, s, e);
    e = __fadd_rn(e, __fadd_rn(sl, pl));
    sh = __fadd_rn(s, e);
    sl = __fsub_rn(e, __fsub_rn(sh, s));
}
// split a double into the nearest FP32 pair
__device__ __forceinline__ void pair_from(double v, float& h, float& l) {
    h = (float)v;
    l = (float)(v - (double)h);
}

// (hi, lo) + x for an FP32 x, renormalised (|lo| <= ulp(hi)/2)
__device__ __forceinline__ float2 pair_add_f(float2 a, float x) {
    float s, e;
    two_sum(a.x, x, s, e);
    e = __fadd_rn(e, a.y);
    float2 r;
    r.x = __fadd_rn(s, e);
    r.y = __fsub_rn(e, __fsub_rn(r.x, s));
    return r;
}
// (hi, lo) + (hi, lo), renormalised
__device__ __forceinline__ float2 pair_add2(float2 a, float2 b) {
    float2 r = a;
    pair_add(r.x, r.y, b.x, b.y);
    return r;
}

// ---- FP64-accurate sums ------------------------------------------------------------
// FP64 in the FP64 mode.  In mixed precision an FP32 pair accumulated with error-free
// additions (about 48 bits), so that no per-cell or per-tile FP64 instruction is
// issued.  Slot is the 8-byte type of a partial sum kept in a global or shared buffer;
// counts below 2^24 are exact in either.
template <class R>
struct DSum;
template <>
struct DSum<double> {
    using Slot = double;
    double v;
    static __device__ __forceinline__ DSum zero() { DSum s; s.v = 0.0; return s; }
    static __device__ __forceinline__ DSum of(Slot x) { DSum s; s.v = x; return s; }
    static __device__ __forceinline__ DSum count(int n) { DSum s; s.v = (double)n; return s; }
    __device__ __forceinline__ void add(double x) { v += x; }
    __device__ __forceinline__ void add(DSum o) { v += o.v; }
    __device__ __forceinline__ void sub(DSum o) { v -= o.v; }
    __device__ __forceinline__ void shfl_add(int o) { v += __shfl_down_sync(0xffffffffu, v, o); }
    __device__ __forceinline__ void shfl_xor_add(int o) { v += __shfl_xor_sync(0xffffffffu, v, o); }
    __device__ __forceinline__ Slot slot() const { return v; }
    __device__ __forceinline__ double value() const { return v; }
};
template <>
struct DSum<float> {
    using Slot = float2;
    float2 v;
    static __device__ __forceinline__ DSum zero() { DSum s; s.v.x = 0.0f; s.v.y = 0.0f; return s; }
    static __device__ __forceinline__ DSum of(Slot x) { DSum s; s.v = x; return s; }
    static __device__ __forceinline__ DSum count(int n) { DSum s; s.v.x = (float)n; s.v.y = 0.0f; return s; }
    __device__ __forceinline__ void add(float x) { v = pair_add_f(v, x); }
    __device__ __forceinline__ void add(float2 x) { v = pair_add2(v, x); }
    __device__ __forceinline__ void add(DSum o) { v = pair_add2(v, o.v); }
    __device__ __forceinline__ void sub(DSum o) {
        float2 m;
        m.x = -o.v.x;
        m.y = -o.v.y;
        v = pair_add2(v, m);
    }
    __device__ __forceinline__ void shfl_add(int o) {
        float2 w;
        w.x = __shfl_down_sync(0xffffffffu, v.x, o);
        w.y = __shfl_down_sync(0xffffffffu, v.y, o);
        v = pair_add2(v, w);
    }
    __device__ __forceinline__ void shfl_xor_add(int o) {
        float2 w;
        w.x = __shfl_xor_sync(0xffffffffu, v.x, o);
        w.y = __shfl_xor_sync(0xffffffffu, v.y, o);
        v = pair_add2(v, w);
    }
    __device__ __forceinline__ Slot slot() const { return v; }
    __device__ __forceinline__ double value() const { return (double)v.x + (double)v.y; }
};

// Block sum in a fixed order (warp shuffles, then the warps in index order); the
// result is valid on thread 0 only.  sh: 32 slots of shared memory.
template <class R>
__device__ __forceinline__ DSum<R> block_sum0(DSum<R> v, typename DSum<R>::Slot* sh) {
    for (int o = 16; o > 0; o >>= 1) v.shfl_add(o);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sh[wid] = v.slot();
    __syncthreads();
    DSum<R> tot = DSum<R>::zero();
    if (threadIdx.x == 0)
        for (int q = 0; q < (int)((blockDim.x + 31) >> 5); ++q) tot.add(DSum<R>::of(sh[q]));
    return tot;
}

// Whether this warp is the last of n to arrive at the ticket, which it then clears.  The warp's
// barriers extend what lane 0's fences order to all its lanes (a shuffle alone orders no memory):
// what any lane wrote before is visible to the last warp, all of whose lanes may read it after.
__device__ __forceinline__ bool last_of(unsigned* ticket, int n, int lane) {
    unsigned last = 0;
    __syncwarp();
    if (lane == 0) {
        __threadfence();
        last = atomicAdd(ticket, 1u) == (unsigned)(n - 1);
        if (last) *ticket = 0u;
        __threadfence();
    }
    __syncwarp();
    return __shfl_sync(0xffffffffu, last, 0) != 0;
}

// load that bypasses L1 (data written by other blocks of the same launch)
__device__ __forceinline__ double ld_cg(const double* p) { return __ldcg(p); }
__device__ __forceinline__ float2 ld_cg(const float2* p) { return __ldcg(p); }

// ---- enthalpy storage ------------------------------------------------------------
// H_e is FP64 in the FP64 mode.  In mixed precision it is an FP32 pair (hi, lo),
// hi = fl32(H_e) and lo = fl32(H_e - hi): about 48 significant bits, read, inverted
// and updated on the FP32 pipes only (GB300's FP64 rate is a small fraction of its
// FP32 rate).  Both take 8 bytes per cell.
template <class R>
struct HeStore;
template <>
struct HeStore<double> {
    using T = double;
};
template <>
struct HeStore<float> {
    using T = float2;
};
__device__ __forceinline__ double he_value(double h) { return h; }
__device__ __forceinline__ double he_value(float2 h) { return (double)h.x + (double)h.y; }
template <class R>
__device__ __forceinline__ double he_get(const void* base, size_t k) {
    return he_value(static_cast<const typename HeStore<R>::T*>(base)[k]);
}
template <class R>
__device__ __forceinline__ void he_set(void* base, size_t k, double v) {
    if constexpr (sizeof(R) == 8) {
        static_cast<double*>(base)[k] = v;
    } else {
        float2 h;
        pair_from(v, h.x, h.y);
        static_cast<float2*>(base)[k] = h;
    }
}

// master potential of cell k in FP64, whichever precision stores it
template <class R>
__device__ __forceinline__ double phi_get(const DevCase* dc, size_t k) {
    if (sizeof(R) == 8) return dc->phi64[k];
    return (double)static_cast<const float*>(dc->phi)[k] + (double)dc->phi_lo[k];
}
template <class R>
__device__ __forceinline__ void phi_set(const DevCase* dc, size_t k, double v) {
    if (sizeof(R) == 8) {
        dc->phi64[k] = v;
    } else {
        float h, l;
        pair_from(v, h, l);
        static_cast<float*>(dc->phi)[k] = h;
        dc->phi_lo[k] = l;
    }
}

}  // namespace lbfs
