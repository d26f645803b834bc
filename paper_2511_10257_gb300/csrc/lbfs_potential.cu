// lbfs_potential.cu -- the magnetic scalar potential, div(mu_m grad phi) = 0 (Eq. 4),
// on the cell-centred five-point stencil with the arithmetic-mean face coefficient:
// the steady state of the paper's magnetic LBFS (Eqs. 12-18) at a half-cell streaming
// step.  Solved by residual refinement: the residual r = b - A phi is formed in FP64, or in
// FP32 pairs in mixed precision, against the master potential, the correction A e = r by one
// multigrid V-cycle in FP32, then phi += e.  The residual alone decides when the potential is
// converged, so the precision of the correction enters only through the number of cycles
// (the contraction of 0.10-0.16 a cycle is far above FP32 rounding); in the FP64 mode the
// residual is scaled by a power of two on its way into the correction, so that FP32's range
// does not matter either.
//
// Operator (per level, homogeneous walls for the correction):
//   (A x)_c = sum_nb mu_f (x_c - x_nb) + sum_Dirichlet-walls 2 mu_c x_c,
//   mu_f = (mu_c + mu_nb)/2, b_c = sum_Dirichlet-walls 2 mu_c phi_wall.
// Coarse levels: 2 x 2 agglomeration with the cell count rounded up, mu averaged over
// the children, residual summed (the 2-D finite-volume operator is scale free),
// bilinear cell-centred prolongation, red-black Gauss-Seidel smoothing, conjugate
// gradients on the coarsest level.  On a level of odd size the last column (row)
// agglomerates a single child and is narrower than the others; its face coefficients
// carry the true face length over centre distance, and the prolongation interpolates
// between the true centres, so every grid size keeps the contraction of the even
// ones.
#include <algorithm>
#include <type_traits>

#include "lbfs_kernels.h"

namespace lbfs {

namespace {

constexpr int kNT = 256;                 // threads of the fine-level cell kernels
constexpr int kRowsPT = kMgTY / (kNT / kMgTX);  // rows of a 32 x 32 tile per thread (4)
static_assert(kRowsPT * (kNT / kMgTX) == kMgTY, "a fine-level tile splits evenly over the threads");

__device__ __forceinline__ bool pot_done(const DevCase* dc) {
    return dc->stats[ST_POT_DONE] >= 1.0;
}

// Neighbour of (i, j) across side w (0 -x, 1 +x, 2 -y, 3 +y) on an nx x ny level.
// Returns 1 if it is a cell (wrapping periodic axes), 0 if the side is a wall.
__device__ __forceinline__ int neighbour(const CaseParams& P, int nx, int ny, int i, int j, int w,
                                         int& ii, int& jj) {
    ii = i + (w == 0 ? -1 : w == 1 ? 1 : 0);
    jj = j + (w == 2 ? -1 : w == 3 ? 1 : 0);
    if (ii < 0 || ii >= nx) {
        if (!P.periodic_x) return 0;
        ii = ii < 0 ? ii + nx : ii - nx;
    }
    if (jj < 0 || jj >= ny) {
        if (!P.periodic_y) return 0;
        jj = jj < 0 ? jj + ny : jj - ny;
    }
    return 1;
}

// ---- geometry of a level whose last column or row may be narrower -------------
template <class M>
__device__ __forceinline__ M cell_wx(const MGLevel& lv, int i) {
    return i == lv.nx - 1 ? M(lv.wlx) : M(1);
}
template <class M>
__device__ __forceinline__ M cell_wy(const MGLevel& lv, int j) {
    return j == lv.ny - 1 ? M(lv.wly) : M(1);
}
// Face length over centre distance, in the level's cell units, for the face of cell
// (i, j) on side w (0 -x, 1 +x, 2 -y, 3 +y): to the neighbour cell, or to the wall half
// the cell's width away.  1 and 2 for regular cells.
template <class M>
__device__ __forceinline__ M face_factor(const MGLevel& lv, int i, int j, int w, bool wall) {
    const M wx = cell_wx<M>(lv, i), wy = cell_wy<M>(lv, j);
    if (w < 2) {
        const M d = wall ? M(0.5) * wx : M(0.5) * (wx + cell_wx<M>(lv, w == 0 ? i - 1 : i + 1));
        return wy / d;
    }
    const M d = wall ? M(0.5) * wy : M(0.5) * (wy + cell_wy<M>(lv, w == 2 ? j - 1 : j + 1));
    return wx / d;
}

// Prolongation along one axis: the fine cell i of a level with nf cells (last width
// wlf) takes 1 - w of its parent I = floor(i/2) on the coarse level (nc cells, last
// width wlc) and w of the coarse neighbour I + d, d in {-1, 0, 1}, by linear
// interpolation between the true centres (in fine-cell units).  Across a wall the
// neighbour is the parent's mirror image about the wall.  Regular cells give w = 1/4.
template <class M>
__device__ __forceinline__ void prolong_axis(int i, int nf, float wlf, int nc, float wlc, int& d, M& w) {
    const M xf = M(i) + (i == nf - 1 ? M(0.5f * wlf) : M(0.5));
    const int I = (i >= 0 ? i : i - 1) / 2;
    const M xp = M(2 * I) + (I == nc - 1 ? M(wlc) : M(1));
    if (xf == xp) {
        d = 0;
        w = M(0);
        return;
    }
    d = xf > xp ? 1 : -1;
    const int N = I + d;
    M xn;
    if (N < 0) xn = -xp;
    else if (N >= nc) xn = M(4 * (nc - 1)) + M(4) * M(wlc) - xp;
    else xn = M(2 * N) + (N == nc - 1 ? M(wlc) : M(1));
    w = (xf - xp) / (xn - xp);
}

template <class T>
__device__ __forceinline__ T block_sum(T v, T* sh) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    __syncthreads();
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    T tot = 0;
    const int nw = (blockDim.x + 31) >> 5;
    for (int q = 0; q < nw; ++q) tot += sh[q];
    return tot;
}

// (A x)_c with the level's coefficient and geometry, homogeneous Dirichlet walls
template <class M>
__device__ __forceinline__ M apply_A(const CaseParams& P, const MGLevel& lv, const M* mu, const M* x, int nx,
                                     int ny, int pitch, int i, int j) {
    const M mc = mu[(size_t)j * pitch + i];
    const M xc = x[(size_t)j * pitch + i];
    M acc = 0;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        int ii, jj;
        if (neighbour(P, nx, ny, i, j, w, ii, jj)) {
            const size_t kn = (size_t)jj * pitch + ii;
            if (lv.ragged) acc += face_factor<M>(lv, i, j, w, false) * M(0.5) * (mc + mu[kn]) * (xc - x[kn]);
            else acc += M(0.5) * (mc + mu[kn]) * (xc - x[kn]);
        } else if (P.mag_dir[w]) {
            acc += (lv.ragged ? face_factor<M>(lv, i, j, w, true) : M(2)) * mc * xc;
        }
    }
    return acc;
}

// ---- residual and check ------------------------------------------------------------
// r = b - A phi written with face terms: T = mu_f (phi_c - phi_nb) on the lower/left face of
// a cell serves the cell on either side, and a Dirichlet wall is a face to the wall value with
// coefficient 2 mu_c (an insulating wall one with coefficient 0), so
//   r_c = T(right) - T(left) + T(top) - T(bottom).
// FP64 mode: in FP64.  Mixed mode: the master potential is the FP32 pair phi + phi_lo, and the
// differences, products and sums are error-free pair operations on the FP32 pipes (about
// 2^-48 relative; GB300's FP64 issue is scarce), both faces of a cell as the two lanes of the
// packed instructions.

// a pair of values per axis: (h, l) each for the left face (x) and the lower face (y)
__device__ __forceinline__ void two_sum2(float2 a, float2 b, float2& s, float2& e) {
    const float2 m1 = make_float2(-1.f, -1.f);
    s = __fadd2_rn(a, b);
    const float2 bb = __ffma2_rn(a, m1, s);
    e = __fadd2_rn(__ffma2_rn(__ffma2_rn(bb, m1, s), m1, a), __ffma2_rn(bb, m1, b));
}

template <class M>
struct FaceTerm;
template <>
struct FaceTerm<double> {
    double x, y;   // T of the left and of the lower face
};
template <>
struct FaceTerm<float> {
    float2 h, l;   // T = h + l; lane x the left face, lane y the lower face
};

template <class M>
struct PotCell;   // one cell's master potential and coefficient
template <>
struct PotCell<double> {
    double v, mu;
};
template <>
struct PotCell<float> {
    float v, lo, mu;
};

// Far field -H0 (x cos a + y sin a) at a wall face.  ix, iy: the face's whole coordinates;
// half: the half cell of its centre belongs to x (0) or y (1).  In mixed precision an FP32
// pair, formed without FP64 instructions while the coordinates are exact in FP32.
__device__ __forceinline__ double far_field(const DevCase* dc, int ix, int iy, int half) {
    const CaseParams& P = dc->P;
    return -P.H0 * ((ix + (half == 0 ? 0.5 : 0.0)) * P.cos_t + (iy + (half == 1 ? 0.5 : 0.0)) * P.sin_t);
}
__device__ __forceinline__ float2 far_pair(const DevCase* dc, int ix, int iy, int half) {
    float2 r;
    if (max(dc->P.nx, dc->P.ny) < (1 << 22)) {
        const float wx = (float)ix + (half == 0 ? 0.5f : 0.0f), wy = (float)iy + (half == 1 ? 0.5f : 0.0f);
        float p, e, q, f, s, t;
        two_prod(dc->far_h[0], wx, p, e);
        two_prod(dc->far_h[1], wy, q, f);
        e = __fmaf_rn(dc->far_l[0], wx, e);
        f = __fmaf_rn(dc->far_l[1], wy, f);
        two_sum(p, q, s, t);
        t = __fadd_rn(t, __fadd_rn(e, f));
        r.x = __fadd_rn(s, t);
        r.y = __fsub_rn(t, __fsub_rn(r.x, s));
    } else {
        pair_from(far_field(dc, ix, iy, half), r.x, r.y);
    }
    return r;
}

// A case's cells as the residual sees them: wall ghosts hold the wall value and the inner
// cell's coefficient.
template <class M>
__device__ __forceinline__ PotCell<M> pot_cell(const DevCase* dc, unsigned k) {
    PotCell<M> c;
    if constexpr (sizeof(M) == 8) {
        c.v = dc->phi64[k];
    } else {
        c.v = static_cast<const float*>(dc->phi)[k];
        c.lo = dc->phi_lo[k];
    }
    c.mu = static_cast<const M*>(dc->lev[0].mu)[k];
    return c;
}
template <class M>
__device__ __forceinline__ void set_wall(PotCell<M>& c, const DevCase* dc, int ix, int iy, int half) {
    if constexpr (sizeof(M) == 8) {
        c.v = far_field(dc, ix, iy, half);
    } else {
        const float2 w = far_pair(dc, ix, iy, half);
        c.v = w.x;
        c.lo = w.y;
    }
}

// The face terms of a cell from its left and lower neighbours; fx, fy: 1/2 for a face between
// cells, 1 for a face to a Dirichlet wall (mu is the inner cell's on both sides), 0 for one to
// an insulating wall.
__device__ __forceinline__ FaceTerm<double> face_terms(const PotCell<double>& c, const PotCell<double>& l,
                                                       const PotCell<double>& b, double fx, double fy) {
    FaceTerm<double> t;
    t.x = fx * (c.mu + l.mu) * (c.v - l.v);
    t.y = fy * (c.mu + b.mu) * (c.v - b.v);
    return t;
}
__device__ __forceinline__ FaceTerm<float> face_terms(const PotCell<float>& c, const PotCell<float>& l,
                                                      const PotCell<float>& b, float fx, float fy) {
    const float2 m1 = make_float2(-1.f, -1.f);
    const float2 k = __fmul2_rn(make_float2(fx, fy), __fadd2_rn(make_float2(c.mu, c.mu), make_float2(l.mu, b.mu)));
    float2 d, e;
    two_sum2(make_float2(c.v, c.v), __fmul2_rn(make_float2(l.v, b.v), m1), d, e);
    e = __fadd2_rn(e, __ffma2_rn(make_float2(l.lo, b.lo), m1, make_float2(c.lo, c.lo)));
    FaceTerm<float> t;
    t.h = __fmul2_rn(k, d);
    t.l = __ffma2_rn(k, e, __ffma2_rn(k, d, __fmul2_rn(t.h, m1)));
    return t;
}
__device__ __forceinline__ double shfl_right(double v) { return __shfl_down_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ float shfl_right(float v) { return __shfl_down_sync(0xffffffffu, v, 1); }

constexpr int kQuadraticFrom = 6;   // steps behind the potential from which three points are extrapolated

// The relative residual of a case is known: converged, failed, or one cycle more.  A case that
// has not converged gets another cycle unless it has had kmax, in which case it is marked as
// failed and left alone.  first: the step's first check (resets the cycle count).
__device__ __forceinline__ void decide(const DevCase* dc, const PotCheck& ck, double rr, double bb, bool scaled) {
    double* st = dc->stats;
    const double rel = bb > 0.0 ? sqrt(rr / bb) : sqrt(rr);
    st[ST_POT_RESID] = rel;
    if (ck.first) {
        st[ST_POT_CYCLES] = 0.0;
        st[ST_EXTRAP] = fmin(st[ST_EXTRAP] + 1.0, (double)kQuadraticFrom);   // steps behind phi_prev (FP64)
        ck.sync[0] = ck.sync[1] = 0u;   // the grid barrier of the cycles that may follow
    }
    if (rel <= ck.tol) {
        st[ST_POT_DONE] = 1.0;
    } else if (st[ST_POT_CYCLES] >= (double)ck.kmax) {
        st[ST_POT_FAIL] = 1.0;
        st[ST_POT_DONE] = 1.0;   // no further kernel of this step touches the case
    } else {
        st[ST_POT_DONE] = 0.0;
        st[ST_POT_CYCLES] += 1.0;
        if (scaled) {   // the power of two that brings the root-mean-square residual to about 1
            int ex = 0;
            const double rms = sqrt(rr / ((double)dc->P.nx * dc->P.ny));
            if (rms > 0.0 && isfinite(rms)) frexp(rms, &ex);
            st[ST_SCALE] = ldexp(1.0, ex < -1000 ? 1000 : -ex);
        }
        if (ck.not_done) atomicAdd(ck.not_done, 1);
    }
}

// One warp per strip of kResidW columns and `rows` rows, one lane per column and one halo
// column on each side, marching up in y with the next row's loads in flight; a strip's norms go
// to its slot, and the warp that finishes last (an atomic ticket per group of strips and one per
// case, no waiting) sums them in a fixed order and decides.  Bound by latency on every grid: a full
// pass on 4096 x 2048 in mixed precision takes 88-91 us at 16 % of the DRAM rate and 45 % of the
// issue slots, where its 16 B a cell (24 in FP64) take 20 us.  72 registers leave 28 warps an SM,
// 4256 places for the 4384 strips of 64 rows, and a warp has two rows in flight.
constexpr int kResidW = kResidStripW;

template <class M>
__device__ __forceinline__ void residual_strip(const DevCase* __restrict__ dc, const TileRef tr, int rows,
                                               const PotCheck& ck, int lane) {
    using Slot = typename DSum<M>::Slot;
    if (!ck.first && pot_done(dc)) return;
    const CaseParams& P = dc->P;
    const int nx = P.nx, ny = P.ny;
    const unsigned pitch = (unsigned)P.pitch;
    const bool per_x = P.periodic_x != 0, per_y = P.periodic_y != 0;
    const int gx = tr.x0 - 1 + lane, y0 = tr.y0, y1 = min(y0 + rows, ny);
    int sx = gx;
    if (per_x) sx = gx < 0 ? gx + nx : (gx >= nx ? gx - nx : gx);
    sx = min(max(sx, 0), nx - 1);
    const bool wall_lo = !per_x && gx == -1, wall_hi = !per_x && gx == nx;
    // factor of the left face: between cells, to the left wall (cell 0) or to the right wall (ghost nx)
    M fx = M(0.5);
    if (!per_x && gx == 0) fx = P.mag_dir[0] ? M(1) : M(0);
    if (wall_hi) fx = P.mag_dir[1] ? M(1) : M(0);
    const bool active = lane >= 1 && lane <= kResidW && gx < nx;
    auto load_row = [&](int j) {
        int sy = j;
        if (per_y) sy = j < 0 ? j + ny : (j >= ny ? j - ny : j);
        sy = min(max(sy, 0), ny - 1);
        return pot_cell<M>(dc, (unsigned)sy * pitch + (unsigned)sx);
    };
    auto ghosts = [&](PotCell<M>& c, int j) {
        if (wall_lo || wall_hi) set_wall<M>(c, dc, wall_lo ? 0 : nx, j, 1);
        if (!per_y && (j == -1 || j == ny)) set_wall<M>(c, dc, sx, j == -1 ? 0 : ny, 0);
    };
    M* r_out = static_cast<M*>(dc->lev[0].r);
    DSum<M> r2 = DSum<M>::zero(), b2 = DSum<M>::zero();
    const auto march = [&](auto edge_tag) {
    constexpr bool EDGE = decltype(edge_tag)::value;   // a wall or a periodic wrap lies in the strip
    PotCell<M> below = load_row(y0 - 1), c0 = load_row(y0), c1 = load_row(y0 + 1);   // two rows in flight
    if (EDGE) ghosts(below, y0 - 1);
    FaceTerm<M> prev{};      // of row j-1
    M rx_h = 0, rx_l = 0;    // T of the right face of row j-1 (FP64: rx_h)
    for (int j = y0; j <= y1; ++j) {
        PotCell<M> c = c0;
        c0 = c1;
        if (j + 2 <= y1) c1 = load_row(j + 2);
        if (EDGE) ghosts(c, j);
        PotCell<M> l;
        l.v = __shfl_up_sync(0xffffffffu, c.v, 1);
        l.mu = __shfl_up_sync(0xffffffffu, c.mu, 1);
        if constexpr (sizeof(M) == 4) l.lo = __shfl_up_sync(0xffffffffu, c.lo, 1);
        M fy = M(0.5);
        if (EDGE && !per_y && j == 0) fy = P.mag_dir[2] ? M(1) : M(0);
        if (EDGE && !per_y && j == ny) fy = P.mag_dir[3] ? M(1) : M(0);
        const FaceTerm<M> t = face_terms(c, l, below, EDGE ? fx : M(0.5), fy);
        if (active && j > y0) {   // row j-1: r = (T(right) - T(left)) + (T(top) - T(bottom))
            M r;
            if constexpr (sizeof(M) == 8) {
                r = (rx_h - prev.x) + (t.y - prev.y);
            } else {
                const float2 m1 = make_float2(-1.f, -1.f);
                float2 s, e;
                two_sum2(make_float2(rx_h, t.h.y), __fmul2_rn(prev.h, m1), s, e);
                e = __fadd2_rn(e, __ffma2_rn(prev.l, m1, make_float2(rx_l, t.l.y)));
                float h, q;
                two_sum(s.x, s.y, h, q);
                r = __fadd_rn(h, __fadd_rn(q, __fadd_rn(e.x, e.y)));
            }
            r_out[(unsigned)(j - 1) * pitch + (unsigned)gx] = r;
            r2.add(r * r);
            // |b|^2 of the step, at cells next to a Dirichlet wall
            const int jj = j - 1;
            if (EDGE && ck.first && (gx == 0 || gx == nx - 1 || jj == 0 || jj == ny - 1)) {
                const bool on[4] = {!per_x && gx == 0 && P.mag_dir[0], !per_x && gx == nx - 1 && P.mag_dir[1],
                                    !per_y && jj == 0 && P.mag_dir[2], !per_y && jj == ny - 1 && P.mag_dir[3]};
                DSum<M> b = DSum<M>::zero();
#pragma unroll
                for (int w = 0; w < 4; ++w)
                    if (on[w]) {
                        const int ix = w == 1 ? nx : (w == 0 ? 0 : gx), iy = w == 3 ? ny : (w == 2 ? 0 : jj);
                        if constexpr (sizeof(M) == 8) b.add(far_field(dc, ix, iy, w < 2));
                        else b.add(far_pair(dc, ix, iy, w < 2));
                    }
                const M m2 = M(2) * below.mu;   // `below` is row j-1, this cell
                if constexpr (sizeof(M) == 8) {
                    const double v = m2 * b.v;
                    b2.add(v * v);
                } else {
                    float h, l, q, ql;
                    two_prod(m2, b.v.x, h, l);
                    l = __fmaf_rn(m2, b.v.y, l);
                    two_prod(h, h, q, ql);
                    b2.add(make_float2(q, __fmaf_rn(2.f * h, l, ql)));
                }
            }
        }
        prev = t;
        if constexpr (sizeof(M) == 8) {
            rx_h = shfl_right(t.x);
        } else {
            rx_h = shfl_right(t.h.x);
            rx_l = shfl_right(t.l.x);
        }
        below = c;
    }
    };
    if (tr.x0 >= 1 && tr.x0 + kResidW < nx && y0 >= 1 && y1 < ny) march(std::false_type{});
    else march(std::true_type{});
    for (int o = 16; o > 0; o >>= 1) {
        r2.shfl_add(o);
        b2.shfl_add(o);
    }
    Slot* red = static_cast<Slot*>(dc->mg_red);
    Slot* groups = static_cast<Slot*>(dc->mg_groups);
    if (lane == 0) {
        red[2 * (size_t)tr.slot] = r2.slot();
        red[2 * (size_t)tr.slot + 1] = b2.slot();
    }
    const int strips = dc->mg_strips;
    const int size = strips <= 1024 ? 1024 : kStageGroup;
    const int g = tr.slot / size, ng = (strips + size - 1) / size, n = min(size, strips - g * size);
    auto sum2 = [&](const Slot* s, int m, DSum<M>& a, DSum<M>& b) {
        a = b = DSum<M>::zero();
        for (int t = lane; t < m; t += 32) {
            a.add(DSum<M>::of(ld_cg(&s[2 * (size_t)t])));
            b.add(DSum<M>::of(ld_cg(&s[2 * (size_t)t + 1])));
        }
        for (int o = 16; o > 0; o >>= 1) {
            a.shfl_add(o);
            b.shfl_add(o);
        }
    };
    if (!last_of(&dc->mg_tickets[1 + g], n, lane)) return;
    sum2(red + 2 * (size_t)g * size, n, r2, b2);
    if (ng > 1) {
        if (lane == 0) {
            groups[2 * (size_t)g] = r2.slot();
            groups[2 * (size_t)g + 1] = b2.slot();
        }
        if (!last_of(&dc->mg_tickets[0], ng, lane)) return;
        sum2(groups, ng, r2, b2);
    }
    if (lane != 0) return;
    if (ck.first) dc->stats[ST_B2] = b2.value();
    decide(dc, ck, r2.value(), ck.first ? b2.value() : dc->stats[ST_B2], sizeof(M) == 8);
}

template <class M>
__global__ void __launch_bounds__(32) k_residual(const DevCase* __restrict__ cases, const TileRef* __restrict__ tiles,
                                                 int rows, const PotCheck ck) {
    const TileRef tr = tiles[blockIdx.x];
    residual_strip<M>(cases + tr.case_id, tr, rows, ck, threadIdx.x);
}

// A case's walls as one word held in a register: bits 0-3 Dirichlet walls, 4 and 5 periodic axes.
__device__ __forceinline__ int wall_mask(const CaseParams& P) {
    return (P.mag_dir[0] ? 1 : 0) | (P.mag_dir[1] ? 2 : 0) | (P.mag_dir[2] ? 4 : 0) | (P.mag_dir[3] ? 8 : 0) |
           (P.periodic_x ? 16 : 0) | (P.periodic_y ? 32 : 0);
}

// coarse value at (I, J), possibly one cell outside: periodic wrap, Dirichlet wall
// (homogeneous) mirrors with a sign change, an insulating wall mirrors evenly
template <class M>
__device__ __forceinline__ M coarse_at(int walls, const M* e, int nx, int ny, int pitch, int I, int J) {
    M sgn = M(1);
    if (I < 0 || I >= nx) {
        if (walls & 16) {
            I = I < 0 ? I + nx : I - nx;
        } else {
            const int w = I < 0 ? 0 : 1;
            I = I < 0 ? 0 : nx - 1;
            if (walls >> w & 1) sgn = -sgn;
        }
    }
    if (J < 0 || J >= ny) {
        if (walls & 32) {
            J = J < 0 ? J + ny : J - ny;
        } else {
            const int w = J < 0 ? 2 : 3;
            J = J < 0 ? 0 : ny - 1;
            if (walls >> w & 1) sgn = -sgn;
        }
    }
    return sgn * e[(unsigned)J * (unsigned)pitch + (unsigned)I];
}

// scale of the fine level's residual on its way into the FP32 correction (FP64 mode)
template <class S>
__device__ __forceinline__ S pot_scale(const DevCase* dc) {
    if constexpr (sizeof(S) == 8) return dc->stats[ST_SCALE];
    else return 1.0f;
}
// phi += e: in FP64, or as a renormalised FP32 pair
template <class M0>
__device__ __forceinline__ void add_correction(const DevCase* dc, unsigned k, float e) {
    if constexpr (sizeof(M0) == 8) {
        dc->phi64[k] += (double)e / dc->stats[ST_SCALE];   // (a power of two)
    } else {
        float* hi = static_cast<float*>(dc->phi);
        float h = hi[k], l = dc->phi_lo[k];
        pair_add(h, l, e, 0.f);
        hi[k] = h;
        dc->phi_lo[k] = l;
    }
}


// ---- fused V-cycle legs ------------------------------------------------------
// A block owns a TX x TY tile of one level (32 x 16, or 16 x 8 on levels with too few
// tiles to fill the GPU) and keeps it with a halo in shared memory.  Red-black Gauss-Seidel half-sweeps shrink the valid region by one cell
// each, so after kFNu full sweeps the tile (plus one cell) holds exactly the values the
// sweeps over the whole level would give.  Down leg: pre-smooth from e = 0, store e,
// restrict r - A e to the next level.  Up leg: add the bilinear prolongation of the
// coarse correction, post-smooth, store eu (neighbouring tiles still read e) or, on the fine level,
// add to phi.
constexpr int kFNu = 2;
constexpr int kHD = 2 * kFNu + 1, kHU = 2 * kFNu;

template <int TX, int TY, int H>
struct FRegion {
    static constexpr int W = TX + 2 * H, Hh = TY + 2 * H, N = W * Hh;
};

// global position of region cell k of a tile at (x0, y0) with halo H; returns 0 if it
// lies beyond a non-periodic wall, else 1 with (sx, sy) the (wrapped) source cell
__device__ __forceinline__ int region_source(const CaseParams& P, int nx, int ny, int x0, int y0, int H,
                                             int W, int k, int& gx, int& gy, int& sx, int& sy) {
    gx = x0 - H + k % W;
    gy = y0 - H + k / W;
    sx = gx;
    sy = gy;
    if (sx < 0 || sx >= nx) {
        if (!P.periodic_x) return 0;
        sx = ((sx % nx) + nx) % nx;
    }
    if (sy < 0 || sy >= ny) {
        if (!P.periodic_y) return 0;
        sy = ((sy % ny) + ny) % ny;
    }
    return 1;
}

// one red-black half-sweep of colour c over the region cells at least h from its edge.
// Threads take only the cells of colour c (every other cell of a row), and a
// neighbour is a cell exactly when its region entry lies inside the domain (in[]),
// which is how the level's walls and periodic wraps were resolved at load time.
// (A x) at region cell k of a tile at (x0, y0), split into its diagonal and the
// neighbour sum: A x = diag x_k - off.  Regular levels take the plain five-point
// coefficients; a ragged level the geometric factors of its narrower last cells.
template <class M, int TX, int TY, int H>
__device__ __forceinline__ void region_stencil(int dirichlet, const MGLevel& lv, int x0, int y0,
                                               const M* mu, const M* x, const unsigned char* in, int k,
                                               M& diag, M& off) {
    using G = FRegion<TX, TY, H>;
    const M mc = mu[k];
    diag = 0;
    off = 0;
    if (!lv.ragged) {
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const int kn = k + (w == 0 ? -1 : w == 1 ? 1 : w == 2 ? -G::W : G::W);
            if (in[kn]) {
                const M mf = M(0.5) * (mc + mu[kn]);
                diag += mf;
                off += mf * x[kn];
            } else if (dirichlet >> w & 1) {
                diag += M(2) * mc;
            }
        }
        return;
    }
    const int gx = x0 - H + k % G::W, gy = y0 - H + k / G::W;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        const int kn = k + (w == 0 ? -1 : w == 1 ? 1 : w == 2 ? -G::W : G::W);
        if (in[kn]) {
            const M mf = face_factor<M>(lv, gx, gy, w, false) * M(0.5) * (mc + mu[kn]);
            diag += mf;
            off += mf * x[kn];
        } else if (dirichlet >> w & 1) {
            diag += face_factor<M>(lv, gx, gy, w, true) * mc;
        }
    }
}

// (A x) at region cell k in difference form, sum_f g mu_f (x_k - x_nb) + walls
template <class M, int TX, int TY, int H>
__device__ __forceinline__ M region_apply(int dirichlet, const MGLevel& lv, int x0, int y0, const M* mu,
                                          const M* x, const unsigned char* in, int k) {
    using G = FRegion<TX, TY, H>;
    const M mc = mu[k], xc = x[k];
    M ax = 0;
    const int gx = x0 - H + k % G::W, gy = y0 - H + k / G::W;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        const int kn = k + (w == 0 ? -1 : w == 1 ? 1 : w == 2 ? -G::W : G::W);
        if (in[kn]) {
            if (lv.ragged) ax += face_factor<M>(lv, gx, gy, w, false) * M(0.5) * (mc + mu[kn]) * (xc - x[kn]);
            else ax += M(0.5) * (mc + mu[kn]) * (xc - x[kn]);
        } else if (dirichlet >> w & 1) {
            ax += (lv.ragged ? face_factor<M>(lv, gx, gy, w, true) : M(2)) * mc * xc;
        }
    }
    return ax;
}

template <class M, int TX, int TY, int H>
__device__ __forceinline__ void region_half_sweep(int dirichlet, const MGLevel& lv, int x0, int y0,
                                                  const M* mu, const M* r, M* e, const unsigned char* in, int c,
                                                  int h, int tid, int nt) {
    using G = FRegion<TX, TY, H>;
    const int VW = G::W - 2 * h, VH = G::Hh - 2 * h, HW = (VW + 1) / 2;
    const int base = (x0 - H) + (y0 - H);
    for (int t = tid; t < HW * VH; t += nt) {
        const int ly = h + t / HW;
        const int lx = h + ((c - base - ly - h) & 1) + 2 * (t % HW);
        if (lx >= G::W - h) continue;
        const int k = ly * G::W + lx;
        if (!in[k]) continue;
        M diag, off;
        region_stencil<M, TX, TY, H>(dirichlet, lv, x0, y0, mu, e, in, k, diag, off);
        e[k] = fdiv(r[k] + off, diag);
    }
}

template <class S, class M, int TX, int TY, int H>
__device__ __forceinline__ void region_load(const CaseParams& P, const MGLevel& lv, int x0, int y0, M* smu,
                                            M* sr, M* se, unsigned char* in, bool load_e, S scale, int tid,
                                            int nt) {
    using G = FRegion<TX, TY, H>;
    const S* mu = static_cast<const S*>(lv.mu);
    const S* r = static_cast<const S*>(lv.r);
    const M* e = static_cast<const M*>(lv.e);
    for (int k = tid; k < G::N; k += nt) {
        int gx, gy, sx, sy;
        const int ok = region_source(P, lv.nx, lv.ny, x0, y0, H, G::W, k, gx, gy, sx, sy);
        const unsigned g = (unsigned)sy * (unsigned)lv.pitch + (unsigned)sx;
        in[k] = (unsigned char)ok;
        smu[k] = ok ? M(mu[g]) : M(0);
        sr[k] = ok ? (sizeof(S) == 8 ? M(r[g] * scale) : M(r[g])) : M(0);
        se[k] = (ok && load_e) ? e[g] : M(0);
    }
}

// S: the type in which the level keeps mu and r (double on the fine level of the FP64 mode,
// whose residual enters scaled); everything else is FP32.
// The tile's nt threads (tid: this one) meet at sync(); mem: kLegBytes<TX, TY> bytes of shared memory.
template <int TX, int TY>
constexpr int kLegBytes = (13 * FRegion<TX, TY, kHD>::N + 15) / 16 * 16;

template <class S, int TX, int TY, class Sync>
__device__ __forceinline__ void vdown_tile(const DevCase* __restrict__ dc, const TileRef tr, int L, unsigned char* mem,
                                           int tid, int nt, Sync sync) {
    using M = float;
    using G = FRegion<TX, TY, kHD>;
    M *smu = reinterpret_cast<M*>(mem), *sr = smu + G::N, *se = sr + G::N;
    unsigned char* in = reinterpret_cast<unsigned char*>(se + G::N);
    if (pot_done(dc)) return;
    const CaseParams& P = dc->P;
    const int dirichlet = wall_mask(P);
    const MGLevel lv = dc->lev[L], cv = dc->lev[L + 1];
    region_load<S, M, TX, TY, kHD>(P, lv, tr.x0, tr.y0, smu, sr, se, in, false, pot_scale<S>(dc), tid, nt);
    sync();
    for (int h = 1; h <= 2 * kFNu; ++h) {
        region_half_sweep<M, TX, TY, kHD>(dirichlet, lv, tr.x0, tr.y0, smu, sr, se, in, (h - 1) & 1, h, tid, nt);
        sync();
    }
    // pre-smoothed correction of the tile
    M* e = static_cast<M*>(lv.e);
    for (int t = tid; t < TX * TY; t += nt) {
        const int gx = tr.x0 + t % TX, gy = tr.y0 + t / TX;
        if (gx < lv.nx && gy < lv.ny)
            e[(unsigned)gy * (unsigned)lv.pitch + (unsigned)gx] = se[(t / TX + kHD) * G::W + t % TX + kHD];
    }
    // restricted residual r - A e over the children of each coarse cell (four, or
    // fewer where the coarse cell is the narrower last one of its row or column), and
    // the coarse coefficient as the mean of the children's
    M* rc = static_cast<M*>(cv.r);
    M* muc = static_cast<M*>(cv.mu);
    for (int t = tid; t < (TX / 2) * (TY / 2); t += nt) {
        const int ci = t % (TX / 2), cj = t / (TX / 2);
        const int I = tr.x0 / 2 + ci, J = tr.y0 / 2 + cj;
        if (I >= cv.nx || J >= cv.ny) continue;
        M acc = 0;
        {
            const int k0 = (kHD + 2 * cj) * G::W + kHD + 2 * ci;
            if (in[k0 + 1] && in[k0 + G::W]) {
                muc[(unsigned)J * (unsigned)cv.pitch + (unsigned)I] =
                    M(0.25) * ((smu[k0] + smu[k0 + 1]) + (smu[k0 + G::W] + smu[k0 + G::W + 1]));
            } else {
                M m = smu[k0];
                int n = 1;
                if (in[k0 + 1]) { m += smu[k0 + 1]; ++n; }
                if (in[k0 + G::W]) { m += smu[k0 + G::W]; ++n; }
                muc[(unsigned)J * (unsigned)cv.pitch + (unsigned)I] = m / M(n);
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int lx = kHD + 2 * ci + (q & 1), ly = kHD + 2 * cj + (q >> 1);
            const int k = ly * G::W + lx;
            if (!in[k]) continue;
            acc += sr[k] - region_apply<M, TX, TY, kHD>(dirichlet, lv, tr.x0, tr.y0, smu, se, in, k);
        }
        rc[(unsigned)J * (unsigned)cv.pitch + (unsigned)I] = acc;
    }
}

// FINE: the fine level, where the smoothed correction goes straight into the master potential
// (M0: its precision) instead of back to e.
template <class S, class M0, bool FINE, int TX, int TY, class Sync>
__device__ __forceinline__ void vup_tile(const DevCase* __restrict__ dc, const TileRef tr, int L, unsigned char* mem,
                                         int tid, int nt, Sync sync) {
    using M = float;
    using G = FRegion<TX, TY, kHU>;
    constexpr int CW = (TX + 2 * kHU) / 2 + 3, CH = (TY + 2 * kHU) / 2 + 3;
    static_assert(13 * G::N + 4 * CW * CH <= kLegBytes<TX, TY>, "the up leg fits the down leg's memory");
    M *smu = reinterpret_cast<M*>(mem), *sr = smu + G::N, *se = sr + G::N, *sc = se + G::N;
    unsigned char* in = reinterpret_cast<unsigned char*>(sc + CW * CH);
    if (pot_done(dc)) return;
    const CaseParams& P = dc->P;
    const int dirichlet = wall_mask(P);
    const MGLevel lv = dc->lev[L], cv = dc->lev[L + 1];
    region_load<S, M, TX, TY, kHU>(P, lv, tr.x0, tr.y0, smu, sr, se, in, true, pot_scale<S>(dc), tid, nt);
    // coarse corrections around the region (one cell beyond its parents)
    const int cx0 = (tr.x0 - kHU) / 2 - 1 - ((tr.x0 - kHU) < 0 ? 1 : 0);
    const int cy0 = (tr.y0 - kHU) / 2 - 1 - ((tr.y0 - kHU) < 0 ? 1 : 0);
    const M* ec = static_cast<const M*>(cv.eu);
    for (int k = tid; k < CW * CH; k += nt) {
        int I = cx0 + k % CW, J = cy0 + k / CW;
        // periodic axes wrap; across a wall only the one-cell ghost is ever used by a
        // cell inside the domain, so the rest is clamped onto it
        if (P.periodic_x) I = ((I % cv.nx) + cv.nx) % cv.nx;
        else I = I < -1 ? -1 : (I > cv.nx ? cv.nx : I);
        if (P.periodic_y) J = ((J % cv.ny) + cv.ny) % cv.ny;
        else J = J < -1 ? -1 : (J > cv.ny ? cv.ny : J);
        sc[k] = coarse_at<M>(dirichlet, ec, cv.nx, cv.ny, cv.pitch, I, J);
    }
    sync();
    for (int k = tid; k < G::N; k += nt) {
        if (!in[k]) continue;
        const int gx = tr.x0 - kHU + k % G::W, gy = tr.y0 - kHU + k / G::W;
        // parent of the region cell in unwrapped level coordinates
        const int I = (gx >= 0 ? gx : gx - 1) / 2, J = (gy >= 0 ? gy : gy - 1) / 2;
        const int a = (J - cy0) * CW + (I - cx0);
        M v;
        if (!lv.ragged && !cv.ragged) {
            const int di = (gx & 1) ? 1 : -1, dj = (gy & 1) ? 1 : -1;
            v = M(9.0 / 16.0) * sc[a] + M(3.0 / 16.0) * sc[a + di] + M(3.0 / 16.0) * sc[a + dj * CW] +
                M(1.0 / 16.0) * sc[a + di + dj * CW];
        } else {
            int di, dj;
            M wx, wy;
            prolong_axis<M>(gx, lv.nx, lv.wlx, cv.nx, cv.wlx, di, wx);
            prolong_axis<M>(gy, lv.ny, lv.wly, cv.ny, cv.wly, dj, wy);
            v = ((M(1) - wx) * (M(1) - wy)) * sc[a] + (wx * (M(1) - wy)) * sc[a + di] +
                ((M(1) - wx) * wy) * sc[a + dj * CW] + (wx * wy) * sc[a + di + dj * CW];
        }
        se[k] += v;
    }
    sync();
    for (int h = 1; h <= 2 * kFNu; ++h) {
        region_half_sweep<M, TX, TY, kHU>(dirichlet, lv, tr.x0, tr.y0, smu, sr, se, in, (h - 1) & 1, h, tid, nt);
        sync();
    }
    M* e = static_cast<M*>(lv.eu);
    for (int t = tid; t < TX * TY; t += nt) {
        const int gx = tr.x0 + t % TX, gy = tr.y0 + t / TX;
        if (gx < lv.nx && gy < lv.ny) {
            const unsigned k = (unsigned)gy * (unsigned)lv.pitch + (unsigned)gx;
            const M v = se[(t / TX + kHU) * G::W + t % TX + kHU];
            if (FINE) add_correction<M0>(dc, k, v);
            else e[k] = v;
        }
    }
}

template <class S, int TX, int TY>
__global__ void __launch_bounds__(256) k_vdown(const DevCase* __restrict__ cases,
                                               const TileRef* __restrict__ tiles, int L) {
    __shared__ __align__(16) unsigned char mem[kLegBytes<TX, TY>];
    const TileRef tr = tiles[blockIdx.x];
    vdown_tile<S, TX, TY>(cases + tr.case_id, tr, L, mem, threadIdx.x, blockDim.x, [] { __syncthreads(); });
}

template <class S, class M0, bool FINE, int TX, int TY>
__global__ void __launch_bounds__(256) k_vup(const DevCase* __restrict__ cases,
                                             const TileRef* __restrict__ tiles, int L) {
    __shared__ __align__(16) unsigned char mem[kLegBytes<TX, TY>];
    const TileRef tr = tiles[blockIdx.x];
    vup_tile<S, M0, FINE, TX, TY>(cases + tr.case_id, tr, L, mem, threadIdx.x, blockDim.x, [] { __syncthreads(); });
}

constexpr int kTailNT = 1024;   // threads of the kernels that take a case's coarse levels, and of the cycles

// conjugate gradients on the coarsest level, one block per case, in shared memory
// (for coarsest levels too large for the tail kernel: a periodic axis that halves to an odd
// size early)
__device__ __forceinline__ void coarsest_case(const DevCase* __restrict__ dc, unsigned char* smem_raw, float* red) {
    using M = float;
    if (pot_done(dc)) return;
    const CaseParams& P = dc->P;
    const MGLevel lv = dc->lev[dc->nlev - 1];
    const int nx = lv.nx, ny = lv.ny, n = nx * ny;
    M* x = reinterpret_cast<M*>(smem_raw);
    M* r = x + n;
    M* p = r + n;
    M* Ap = p + n;
    M* mu = Ap + n;
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
        const int i = k % nx, j = k / nx;
        mu[k] = static_cast<const M*>(lv.mu)[(size_t)j * lv.pitch + i];
        r[k] = static_cast<const M*>(lv.r)[(size_t)j * lv.pitch + i];
        p[k] = r[k];
        x[k] = 0;
    }
    __syncthreads();
    M rr = 0;
    for (int k = threadIdx.x; k < n; k += blockDim.x) rr += r[k] * r[k];
    rr = block_sum(rr, red);
    const M rr0 = rr;
    // the coarse correction of a V-cycle needs only a few digits: 1e-3 relative (the cycle
    // contracts as with an exact coarse solve; the fine-level residual test alone decides
    // when the potential is converged)
    const M tol2 = M(1e-6);
    const int maxit = 4 * (nx + ny) + 100;
    for (int it = 0; it < maxit && rr > tol2 * rr0 && rr > M(0); ++it) {
        M pAp = 0;
        for (int k = threadIdx.x; k < n; k += blockDim.x) {
            const M a = apply_A<M>(P, lv, mu, p, nx, ny, nx, k % nx, k / nx);
            Ap[k] = a;
            pAp += p[k] * a;
        }
        pAp = block_sum(pAp, red);
        const M alpha = rr / pAp;
        M rn = 0;
        for (int k = threadIdx.x; k < n; k += blockDim.x) {
            x[k] += alpha * p[k];
            r[k] -= alpha * Ap[k];
            rn += r[k] * r[k];
        }
        rn = block_sum(rn, red);
        const M beta = rn / rr;
        rr = rn;
        for (int k = threadIdx.x; k < n; k += blockDim.x) p[k] = r[k] + beta * p[k];
        __syncthreads();
    }
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
        const int i = k % nx, j = k / nx;
        static_cast<M*>(lv.e)[(size_t)j * lv.pitch + i] = x[k];
    }
}

__global__ void __launch_bounds__(kTailNT) k_coarsest(const DevCase* __restrict__ cases, const int* __restrict__ ids) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ float red[32];
    coarsest_case(cases + ids[blockIdx.x], smem_raw, red);
}

// ---- the coarse levels in one kernel ---------------------------------------------------
// One block per case takes the V-cycle from level dc->tail (at most kTailCells cells) down to
// the coarsest level and back, all in shared memory: on small levels a kernel per leg is all
// launch latency.  Red-black Gauss-Seidel sweeps, restriction and prolongation are those of the
// fused legs.  What bounds it is the chain of some 80 dependent half-sweeps, so a half-sweep is
// kept short: cells 2t and 2t + 1 of a level, one of each colour, belong to thread t, which holds
// their coefficients, right-hand side and neighbours' places in registers for a whole leg; only
// the warps that own cells meet at the level's barrier, and levels of one warp need none.
// (With every sweep reading all of it from shared memory a solve took 46.8 us on 128 x 64, each launch
// profiled from cold caches; now 33.7.)
// The coarsest level is swept 2 kFNu times when it has at most kTinyCells cells and solved by
// conjugate gradients in one warp otherwise (grids whose one axis runs out first).  The part of at
// most kPassCells cells runs twice, so that it stands for an exact solve: with one pass the
// potential's error at the same residual is half as large again.  A case whose tail starts at
// level 0 adds the correction to its potential here.
constexpr int kTailPasses = 2, kTinyCells = 16;
static_assert(kTailCells <= 2 * kTailNT, "two cells a thread on the first level");

struct TailLevel {
    int nx, ny, off, ragged;   // off: of its cells in the arrays below
    int nt;                    // threads that own cells, in whole warps
};

template <class M>
__device__ __forceinline__ M warp_allsum(M v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// all cells of a level by the block's warps, row by row: f(i, j, k)
template <class F>
__device__ __forceinline__ void tail_cells(int nx, int ny, F f) {
    for (int j = threadIdx.x >> 5; j < ny; j += kTailNT >> 5)
        for (int i = threadIdx.x & 31; i < nx; i += 32) f(i, j, j * nx + i);
}

// places of a cell's left, right, lower and upper neighbour (the far end of the axis beyond a wall)
__device__ __forceinline__ void tail_neighbours(int nx, int ny, int i, int j, int k, int (&n)[4]) {
    n[0] = i > 0 ? k - 1 : k + nx - 1;
    n[1] = i < nx - 1 ? k + 1 : k - nx + 1;
    n[2] = j > 0 ? k - nx : k + (ny - 1) * nx;
    n[3] = j < ny - 1 ? k + nx : k - (ny - 1) * nx;
}

// A thread's two cells of a level, by colour: place (-1: none), row and column, neighbours, face
// coefficients (0 at a wall), inverse diagonal, Dirichlet-wall coefficient, right-hand side.
struct TailPair {
    int k[2], i[2], j[2], n[2][4];
    float c[2][4], d[2], w[2], r[2];
};

template <class M0>
__device__ __forceinline__ void tail_case(const DevCase* __restrict__ dc, int max_cells, int max_small,
                                          unsigned char* smem_raw, TailLevel* lv, MGLevel* geo) {
    if (pot_done(dc)) return;
    const CaseParams& P = dc->P;
    const int L0 = dc->tail, n_lev = dc->nlev - L0, t = threadIdx.x;
    // per level, cell by cell: mu, right-hand side, correction, coefficients of the right and
    // upper faces (0 at a wall) and of Dirichlet walls, inverse diagonal; the residual of one
    // level at a time; p and A p of the conjugate gradients
    float* mu = reinterpret_cast<float*>(smem_raw);
    float *r = mu + max_cells, *e = r + max_cells, *cx = e + max_cells, *cy = cx + max_cells, *wl = cy + max_cells;
    float *di = wl + max_cells, *res = di + max_cells, *p = res + max_cells, *Ap = p + max_small;
    if (t < n_lev) {
        int off = 0;
        for (int l = 0; l < t; ++l) off += dc->lev[L0 + l].nx * dc->lev[L0 + l].ny;
        const MGLevel g = dc->lev[L0 + t];
        geo[t] = g;
        lv[t] = TailLevel{g.nx, g.ny, off, g.ragged, max(32, ((g.nx * g.ny + 1) / 2 + 31) / 32 * 32)};
    }
    {
        const MGLevel& g = dc->lev[L0];
        if (sizeof(M0) == 8 && L0 == 0) {
            const double sc = dc->stats[ST_SCALE];
            tail_cells(g.nx, g.ny, [&](int i, int j, int k) {
                const size_t q = (size_t)j * g.pitch + i;
                mu[k] = (float)static_cast<const double*>(g.mu)[q];
                r[k] = (float)(static_cast<const double*>(g.r)[q] * sc);
            });
        } else {
            tail_cells(g.nx, g.ny, [&](int i, int j, int k) {
                const size_t q = (size_t)j * g.pitch + i;
                mu[k] = static_cast<const float*>(g.mu)[q];
                r[k] = static_cast<const float*>(g.r)[q];
            });
        }
    }
    const int walls = wall_mask(P), dirichlet = walls & 15;
    const bool per_x = (walls & 16) != 0, per_y = (walls & 32) != 0;
    __syncthreads();
    // mu of the coarser levels: the mean of the children
    for (int l = 0; l + 1 < n_lev; ++l) {
        const TailLevel v = lv[l], c = lv[l + 1];
        const float* m = mu + v.off;
        tail_cells(c.nx, c.ny, [&](int I, int J, int K) {
            const int i0 = 2 * I, j0 = 2 * J, i1 = i0 + 1 < v.nx, j1 = j0 + 1 < v.ny;
            const float* q = m + j0 * v.nx + i0;
            float s = q[0];
            if (i1) s += q[1];
            if (j1) s += i1 ? q[v.nx] + q[v.nx + 1] : q[v.nx];
            mu[c.off + K] = s * (i1 && j1 ? 0.25f : (i1 || j1 ? 0.5f : 1.f));
        });
        __syncthreads();
    }
    // coefficients of every level
    for (int l = 0; l < n_lev; ++l) {
        const TailLevel v = lv[l];
        const MGLevel& g = geo[l];
        const float* m = mu + v.off;
        tail_cells(v.nx, v.ny, [&](int i, int j, int k) {
            int n[4];
            tail_neighbours(v.nx, v.ny, i, j, k, n);
            const bool in[4] = {per_x || i > 0, per_x || i < v.nx - 1, per_y || j > 0, per_y || j < v.ny - 1};
            const float mc = m[k];
            float d = 0.f, wall = 0.f, c4[4];
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                c4[w] = 0.f;
                if (in[w]) {
                    c4[w] = 0.5f * (mc + m[n[w]]);
                    if (v.ragged) c4[w] *= face_factor<float>(g, i, j, w, false);
                    d += c4[w];
                } else if (dirichlet >> w & 1) {
                    wall += (v.ragged ? face_factor<float>(g, i, j, w, true) : 2.f) * mc;
                }
            }
            cx[v.off + k] = c4[1];
            cy[v.off + k] = c4[3];
            wl[v.off + k] = wall;
            di[v.off + k] = fdiv(1.f, d + wall);
        });
    }
    __syncthreads();
    auto meet = [&](int l) {   // the threads that own cells of level l
        if (lv[l].nt == 32) __syncwarp();
        else asm volatile("bar.sync %0, %1;" ::"r"(2 + l), "r"(lv[l].nt) : "memory");
    };
    TailPair q;
    auto load = [&](int l) {
        const TailLevel v = lv[l];
        const float *a = cx + v.off, *b = cy + v.off;
        const int n = v.nx * v.ny;
        // colour of cell 2t: (i + j) & 1, which is k & 1 on rows of odd length
        const int j0 = 2 * t / v.nx, c0 = v.nx & 1 ? 0 : j0 & 1;
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int k = 2 * t + (s ^ c0);
            q.k[s] = k < n ? k : -1;
            if (k >= n) continue;
            const int j = k / v.nx, i = k - j * v.nx;
            q.i[s] = i;
            q.j[s] = j;
            tail_neighbours(v.nx, v.ny, i, j, k, q.n[s]);
            q.c[s][0] = a[q.n[s][0]];
            q.c[s][1] = a[k];
            q.c[s][2] = b[q.n[s][2]];
            q.c[s][3] = b[k];
            q.d[s] = di[v.off + k];
            q.w[s] = wl[v.off + k];
            q.r[s] = r[v.off + k];
        }
    };
    auto relaxed = [&](int s, const float* x) {   // the sweep's new value of the cell of colour s
        return (q.r[s] + ((q.c[s][0] * x[q.n[s][0]] + q.c[s][1] * x[q.n[s][1]]) +
                          (q.c[s][2] * x[q.n[s][2]] + q.c[s][3] * x[q.n[s][3]]))) * q.d[s];
    };
    auto half = [&](int l, int s, float* x) {
        if (q.k[s] >= 0) x[q.k[s]] = relaxed(s, x);
        meet(l);
    };
    auto restrict_to = [&](int l, int k) {   // cell k of level l: the residual of its children on level l - 1
        const TailLevel v = lv[l - 1], c = lv[l];
        const int J = k / c.nx, I = k - J * c.nx, i1 = 2 * I + 1 < v.nx, j1 = 2 * J + 1 < v.ny;
        const float* y = res + 2 * J * v.nx + 2 * I;
        float s = y[0];
        if (i1) s += y[1];
        if (j1) s += i1 ? y[v.nx] + y[v.nx + 1] : y[v.nx];
        r[c.off + k] = s;
    };
    auto down = [&](int l, bool fresh) {
        load(l);
        float* x = e + lv[l].off;
        if (fresh) {   // from zero: the first colour's neighbours are zero
            if (q.k[0] >= 0) x[q.k[0]] = q.r[0] * q.d[0];
            if (q.k[1] >= 0) x[q.k[1]] = 0.f;   // (read with a zero coefficient across a wall)
            meet(l);
        } else {
            half(l, 0, x);
        }
        half(l, 1, x);
#pragma unroll
        for (int n = 1; n < kFNu; ++n) {
            half(l, 0, x);
            half(l, 1, x);
        }
#pragma unroll
        for (int s = 0; s < 2; ++s)   // r - A x in differences, so that smooth x keeps its digits
            if (q.k[s] >= 0) {
                const float xc = x[q.k[s]];
                res[q.k[s]] = q.r[s] - (((q.c[s][0] * (xc - x[q.n[s][0]]) + q.c[s][1] * (xc - x[q.n[s][1]])) +
                                         (q.c[s][2] * (xc - x[q.n[s][2]]) + q.c[s][3] * (xc - x[q.n[s][3]]))) + q.w[s] * xc);
            }
        meet(l);
        const TailLevel c = lv[l + 1];
        const int n = c.nx * c.ny;
        if (l + 1 < n_lev - 1) {   // each owner its own cells, which it loads next
            if (2 * t < n) restrict_to(l + 1, 2 * t);
            if (2 * t + 1 < n) restrict_to(l + 1, 2 * t + 1);
        } else if (t < 32) {
            for (int k = t; k < n; k += 32) restrict_to(l + 1, k);
        }
    };
    auto up = [&](int l) {
        meet(l);   // the coarser level is done
        load(l);
        const TailLevel v = lv[l], c = lv[l + 1];
        float* x = e + v.off;
        const float* xc = e + c.off;
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            if (q.k[s] < 0) continue;
            const int i = q.i[s], j = q.j[s], I = i >> 1, J = j >> 1;
            int di_ = (i & 1) ? 1 : -1, dj_ = (j & 1) ? 1 : -1;
            float wx = 0.25f, wy = 0.25f;
            if (v.ragged || c.ragged) {
                prolong_axis<float>(i, v.nx, geo[l].wlx, c.nx, geo[l + 1].wlx, di_, wx);
                prolong_axis<float>(j, v.ny, geo[l].wly, c.ny, geo[l + 1].wly, dj_, wy);
            }
            x[q.k[s]] += ((1.f - wx) * (1.f - wy)) * xc[J * c.nx + I] +
                         (wx * (1.f - wy)) * coarse_at<float>(walls, xc, c.nx, c.ny, c.nx, I + di_, J) +
                         ((1.f - wx) * wy) * coarse_at<float>(walls, xc, c.nx, c.ny, c.nx, I, J + dj_) +
                         (wx * wy) * coarse_at<float>(walls, xc, c.nx, c.ny, c.nx, I + di_, J + dj_);
        }
        meet(l);
#pragma unroll
        for (int n = 0; n < kFNu; ++n) {
            half(l, 0, x);
            half(l, 1, x);
        }
    };
    auto coarsest = [&] {   // one warp
        const int l = n_lev - 1;
        const TailLevel v = lv[l];
        const int n = v.nx * v.ny;
        float *x = e + v.off, *b = r + v.off;
        __syncwarp();
        for (int k = t; k < n; k += 32) x[k] = 0.f;
        __syncwarp();
        if (n <= kTinyCells) {
            load(l);
            for (int h = 0; h < 4 * kFNu; ++h) {
                const int s = h & 1;
                const float y = q.k[s] >= 0 ? relaxed(s, x) : 0.f;
                __syncwarp();   // (a periodic axis of odd length joins cells of one colour)
                if (q.k[s] >= 0) x[q.k[s]] = y;
                __syncwarp();
            }
            return;
        }
        // conjugate gradients
        const float *a = cx + v.off, *c = cy + v.off, *dg = di + v.off;
        float rr = 0.f;
        for (int k = t; k < n; k += 32) {
            p[k] = b[k];
            rr += b[k] * b[k];
        }
        rr = warp_allsum(rr);
        __syncwarp();
        const float rr0 = rr;
        const float tol2 = 1e-6f;   // a coarse correction needs only a few digits (as the block version)
        const int maxit = 4 * (v.nx + v.ny) + 100;
        for (int it = 0; it < maxit && rr > tol2 * rr0 && rr > 0.f; ++it) {
            float pAp = 0.f;
            for (int k = t; k < n; k += 32) {
                const int j = k / v.nx, i = k - j * v.nx;
                int m[4];
                tail_neighbours(v.nx, v.ny, i, j, k, m);
                const float y = fdiv(p[k], dg[k]) - ((a[m[0]] * p[m[0]] + a[k] * p[m[1]]) + (c[m[2]] * p[m[2]] + c[k] * p[m[3]]));
                Ap[k] = y;
                pAp += p[k] * y;
            }
            pAp = warp_allsum(pAp);
            const float alpha = rr / pAp;
            float rn = 0.f;
            for (int k = t; k < n; k += 32) {
                x[k] += alpha * p[k];
                const float rk = b[k] - alpha * Ap[k];
                b[k] = rk;
                rn += rk * rk;
            }
            rn = warp_allsum(rn);
            const float beta = rn / rr;
            rr = rn;
            __syncwarp();   // every lane's reads of p for A p are done
            for (int k = t; k < n; k += 32) p[k] = b[k] + beta * p[k];
            __syncwarp();
        }
    };
    // levels [0, mine) are the ones this thread owns cells of; from level `twice` the part that
    // runs twice
    int twice = 0, mine = 0;
    while (twice < n_lev - 1 && lv[twice].nx * lv[twice].ny > kPassCells) ++twice;
    while (mine < n_lev - 1 && t < lv[mine].nt) ++mine;
    const int top = min(twice, mine);
    for (int l = 0; l < top; ++l) down(l, true);
    if (twice < n_lev - 1 ? mine > twice : t < 32) {
        const int passes = twice < n_lev - 1 ? kTailPasses : 1;
        for (int pass = 0; pass < passes; ++pass) {
            for (int l = twice; l < mine; ++l) down(l, pass == 0 || l > twice);
            if (t < 32) coarsest();
            for (int l = mine - 1; l >= twice; --l) up(l);
        }
    }
    for (int l = top - 1; l >= 0; --l) up(l);
    __syncthreads();
    const MGLevel& g = geo[0];
    tail_cells(g.nx, g.ny, [&](int i, int j, int k) {
        const unsigned o = (unsigned)j * (unsigned)g.pitch + (unsigned)i;
        if (L0 == 0) add_correction<M0>(dc, o, e[k]);
        else static_cast<float*>(g.e)[o] = e[k];
    });
}

template <class M0>
__global__ void __launch_bounds__(kTailNT) k_tail(const DevCase* __restrict__ cases, const int* __restrict__ ids,
                                                  int max_cells, int max_small) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ TailLevel lv[kMaxLevels];
    __shared__ MGLevel geo[kMaxLevels];
    tail_case<M0>(cases + ids[blockIdx.x], max_cells, max_small, smem_raw, lv, geo);
}

// ---- refinement cycles until every case has converged, in one cooperative kernel --------
// The kernels above as phases of one grid, a block an SM, with a grid barrier between
// dependent phases: a leg's tile takes kLegNT threads, a coarse solve a block, a residual strip
// a warp.  When the check before it found every case converged the kernel returns at once.
// The phases run the same code on the same data as the kernels of their own: the potential is
// the same bit for bit.  Bound by latency: a cycle on 128 x 64 takes 57 us, against 46 as kernels of a
// recorded graph, for its grid barriers and for its spills (64 registers a thread at 1024 threads: 456 B
// of stores and 508 of loads in mixed precision, 640 and 1332 in FP64; the kernels of their own spill
// nothing), but a step that needs none pays 5 us where a conditional graph node took 16.
constexpr int kLegNT = 256, kLegGroups = kTailNT / kLegNT;

// All blocks of the grid arrive (sync[0] counts them; it starts a launch at zero and only
// grows).  The blocks of a cooperative launch run at the same time, so the wait ends; should it
// not within `limit` polls, sync[1] tells every block to give up.
__device__ __forceinline__ bool grid_sync(unsigned* sync, unsigned& target, int limit, int* ok) {
    target += gridDim.x;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(sync, 1u);
        int polls = 0;
        while (*static_cast<volatile unsigned*>(sync) < target && ++polls < limit &&
               *static_cast<volatile unsigned*>(sync + 1) == 0u) {
        }
        __threadfence();
        *ok = *static_cast<volatile unsigned*>(sync) >= target;
        if (!*ok) atomicExch(sync + 1, 1u);
    }
    __syncthreads();
    return *ok != 0;
}

template <class M0>
__global__ void __launch_bounds__(kTailNT, 1) k_cycles(const __grid_constant__ CycleArgs a, const PotCheck ck) {
    extern __shared__ __align__(16) unsigned char mem[];
    __shared__ TailLevel lv[kMaxLevels];
    __shared__ MGLevel geo[kMaxLevels];
    __shared__ float red[32];
    __shared__ int ok;
    const int nb = gridDim.x, b = blockIdx.x, cases_n = a.n_tail + a.n_coarsest;
    auto case_of = [&](int q) { return a.cases + (q < a.n_tail ? a.tail[q] : a.coarsest[q - a.n_tail]); };
    auto pending = [&] {   // does a case still need a cycle?
        int n = 0;
        for (int q = threadIdx.x; q < cases_n; q += kTailNT) n |= !pot_done(case_of(q));
        return __syncthreads_or(n) != 0;
    };
    if (!pending()) return;
    unsigned target = 0;
    const int group = threadIdx.x / kLegNT, tid = threadIdx.x % kLegNT;
    auto sync = [&] { asm volatile("bar.sync %0, %1;" ::"r"(2 + group), "n"(kLegNT) : "memory"); };
    unsigned char* const leg = mem + group * kLegBytes<kFusedTX, kFusedTY>;
    bool more;
    do {
        bool alive = true;
        for (int L = 0; L < a.depth && alive; ++L) {
            for (int t = group * nb + b; t < a.n_tiles[L]; t += kLegGroups * nb) {
                const TileRef tr = a.tiles[L][t];
                const DevCase* dc = a.cases + tr.case_id;
                const bool wide = sizeof(M0) == 8 && L == 0;
                if (a.small[L]) {
                    if (wide) vdown_tile<M0, kFusedSmallTX, kFusedSmallTY>(dc, tr, L, leg, tid, kLegNT, sync);
                    else vdown_tile<float, kFusedSmallTX, kFusedSmallTY>(dc, tr, L, leg, tid, kLegNT, sync);
                } else {
                    if (wide) vdown_tile<M0, kFusedTX, kFusedTY>(dc, tr, L, leg, tid, kLegNT, sync);
                    else vdown_tile<float, kFusedTX, kFusedTY>(dc, tr, L, leg, tid, kLegNT, sync);
                }
                sync();   // the tile's memory is free again
            }
            alive = grid_sync(ck.sync, target, ck.wait_polls, &ok);
        }
        for (int q = b; q < cases_n && alive; q += nb) {
            if (q < a.n_tail) tail_case<M0>(case_of(q), a.tail_cells, a.tail_small, mem, lv, geo);
            else coarsest_case(case_of(q), mem, red);
            __syncthreads();
        }
        alive = alive && grid_sync(ck.sync, target, ck.wait_polls, &ok);
        for (int L = a.depth - 1; L >= 0 && alive; --L) {
            for (int t = group * nb + b; t < a.n_tiles[L]; t += kLegGroups * nb) {
                const TileRef tr = a.tiles[L][t];
                const DevCase* dc = a.cases + tr.case_id;
                if (L > 0) {
                    if (a.small[L]) vup_tile<float, float, false, kFusedSmallTX, kFusedSmallTY>(dc, tr, L, leg, tid, kLegNT, sync);
                    else vup_tile<float, float, false, kFusedTX, kFusedTY>(dc, tr, L, leg, tid, kLegNT, sync);
                } else {
                    if (a.small[L]) vup_tile<M0, M0, true, kFusedSmallTX, kFusedSmallTY>(dc, tr, L, leg, tid, kLegNT, sync);
                    else vup_tile<M0, M0, true, kFusedTX, kFusedTY>(dc, tr, L, leg, tid, kLegNT, sync);
                }
                sync();
            }
            alive = grid_sync(ck.sync, target, ck.wait_polls, &ok);
        }
        if (alive) {
            for (int t = (threadIdx.x >> 5) * nb + b; t < a.n_strips; t += (kTailNT >> 5) * nb) {
                const TileRef tr = a.strips[t];
                residual_strip<M0>(a.cases + tr.case_id, tr, a.rows, ck, threadIdx.x & 31);
            }
            alive = grid_sync(ck.sync, target, ck.wait_polls, &ok);
        }
        if (!alive) {   // the host reports it and clears the tickets of a residual some blocks did not take
            if (threadIdx.x == 0) atomicExch(ck.sync + 2, 1u);
            return;
        }
        more = pending();
    } while (more);
}

// The FP64 warm start, extrapolated in time, cell by cell, from the potentials of the previous
// steps: linearly, 2 phi - phi_prev, once one is known, and through the last three points,
// 3 (phi - phi_prev) + phi_prev2, from the kQuadraticFrom-th step after a state was set (the first
// steps settle too fast for a second difference).  ST_EXTRAP counts the steps.  A start closer to the
// step's potential needs fewer refinement cycles to reach the FP64 tolerance; the converged
// potential is the same.  On 128 x 64 the start's error is 2.5e-7 of the potential linearly and
// 1.2e-8 with three points, 1.2e-8 and 2e-9 on 512 x 256: 4.4 cycles a step instead of 5.7, and 3.4
// instead of 5.0.  (The mixed path gains nothing from it:
// its potential moves only on steps that run a cycle.)
__global__ void __launch_bounds__(kNT) k_extrapolate(const DevCase* __restrict__ cases,
                                                     const TileRef* __restrict__ tiles) {
    const TileRef tr = tiles[blockIdx.x];
    const DevCase* dc = cases + tr.case_id;
    const MGLevel lv = dc->lev[0];
    const int i = tr.x0 + threadIdx.x % kMgTX;
    if (i >= lv.nx) return;
    const double steps = dc->stats[ST_EXTRAP];
    double *phi = dc->phi64, *prev = dc->phi_prev64, *prev2 = prev + (size_t)lv.pitch * lv.ny;
#pragma unroll
    for (int q = 0; q < kRowsPT; ++q) {
        const int j = tr.y0 + threadIdx.x / kMgTX + q * (kNT / kMgTX);
        if (j >= lv.ny) break;
        const size_t k = (size_t)j * lv.pitch + i;
        const double v = phi[k], v1 = prev[k];
        if (steps >= kQuadraticFrom) phi[k] = 3.0 * (v - v1) + prev2[k];
        else if (steps > 0.0) phi[k] = 2.0 * v - v1;
        prev2[k] = v1;
        prev[k] = v;
    }
}

// ---- the paper's own magnetic solver (Sec. 3.2, Eqs. 12-18) ----------------------
// Explicit pseudo-time relaxation of Eq. 17, phi <- phi - dtau div F, with the LBFS
// face flux of the magnetic distribution.  Per face (cell A below/left, B above/right,
// normal n): the equilibrium w_a phi (Eq. 13) at the points x_f - e_a dts, each
// reconstructed from its upwind cell with central gradients (Eq. 44); interface value
// Eq. 45; tau = 1/2 + mu_f/(c_s^2 dts) (Eq. 12 with the arithmetic-mean face mu); the
// starred distribution of Eq. 16.  Summed over the D2Q9 directions, the flux
//   F = sum_a e_a.n phi*_a = (tau - 1/2) sum_a e_a.n w_a phi(x_f - e_a dts)
// (the interface part carries sum_a e_a.n w_a = 0), and the three points on each side
// average their tangential slopes out, leaving
//   F = mu_f/(2 dts) [phi_A - phi_B + (1/2 - dts)(g_A + g_B)],  g = normal central slope,
// the compact -mu_f (phi_B - phi_A) at dts = 1/2.  Walls: a Dirichlet face carries the
// compact flux to the wall value half a cell away, an insulating face none; the ghost
// layer for the slopes is 2 phi_w - phi (Dirichlet) or phi (insulating).  FP64
// arithmetic in both precisions; out receives the new potential.
template <class M>
__device__ __forceinline__ double phi_cell(const DevCase* dc, const CaseParams& P, int nx, int ny, int i, int j) {
    // phi at (i, j), which may be one cell outside the grid (ghost rules above)
    int w = -1;
    if (i < 0 || i >= nx) {
        if (P.periodic_x) i = i < 0 ? i + nx : i - nx;
        else w = i < 0 ? 0 : 1;
    }
    if (j < 0 || j >= ny) {
        if (P.periodic_y) j = j < 0 ? j + ny : j - ny;
        else w = j < 0 ? 2 : 3;
    }
    if (w < 0) return phi_get<M>(dc, (size_t)j * P.pitch + i);
    const int ii = i < 0 ? 0 : (i >= nx ? nx - 1 : i), jj = j < 0 ? 0 : (j >= ny ? ny - 1 : j);
    const double pin = phi_get<M>(dc, (size_t)jj * P.pitch + ii);
    if (!P.mag_dir[w]) return pin;
    const double wx = w == 0 ? 0.0 : (w == 1 ? (double)nx : ii + 0.5);
    const double wy = w == 2 ? 0.0 : (w == 3 ? (double)ny : jj + 0.5);
    return 2.0 * (-P.H0 * (wx * P.cos_t + wy * P.sin_t)) - pin;
}

template <class M>
__global__ void k_pseudo_step(const DevCase* __restrict__ dc, double dtau, double* __restrict__ out) {
    const CaseParams& P = dc->P;
    const int nx = P.nx, ny = P.ny;
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
    if (i >= nx) return;
    const M* mu = static_cast<const M*>(dc->lev[0].mu);
    const int mp = dc->lev[0].pitch;
    const double dts = P.dts, c1 = 0.5 - dts;
    const double pc = phi_cell<M>(dc, P, nx, ny, i, j);
    const double mc = (double)mu[(size_t)j * mp + i];
    double div = 0.0;
    // faces 0 left, 1 right, 2 bottom, 3 top; F is the flux along +x / +y
    for (int f = 0; f < 4; ++f) {
        const bool xf = f < 2, hi = (f & 1) != 0;
        const int ni = i + (xf ? (hi ? 1 : -1) : 0), nj = j + (xf ? 0 : (hi ? 1 : -1));
        const bool wall = xf ? (!P.periodic_x && (ni < 0 || ni >= nx)) : (!P.periodic_y && (nj < 0 || nj >= ny));
        double F;
        if (wall) {
            if (!P.mag_dir[f]) continue;
            const double wx = f == 0 ? 0.0 : (f == 1 ? (double)nx : i + 0.5);
            const double wy = f == 2 ? 0.0 : (f == 3 ? (double)ny : j + 0.5);
            const double pw = -P.H0 * (wx * P.cos_t + wy * P.sin_t);
            // compact flux to the wall half a cell away, along +x / +y
            F = hi ? 2.0 * mc * (pc - pw) : -2.0 * mc * (pc - pw);
        } else {
            const int wi = ni < 0 ? ni + nx : (ni >= nx ? ni - nx : ni);
            const int wj = nj < 0 ? nj + ny : (nj >= ny ? nj - ny : nj);
            const double mn = (double)mu[(size_t)wj * mp + wi];
            const double muf = 0.5 * (mc + mn);
            // A is the lower/left cell of the face, B the upper/right one
            const int ai = hi ? i : ni, aj = hi ? j : nj, bi = hi ? ni : i, bj = hi ? nj : j;
            const int dx = xf ? 1 : 0, dy = xf ? 0 : 1;
            const double pA = hi ? pc : phi_cell<M>(dc, P, nx, ny, ai, aj);
            const double pB = hi ? phi_cell<M>(dc, P, nx, ny, bi, bj) : pc;
            double gsum = 0.0;
            if (c1 != 0.0) {
                const double gA = 0.5 * (phi_cell<M>(dc, P, nx, ny, ai + dx, aj + dy) -
                                         phi_cell<M>(dc, P, nx, ny, ai - dx, aj - dy));
                const double gB = 0.5 * (phi_cell<M>(dc, P, nx, ny, bi + dx, bj + dy) -
                                         phi_cell<M>(dc, P, nx, ny, bi - dx, bj - dy));
                gsum = gA + gB;
            }
            F = muf / (2.0 * dts) * ((pA - pB) + c1 * gsum);
        }
        div += hi ? F : -F;
    }
    out[(size_t)j * nx + i] = pc - dtau * div;
}

template <class M>
__global__ void k_pseudo_store(const DevCase* __restrict__ dc, const double* __restrict__ in) {
    const CaseParams& P = dc->P;
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
    if (i >= P.nx) return;
    phi_set<M>(dc, (size_t)j * P.pitch + i, in[(size_t)j * P.nx + i]);
}

}  // namespace

cudaError_t launch_pseudo_time(int prec, const DevCase* d, int nx, int ny, int iters, double dtau, double* tmp,
                               cudaStream_t st) {
    const dim3 grid((nx + 127) / 128, ny);
    for (int it = 0; it < iters; ++it) {
        if (prec == 0) {
            k_pseudo_step<double><<<grid, 128, 0, st>>>(d, dtau, tmp);
            k_pseudo_store<double><<<grid, 128, 0, st>>>(d, tmp);
        } else {
            k_pseudo_step<float><<<grid, 128, 0, st>>>(d, dtau, tmp);
            k_pseudo_store<float><<<grid, 128, 0, st>>>(d, tmp);
        }
    }
    return cudaGetLastError();
}

cudaError_t launch_mg_residual(int prec, const DevCase* cases, const TileRef* tiles, int n, int rows, const PotCheck& ck,
                               cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    if (prec == 0) k_residual<double><<<n, 32, 0, st>>>(cases, tiles, rows, ck);
    else k_residual<float><<<n, 32, 0, st>>>(cases, tiles, rows, ck);
    return cudaGetLastError();
}

template <int TX, int TY>
static void vdown(int wide, const DevCase* cases, const TileRef* tiles, int n, int L, cudaStream_t st) {
    constexpr int NT = TX * TY >= 512 ? 256 : 128;
    if (wide) k_vdown<double, TX, TY><<<n, NT, 0, st>>>(cases, tiles, L);
    else k_vdown<float, TX, TY><<<n, NT, 0, st>>>(cases, tiles, L);
}

cudaError_t launch_mg_vdown(int prec, const DevCase* cases, const TileRef* tiles, int n, int L, int small,
                            cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    const int wide = prec == 0 && L == 0;
    if (small) vdown<kFusedSmallTX, kFusedSmallTY>(wide, cases, tiles, n, L, st);
    else vdown<kFusedTX, kFusedTY>(wide, cases, tiles, n, L, st);
    return cudaGetLastError();
}

template <int TX, int TY>
static void vup(int prec, const DevCase* cases, const TileRef* tiles, int n, int L, cudaStream_t st) {
    constexpr int NT = TX * TY >= 512 ? 256 : 128;
    if (L > 0) k_vup<float, float, false, TX, TY><<<n, NT, 0, st>>>(cases, tiles, L);
    else if (prec == 0) k_vup<double, double, true, TX, TY><<<n, NT, 0, st>>>(cases, tiles, L);
    else k_vup<float, float, true, TX, TY><<<n, NT, 0, st>>>(cases, tiles, L);
}

cudaError_t launch_mg_vup(int prec, const DevCase* cases, const TileRef* tiles, int n, int L, int small,
                          cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    if (small) vup<kFusedSmallTX, kFusedSmallTY>(prec, cases, tiles, n, L, st);
    else vup<kFusedTX, kFusedTY>(prec, cases, tiles, n, L, st);
    return cudaGetLastError();
}

static constexpr size_t tail_bytes(int max_cells, int max_small) {
    return ((size_t)8 * max_cells + (size_t)2 * max_small) * sizeof(float);
}
static constexpr size_t coarsest_bytes(int max_cells) { return (size_t)5 * max_cells * sizeof(float); }

// The dynamic shared memory a kernel may ask for belongs to the kernel on its device, not to a
// context or a launch, and other threads' contexts launch the same kernels: it is set to what the
// largest cases need (a level has at most 9/25 of the cells above it, so a tail fewer than twice
// its first level's), always the same, and never by a step.
constexpr size_t kTailLimit = tail_bytes(2 * kTailCells, kTailCoarsest), kCoarsestLimit = coarsest_bytes(kCoarsestMax);
constexpr size_t kCyclesLimit =
    std::max({(size_t)kLegGroups * kLegBytes<kFusedTX, kFusedTY>, kTailLimit, kCoarsestLimit});
static_assert(kCyclesLimit <= 220 * 1024, "leaves the static shared memory its place in a block's 227 KB");

cudaError_t prepare_potential(int prec) {
    const auto limit = [](const void* kern, size_t bytes) {
        return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    };
    const void* tail = prec == 0 ? (const void*)k_tail<double> : (const void*)k_tail<float>;
    const void* cycles = prec == 0 ? (const void*)k_cycles<double> : (const void*)k_cycles<float>;
    cudaError_t e = limit(tail, kTailLimit);
    if (e == cudaSuccess) e = limit((const void*)k_coarsest, kCoarsestLimit);
    if (e == cudaSuccess) e = limit(cycles, kCyclesLimit);
    return e;
}

cudaError_t launch_mg_tail(int prec, const DevCase* cases, const int* ids, int ncases, int max_cells, int max_small,
                           cudaStream_t st) {
    if (ncases <= 0) return cudaSuccess;
    const size_t sm = tail_bytes(max_cells, max_small);
    auto kern = prec == 0 ? k_tail<double> : k_tail<float>;
    kern<<<ncases, kTailNT, sm, st>>>(cases, ids, max_cells, max_small);
    return cudaGetLastError();
}

cudaError_t launch_mg_coarsest(const DevCase* cases, const int* ids, int ncases, int max_cells, cudaStream_t st) {
    if (ncases <= 0) return cudaSuccess;
    k_coarsest<<<ncases, kTailNT, coarsest_bytes(max_cells), st>>>(cases, ids);
    return cudaGetLastError();
}

cudaError_t launch_mg_cycles(int prec, const CycleArgs& a, int blocks, int max_coarsest, const PotCheck& ck,
                             cudaStream_t st) {
    const size_t sm = std::max({(size_t)kLegGroups * kLegBytes<kFusedTX, kFusedTY>, tail_bytes(a.tail_cells, a.tail_small),
                                coarsest_bytes(max_coarsest)});
    auto kern = prec == 0 ? k_cycles<double> : k_cycles<float>;
    void* args[] = {const_cast<CycleArgs*>(&a), const_cast<PotCheck*>(&ck)};
    return cudaLaunchCooperativeKernel(kern, dim3(blocks), dim3(kTailNT), args, sm, st);
}

cudaError_t launch_mg_extrapolate(const DevCase* cases, const TileRef* tiles, int n, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    k_extrapolate<<<n, kNT, 0, st>>>(cases, tiles);
    return cudaGetLastError();
}

}  // namespace lbfs
