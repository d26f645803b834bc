// lbfs_fields.cu -- per-case utility kernels: initial condition, field export and
// import in FP64, the potential coefficient of a state, its statistics (Eq. 51 liquid
// fraction of the droplet, sums of C and H_e) and the Sec. 5 diagnostics.
#include "lbfs_kernels.h"

namespace lbfs {

namespace {


__device__ __forceinline__ bool cell_of(int nx, int ny, int& i, int& j) {
    i = blockIdx.x * blockDim.x + threadIdx.x;
    j = blockIdx.y;
    return i < nx && j < ny;
}

// Table 1 "Initialization": droplet C = 1/2 + 1/2 tanh(2 (R - r)/xi) (the equilibrium
// profile of the Cahn-Hilliard free energy), uniform T_init, liquid everywhere so
// H_e = C_p T + L, p = 0, u = 0, uniform far-field potential.
template <class R>
__global__ void k_init(const DevCase* __restrict__ dc, InitArgs a) {
    int i, j;
    const CaseParams& P = dc->P;
    if (!cell_of(P.nx, P.ny, i, j)) return;
    const double x = i + 0.5, y = j + 0.5;
    double C = 1.0;
    if (a.kind != 2) {
        const double dx = x - a.cx, dy = y - a.cy;
        C = 0.5 + 0.5 * tanh(2.0 * (a.radius - sqrt(dx * dx + dy * dy)) / a.xi);
    }
    const double cp = mixture<double>(0.0, C, P.cp_s, P.cp_l, P.cp_g);
    const double He = cp * a.T_init + P.L;
    const size_t k = (size_t)j * P.pitch + i;
    he_set<R>(dc->He[0], k, He);
    typename Quad<R>::T w;
    w.x = w.y = w.z = R(0);
    w.w = R(C);
    static_cast<typename Quad<R>::T*>(dc->W[0])[k] = w;
    phi_set<R>(dc, k, -P.H0 * (x * P.cos_t + y * P.sin_t));
    R T, Fl;
    invert_enthalpy<R, double>(P, He, R(C), T, Fl);
    static_cast<R*>(dc->Fs_prev)[k] = R(1) - Fl;
}

template <class R>
__global__ void k_mu_from_state(const DevCase* __restrict__ dc) {
    int i, j;
    const CaseParams& P = dc->P;
    if (!cell_of(P.nx, P.ny, i, j)) return;
    const size_t k = (size_t)j * P.pitch + i;
    const R C = static_cast<const typename Quad<R>::T*>(dc->W[0])[k].w;
    R T, Fl;
    invert_enthalpy<R, double>(P, he_get<R>(dc->He[0], k), C, T, Fl);
    static_cast<R*>(dc->lev[0].mu)[(size_t)j * dc->lev[0].pitch + i] =
        R(1) + mixture(R(1) - Fl, C, P.chi_s, P.chi_l, P.chi_g);
}

template <class R>
__device__ __forceinline__ R C_at(const CaseParams& P, const typename Quad<R>::T* W, int i, int j) {
    // C with the wall ghost rule (wetting; zero gradient at 90 degrees) or periodic wrap
    bool wall = false;
    if (i < 0) { wall = !P.periodic_x; i = P.periodic_x ? i + P.nx : 0; }
    if (i >= P.nx) { wall = !P.periodic_x; i = P.periodic_x ? i - P.nx : P.nx - 1; }
    if (j < 0) { wall = wall || !P.periodic_y; j = P.periodic_y ? j + P.ny : 0; }
    if (j >= P.ny) { wall = wall || !P.periodic_y; j = P.periodic_y ? j - P.ny : P.ny - 1; }
    const R c = W[(size_t)j * P.pitch + i].w;
    return wall ? c + R(P.wet) * c * (R(1) - c) : c;
}

template <class R>
__global__ void k_derive(const DevCase* __restrict__ dc, uint32_t mask, double* __restrict__ out) {
    int i, j;
    const CaseParams& P = dc->P;
    if (!cell_of(P.nx, P.ny, i, j)) return;
    const size_t k = (size_t)j * P.pitch + i;
    const size_t N = (size_t)P.nx * P.ny, o = (size_t)j * P.nx + i;
    const double He = he_get<R>(dc->He[0], k);
    const typename Quad<R>::T* Wg = static_cast<const typename Quad<R>::T*>(dc->W[0]);
    const typename Quad<R>::T w = Wg[k];
    const R C = w.w;
    R T, Fl;
    invert_enthalpy<R, double>(P, He, C, T, Fl);
    const R rho = mixture(R(1) - Fl, C, P.rho_s, P.rho_l, P.rho_g);
    const R mx = w.y, my = w.z;
    int slot = 0;
    for (int f = 0; f < 13; ++f) {
        if (!(mask & (1u << f))) continue;
        double v = 0.0;
        switch (f) {
        case 0: v = phi_get<R>(dc, k); break;
        case 1: v = He; break;
        case 2: v = (double)T; break;
        case 3: v = (double)Fl; break;
        case 4: v = (double)w.x; break;
        case 5: v = (double)(mx * R(3) / rho); break;
        case 6: v = (double)(my * R(3) / rho); break;
        case 7: v = (double)C; break;
        case 8: {
            const R lap = C_at<R>(P, Wg, i + 1, j) + C_at<R>(P, Wg, i - 1, j) + C_at<R>(P, Wg, i, j + 1) +
                          C_at<R>(P, Wg, i, j - 1) - R(4) * C;
            v = (double)(R(2) * R(P.beta) * C * (C - R(1)) * (R(2) * C - R(1)) - R(P.kappa) * lap);
            break;
        }
        case 9: v = (double)rho; break;
        case 10: v = (double)mx; break;
        case 11: v = (double)my; break;
        case 12: v = (double)static_cast<const R*>(dc->Fs_prev)[k]; break;
        }
        out[slot * N + o] = v;
        ++slot;
    }
}

// Sec. 5 diagnostics, 32 columns a block, one lane per column; each of the 32 warps marches down
// its share of the rows:
//  - the column's droplet height: the highest point where C crosses 1/2, linear in y
//    between the cell centres on either side, ny when the top cell has C >= 1/2;
//  - the largest speed |u| over the block's droplet cells (C >= 1/2), in each of its columns;
//  - the local heat flux on a cold (Dirichlet) bottom wall, Q = -lambda dT/dy at y = 0
//    (Sec. 5.2).  The slope is that of the quadratic through the wall value at y = 0 and
//    the first two cell centres (y = 1/2, 3/2): (-8 T_w + 9 T_0 - T_1)/3; a single row
//    uses (T_0 - T_w)/(1/2).  lambda is the first cell's Eq. 11 conductivity.
// Everything is evaluated in FP64 from the stored state.  cols holds three rows of nx.
// Bound by HBM: the speeds are compared as an upper bound first, formed from the stored quad alone
// with the smaller of the cell's solid and liquid mixture densities, and only a cell whose bound
// exceeds the largest speed so far is evaluated (FP64, enthalpy inversion), which leaves the
// maximum as it was.
// The bound's margin of 1e-3 is far above its rounding; cells outside the range in which that
// is so (cancelling densities, C > 2, NaN) are always evaluated.
// One thread a column, serial over the rows in FP64, had 8 blocks on 1024 x 512 and took about
// half of a monitoring pass (diagnostics and six derived fields): 1157 us, now 580 to 680 with
// the host link's spread.
constexpr int kDiagWarps = 32, kDiagAhead = 4;

template <class R>
__global__ void __launch_bounds__(32 * kDiagWarps) k_diag_columns(const DevCase* __restrict__ dc,
                                                                 double* __restrict__ cols) {
    __shared__ double top[kDiagWarps][32], fastest[kDiagWarps];
    const CaseParams& P = dc->P;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
    const bool in = i < P.nx;
    using Q4 = typename Quad<R>::T;
    const Q4* Wg = static_cast<const Q4*>(dc->W[0]) + (in ? i : P.nx - 1);
    const void* Heg = dc->He[0];
    const R rho_s = R(P.rho_s), rho_l = R(P.rho_l), rho_g = R(P.rho_g), floor_rho = R(0.01) * (R(2) * rho_l + rho_g);
    double h = -1.0, umax = 0.0, C_above = 0.0;   // h < 0: no droplet cell yet
    R bar = R(0);                                 // umax in the bound's precision, 0 while it is tiny
    const int j0 = (int)((long long)P.ny * w / kDiagWarps), j1 = (int)((long long)P.ny * (w + 1) / kDiagWarps);
    if (j1 < P.ny) C_above = (double)Wg[(size_t)j1 * P.pitch].w;
    for (int jb = j1 - 1; jb >= j0; jb -= kDiagAhead) {
        Q4 row[kDiagAhead];
#pragma unroll
        for (int q = 0; q < kDiagAhead; ++q) row[q] = Wg[(size_t)max(jb - q, j0) * P.pitch];
#pragma unroll
        for (int q = 0; q < kDiagAhead; ++q) {
            const int j = jb - q;
            const double C = (double)row[q].w;
            const bool drop = in && j >= j0 && C >= 0.5;
            if (drop && h < 0.0)
                h = (j == P.ny - 1) ? (double)P.ny : (j + 0.5) + (C - 0.5) / (C - C_above);
            C_above = C;
            const R c = row[q].w, a = fabs(row[q].y), b = fabs(row[q].z);
            const R rho = fmin(rho_s, c * rho_l + (R(1) - c) * rho_g);
            // |(a, b)| <= max + (sqrt(2) - 1) min
            const R bound = R(3.003) * (fmax(a, b) + R(0.41422) * fmin(a, b));
            const bool look = drop && !(c <= R(2) && rho > floor_rho && bar > R(0) && bound <= bar * rho);
            if (__any_sync(0xffffffffu, look)) {
                double speed = 0.0;
                if (look) {
                    double T, Fl;
                    invert_enthalpy<double, double>(P, he_get<R>(Heg, (size_t)j * P.pitch + i), C, T, Fl);
                    const double r = mixture<double>(1.0 - Fl, C, P.rho_s, P.rho_l, P.rho_g);
                    const double u = (double)row[q].y * 3.0 / r, v = (double)row[q].z * 3.0 / r;
                    speed = sqrt(u * u + v * v);
                }
                umax = fmax(umax, speed);
                for (int o = 16; o > 0; o >>= 1) umax = fmax(umax, __shfl_xor_sync(0xffffffffu, umax, o));
                bar = umax > 1e-30 && umax < 1e30 ? R(umax) : R(0);
            }
        }
    }
    top[w][lane] = h;
    if (lane == 0) fastest[w] = umax;
    __syncthreads();
    if (w != 0 || !in) return;
    h = 0.0;
    for (int q = kDiagWarps - 1; q >= 0; --q)
        if (!(top[q][lane] < 0.0)) {   // the highest rows with a droplet cell
            h = top[q][lane];
            break;
        }
    for (int q = 0; q < kDiagWarps; ++q) umax = fmax(umax, fastest[q]);
    const Q4 *W0 = static_cast<const Q4*>(dc->W[0]);
    double Q = 0.0;
    if (!P.periodic_y && P.thermal_dir[2]) {
        const double C0 = (double)W0[i].w;
        double T0, Fl0;
        invert_enthalpy<double, double>(P, he_get<R>(Heg, i), C0, T0, Fl0);
        const double lam = mixture<double>(1.0 - Fl0, C0, P.lam_s, P.lam_l, P.lam_g);
        const double Tw = P.wall_T[2];
        double slope;
        if (P.ny >= 2) {
            const size_t k1 = (size_t)P.pitch + i;
            double T1, Fl1;
            invert_enthalpy<double, double>(P, he_get<R>(Heg, k1), (double)W0[k1].w, T1, Fl1);
            slope = (-8.0 * Tw + 9.0 * T0 - T1) / 3.0;
        } else {
            slope = (T0 - Tw) / 0.5;
        }
        Q = -lam * slope;
    }
    cols[i] = h;
    cols[P.nx + i] = umax;
    cols[2 * (size_t)P.nx + i] = Q;
}

// Reduces the per-column diagnostics of one case with one block of kDiagThreads
// threads in a fixed order: H_m and U_max are maxima, Q_wall the sum of Q dx over the
// wall faces.  Pe = U_max D / alpha_l with D = 2 R_0 and alpha_l = lambda_l/(rho_l C_p,l)
// (Eq. 50, read with the largest droplet speed); Fo = lambda_l t/(rho_l C_p,l R_0^2).
constexpr int kDiagThreads = 256;

__global__ void __launch_bounds__(kDiagThreads) k_diag_finalize(const DevCase* __restrict__ dc,
                                                                 const double* __restrict__ cols,
                                                                 double R0, double* __restrict__ out) {
    __shared__ double sh[3][kDiagThreads];
    const int nx = dc->P.nx;
    double h = 0.0, u = 0.0, q = 0.0;
    for (int i = threadIdx.x; i < nx; i += kDiagThreads) {
        h = fmax(h, cols[i]);
        u = fmax(u, cols[nx + i]);
        q += cols[2 * (size_t)nx + i];
    }
    sh[0][threadIdx.x] = h;
    sh[1][threadIdx.x] = u;
    sh[2][threadIdx.x] = q;
    __syncthreads();
    for (int w = kDiagThreads / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) {
            sh[0][threadIdx.x] = fmax(sh[0][threadIdx.x], sh[0][threadIdx.x + w]);
            sh[1][threadIdx.x] = fmax(sh[1][threadIdx.x], sh[1][threadIdx.x + w]);
            sh[2][threadIdx.x] += sh[2][threadIdx.x + w];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const CaseParams& P = dc->P;
        const double alpha_l = P.lam_l / (P.rho_l * P.cp_l);
        out[0] = sh[0][0];
        out[1] = sh[1][0];
        out[2] = sh[1][0] * 2.0 * R0 / alpha_l;
        out[3] = P.lam_l * dc->stats[ST_T] / (P.rho_l * P.cp_l * R0 * R0);
        out[4] = sh[2][0];
    }
}

template <class R>
__global__ void k_store(const DevCase* __restrict__ dc, uint32_t mask, const double* __restrict__ in) {
    int i, j;
    const CaseParams& P = dc->P;
    if (!cell_of(P.nx, P.ny, i, j)) return;
    const size_t k = (size_t)j * P.pitch + i;
    const size_t N = (size_t)P.nx * P.ny, o = (size_t)j * P.nx + i;
    typename Quad<R>::T* W = static_cast<typename Quad<R>::T*>(dc->W[0]) + k;
    int slot = 0;
    for (int f = 0; f < 13; ++f) {
        if (!(mask & (1u << f))) continue;
        const double v = in[slot * N + o];
        switch (f) {
        case 0: phi_set<R>(dc, k, v); break;
        case 1: he_set<R>(dc->He[0], k, v); break;
        case 4: W->x = R(v); break;
        case 7: W->w = R(v); break;
        case 10: W->y = R(v); break;
        case 11: W->z = R(v); break;
        case 12: static_cast<R*>(dc->Fs_prev)[k] = R(v); break;
        default: break;
        }
        ++slot;
    }
}

// statistics of the stored state, after initialisation or import: kFinChunks blocks
// each sum a fixed range of rows (FP64, or FP32 pairs in mixed precision); the last
// block to finish (a ticket, no waiting) sums the chunks in order and writes sum C,
// sum H_e, the droplet sums and Q_L (Eq. 51), which also seeds the freezing-time
// interpolation
template <class R>
__global__ void k_stats_init(const DevCase* __restrict__ dc) {
    using Slot = typename DSum<R>::Slot;
    using HS = typename HeStore<R>::T;
    __shared__ Slot sh[32];
    __shared__ bool last;
    const CaseParams& P = dc->P;
    const int c = blockIdx.x;
    const int j0 = (int)((long long)P.ny * c / kFinChunks), j1 = (int)((long long)P.ny * (c + 1) / kFinChunks);
    DSum<R> acc[5];
    for (int q = 0; q < 5; ++q) acc[q] = DSum<R>::zero();
    const HS* He = static_cast<const HS*>(dc->He[0]);
    const typename Quad<R>::T* Wg = static_cast<const typename Quad<R>::T*>(dc->W[0]);
    for (int j = j0; j < j1; ++j)
        for (int i = threadIdx.x; i < P.nx; i += blockDim.x) {
            const size_t k = (size_t)j * P.pitch + i;
            const R C = Wg[k].w;
            R T, Fl;
            invert_enthalpy<R, double>(P, he_value(He[k]), C, T, Fl);
            acc[0].add(C);
            acc[1].add(He[k]);
            if (C >= R(0.5)) {
                acc[2].add(Fl);
                acc[3].add(R(1));
                acc[4].add(R(1) - Fl);
            }
        }
    for (int q = 0; q < 5; ++q) acc[q] = block_sum0<R>(acc[q], sh);
    Slot* ch = static_cast<Slot*>(dc->chunk);
    if (threadIdx.x == 0) {
        for (int q = 0; q < 5; ++q) ch[c * kRedN + q] = acc[q].slot();
        __threadfence();
        last = atomicAdd(&dc->tickets[0], 1u) == (unsigned)(kFinChunks - 1);
    }
    __syncthreads();
    if (!last || threadIdx.x != 0) return;
    __threadfence();
    double a[5];
    for (int q = 0; q < 5; ++q) {
        DSum<R> v = DSum<R>::zero();
        for (int k = 0; k < kFinChunks; ++k) v.add(DSum<R>::of(ld_cg(&ch[k * kRedN + q])));
        a[q] = v.value();
    }
    dc->tickets[0] = 0u;
    double* st = dc->stats;
    st[ST_SUM_C] = a[0];
    st[ST_SUM_HE] = a[1];
    st[ST_SUM_FL_DROP] = a[2];
    st[ST_N_DROP] = a[3];
    st[ST_Q_L] = a[3] > 0 ? a[4] / a[3] : 0.0;
    st[ST_QL_PREV] = st[ST_Q_L];
}

}  // namespace

static dim3 cell_grid(int nx, int ny) { return dim3((nx + 127) / 128, ny); }

cudaError_t launch_init(int prec, const DevCase* d, int nx, int ny, InitArgs a, cudaStream_t st) {
    if (prec == 0) k_init<double><<<cell_grid(nx, ny), 128, 0, st>>>(d, a);
    else k_init<float><<<cell_grid(nx, ny), 128, 0, st>>>(d, a);
    return cudaGetLastError();
}

cudaError_t launch_mu_from_state(int prec, const DevCase* d, int nx, int ny, cudaStream_t st) {
    if (prec == 0) k_mu_from_state<double><<<cell_grid(nx, ny), 128, 0, st>>>(d);
    else k_mu_from_state<float><<<cell_grid(nx, ny), 128, 0, st>>>(d);
    return cudaGetLastError();
}

cudaError_t launch_derive_fields(int prec, const DevCase* d, int nx, int ny, uint32_t mask, double* out,
                                 cudaStream_t st) {
    if (prec == 0) k_derive<double><<<cell_grid(nx, ny), 128, 0, st>>>(d, mask, out);
    else k_derive<float><<<cell_grid(nx, ny), 128, 0, st>>>(d, mask, out);
    return cudaGetLastError();
}

cudaError_t launch_diagnostics(int prec, const DevCase* d, int nx, double R0, double* cols, double* out5,
                               cudaStream_t st) {
    const int nb = (nx + 31) / 32;
    if (prec == 0) k_diag_columns<double><<<nb, 32 * kDiagWarps, 0, st>>>(d, cols);
    else k_diag_columns<float><<<nb, 32 * kDiagWarps, 0, st>>>(d, cols);
    k_diag_finalize<<<1, kDiagThreads, 0, st>>>(d, cols, R0, out5);
    return cudaGetLastError();
}

cudaError_t launch_store_fields(int prec, const DevCase* d, int nx, int ny, uint32_t mask,
                                const double* in, cudaStream_t st) {
    if (prec == 0) k_store<double><<<cell_grid(nx, ny), 128, 0, st>>>(d, mask, in);
    else k_store<float><<<cell_grid(nx, ny), 128, 0, st>>>(d, mask, in);
    return cudaGetLastError();
}

cudaError_t launch_stats_init(int prec, const DevCase* d, int nx, int ny, cudaStream_t st) {
    (void)nx;
    (void)ny;
    if (prec == 0) k_stats_init<double><<<kFinChunks, 512, 0, st>>>(d);
    else k_stats_init<float><<<kFinChunks, 512, 0, st>>>(d);
    return cudaGetLastError();
}

}  // namespace lbfs
