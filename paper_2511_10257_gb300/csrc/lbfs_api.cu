// lbfs_api.cu -- host implementation of the C ABI declared in include/lbfs.h:
// context and case management, device memory layout, lists of strips and tiles for batched
// cases, and the per-step schedule (potential refinement, three Runge-Kutta stages, the last
// with the step's statistics), optionally recorded once as a CUDA graph and replayed.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "lbfs.h"
#include "lbfs_kernels.h"

using namespace lbfs;

namespace {

constexpr int kCoarsenCells = 4;      // stop coarsening at or below this many cells

constexpr size_t kFieldAlign = 32;    // of a case's arrays: one load of a cell's four FP64 quantities
static_assert(kFieldAlign % alignof(Quad64) == 0, "a case's quads lie on their own boundary");
constexpr int kFlags = 4;             // words of lbfs_ctx::d_flag

size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

struct Slot {
    bool defined = false;
    lbfs_case_desc desc{};
    DevCase hd{};
    StageCase<float> sf{};    // the stage kernel's view, in the context's precision
    StageCase<double> sd{};
    void* block = nullptr;
    size_t ticket_bytes = 0;  // of hd.mg_tickets
};

}  // namespace

struct lbfs_ctx {
    lbfs_config cfg{};
    int prec = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    std::vector<Slot> slots;
    DevCase* d_cases = nullptr;
    double* d_stats = nullptr;
    void* d_stage_cases = nullptr;   // StageCase of every slot, in the context's precision
    TileRef* d_stage_tiles = nullptr;
    int n_stage_tiles = 0;
    TileRef* d_mg_tiles = nullptr;      // fine-level 32 x 32 tiles (FP64: the extrapolated start)
    int n_mg_tiles = 0;
    TileRef* d_res_tiles = nullptr;     // the residual's strips
    int n_res_tiles = 0, res_rows = 0;
    std::vector<TileRef*> d_ft_tiles;   // fused V-cycle tiles per level
    std::vector<int> n_ft_tiles;
    std::vector<int> ft_small;          // per level: 16 x 8 fused tiles instead of 32 x 16
    int n_active = 0;
    int n_pot = 0;
    int* d_tail = nullptr;              // cases whose coarse levels run in one kernel
    int n_tail = 0, tail_cells = 0, tail_small = 0;
    int* d_coarsest = nullptr;          // the others: their coarsest level
    int n_coarsest = 0, coarsest_cells = 0;
    int max_depth = 0;                  // levels with a kernel per leg
    int sm_count = 152;               // multiprocessors of the context's device
    // after the statistics, copied to the host with them: [0] votes of host-counted cycles, [1] and
    // [2] the cycles' grid barrier, [3] a wait in it ran out
    int* d_flag = nullptr;
    size_t stats_bytes = 0;   // of the statistics, to the flags
    int* h_flag = nullptr;
    double* h_stats = nullptr;
    double* d_scratch = nullptr;
    size_t scratch_bytes = 0;
    bool dirty = true;
    bool pot_fail = false;
    std::string err;
    int64_t launches = 0;
    double mg_tol = 0.0;
    int mg_max_cycles = 0;
    int mg_warm_cycles = 0;
    int mg_wait_polls = 0;
    int half = 0;          // every defined case has dts = 1/2
    int tile = 0;          // stage-kernel strip shape id (config or autotuner)
    int rows = 0;          // rows of a strip, by the shape id or its rule
    bool pot_fresh = true; // a state was set since the last full potential solve
    // whether all blocks of the cycles' kernel run at once on the context's stream: -1 not known
    // yet, 1 it has run, 0 it was refused or a wait of its ran out
    int coop = -1;
    cudaGraphExec_t gexec = nullptr;
    cudaGraph_t graph = nullptr;
    int64_t graph_launches = 0;       // kernel nodes in one recorded step
    cudaStream_t cap_stream = nullptr; // private stream used to record the graph
    // kernel timing (events on the context stream)
    bool timing = false;
    double t_ms[3] = {0, 0, 0};
    int64_t t_cnt[3] = {0, 0, 0};
    std::vector<cudaEvent_t> ev_pool;
    std::vector<std::pair<int, std::pair<cudaEvent_t, cudaEvent_t>>> ev_pending;
};

namespace {

lbfs_status fail(lbfs_ctx* c, lbfs_status s, const std::string& msg) {
    if (c) c->err = msg;
    return s;
}

#define CK(call)                                                                                  \
    do {                                                                                          \
        cudaError_t e_ = (call);                                                                  \
        if (e_ != cudaSuccess)                                                                    \
            return fail(ctx, LBFS_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_));     \
    } while (0)

void* dalloc(lbfs_ctx* ctx, size_t bytes) {
    if (bytes == 0) bytes = 256;
    if (ctx->cfg.dev_alloc) return ctx->cfg.dev_alloc(bytes, ctx->cfg.alloc_user);
    void* p = nullptr;
    if (cudaMalloc(&p, bytes) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    return p;
}

void dfree(lbfs_ctx* ctx, void* p) {
    if (!p) return;
    if (ctx->cfg.dev_free) ctx->cfg.dev_free(p, ctx->cfg.alloc_user);
    else cudaFree(p);
}

void drop_graph(lbfs_ctx* ctx) {
    if (ctx->gexec) cudaGraphExecDestroy(ctx->gexec);
    if (ctx->graph) cudaGraphDestroy(ctx->graph);
    ctx->gexec = nullptr;
    ctx->graph = nullptr;
}

cudaEvent_t take_event(lbfs_ctx* ctx) {
    if (!ctx->ev_pool.empty()) {
        cudaEvent_t e = ctx->ev_pool.back();
        ctx->ev_pool.pop_back();
        return e;
    }
    cudaEvent_t e = nullptr;
    cudaEventCreate(&e);
    return e;
}

// open an event bracket of class cls (no-op unless timing is on)
cudaEvent_t tic(lbfs_ctx* ctx) {
    if (!ctx->timing) return nullptr;
    cudaEvent_t e = take_event(ctx);
    cudaEventRecord(e, ctx->stream);
    return e;
}

void toc(lbfs_ctx* ctx, int cls, cudaEvent_t start) {
    if (!ctx->timing || !start) return;
    cudaEvent_t e = take_event(ctx);
    cudaEventRecord(e, ctx->stream);
    ctx->ev_pending.push_back({cls, {start, e}});
}

// after a stream synchronisation: accumulate and recycle the event pairs
void harvest(lbfs_ctx* ctx) {
    for (auto& pe : ctx->ev_pending) {
        float ms = 0.f;
        if (cudaEventElapsedTime(&ms, pe.second.first, pe.second.second) == cudaSuccess) {
            ctx->t_ms[pe.first] += ms;
            ctx->t_cnt[pe.first] += 1;
        }
        ctx->ev_pool.push_back(pe.second.first);
        ctx->ev_pool.push_back(pe.second.second);
    }
    ctx->ev_pending.clear();
}

// Resolve the case parameters (Eq. 50 groups, mu_c coefficients, boundary flags).
lbfs_status resolve(lbfs_ctx* ctx, const lbfs_case_desc& d, CaseParams& P) {
    std::memset(&P, 0, sizeof(P));
    if (d.nx < 4 || d.ny < 4) return fail(ctx, LBFS_EINVAL, "nx and ny must be >= 4");
    // cell indices (row pitch a multiple of 32 times ny) stay below 2^31 in 32-bit arithmetic
    if ((int64_t)align_up((size_t)d.nx, 32) * d.ny >= (int64_t)1 << 31)
        return fail(ctx, LBFS_EINVAL, "grid too large");
    if (d.flags != 0) return fail(ctx, LBFS_EINVAL, "flags must be 0");
    if (d.init < 0 || d.init > 2) return fail(ctx, LBFS_EINVAL, "init must be 0, 1 or 2");
    if (d.mag_bc < 0 || d.mag_bc > 1) return fail(ctx, LBFS_EINVAL, "mag_bc must be 0 or 1");
    if (!(d.dt > 0 && d.dts > 0 && d.Q_g > 0 && d.xi > 0 && d.sigma >= 0 && d.mobility >= 0))
        return fail(ctx, LBFS_EINVAL, "dt, dts, Q_g, xi must be > 0; sigma, mobility >= 0");
    const double pos[] = {d.rho_l, d.rho_g, d.rho_s, d.cp_l, d.cp_g, d.cp_s};
    for (double v : pos)
        if (!(v > 0)) return fail(ctx, LBFS_EINVAL, "densities and heat capacities must be > 0");
    const double nonneg[] = {d.mu_l, d.mu_g, d.mu_s, d.lam_l, d.lam_g, d.lam_s};
    for (double v : nonneg)
        if (!(v >= 0)) return fail(ctx, LBFS_EINVAL, "viscosities and conductivities must be >= 0");
    if (d.init == 0 || d.init == 1) {
        if (!(d.radius > 0)) return fail(ctx, LBFS_EINVAL, "radius must be > 0");
    }
    P.nx = d.nx;
    P.ny = d.ny;
    P.pitch = (int)align_up((size_t)d.nx, 32);
    P.periodic_x = d.periodic_x ? 1 : 0;
    P.periodic_y = d.periodic_y ? 1 : 0;
    for (int w = 0; w < 4; ++w) {
        const bool on_periodic = (w < 2) ? P.periodic_x : P.periodic_y;
        P.thermal_dir[w] = (!on_periodic && d.thermal_dirichlet[w]) ? 1 : 0;
        P.wall_T[w] = d.wall_T[w];
        P.mag_dir[w] = on_periodic ? 0 : (d.mag_bc == 1 && w < 2 ? 0 : 1);
    }
    P.rho_l = d.rho_l; P.rho_g = d.rho_g; P.rho_s = d.rho_s;
    P.mu_l = d.mu_l; P.mu_g = d.mu_g; P.mu_s = d.mu_s;
    P.cp_l = d.cp_l; P.cp_g = d.cp_g; P.cp_s = d.cp_s;
    P.lam_l = d.lam_l; P.lam_g = d.lam_g; P.lam_s = d.lam_s;
    P.chi_l = d.chi_l; P.chi_g = d.chi_g; P.chi_s = d.chi_s;
    P.beta = 12.0 * d.sigma / d.xi;
    P.kappa = 1.5 * d.xi * d.sigma;
    P.mobility = d.mobility;
    P.Q_g = d.Q_g;
    P.gravity = d.gravity;
    P.T_m = d.T_m;
    // Eq. 50: Ste = C_p,l (T_m - T_w) / L with the cold bottom wall, and
    // Bo_m = mu_0 H^2 D / sigma on the droplet diameter D = 2 R (mu_0 = 1)
    P.L = d.stefan > 0.0 ? d.cp_l * (d.T_m - d.wall_T[2]) / d.stefan : d.latent;
    if (!(P.L > 0)) return fail(ctx, LBFS_EINVAL, "latent heat must be > 0");
    P.H0 = d.bo_m > 0.0 ? std::sqrt(d.bo_m * d.sigma / (2.0 * d.radius)) : d.H0;
    const double ang = d.field_angle_deg * 3.14159265358979323846 / 180.0;
    P.cos_t = std::cos(ang);
    P.sin_t = std::sin(ang);
    P.dt = d.dt;
    P.dts = d.dts;
    if (!(d.contact_angle_deg > 0.0 && d.contact_angle_deg < 180.0))
        return fail(ctx, LBFS_EINVAL, "contact_angle_deg must lie in (0, 180)");
    // wetting: the equilibrium profile C = (1 + tanh(2 d/xi))/2 meets a wall at theta_w when
    // dC/dn = -(4/xi) cos(theta_w) C (1 - C); 90 degrees is exactly the no-flux wall
    P.wet = d.contact_angle_deg == 90.0 ? 0.0 : 4.0 * std::cos(d.contact_angle_deg * 3.14159265358979323846 / 180.0) / d.xi;
    P.cp_ref = 0.5 * (d.cp_s + d.cp_l);
    P.vol_ratio = 1.0 - d.rho_s / d.rho_l;
    bool chi = d.chi_l != 0.0 || d.chi_s != 0.0 || d.chi_g != 0.0;
    bool dir = false;
    for (int w = 0; w < 4; ++w) dir = dir || P.mag_dir[w];
    P.solve_potential = (chi && dir) ? 1 : 0;
    // explicit stability of the diffusive terms (RK3 real-axis bound ~2.51, five-point
    // eigenvalue up to 8 D / dx^2)
    double Dmax = 0.0;
    const double rho[3] = {d.rho_l, d.rho_g, d.rho_s}, lam[3] = {d.lam_l, d.lam_g, d.lam_s};
    const double cp[3] = {d.cp_l, d.cp_g, d.cp_s}, mu[3] = {d.mu_l, d.mu_g, d.mu_s};
    for (int k = 0; k < 3; ++k) {
        Dmax = std::fmax(Dmax, lam[k] / (rho[k] * cp[k]));
        Dmax = std::fmax(Dmax, mu[k] / rho[k]);
    }
    if (d.dt * 8.0 * Dmax > 2.51)
        return fail(ctx, LBFS_EINVAL, "dt exceeds the explicit diffusion limit 2.51/(8 D_max)");
    if (P.solve_potential && ((P.periodic_x && (d.nx & 1)) || (P.periodic_y && (d.ny & 1))))
        return fail(ctx, LBFS_EINVAL, "periodic axes of a case with a potential solve need even sizes");
    return LBFS_OK;
}

template <class R>
void fill_phys(const CaseParams& P, PhysT<R>& q) {
    q.rho_s = R(P.rho_s); q.rho_g = R(P.rho_g);
    q.mu_s = R(P.mu_s); q.mu_l = R(P.mu_l); q.mu_g = R(P.mu_g);
    q.lam_s = R(P.lam_s); q.lam_l = R(P.lam_l); q.lam_g = R(P.lam_g);
    q.cp_s = R(P.cp_s); q.cp_g = R(P.cp_g);
    q.chi_s = R(P.chi_s); q.chi_g = R(P.chi_g);
    q.kappa = R(P.kappa); q.cp_ref = R(P.cp_ref);
    q.inv_dts = R(1.0 / P.dts); q.inv_cpref_dts = R(1.0 / (P.cp_ref * P.dts));
    q.dt = R(P.dt); q.vol_ratio = R(P.vol_ratio); q.gravity = R(P.gravity); q.T_m = R(P.T_m); q.L = R(P.L);
    for (int w = 0; w < 4; ++w) q.wall_T[w] = R(P.wall_T[w]);
    q.wet = R(P.wet);
    const double Hes = P.cp_s * P.T_m;
    q.Hes_hi = R(Hes);
    q.Hes_lo = R(Hes - double(q.Hes_hi));
    q.L_hi = R(P.L);
    q.L_lo = R(P.L - double(q.L_hi));
    q.rho_sg = q.rho_s - q.rho_g; q.rho_lg = R(P.rho_l) - q.rho_g;
    q.cp_sg = q.cp_s - q.cp_g; q.cp_lg = R(P.cp_l) - q.cp_g;
    q.mu_sg = q.mu_s - q.mu_g; q.mu_lg = q.mu_l - q.mu_g;
    q.lam_sg = q.lam_s - q.lam_g; q.lam_lg = q.lam_l - q.lam_g; q.chi_lg = R(P.chi_l) - q.chi_g;
    q.m_Qg = -R(P.Q_g); q.m_cp_ref3 = R(-P.cp_ref / 3.0);
    q.inv_cps = R(1.0 / P.cp_s);
    q.x_g = R(P.mobility / (P.Q_g * P.dts)); q.om_x_g = R(1) - q.x_g; q.beta2 = R(2.0 * P.beta); q.Qg3 = R(3.0 * P.Q_g);
    q.mhd = R(-0.5 * P.dts); q.off = R(0.5 * (0.5 - P.dts)); q.inv_dt = R(1.0 / P.dt);
}

template <class R>
void fill_stage(const DevCase& d, StageCase<R>& c) {
    const CaseParams& P = d.P;
    std::memset(&c, 0, sizeof(c));
    fill_phys<R>(P, c.Q);
    for (int k = 0; k < 3; ++k) {
        c.He[k] = d.He[k];
        c.W[k] = d.W[k];
    }
    c.phi = d.phi;
    c.Fs_prev = d.Fs_prev;
    c.Sdot = d.Sdot;
    c.mu = d.lev[0].mu;
    c.red = d.red;
    c.red_groups = d.red_groups;
    c.tickets = d.red_tickets;
    c.stats = d.stats;
    c.dt = P.dt;
    c.solve_potential = P.solve_potential;
    c.far_x = -2.0 * P.H0 * P.cos_t;
    c.far_y = -2.0 * P.H0 * P.sin_t;
    const double far[2] = {c.far_x, c.far_y};
    for (int k = 0; k < 2; ++k) {
        c.far_h[k] = (float)far[k];
        c.far_l[k] = (float)(far[k] - (double)c.far_h[k]);
    }
    c.nx = P.nx; c.ny = P.ny; c.pitch = P.pitch;
    c.periodic_x = P.periodic_x; c.periodic_y = P.periodic_y;
    for (int w = 0; w < 4; ++w) {
        c.thermal_dir[w] = P.thermal_dir[w];
        c.mag_dir[w] = P.mag_dir[w];
    }
}

// The lists of strips, tiles and cases that the kernels read, on the host.
struct Lists {
    std::vector<TileRef> stage, resid, mg;
    std::vector<int> tails, others;
    std::vector<std::vector<TileRef>> legs;   // fused V-cycle tiles per level
};

// Make the concatenated lists of all defined cases and send them, with the counts in the cases'
// tables that depend on them, in the order of the stream whose kernels read them (a copy on the
// default stream may return before its data has arrived, and a non-blocking stream does not wait
// for it).
lbfs_status make_lists(lbfs_ctx* ctx, Lists& lists) {
    auto send = [&](void* dst, const void* src, size_t bytes) {
        return cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, ctx->stream) == cudaSuccess;
    };
    std::vector<TileRef>& st = lists.stage;
    long long row_warps = 0;   // strips of one row's height over all cases
    for (const Slot& s : ctx->slots)
        if (s.defined) row_warps += (long long)((s.hd.P.nx + kStripW - 1) / kStripW) * s.hd.P.ny;
    const int TX = kStripW, TY = stage_rows(ctx->prec, ctx->tile, row_warps, ctx->sm_count);
    ctx->rows = TY;
    std::vector<int> pot;
    std::vector<int>&tails = lists.tails, &others = lists.others;
    int active = 0, depth = 0, tail_cells = 0, tail_small = 0, coarsest = 0;
    int half = 1;
    // The residual's strips: 64 rows, or fewer while all of them run at once (24 warps an SM)
    long long res_warps = 0;
    for (const Slot& s : ctx->slots)
        if (s.defined && s.hd.P.solve_potential)
            res_warps += (long long)((s.hd.P.nx + kResidStripW - 1) / kResidStripW) * s.hd.P.ny;
    int res_rows = kResidMinRows;
    while (res_rows < 64 && res_warps > 24LL * ctx->sm_count * res_rows) res_rows *= 2;
    std::vector<TileRef>& rt = lists.resid;
    for (int c = 0; c < (int)ctx->slots.size(); ++c) {
        Slot& s = ctx->slots[c];
        if (!s.defined) continue;
        // the counts of the kernels' last-arriver sums, on the device after every rebuild, whatever
        // the tables held (lbfs_set_case clears them)
        s.hd.mg_strips = ((s.hd.P.nx + kResidStripW - 1) / kResidStripW) * ((s.hd.P.ny + res_rows - 1) / res_rows);
        s.sf.strips = s.sd.strips = ((s.hd.P.nx + TX - 1) / TX) * ((s.hd.P.ny + TY - 1) / TY);
        const void* sc = ctx->prec == 0 ? (const void*)&s.sd : (const void*)&s.sf;
        const size_t scb = ctx->prec == 0 ? sizeof(s.sd) : sizeof(s.sf);
        if (!send(ctx->d_cases + c, &s.hd, sizeof(DevCase)) ||
            !send(static_cast<char*>(ctx->d_stage_cases) + c * scb, sc, scb))
            return fail(ctx, LBFS_ECUDA, "case table update failed");
        ++active;
        if (s.hd.P.dts != 0.5) half = 0;
        int slot = 0;
        for (int y = 0; y < s.hd.P.ny; y += TY)
            for (int x = 0; x < s.hd.P.nx; x += TX) st.push_back(TileRef{c, x, y, slot++});
        if (s.hd.P.solve_potential) {
            pot.push_back(c);
            depth = std::max(depth, s.hd.tail);
            const MGLevel& lc = s.hd.lev[s.hd.nlev - 1];
            if (lc.nx * lc.ny <= kTailCoarsest) {
                tails.push_back(c);
                int cells = 0;
                for (int L = s.hd.tail; L < s.hd.nlev; ++L) cells += s.hd.lev[L].nx * s.hd.lev[L].ny;
                tail_cells = std::max(tail_cells, cells);
                tail_small = std::max(tail_small, lc.nx * lc.ny);
            } else {
                others.push_back(c);
                coarsest = std::max(coarsest, lc.nx * lc.ny);
            }
            slot = 0;
            for (int y = 0; y < s.hd.P.ny; y += res_rows)
                for (int x = 0; x < s.hd.P.nx; x += kResidStripW) rt.push_back(TileRef{c, x, y, slot++});
        }
    }
    std::vector<TileRef>& mg = lists.mg;
    std::vector<std::vector<TileRef>>& ft = lists.legs;
    ft.resize(depth);
    if (ctx->prec == 0)
        for (int c : pot) {
            const CaseParams& P = ctx->slots[c].hd.P;
            int slot = 0;
            for (int y = 0; y < P.ny; y += kMgTY)
                for (int x = 0; x < P.nx; x += kMgTX) mg.push_back(TileRef{c, x, y, slot++});
        }
    // A level takes 16 x 8 fused tiles when its 32 x 16 tiles over all cases would
    // leave most SMs idle (fewer than two a multiprocessor): the legs of a small grid
    // then spread over four times as many SMs, at a larger halo share.
    std::vector<int> small(depth, 0);
    for (int L = 0; L < depth; ++L) {
        long long big = 0;
        for (int c : pot) {
            const Slot& s = ctx->slots[c];
            if (s.hd.tail > L)
                big += (long long)((s.hd.lev[L].nx + kFusedTX - 1) / kFusedTX) *
                       ((s.hd.lev[L].ny + kFusedTY - 1) / kFusedTY);
        }
        small[L] = big > 0 && big < 2LL * ctx->sm_count ? 1 : 0;
    }
    for (int L = 0; L < depth; ++L) {
        const int fx = small[L] ? kFusedSmallTX : kFusedTX, fy = small[L] ? kFusedSmallTY : kFusedTY;
        for (int c : pot) {
            const Slot& s = ctx->slots[c];
            if (s.hd.tail <= L) continue;
            int slot = 0;
            for (int y = 0; y < s.hd.lev[L].ny; y += fy)
                for (int x = 0; x < s.hd.lev[L].nx; x += fx) ft[L].push_back(TileRef{c, x, y, slot++});
        }
    }
    ctx->ft_small = small;
    auto upload = [&](void** dst, const void* src, size_t bytes) -> bool {
        if (*dst) dfree(ctx, *dst);
        *dst = nullptr;
        if (bytes == 0) return true;
        *dst = dalloc(ctx, bytes);
        if (!*dst) return false;
        return send(*dst, src, bytes);
    };
    if (!upload((void**)&ctx->d_stage_tiles, st.data(), st.size() * sizeof(TileRef)) ||
        !upload((void**)&ctx->d_mg_tiles, mg.data(), mg.size() * sizeof(TileRef)) ||
        !upload((void**)&ctx->d_res_tiles, rt.data(), rt.size() * sizeof(TileRef)) ||
        !upload((void**)&ctx->d_tail, tails.data(), tails.size() * sizeof(int)) ||
        !upload((void**)&ctx->d_coarsest, others.data(), others.size() * sizeof(int)))
        return fail(ctx, LBFS_ENOMEM, "tile list upload failed");
    for (auto* p : ctx->d_ft_tiles) dfree(ctx, p);
    ctx->d_ft_tiles.assign(depth, nullptr);
    ctx->n_ft_tiles.assign(depth, 0);
    for (int L = 0; L < depth; ++L) {
        if (!upload((void**)&ctx->d_ft_tiles[L], ft[L].data(), ft[L].size() * sizeof(TileRef)))
            return fail(ctx, LBFS_ENOMEM, "multigrid tile list upload failed");
        ctx->n_ft_tiles[L] = (int)ft[L].size();
    }
    ctx->n_mg_tiles = (int)mg.size();
    ctx->n_res_tiles = (int)rt.size();
    ctx->res_rows = res_rows;
    ctx->n_tail = (int)tails.size();
    ctx->tail_cells = tail_cells;
    ctx->tail_small = tail_small;
    ctx->n_coarsest = (int)others.size();
    ctx->n_stage_tiles = (int)st.size();
    ctx->n_active = active;
    ctx->n_pot = (int)pot.size();
    ctx->max_depth = depth;
    ctx->coarsest_cells = coarsest;
    ctx->half = half;
    return LBFS_OK;
}

lbfs_status rebuild(lbfs_ctx* ctx) {
    drop_graph(ctx);
    Lists lists;
    const lbfs_status r = make_lists(ctx, lists);
    const cudaError_t e = cudaStreamSynchronize(ctx->stream);   // `lists` outlives its copies
    if (r != LBFS_OK) return r;
    if (e != cudaSuccess) return fail(ctx, LBFS_ECUDA, std::string("tile list upload: ") + cudaGetErrorString(e));
    ctx->dirty = false;
    return LBFS_OK;
}

#define LK(call)                                   \
    do {                                           \
        cudaError_t e_ = (call);                   \
        ++ctx->launches;                           \
        if (e_ != cudaSuccess)                     \
            return fail(ctx, LBFS_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

// One V-cycle on the correction equation A e = r of every solving case, ending with phi += e:
// a fused pre-smooth + restriction kernel per level on the way down, the coarse levels in one
// kernel per case (or conjugate gradients on a coarsest level too large for it), a fused
// prolongation + post-smooth kernel per level up.
lbfs_status vcycle(lbfs_ctx* ctx) {
    const int p = ctx->prec;
    cudaStream_t s = ctx->stream;
    const int D = ctx->max_depth;
    for (int L = 0; L < D; ++L)
        LK(launch_mg_vdown(p, ctx->d_cases, ctx->d_ft_tiles[L], ctx->n_ft_tiles[L], L, ctx->ft_small[L], s));
    if (ctx->n_tail > 0) LK(launch_mg_tail(p, ctx->d_cases, ctx->d_tail, ctx->n_tail, ctx->tail_cells, ctx->tail_small, s));
    if (ctx->n_coarsest > 0) LK(launch_mg_coarsest(ctx->d_cases, ctx->d_coarsest, ctx->n_coarsest, ctx->coarsest_cells, s));
    for (int L = D - 1; L >= 0; --L)
        LK(launch_mg_vup(p, ctx->d_cases, ctx->d_ft_tiles[L], ctx->n_ft_tiles[L], L, ctx->ft_small[L], s));
    return LBFS_OK;
}

PotCheck pot_check(const lbfs_ctx* ctx, int first, int kmax, int* not_done) {
    return PotCheck{first, ctx->mg_tol, kmax, not_done, reinterpret_cast<unsigned*>(ctx->d_flag + 1), ctx->mg_wait_polls};
}

// the residual of the master potential and each case's check
cudaError_t check_residual(lbfs_ctx* ctx, int first, int kmax, int* not_done) {
    return launch_mg_residual(ctx->prec, ctx->d_cases, ctx->d_res_tiles, ctx->n_res_tiles, ctx->res_rows,
                              pot_check(ctx, first, kmax, not_done), ctx->stream);
}

// refinement cycles until every case has converged or had kmax
cudaError_t cycles(lbfs_ctx* ctx, int kmax) {
    CycleArgs a{};
    a.cases = ctx->d_cases;
    a.depth = ctx->max_depth;
    int units = std::max(ctx->n_tail + ctx->n_coarsest, (ctx->n_res_tiles + 7) / 8);
    for (int L = 0; L < a.depth; ++L) {
        a.tiles[L] = ctx->d_ft_tiles[L];
        a.n_tiles[L] = ctx->n_ft_tiles[L];
        a.small[L] = ctx->ft_small[L];
        units = std::max(units, a.n_tiles[L]);
    }
    a.tail = ctx->d_tail;
    a.coarsest = ctx->d_coarsest;
    a.n_tail = ctx->n_tail;
    a.n_coarsest = ctx->n_coarsest;
    a.tail_cells = ctx->tail_cells;
    a.tail_small = ctx->tail_small;
    a.strips = ctx->d_res_tiles;
    a.n_strips = ctx->n_res_tiles;
    a.rows = ctx->res_rows;
    return launch_mg_cycles(ctx->prec, a, std::min(units, ctx->sm_count), ctx->n_coarsest > 0 ? ctx->coarsest_cells : 0,
                            pot_check(ctx, 0, kmax, nullptr), ctx->stream);
}

// Cycles launched phase by phase before the kernel that runs as many as are still needed; what is
// launched for a converged case returns at once.  A grid barrier costs more than a launch of a
// recorded graph (a cycle on 128 x 64 takes 46 us by launches, 57 in one kernel), so the first
// cycles of a step that is likely to need them are launched: four in FP64, whose warm steps take
// three to six (3 to 6 launched are within 3%), and one in a batch of at least four cases, of which
// one needs a cycle in every other step (64 cases: 780 us a step against 911; 4: 150 against 166).
// A single mixed case mostly takes none, for which the one kernel alone is the cheaper: 5 us, against
// 16 for a conditional graph node (512 x 256: 89 us a step, 93 with a launched cycle).
int phased_cycles(int prec, int cases) {
    return prec == 0 ? 4 : (cases >= 4 ? 1 : 0);
}

// whether all cycles are launched phase by phase: as configured, or because the kernel that takes
// them in one launch needs all its blocks to run at once and cannot have that on this stream
bool launched_cycles(const lbfs_ctx* ctx) { return ctx->cfg.mg_plain_cycles || ctx->coop == 0; }

// The potential of the current state: in FP64 a warm step starts from the potential
// extrapolated in time; then the step's first residual and check, then refinement cycles
// (V-cycle, correction, residual of the corrected potential, check), which the checks end on the
// device, so a step whose start already meets mg_tol runs none and no host round trip is
// made.  At most mg_warm_cycles cycles, or mg_max_cycles after a state was set (pot_fresh); a
// case still above mg_tol then is marked as failed (LBFS_ENOTCONVERGED at the end of lbfs_step).
// So the reported residual is always that of the potential the thermo-fluid stages use.
lbfs_status potential_solve(lbfs_ctx* ctx) {
    if (ctx->n_pot == 0) return LBFS_OK;
    const int kmax = ctx->pot_fresh ? ctx->mg_max_cycles : ctx->mg_warm_cycles;
    cudaStream_t s = ctx->stream;
    if (ctx->prec == 0 && !ctx->pot_fresh)
        LK(launch_mg_extrapolate(ctx->d_cases, ctx->d_mg_tiles, ctx->n_mg_tiles, s));
    const bool launched = launched_cycles(ctx);
    if (launched && ctx->pot_fresh) {   // as many as are needed, counted on the host
        for (int it = 0;; ++it) {
            CK(cudaMemsetAsync(ctx->d_flag, 0, sizeof(int), s));
            LK(check_residual(ctx, it == 0, kmax, ctx->d_flag));
            CK(cudaMemcpyAsync(ctx->h_flag, ctx->d_flag, sizeof(int), cudaMemcpyDeviceToHost, s));
            CK(cudaStreamSynchronize(s));
            if (*ctx->h_flag == 0) break;
            lbfs_status r = vcycle(ctx);
            if (r != LBFS_OK) return r;
        }
    } else {
        const int phased = launched ? kmax : std::min(kmax, phased_cycles(ctx->prec, ctx->n_pot));
        LK(check_residual(ctx, 1, kmax, nullptr));
        for (int c = 0; c < kmax; ++c) {
            if (c == phased) {
                const cudaError_t e = cycles(ctx, kmax);
                if (e != cudaErrorCooperativeLaunchTooLarge) {
                    LK(e);
                    ctx->coop = 1;
                    break;
                }
                cudaGetLastError();   // the stream has fewer multiprocessors than the device: launch the rest
                ctx->coop = 0;
            }
            lbfs_status r = vcycle(ctx);
            if (r != LBFS_OK) return r;
            LK(check_residual(ctx, 0, kmax, nullptr));
        }
    }
    if (ctx->pot_fresh) {
        // the warm steps that follow extrapolate only once they have stored a potential
        for (size_t c = 0; c < ctx->slots.size(); ++c)
            if (ctx->slots[c].defined)
                CK(cudaMemsetAsync(ctx->d_stats + c * kStatN + ST_EXTRAP, 0, sizeof(double), s));
        ctx->pot_fresh = false;
    }
    return LBFS_OK;
}

// stage k of every case
cudaError_t stage(lbfs_ctx* ctx, int k) {
    const Slot* one = nullptr;
    if (ctx->n_active == 1)
        for (const Slot& s : ctx->slots)
            if (s.defined) one = &s;
    if (ctx->prec == 0)
        return launch_stage<double>(ctx->half, one ? &one->sd : nullptr, static_cast<StageCase<double>*>(ctx->d_stage_cases),
                                    ctx->d_stage_tiles, ctx->n_stage_tiles, ctx->rows, k, ctx->stream);
    return launch_stage<float>(ctx->half, one ? &one->sf : nullptr, static_cast<StageCase<float>*>(ctx->d_stage_cases),
                               ctx->d_stage_tiles, ctx->n_stage_tiles, ctx->rows, k, ctx->stream);
}

lbfs_status one_step(lbfs_ctx* ctx) {
    cudaEvent_t t0 = tic(ctx);
    lbfs_status r = potential_solve(ctx);
    if (r != LBFS_OK) return r;
    toc(ctx, LBFS_TIMING_POTENTIAL, t0);
    for (int k = 0; k < 3; ++k) {
        cudaEvent_t t1 = tic(ctx);
        LK(stage(ctx, k));
        toc(ctx, LBFS_TIMING_STAGE, t1);
    }
    cudaEvent_t t2 = tic(ctx);   // (the step-end statistics are part of stage 3)
    toc(ctx, LBFS_TIMING_FINALIZE, t2);
    return LBFS_OK;
}

// Record one warm step as a CUDA graph on a private stream (capture is not allowed
// on the legacy default stream a caller may lend us); replay it on ctx->stream.
lbfs_status record_graph(lbfs_ctx* ctx) {
    drop_graph(ctx);
    if (!ctx->cap_stream) CK(cudaStreamCreateWithFlags(&ctx->cap_stream, cudaStreamNonBlocking));
    cudaStream_t user = ctx->stream;
    const int64_t l0 = ctx->launches;
    ctx->stream = ctx->cap_stream;
    cudaError_t e = cudaStreamBeginCapture(ctx->cap_stream, cudaStreamCaptureModeThreadLocal);
    lbfs_status r = e == cudaSuccess ? one_step(ctx) : LBFS_ECUDA;
    cudaGraph_t g = nullptr;
    cudaError_t e2 = cudaStreamEndCapture(ctx->cap_stream, &g);
    ctx->stream = user;
    ctx->graph_launches = ctx->launches - l0;
    ctx->launches = l0;
    if (e != cudaSuccess) return fail(ctx, LBFS_ECUDA, std::string("cudaStreamBeginCapture: ") + cudaGetErrorString(e));
    if (r != LBFS_OK) {
        if (g) cudaGraphDestroy(g);
        return r;
    }
    if (e2 != cudaSuccess) return fail(ctx, LBFS_ECUDA, std::string("cudaStreamEndCapture: ") + cudaGetErrorString(e2));
    ctx->graph = g;
    CK(cudaGraphInstantiate(&ctx->gexec, g, 0));
    return LBFS_OK;
}

lbfs_status check_case(lbfs_ctx* ctx, int32_t id) {
    if (!ctx) return LBFS_EINVAL;
    if (id < 0 || id >= (int)ctx->slots.size()) return fail(ctx, LBFS_EINVAL, "case_id out of range");
    return LBFS_OK;
}

void free_slot(lbfs_ctx* ctx, Slot& s) {
    if (s.block) dfree(ctx, s.block);
    s.block = nullptr;
    s.defined = false;
}

}  // namespace

extern "C" {

lbfs_status lbfs_create(const lbfs_config* cfg, lbfs_ctx** out) {
    if (!out) return LBFS_EINVAL;
    *out = nullptr;
    if (!cfg || cfg->max_cases < 1 || cfg->max_cases > 65536 || cfg->precision < 0 || cfg->precision > 1 ||
        (cfg->dev_alloc == nullptr) != (cfg->dev_free == nullptr) || cfg->mg_warm_cycles < 0 ||
        cfg->mg_warm_cycles > 64)
        return LBFS_EINVAL;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || cfg->device < 0 || cfg->device >= ndev) {
        cudaGetLastError();
        return LBFS_ECUDA;
    }
    if (cudaSetDevice(cfg->device) != cudaSuccess || prepare_potential(cfg->precision) != cudaSuccess) {
        cudaGetLastError();
        return LBFS_ECUDA;
    }
    lbfs_ctx* ctx = new lbfs_ctx();
    ctx->cfg = *cfg;
    ctx->prec = cfg->precision;
    ctx->mg_tol = cfg->mg_tol > 0 ? cfg->mg_tol : (ctx->prec == 0 ? 1e-13 : 1e-6);
    ctx->mg_max_cycles = cfg->mg_max_cycles > 0 ? cfg->mg_max_cycles : 40;
    ctx->mg_warm_cycles = cfg->mg_warm_cycles > 0 ? cfg->mg_warm_cycles : (ctx->prec == 0 ? 12 : 3);
    ctx->mg_wait_polls = cfg->mg_wait_polls > 0 ? cfg->mg_wait_polls : kWaitPolls;
    ctx->slots.resize(cfg->max_cases);
    ctx->tile = (cfg->tile >= 0 && cfg->tile < stage_tile_shapes()) ? cfg->tile : 0;
    {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, cfg->device) == cudaSuccess && n > 0)
            ctx->sm_count = n;
        cudaGetLastError();
    }
    if (cfg->cuda_stream) {
        ctx->stream = static_cast<cudaStream_t>(cfg->cuda_stream);
    } else {
        if (cudaStreamCreateWithFlags(&ctx->stream, cudaStreamNonBlocking) != cudaSuccess) {
            delete ctx;
            return LBFS_ECUDA;
        }
        ctx->own_stream = true;
    }
    // the context's tables in one allocation
    const size_t cases_b = align_up(sizeof(DevCase) * cfg->max_cases, 256);
    const size_t stage_b =
        align_up((ctx->prec == 0 ? sizeof(StageCase<double>) : sizeof(StageCase<float>)) * cfg->max_cases, 256);
    const size_t stats_b = align_up(sizeof(double) * kStatN * cfg->max_cases, 256);
    ctx->d_cases = static_cast<DevCase*>(dalloc(ctx, cases_b + stage_b + stats_b + 256));
    if (ctx->d_cases) {
        char* base = reinterpret_cast<char*>(ctx->d_cases);
        ctx->d_stage_cases = base + cases_b;
        ctx->d_stats = reinterpret_cast<double*>(base + cases_b + stage_b);
        ctx->d_flag = reinterpret_cast<int*>(base + cases_b + stage_b + stats_b);
    }
    if (!ctx->d_cases ||
        cudaMallocHost(&ctx->h_flag, sizeof(int)) != cudaSuccess ||
        cudaMallocHost(&ctx->h_stats, stats_b + kFlags * sizeof(int)) != cudaSuccess) {
        lbfs_destroy(ctx);
        return LBFS_ENOMEM;
    }
    ctx->stats_bytes = stats_b;
    cudaMemset(ctx->d_cases, 0, cases_b + stage_b + stats_b + 256);
    if (cudaDeviceSynchronize() != cudaSuccess) {
        lbfs_destroy(ctx);
        return LBFS_ECUDA;
    }
    *out = ctx;
    return LBFS_OK;
}

lbfs_status lbfs_set_case(lbfs_ctx* ctx, int32_t id, const lbfs_case_desc* desc) {
    lbfs_status r = check_case(ctx, id);
    if (r != LBFS_OK) return r;
    if (!desc) return fail(ctx, LBFS_EINVAL, "desc is NULL");
    CaseParams P;
    r = resolve(ctx, *desc, P);
    if (r != LBFS_OK) return r;
    CK(cudaSetDevice(ctx->cfg.device));
    // multigrid hierarchy
    DevCase hd;
    std::memset(&hd, 0, sizeof(hd));
    hd.P = P;
    // Each coarser level halves both cell counts, rounding up: level L's column I covers
    // the fine columns [I 2^L, min((I + 1) 2^L, nx)), so only the last column (row) can
    // be narrower; wlx (wly) is its width relative to the level's other cells.  A
    // periodic axis of odd size cannot agglomerate across its wrap, so coarsening stops
    // there.
    int nx = P.nx, ny = P.ny, nlev = 1;
    hd.lev[0].nx = nx;
    hd.lev[0].ny = ny;
    hd.lev[0].wlx = hd.lev[0].wly = 1.0f;
    hd.lev[0].ragged = 0;
    while (nlev < kMaxLevels && nx * ny > kCoarsenCells && nx >= 4 && ny >= 4 && !(P.periodic_x && (nx & 1)) &&
           !(P.periodic_y && (ny & 1))) {
        nx = (nx + 1) / 2;
        ny = (ny + 1) / 2;
        const int sc = 1 << nlev;
        MGLevel& lv = hd.lev[nlev];
        lv.nx = nx;
        lv.ny = ny;
        lv.wlx = (float)(P.nx - (nx - 1) * sc) / (float)sc;
        lv.wly = (float)(P.ny - (ny - 1) * sc) / (float)sc;
        lv.ragged = (lv.wlx < 1.0f || lv.wly < 1.0f) ? 1 : 0;
        ++nlev;
    }
    if (P.solve_potential && nx * ny > kCoarsestMax)
        return fail(ctx, LBFS_EINVAL,
                    "the potential's coarsest level would exceed 4096 cells (a periodic axis whose size "
                    "halves to an odd number early, or an extreme aspect ratio)");
    hd.nlev = nlev;
    // partial-sum slots for the lowest strips
    const int red_cap = ((P.nx + kStripW - 1) / kStripW) * ((P.ny + kStageMinRows - 1) / kStageMinRows);
    const int res_cap = ((P.nx + kResidStripW - 1) / kResidStripW) * ((P.ny + kResidMinRows - 1) / kResidMinRows);
    const int res_groups = (res_cap + kStageGroup - 1) / kStageGroup;
    // the levels that run in one kernel per case
    hd.tail = nlev - 1;
    if (nx * ny <= kTailCoarsest)
        while (hd.tail > 0 && hd.lev[hd.tail - 1].nx * hd.lev[hd.tail - 1].ny <= kTailCells) --hd.tail;
    hd.far_h[0] = (float)(-P.H0 * P.cos_t);
    hd.far_l[0] = (float)(-P.H0 * P.cos_t - (double)hd.far_h[0]);
    hd.far_h[1] = (float)(-P.H0 * P.sin_t);
    hd.far_l[1] = (float)(-P.H0 * P.sin_t - (double)hd.far_h[1]);
    // one device block per case
    const size_t rs = ctx->prec == 0 ? sizeof(double) : sizeof(float);
    const size_t cells = (size_t)P.pitch * P.ny;
    size_t off = 0;
    std::vector<std::pair<void**, size_t>> plan;
    auto add = [&](void** dst, size_t bytes) {
        plan.push_back({dst, off});
        off = align_up(off + bytes, 256);
    };
    for (int k = 0; k < 3; ++k) {
        add(&hd.He[k], cells * sizeof(double));
        add(&hd.W[k], cells * 4 * rs);
    }
    if (ctx->prec == 0) {
        add((void**)&hd.phi64, cells * sizeof(double));
        add((void**)&hd.phi_prev64, 2 * cells * sizeof(double));
    } else {
        add(&hd.phi, cells * rs);
        add((void**)&hd.phi_lo, cells * sizeof(float));
    }
    add(&hd.Fs_prev, cells * rs);
    add(&hd.Sdot, cells * rs);
    for (int L = 0; L < nlev; ++L) {
        hd.lev[L].pitch = (int)align_up((size_t)hd.lev[L].nx, 32);
        const size_t lc = (size_t)hd.lev[L].pitch * hd.lev[L].ny;
        add(&hd.lev[L].mu, lc * (L == 0 ? rs : sizeof(float)));
        add(&hd.lev[L].e, lc * sizeof(float));
        add(&hd.lev[L].r, lc * (L == 0 ? rs : sizeof(float)));
        if (L > 0 && L < hd.tail) add(&hd.lev[L].eu, lc * sizeof(float));
    }
    const int red_groups = (red_cap + kStageGroup - 1) / kStageGroup;
    add((void**)&hd.red, (size_t)red_cap * kRedN * sizeof(double));
    add((void**)&hd.red_groups, (size_t)red_groups * kRedN * sizeof(double));
    add((void**)&hd.red_tickets, (size_t)(1 + red_groups) * sizeof(unsigned));
    add((void**)&hd.mg_red, (size_t)res_cap * 2 * sizeof(double));
    add((void**)&hd.mg_groups, (size_t)res_groups * 2 * sizeof(double));
    const size_t ticket_bytes = (size_t)(1 + res_groups) * sizeof(unsigned);
    add((void**)&hd.mg_tickets, ticket_bytes);
    add((void**)&hd.chunk, (size_t)kFinChunks * kRedN * sizeof(double));
    add((void**)&hd.tickets, sizeof(unsigned));
    Slot& s = ctx->slots[id];
    free_slot(ctx, s);
    drop_graph(ctx);
    ctx->dirty = true;
    // cudaMalloc aligns to 256 bytes; an allocator of the caller's to 8 at least, from where the
    // arrays are moved up to the next multiple of a field's widest load
    s.block = dalloc(ctx, off + (ctx->cfg.dev_alloc ? kFieldAlign : 0));
    if (!s.block) return fail(ctx, LBFS_ENOMEM, "device allocation of the case failed");
    char* base = reinterpret_cast<char*>(align_up(reinterpret_cast<size_t>(s.block), kFieldAlign));
    for (auto& pr : plan) *pr.first = base + pr.second;
    for (int L = 0; L < nlev; ++L)
        if (!hd.lev[L].eu) hd.lev[L].eu = hd.lev[L].e;
    if (ctx->prec == 0) hd.phi = hd.phi64;
    hd.stats = ctx->d_stats + (size_t)id * kStatN;
    s.hd = hd;
    s.ticket_bytes = ticket_bytes;
    s.desc = *desc;
    const void* sc = &s.sf;
    size_t scb = sizeof(s.sf);
    if (ctx->prec == 0) {
        fill_stage<double>(hd, s.sd);
        sc = &s.sd;
        scb = sizeof(s.sd);
    } else {
        fill_stage<float>(hd, s.sf);
    }
    CK(cudaMemsetAsync(base, 0, off, ctx->stream));
    CK(cudaMemcpyAsync(ctx->d_cases + id, &s.hd, sizeof(DevCase), cudaMemcpyHostToDevice, ctx->stream));
    CK(cudaMemcpyAsync(static_cast<char*>(ctx->d_stage_cases) + id * scb, sc, scb, cudaMemcpyHostToDevice, ctx->stream));
    double st0[kStatN];
    for (double& v : st0) v = 0.0;
    st0[ST_T_FREEZE] = -1.0;
    CK(cudaMemcpyAsync(hd.stats, st0, sizeof(st0), cudaMemcpyHostToDevice, ctx->stream));
    InitArgs a;
    a.kind = desc->init;
    a.radius = desc->radius;
    a.cx = desc->init == 0 ? 0.5 * P.nx : desc->drop_x;
    a.cy = desc->init == 0 ? 0.0 : desc->drop_y;
    a.T_init = desc->T_init;
    a.xi = desc->xi;
    const DevCase* dcase = ctx->d_cases + id;
    CK(launch_init(ctx->prec, dcase, P.nx, P.ny, a, ctx->stream));
    CK(launch_mu_from_state(ctx->prec, dcase, P.nx, P.ny, ctx->stream));
    CK(launch_stats_init(ctx->prec, dcase, P.nx, P.ny, ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    s.defined = true;
    ctx->pot_fresh = true;
    return LBFS_OK;
}

static lbfs_status ensure_scratch(lbfs_ctx* ctx, size_t bytes) {
    if (ctx->scratch_bytes >= bytes) return LBFS_OK;
    dfree(ctx, ctx->d_scratch);
    ctx->d_scratch = static_cast<double*>(dalloc(ctx, bytes));
    ctx->scratch_bytes = ctx->d_scratch ? bytes : 0;
    return ctx->d_scratch ? LBFS_OK : fail(ctx, LBFS_ENOMEM, "scratch allocation failed");
}

lbfs_status lbfs_set_fields(lbfs_ctx* ctx, int32_t id, uint32_t mask, const double* host_in) {
    lbfs_status r = check_case(ctx, id);
    if (r != LBFS_OK) return r;
    Slot& s = ctx->slots[id];
    if (!s.defined) return fail(ctx, LBFS_EINVAL, "case not defined");
    const uint32_t settable = (1u << LBFS_FIELD_PHI) | (1u << LBFS_FIELD_HE) | (1u << LBFS_FIELD_P) |
                              (1u << LBFS_FIELD_C) | (1u << LBFS_FIELD_MX) | (1u << LBFS_FIELD_MY) |
                              (1u << LBFS_FIELD_FSPREV);
    if ((mask & ~settable) || mask == 0 || !host_in) return fail(ctx, LBFS_EINVAL, "bad field mask or buffer");
    CK(cudaSetDevice(ctx->cfg.device));
    const int nf = __builtin_popcount(mask);
    const size_t N = (size_t)s.hd.P.nx * s.hd.P.ny;
    r = ensure_scratch(ctx, nf * N * sizeof(double));
    if (r != LBFS_OK) return r;
    CK(cudaMemcpyAsync(ctx->d_scratch, host_in, nf * N * sizeof(double), cudaMemcpyHostToDevice, ctx->stream));
    const DevCase* dcase = ctx->d_cases + id;
    CK(launch_store_fields(ctx->prec, dcase, s.hd.P.nx, s.hd.P.ny, mask, ctx->d_scratch, ctx->stream));
    CK(launch_mu_from_state(ctx->prec, dcase, s.hd.P.nx, s.hd.P.ny, ctx->stream));
    CK(launch_stats_init(ctx->prec, dcase, s.hd.P.nx, s.hd.P.ny, ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    ctx->pot_fresh = true;
    return LBFS_OK;
}

lbfs_status lbfs_fields(lbfs_ctx* ctx, int32_t id, uint32_t mask, double* host_out) {
    lbfs_status r = check_case(ctx, id);
    if (r != LBFS_OK) return r;
    Slot& s = ctx->slots[id];
    if (!s.defined) return fail(ctx, LBFS_EINVAL, "case not defined");
    if (mask == 0 || (mask >> 13) || !host_out) return fail(ctx, LBFS_EINVAL, "bad field mask or buffer");
    CK(cudaSetDevice(ctx->cfg.device));
    const int nf = __builtin_popcount(mask);
    const size_t N = (size_t)s.hd.P.nx * s.hd.P.ny;
    r = ensure_scratch(ctx, nf * N * sizeof(double));
    if (r != LBFS_OK) return r;
    CK(launch_derive_fields(ctx->prec, ctx->d_cases + id, s.hd.P.nx, s.hd.P.ny, mask, ctx->d_scratch,
                            ctx->stream));
    CK(cudaMemcpyAsync(host_out, ctx->d_scratch, nf * N * sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    return LBFS_OK;
}

lbfs_status lbfs_diagnostics(lbfs_ctx* ctx, int32_t id, lbfs_case_diag* out, double* q_wall) {
    lbfs_status r = check_case(ctx, id);
    if (r != LBFS_OK) return r;
    Slot& s = ctx->slots[id];
    if (!s.defined) return fail(ctx, LBFS_EINVAL, "case not defined");
    if (!out) return fail(ctx, LBFS_EINVAL, "out is NULL");
    CK(cudaSetDevice(ctx->cfg.device));
    const int nx = s.hd.P.nx;
    r = ensure_scratch(ctx, (3 * (size_t)nx + 5) * sizeof(double));
    if (r != LBFS_OK) return r;
    double* cols = ctx->d_scratch;
    double* res = ctx->d_scratch + 3 * (size_t)nx;
    CK(launch_diagnostics(ctx->prec, ctx->d_cases + id, nx, s.desc.radius, cols, res, ctx->stream));
    double h[5];
    CK(cudaMemcpyAsync(h, res, sizeof(h), cudaMemcpyDeviceToHost, ctx->stream));
    if (q_wall)
        CK(cudaMemcpyAsync(q_wall, cols + 2 * (size_t)nx, nx * sizeof(double), cudaMemcpyDeviceToHost,
                           ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    out->H_m = h[0];
    out->U_max = h[1];
    out->Pe = h[2];
    out->Fo = h[3];
    out->Q_wall = h[4];
    return LBFS_OK;
}

lbfs_status lbfs_potential_pseudo_time(lbfs_ctx* ctx, int32_t id, int32_t iters, double dtau) {
    lbfs_status r = check_case(ctx, id);
    if (r != LBFS_OK) return r;
    Slot& s = ctx->slots[id];
    if (!s.defined) return fail(ctx, LBFS_EINVAL, "case not defined");
    if (iters < 0 || !(dtau > 0.0)) return fail(ctx, LBFS_EINVAL, "iters must be >= 0 and dtau > 0");
    CK(cudaSetDevice(ctx->cfg.device));
    const int nx = s.hd.P.nx, ny = s.hd.P.ny;
    r = ensure_scratch(ctx, (size_t)nx * ny * sizeof(double));
    if (r != LBFS_OK) return r;
    CK(launch_mu_from_state(ctx->prec, ctx->d_cases + id, nx, ny, ctx->stream));
    CK(launch_pseudo_time(ctx->prec, ctx->d_cases + id, nx, ny, iters, dtau, ctx->d_scratch, ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    ctx->pot_fresh = true;   // the next step re-converges the potential from this state
    return LBFS_OK;
}

lbfs_status lbfs_step(lbfs_ctx* ctx, int32_t nsteps, lbfs_case_stats* out) {
    if (!ctx) return LBFS_EINVAL;
    if (nsteps < 0) return fail(ctx, LBFS_EINVAL, "nsteps must be >= 0");
    CK(cudaSetDevice(ctx->cfg.device));
    if (ctx->dirty) {
        lbfs_status r = rebuild(ctx);
        if (r != LBFS_OK) return r;
    }
    ctx->launches = 0;
    ctx->pot_fail = false;
    for (size_t c = 0; c < ctx->slots.size(); ++c)
        if (ctx->slots[c].defined) {
            CK(cudaMemsetAsync(ctx->d_stats + c * kStatN + ST_POT_FAIL, 0, sizeof(double), ctx->stream));
            // ST_POT_RESID_MAX, ST_POT_CYCLES_SUM, ST_STEPS_CALL: per-call accumulators
            CK(cudaMemsetAsync(ctx->d_stats + c * kStatN + ST_POT_RESID_MAX, 0, 3 * sizeof(double), ctx->stream));
        }
    for (int n = 0; n < nsteps && ctx->n_active > 0; ++n) {
        // a step after the first potential solve has no host round trip and can be replayed
        // (not before it is known whether the cycles' kernel can run: a refusal would end the recording)
        const bool known = launched_cycles(ctx) || ctx->coop == 1 || phased_cycles(ctx->prec, ctx->n_pot) >= ctx->mg_warm_cycles;
        const bool graphable = ctx->cfg.use_graph && !ctx->timing && !(ctx->n_pot > 0 && (ctx->pot_fresh || !known));
        if (graphable) {
            if (!ctx->gexec) {
                lbfs_status r = record_graph(ctx);
                if (r != LBFS_OK) return r;
            }
            CK(cudaGraphLaunch(ctx->gexec, ctx->stream));
            ctx->launches += ctx->graph_launches;
            continue;
        }
        lbfs_status r = one_step(ctx);
        if (r != LBFS_OK) return r;
    }
    CK(cudaMemcpyAsync(ctx->h_stats, ctx->d_stats, ctx->stats_bytes + kFlags * sizeof(int), cudaMemcpyDeviceToHost,
                       ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    harvest(ctx);
    const bool timed_out = reinterpret_cast<const int*>(reinterpret_cast<const char*>(ctx->h_stats) + ctx->stats_bytes)[3] != 0;
    if (timed_out) {   // blocks left the cycles at different places: no ticket keeps a count, the next step solves afresh,
                       // with launched cycles
        for (const Slot& s : ctx->slots)
            if (s.defined) CK(cudaMemsetAsync(s.hd.mg_tickets, 0, s.ticket_bytes, ctx->stream));
        CK(cudaMemsetAsync(ctx->d_flag, 0, kFlags * sizeof(int), ctx->stream));
        CK(cudaStreamSynchronize(ctx->stream));
        ctx->pot_fresh = true;
        ctx->coop = 0;
        drop_graph(ctx);
    }
    bool bad = false;
    for (size_t c = 0; c < ctx->slots.size(); ++c) {
        const double* st = ctx->h_stats + c * kStatN;
        if (ctx->slots[c].defined && st[ST_NONFINITE] > 0) bad = true;
        if (ctx->slots[c].defined && st[ST_POT_FAIL] > 0) ctx->pot_fail = true;
        if (out) {
            lbfs_case_stats& o = out[c];
            std::memset(&o, 0, sizeof(o));
            if (!ctx->slots[c].defined) continue;
            o.sum_C = st[ST_SUM_C];
            o.sum_He = st[ST_SUM_HE];
            o.sum_Fl_drop = st[ST_SUM_FL_DROP];
            o.n_drop = st[ST_N_DROP];
            o.Q_L = st[ST_Q_L];
            o.t = st[ST_T];
            o.t_freeze = st[ST_T_FREEZE];
            o.pot_resid = st[ST_POT_RESID];
            o.pot_cycles = (int32_t)st[ST_POT_CYCLES];
            o.nonfinite = st[ST_NONFINITE] > 0 ? 1 : 0;
            o.pot_resid_max = st[ST_POT_RESID_MAX];
            o.pot_cycles_mean = st[ST_STEPS_CALL] > 0 ? st[ST_POT_CYCLES_SUM] / st[ST_STEPS_CALL] : 0.0;
        }
    }
    if (timed_out)
        return fail(ctx, LBFS_ETIMEOUT, "a wait between the blocks of the potential's cycles ran out of its polls (mg_wait_polls)");
    if (bad) return fail(ctx, LBFS_EDIVERGED, "a non-finite value appeared in a case's state");
    if (ctx->pot_fail)
        return fail(ctx, LBFS_ENOTCONVERGED,
                    "the potential solve missed mg_tol within mg_max_cycles (first solve) or mg_warm_cycles");
    return LBFS_OK;
}

int64_t lbfs_last_launch_count(const lbfs_ctx* ctx) { return ctx ? ctx->launches : 0; }

lbfs_status lbfs_autotune(lbfs_ctx* ctx, int32_t reps, int32_t* chosen, double* ms, int32_t n) {
    if (!ctx || reps < 1 || n < 0) return LBFS_EINVAL;
    CK(cudaSetDevice(ctx->cfg.device));
    if (ctx->dirty) {
        lbfs_status r = rebuild(ctx);
        if (r != LBFS_OK) return r;
    }
    if (ctx->n_active == 0) return fail(ctx, LBFS_EINVAL, "no case defined");
    cudaEvent_t a = take_event(ctx), b = take_event(ctx);
    int best = ctx->tile;
    double best_ms = 1e300;
    for (int t = 0; t < stage_tile_shapes(); ++t) {
        ctx->tile = t;
        lbfs_status r = rebuild(ctx);
        if (r != LBFS_OK) return r;
        // Runge-Kutta stage 2 reads sets 0 and 1 and dF_s/dt and writes only the stage
        // buffer 2, so timing it leaves the state untouched
        CK(stage(ctx, 1));
        CK(cudaEventRecord(a, ctx->stream));
        for (int k = 0; k < reps; ++k)
            CK(stage(ctx, 1));
        CK(cudaEventRecord(b, ctx->stream));
        CK(cudaEventSynchronize(b));
        float el = 0.f;
        CK(cudaEventElapsedTime(&el, a, b));
        const double per = el / reps;
        if (t < n && ms) ms[t] = per;
        // a later shape must be more than 2 % faster to replace the current choice, so
        // near-ties resolve to the same shape from run to run
        if (per < 0.98 * best_ms) {
            best_ms = per;
            best = t;
        }
    }
    ctx->ev_pool.push_back(a);
    ctx->ev_pool.push_back(b);
    ctx->tile = best;
    lbfs_status r = rebuild(ctx);
    if (r != LBFS_OK) return r;
    if (chosen) *chosen = best;
    return LBFS_OK;
}

lbfs_status lbfs_timing(lbfs_ctx* ctx, int32_t enable) {
    if (!ctx) return LBFS_EINVAL;
    CK(cudaStreamSynchronize(ctx->stream));
    harvest(ctx);
    ctx->timing = enable != 0;
    for (int k = 0; k < 3; ++k) {
        ctx->t_ms[k] = 0.0;
        ctx->t_cnt[k] = 0;
    }
    return LBFS_OK;
}

lbfs_status lbfs_timing_read(lbfs_ctx* ctx, double* ms, int64_t* counts, int32_t n) {
    if (!ctx || n < 0 || n > 3) return LBFS_EINVAL;
    for (int k = 0; k < n; ++k) {
        if (ms) ms[k] = ctx->t_ms[k];
        if (counts) counts[k] = ctx->t_cnt[k];
    }
    return LBFS_OK;
}

void lbfs_destroy(lbfs_ctx* ctx) {
    if (!ctx) return;
    cudaSetDevice(ctx->cfg.device);
    if (ctx->stream) cudaStreamSynchronize(ctx->stream);
    drop_graph(ctx);
    harvest(ctx);
    for (cudaEvent_t e : ctx->ev_pool) cudaEventDestroy(e);
    if (ctx->cap_stream) cudaStreamDestroy(ctx->cap_stream);
    for (Slot& s : ctx->slots) free_slot(ctx, s);
    for (auto* p : ctx->d_ft_tiles) dfree(ctx, p);
    dfree(ctx, ctx->d_mg_tiles);
    dfree(ctx, ctx->d_res_tiles);
    dfree(ctx, ctx->d_tail);
    dfree(ctx, ctx->d_coarsest);
    dfree(ctx, ctx->d_stage_tiles);
    dfree(ctx, ctx->d_cases);
    dfree(ctx, ctx->d_scratch);
    if (ctx->h_flag) cudaFreeHost(ctx->h_flag);
    if (ctx->h_stats) cudaFreeHost(ctx->h_stats);
    if (ctx->own_stream && ctx->stream) cudaStreamDestroy(ctx->stream);
    delete ctx;
}

const char* lbfs_last_error(const lbfs_ctx* ctx) { return ctx ? ctx->err.c_str() : "null context"; }

}  // extern "C"
